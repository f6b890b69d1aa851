"""The ray-tracing roofline of bench.py (no GPU): counts from the profile summary of the kernel in use, none for another one."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_counts_are_those_of_the_kernel_in_use(tmp_path, monkeypatch):
    seg, t = 17_980_808, 2.0e-3
    roof = bench.ray_roofline(seg, t, 2070.0)
    src = open(os.path.join(ROOT, "paper_0902_3092_gb300", "csrc", "raytrace.cu"), encoding="utf-8").read()
    kernel = re.match(r"(\w+)<", roof["kernel"]).group(1)
    assert re.search(rf"__global__[^;{{]*\b{kernel}\b", src, re.S)
    for k in re.findall(r"\bk_\w+", roof["kernel"]):
        assert k in src
    c = bench.transport_counts(bench.RAY_COUNTS_FILE)
    assert len(c["source_sha16"]) == 16 and c["dram_bytes_per_launch"] > 0
    if c["source_sha16"] == bench.ray_source_hash():
        assert roof["achieved"] == pytest.approx(c["warp_inst_per_segment"] * seg / t)
        assert 0 < roof["frac"] < 1 and 0 < roof["thread_inst_frac"] < 1
    # counts of other code are not used
    f = tmp_path / "counts.md"
    f.write_text(open(bench.RAY_COUNTS_FILE, encoding="utf-8").read().replace(c["source_sha16"], "0" * 16))
    monkeypatch.setattr(bench, "RAY_COUNTS_FILE", str(f))
    roof = bench.ray_roofline(seg, t, 2070.0)
    assert roof["frac"] is None and roof["achieved"] is None and roof["traffic"] is None


@pytest.mark.parametrize("name", ["common.cuh", "raymarch.cuh", "raytrace.cu"])
def test_hash_follows_the_code(tmp_path, name):
    csrc = tmp_path / "paper_0902_3092_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for f in ("common.cuh", "raymarch.cuh", "raytrace.cu"):
        (csrc / f).write_text(open(os.path.join(ROOT, "paper_0902_3092_gb300", "csrc", f), encoding="utf-8").read(),
                              encoding="utf-8")
    h = bench.ray_source_hash(str(tmp_path))
    assert h == bench.ray_source_hash()
    (csrc / name).write_text((csrc / name).read_text(encoding="utf-8") + "\nstatic int added;\n", encoding="utf-8")
    assert bench.ray_source_hash(str(tmp_path)) != h
