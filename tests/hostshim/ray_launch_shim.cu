// Host build of the ray tracer's launches (raytrace.cu) over a stand-in for the call that raises a kernel's
// shared-memory limit, which the process keeps: the limit that a launch leaves behind.
#include <cuda_runtime.h>

namespace fake {
int limit = 0;
template <class F>
cudaError_t set_attribute(F*, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit = v;
  return cudaSuccess;
}
}  // namespace fake
#define cudaFuncSetAttribute fake::set_attribute
#include "raytrace.cu"

// (of the library's other files, not reached here)
namespace mcrt {
mcrt_status set_error(mcrt_disk*, mcrt_status s, const std::string&) { return s; }
mcrt_status cuda_fail(mcrt_disk*, cudaError_t, const char*) { return MCRT_ECUDA; }
mcrt_status compute_temperatures(mcrt_disk*) { return MCRT_OK; }
void pda_free(PdaState*) {}
}  // namespace mcrt
mcrt::DevModel<float> mcrt_disk::model32() const { return {}; }
mcrt::DevModel<double> mcrt_disk::model64() const { return {}; }

// The limit that a launch over nt polar cells leaves, and the shared memory that it asks for.
extern "C" int host_ray_limit(int prec, int nt, int nlam, int before, long long* smem) {
  mcrt_disk* d = new mcrt_disk();
  mcrt::RayState* rs = new mcrt::RayState();
  d->nr = 1;
  d->nt = nt;
  d->nlam = nlam;
  d->l_unit = 1.0;
  rs->n = 1;
  fake::limit = before;
  if (prec == 64) {
    *smem = (long long)mcrt::ray_smem<double>(nt);
    mcrt::launch_trace<double>(d, rs, mcrt::DevModel<double>(), nullptr, 152);
  } else {
    *smem = (long long)mcrt::ray_smem<float>(nt);
    mcrt::launch_trace<float>(d, rs, mcrt::DevModel<float>(), nullptr, 152);
  }
  return fake::limit;
}
