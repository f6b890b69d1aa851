// firstflight.cuh -- the first flights of a run's packets, from the star along a radius, found at once (FP32).
#pragma once
#include "transport.cuh"

namespace mcrt {

// The packets' first flights. A packet from the star moves along a radius: it stays in its polar row, and its
// first interaction lies in the shell where the row's column sum passes tau / chi, or the packet leaves the
// grid. One thread per packet finds the shell by binary search in the row's sums instead of crossing
// shell after shell in a transport kernel; the entries of the shells it passed are counted per (row, last
// shell) and added to the visits by k_first_visits(), packets that leave the grid are done, the others are
// listed for the transport. 40x40 gray disk, tau_mid = 100, 1e6 packets: 1.47 -> 0.89 ms for the whole step
// (reset, run, temperatures, spectrum), the same tallies as the marches'.
//
// For gray plain Monte Carlo runs of up to 12 packets per lane (one chi; packets of a few hundred steps). Not with the MRW: there the long
// packets' deposits would fall behind the short packets that get faster alone, and the re-emission bins drawn at
// escape see that (200x120, tau_mid = 1e6, 1e8 packets: 1.19 -> 0.94 s, but the escape spectrum 1e-3 from the
// marches', eight times what two runs differ by). Nor for runs that keep a path-length tally or polarization,
// start packets inside the disk, or must repeat the packets' marches bit for bit (tail_warps_per_sm = -1).
//
// The packets are taken, 64 at a time, and so listed, nearly in the order of their numbers: the re-emission bins of
// gray dust, drawn at escape, see the tallies in the state that packets of lower numbers left. Latency-bound (two
// binary searches in cached tables); one block of 128 threads per SM keeps the order within 4e4 packets and
// takes about 0.05 ms per 1e6.
constexpr int kStarBlock = 128;
static __global__ void __launch_bounds__(kStarBlock) k_star_flights(const KParams<float> P, unsigned long long* __restrict__ list,
                                                             int shared_rows) {
  extern __shared__ unsigned sh[];  // escapes per (bin, inclination), then (shared_rows) per polar row
  const DevModel<float>& M = P.m0;
  const int nsed = M.nlam * kNInc, nsh = nsed + (shared_rows ? M.nt : 0);
  for (int i = threadIdx.x; i < nsh; i += blockDim.x) sh[i] = 0u;
  __syncthreads();
  const unsigned lane = threadIdx.x & 31u;
  const int rows = M.nr + 1;
  Acc acc = Acc{};
  unsigned long long id = 0;
  for (unsigned step = 0;; ++step, id += 32ull) {
    if ((step & 1u) == 0u) {
      if (lane == 0) id = atomicAdd(P.queue + 2, 64ull);
      id = __shfl_sync(0xffffffffu, id, 0) + lane;
    }
    if (id - lane >= P.total) break;
    bool keep = false;
    unsigned long long entry = 0;
    if (id < P.total) {
      const unsigned long long k = M.first_id + id;
      const uint4 w = philox_block(0u, M.model_id, (uint32_t)k, (uint32_t)(k >> 32), (uint32_t)P.seed,
                                   (uint32_t)(P.seed >> 32));
      const int lam = sample_star(M, uni<float>(w.x));
      float ux, uy, uz;
      iso_dir<float>(w.y, w.z, ux, uy, uz);
      const float t = neg_log<float>(uni<float>(w.w)) / M.chi0;
      int it = 0, hi = M.nt;
      while (hi - it > 1) {  // theta_cell of the direction
        const int mid = (it + hi) >> 1;
        if (M.cf[mid] >= uz) it = mid; else hi = mid;
      }
      const float* N = M.ncol + (size_t)it * rows;
      int ir = 0;
      hi = rows;  // N[ir] <= t < N[hi] (hi = nr + 1: past the last face)
      while (hi - ir > 1) {
        const int mid = (ir + hi) >> 1;
        if (ldg(N + mid) <= t) ir = mid; else hi = mid;
      }
      acc.packets++;
      if (ir == M.nr) {
        int ib = (int)(fabsf(uz) * (float)kNInc);
        ib = ib < kNInc ? ib : kNInc - 1;
        atomicAdd(sh + lam * kNInc + ib, 1u);
        if (shared_rows) atomicAdd(sh + nsed + it, 1u);
        else atomicAdd(M.first + (size_t)it * rows + ir, 1ull);
        acc.escaped++;
        const unsigned long long packed = ((unsigned long long)(rows + 1) << 24) | ((uint32_t)k & 0xffffffu);
        acc.longest = packed > acc.longest ? packed : acc.longest;
      } else {
        if (ir > 0) atomicAdd(M.first + (size_t)it * rows + ir, 1ull);
        keep = true;
        entry = id | (unsigned long long)ir << 32 | (unsigned long long)it << 48;
      }
      if (ir > 0) acc.cross += (unsigned)ir + 1u;
    }
    const unsigned kept = __ballot_sync(0xffffffffu, keep);
    if (kept) {
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(P.queue + 1, (unsigned long long)__popc(kept));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (keep) list[base + __popc(kept & ((1u << lane) - 1u))] = entry;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nsed; i += blockDim.x)
    if (sh[i]) atomicAdd(M.sed + i, (unsigned long long)sh[i]);
  for (int i = nsed + threadIdx.x; i < nsh; i += blockDim.x)
    if (sh[i]) atomicAdd(M.first + (size_t)(i - nsed) * rows + M.nr, (unsigned long long)sh[i]);
  flush(M, acc, true);
}

// Entries of the first flights into the visits: cell (i, row) was entered by every packet whose flight ended
// in a shell k >= max(i, 1). One warp per row, from the last shell inwards; clears the counts.
static __global__ void k_first_visits(int nr, int nt, unsigned long long* __restrict__ first,
                                      unsigned long long* __restrict__ visits) {
  const int lane = (int)(threadIdx.x & 31u);
  const int nw = (int)(gridDim.x * blockDim.x) >> 5;
  for (int it = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < nt; it += nw) {
    unsigned long long* f = first + (size_t)it * (nr + 1);
    unsigned long long beyond = 0;  // flights that ended past the lanes' shells
    for (int k0 = nr; k0 >= 0; k0 -= 32) {
      const int k = k0 - lane;
      unsigned long long v = k >= 0 ? f[k] : 0ull;
      if (k >= 0 && v) f[k] = 0ull;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long w = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += w;
      }
      v += beyond;
      if (k >= 0 && k < nr && v) visits[(size_t)k * nt + it] += v;
      beyond = __shfl_sync(0xffffffffu, v, 31);
    }
  }
}

}  // namespace mcrt
