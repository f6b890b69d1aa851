// cgcluster.cuh -- a whole inner conjugate-gradient solve of the PDA in one launch: one thread-block cluster
// holds the system in its shared memory and registers.
//
// An iteration of the tile kernels (pda.cu) is three graph nodes of a few microseconds each, whatever the
// system's size (11 us at 20,000 cells, where the arithmetic is 0.1 us). Here the box of rows and columns that
// holds the unknown cells is split by rows over the CTAs of one cluster (1 to 16, one per SM). A CTA keeps p and the
// couplings of its rows in shared memory, r and y of its cells in registers, and a copy of p for the row above
// and below it, which it updates itself (p = r + beta p needs only those rows' r, written by the neighbour
// CTA into distributed shared memory when it updates them). So an iteration needs two cluster barriers, those of
// its two dot products.
//
// What bounds an iteration is the latency of the two dot products and the barriers, so the sums are built
// for it: FP32 in a warp and over the warps of a CTA (every warp adds the warps' sums itself, no broadcast), the
// CTAs' sums as pairs of floats (FP64 adds and divides have several times the latency here), few warps per CTA with
// several cells per thread. Sums are in a fixed order: the same system gives the same bits. Cells of the box
// that are no unknowns have zero couplings and a zero right-hand side, and stay zero.
//
// Limit: 8192 cells per CTA, 131072 in the box; beyond it the tile kernels use the whole GPU.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

namespace mcrt {

// threads of a CTA at most when each carries K cells (the register budget of K cells' vectors)
__host__ __device__ constexpr int cg_threads(int K) { return K <= 4 ? 1024 : 512; }
constexpr int kCgMaxCluster = 16;
constexpr int kCgMaxIter = 200000;  // iterations of one launch at most (about 0.4 s)

struct CgBox {
  int nt;              // columns of the grid
  int i0, j0;          // first row and column of the box
  int rows, w;         // its size
  const float *ar, *at;  // scaled couplings to the next row / column (whole grid)
  const double* rs;    // scaled residual (whole grid)
  double inv_scale;    // right-hand side r = rs * inv_scale
  float* y;            // solution (whole grid, box cells written)
  double tol2;         // stop at rr <= tol2 rr0
  int max_iter;
  int* iters;          // out: iterations made
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared-memory address of `p` in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void peer_store(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// A sum of floats kept as an unevaluated pair (hi + lo; Knuth's two-sum, Dekker's quotient): about 48 bits.
struct FloatPair {
  float hi, lo;
};
__device__ __forceinline__ FloatPair pair_add(FloatPair a, FloatPair b) {
  const float s = a.hi + b.hi, t = s - a.hi;
  const float e = (a.hi - (s - t)) + (b.hi - t) + (a.lo + b.lo);
  const float h = s + e;
  return {h, e - (h - s)};
}
__device__ __forceinline__ float pair_ratio(FloatPair a, FloatPair b) {
  const float c = __fdividef(1.f, b.hi), q = a.hi * c;
  const float r = fmaf(-q, b.hi, a.hi) + (a.lo - q * b.lo);  // the remainder makes up for the quick reciprocal
  return fmaf(r, c, q);
}

// floats of shared memory a CTA of `rows` rows needs: the halo rows' r, p with its two halo rows (a guard element at
// each end), the couplings
__host__ __device__ inline size_t cg_floats(int rows, int w) {
  return 2 * (size_t)w + (size_t)(rows + 2) * w + 2 + (size_t)(rows + 1) * w + 1 + (size_t)rows * w;
}

template <int K>
__global__ void __launch_bounds__(cg_threads(K), 1) k_cg_cluster(const CgBox B) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float wsum[2][32];             // the warps' and the CTAs' sums, a slot for each dot product (a
  __shared__ float part[2][kCgMaxCluster];  // slot is written again only after a barrier past its readers)
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = (int)blockDim.x, nw = nthr >> 5;
  const uint32_t rank = cluster_rank();
  const int nc = (int)gridDim.x;  // one cluster
  const int r0 = (int)((long long)B.rows * rank / nc), r1 = (int)((long long)B.rows * (rank + 1) / nc);
  const int rows = r1 - r0, w = B.w, cells = rows * w;
  float* rh = sm;                                // r of the row below and of the row above (w each)
  float* p = rh + 2 * w + 1;                     // (rows + 2) x w
  float* cr = p + (size_t)(rows + 2) * w + 1;    // coupling of row k - 1 to row k, k = 0 .. rows
  float* ct = cr + (size_t)(rows + 1) * w + 1;   // coupling to the next column, one guard element before
  auto grid_cell = [&](int row, int col) { return (size_t)(B.i0 + r0 + row) * B.nt + B.j0 + col; };

  for (int i = tid; i < (rows + 2) * w + 2; i += nthr) p[i - 1] = 0.f;
  for (int i = tid; i < (rows + 1) * w; i += nthr) {
    const int row = i / w - 1, col = i - (row + 1) * w;
    cr[i] = r0 + row >= 0 && r0 + row + 1 < B.rows ? B.ar[grid_cell(row, col)] : 0.f;
  }
  for (int i = tid; i < cells; i += nthr) {
    const int row = i / w, col = i - row * w;
    ct[i] = col + 1 < w ? B.at[grid_cell(row, col)] : 0.f;
  }
  if (tid == 0) ct[-1] = 0.f;
  for (int i = tid; i < 2 * w; i += nthr) {
    const int row = i < w ? -1 : rows, col = i < w ? i : i - w;
    rh[i] = r0 + row >= 0 && r0 + row < B.rows ? (float)(B.rs[grid_cell(row, col)] * B.inv_scale) : 0.f;
  }
  float r[K], y[K], ap[K], pc[K];
  float v = 0.f;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int c = tid + k * nthr;
    r[k] = y[k] = ap[k] = pc[k] = 0.f;
    if (c < cells) {
      const int row = c / w;
      r[k] = (float)(B.rs[grid_cell(row, c - row * w)] * B.inv_scale);
    }
    v += r[k] * r[k];
  }
  __syncthreads();
  // the cells' couplings in registers, if there are few
  constexpr bool kRegs = K <= 4;
  float cd[kRegs ? K : 1], cu[kRegs ? K : 1], cl[kRegs ? K : 1], ch[kRegs ? K : 1];
  if constexpr (kRegs) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int c = tid + k * nthr;
      const bool in = c < cells;
      cd[k] = in ? cr[c] : 0.f;
      cu[k] = in ? cr[c + w] : 0.f;
      cl[k] = in ? ct[c - 1] : 0.f;
      ch[k] = in ? ct[c] : 0.f;
    }
  }
  if (nc > 1) cluster_barrier();  // every CTA of the cluster runs: its shared memory may be written

  // the cluster's sum of v, in every thread
  auto total = [&](float x, int slot) -> FloatPair {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) wsum[slot][warp] = x;
    __syncthreads();
    if (nc == 1 || warp == 0) {  // (lanes below the next power of two of nw hold the sum)
      x = lane < nw ? wsum[slot][lane] : 0.f;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1)
        if (o < nw) x += __shfl_xor_sync(0xffffffffu, x, o);
    }
    FloatPair s{__shfl_sync(0xffffffffu, x, 0), 0.f};
    if (nc > 1) {
      x = s.hi;
      if (warp == 0 && lane < nc) peer_store(peer_addr(&part[slot][rank], (uint32_t)lane), x);
      cluster_barrier();
      s.hi = lane < nc ? part[slot][lane] : 0.f;
#pragma unroll
      for (int o = 1; o < kCgMaxCluster; o <<= 1) {
        if (o < nc) {
          const FloatPair b{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o)};
          s = pair_add(s, b);
        }
      }
      s.hi = __shfl_sync(0xffffffffu, s.hi, 0);  // (lanes past the cluster's size hold other sums)
      s.lo = __shfl_sync(0xffffffffu, s.lo, 0);
    }
    return s;
  };

  FloatPair rr = total(v, 0), rr_old = rr;
  const float rr_stop = (float)(B.tol2 * ((double)rr.hi + (double)rr.lo));
  int it = 0;
  for (;; ++it) {
    if (it >= B.max_iter || !(rr.hi > rr_stop)) break;  // (also ends where rr is no number)
    const float beta = it == 0 ? 0.f : pair_ratio(rr, rr_old);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int c = tid + k * nthr;
      pc[k] = r[k] + beta * pc[k];
      if (c < cells) p[w + c] = pc[k];
    }
    for (int i = tid; i < 2 * w; i += nthr) {
      float* h = i < w ? p + i : p + (size_t)rows * w + i;  // (i - w into row rows + 1)
      *h = rh[i] + beta * *h;
    }
    __syncthreads();
    v = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int c = tid + k * nthr;
      if (c < cells) {
        const float* q = p + w + c;
        float a;
        if constexpr (kRegs) a = pc[k] + cd[k] * q[-w] + cu[k] * q[w] + cl[k] * q[-1] + ch[k] * q[1];
        else a = pc[k] + cr[c] * q[-w] + cr[c + w] * q[w] + ct[c - 1] * q[-1] + ct[c] * q[1];
        ap[k] = a;
        v += pc[k] * a;
      }
    }
    const float alpha = pair_ratio(rr, total(v, 1));
    v = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int c = tid + k * nthr;
      if (c < cells) {
        y[k] += alpha * pc[k];
        r[k] -= alpha * ap[k];
        v += r[k] * r[k];
      }
    }
    if (nc > 1) {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int c = tid + k * nthr;
        // the neighbours' copies of the first and the last row
        if (rank > 0 && c < w) peer_store(peer_addr(rh + w + c, rank - 1), r[k]);
        if ((int)rank + 1 < nc && c >= cells - w && c < cells) peer_store(peer_addr(rh + (c - (cells - w)), rank + 1), r[k]);
      }
    }
    rr_old = rr;
    rr = total(v, 0);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int c = tid + k * nthr;
    if (c < cells) {
      const int row = c / w;
      B.y[grid_cell(row, c - row * w)] = y[k];
    }
  }
  if (rank == 0 && tid == 0) *B.iters = it;
}

// CTAs of the cluster, cells and threads for a box. nc = 0: it does not fit (the tile kernels take it).
struct CgPlan {
  int nc = 0, k = 0, threads = 0;
  size_t smem = 0;
};

template <int K>
cudaError_t cg_launch(const CgBox& B, const CgPlan& L, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_cg_cluster<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cg_cluster<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)L.nc);
  cfg.blockDim = dim3((unsigned)L.threads);
  cfg.dynamicSmemBytes = L.smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)L.nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_cg_cluster<K>, B);
}

// whether the device can hold a cluster of the plan
template <int K>
bool cg_resident(const CgPlan& L) {
  if (cudaFuncSetAttribute(k_cg_cluster<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.smem) != cudaSuccess ||
      cudaFuncSetAttribute(k_cg_cluster<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)L.nc);
  cfg.blockDim = dim3((unsigned)L.threads);
  cfg.dynamicSmemBytes = L.smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)L.nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_cg_cluster<K>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= 1;
}

// The smallest cluster whose CTAs have at most 1024 cells (two per thread), as large as 16, then more cells per
// thread; up to 4096 cells one CTA alone, which needs no cluster barrier. Measured (whole solve of an m x n system, 1 / 4 /
// 8 / 16 CTAs, ms): 38x38 0.50 / 0.66 / 0.69 / 0.79; 10x201 0.88 / 1.17 / 1.18 / -; 98x58 1.69 / 1.20 / 1.14 / 1.28;
// 198x118 - / 4.4 / 2.8 / 2.7. The tile kernels: 2.9, 5.9, 5.9, 10.1.
inline CgPlan cg_plan(int rows, int w, int max_iter) {
  if (rows < 1 || w < 1 || (long long)rows * w > 8192ll * kCgMaxCluster || max_iter > kCgMaxIter) return CgPlan();
  const long long all = (long long)rows * w;
  for (int nc = 1; nc <= kCgMaxCluster && nc <= rows; nc *= 2) {
    const int per = (rows + nc - 1) / nc;  // rows of the largest CTA
    const long long cells = (long long)per * w;
    const bool last = 2 * nc > kCgMaxCluster || 2 * nc > rows;
    if (!last && cells > (nc == 1 ? 4096 : 1024)) continue;
    for (int k = 2; k <= 16; k *= 2) {
      if (cells > (long long)k * cg_threads(k) || (k == 2 && all > 2048 && nc == 1)) continue;
      CgPlan L;
      L.nc = nc;
      L.k = k;
      L.threads = (int)(((cells + k - 1) / k + 31) / 32 * 32);
      L.smem = cg_floats(per, w) * sizeof(float);
      if (L.smem > 220 * 1024) return CgPlan();
      const bool ok = k == 2 ? cg_resident<2>(L) : k == 4 ? cg_resident<4>(L) : k == 8 ? cg_resident<8>(L) : cg_resident<16>(L);
      if (ok) return L;
    }
  }
  return CgPlan();
}

inline cudaError_t cg_solve(const CgBox& B, const CgPlan& L, cudaStream_t st) {
  switch (L.k) {
    case 2: return cg_launch<2>(B, L, st);
    case 4: return cg_launch<4>(B, L, st);
    case 8: return cg_launch<8>(B, L, st);
    default: return cg_launch<16>(B, L, st);
  }
}

}  // namespace mcrt
