// cgcluster.cuh -- a whole inner conjugate-gradient solve of the PDA in one launch: one thread-block cluster
// holds the system in its shared memory and registers.
//
// An iteration of the tile kernels (pda.cu) is three graph nodes of a few microseconds each, whatever the
// system's size (11 us at 20,000 cells, where the arithmetic is 0.1 us). Here the box of rows and columns that
// holds the unknown cells is split by rows over the CTAs of one cluster (1 to 16, one per SM), its vectors in registers and
// shared memory.
//
// What bounds an iteration is the latency of its barriers and sums, so there is one cluster barrier in it: all dot products
// at once, those of r and A r alone (Chronopoulos and Gear's form of the method; p.Ap follows from them), and A p by the
// recurrence s = A r + beta s. The barrier that brings the sums also brings A r of the neighbour CTAs' rows beside this CTA's,
// whose r it updates itself. (With a barrier each for p.Ap and r.r a whole solve of the 400x200 disk's PDA took 6.4 ms
// against 5.2.) The sums are FP32 in a CTA, the CTAs' sums pairs of floats (FP64 adds and divides have several times
// the latency here), in a fixed order: the same system gives the same bits. (Systems of very high contrast that this does
// not carry are left to the tile kernels: Refinement in pda.cu.) Cells of the box that are no unknowns have zero
// couplings and a zero right-hand side, and stay zero.
//
// Limit: about 100 rows of 32 columns to 14 of 288 per CTA with the line preconditioner, else 8192 cells per CTA; beyond it
// the tile kernels use the whole GPU.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

namespace mcrt {

// threads of a CTA at most when each carries K cells (the register budget of K cells' vectors)
__host__ __device__ constexpr int cg_threads(int K) { return K <= 4 ? 1024 : 512; }
constexpr int kCgMaxCluster = 16;
constexpr int kCgMaxIter = 200000;  // iterations of one launch at most (about 0.6 s)

struct CgBox {
  int nt;              // columns of the grid
  int i0, j0;          // first row and column of the box
  int rows, w;         // its size
  const float *ar, *at;  // scaled couplings to the next row / column (whole grid)
  const double* rs;    // scaled residual (whole grid)
  double inv_scale;    // right-hand side r = rs * inv_scale
  float* y;            // solution (whole grid, box cells written)
  double tol2;         // stop at rr <= kCgStop tol2 rr0
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

// The cluster's sums of v[0 .. N), in every thread. wsum: the CTA's warps; part: the CTAs' sums here. part may be written
// again only in the next but one call (a CTA may be a call ahead of one that still reads).
template <int N>
__device__ __forceinline__ void cluster_sums(float* v, FloatPair* s, float (*wsum)[32], float (*part)[kCgMaxCluster],
                                             int nc, uint32_t rank) {
  const unsigned full = 0xffffffffu;
  const int lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] += __shfl_xor_sync(full, v[i], o);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) wsum[i][warp] = v[i];
  }
  __syncthreads();
  if (nc == 1 || warp == 0) {  // (lanes below the next power of two of nw hold the sum)
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = lane < nw ? wsum[i][lane] : 0.f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
      if (o < nw) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] += __shfl_xor_sync(full, v[i], o);
      }
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = __shfl_sync(full, v[i], 0);
  }
#pragma unroll
  for (int i = 0; i < N; ++i) s[i] = {v[i], 0.f};
  if (nc > 1) {
    if (warp == 0 && lane < nc) {
      const uint32_t a = peer_addr(&part[0][rank], (uint32_t)lane);
#pragma unroll
      for (int i = 0; i < N; ++i) peer_store(a + i * (uint32_t)(kCgMaxCluster * sizeof(float)), v[i]);
    }
    cluster_barrier();
#pragma unroll
    for (int i = 0; i < N; ++i) s[i].hi = lane < nc ? part[i][lane] : 0.f;
#pragma unroll
    for (int o = 1; o < kCgMaxCluster; o <<= 1)
      if (o < nc) {
#pragma unroll
        for (int i = 0; i < N; ++i)
          s[i] = pair_add(s[i], {__shfl_xor_sync(full, s[i].hi, o), __shfl_xor_sync(full, s[i].lo, o)});
      }
#pragma unroll
    for (int i = 0; i < N; ++i) {  // (lanes past the cluster's size hold other sums)
      s[i].hi = __shfl_sync(full, s[i].hi, 0);
      s[i].lo = __shfl_sync(full, s[i].lo, 0);
    }
  }
}

// The preconditioned iterations leave more of the error in the slow components than the tile kernels' at the same
// residual, so they stop at a third of the residual asked for: a few more iterations instead of a larger error of the
// whole solve. Relative error of the PDA temperatures against a 64-bit direct solve, tile kernels / 1 / 0.1 here:
// 400x200 non-gray 1.3e-13 / 3.8e-13 / 2.5e-14, 300x160 gray 5.9e-14 / 7.3e-14 / 1.5e-14, 68x160 non-gray 7e-14 / 2e-13 /
// 2e-14; time of the call 21.8 / 3.91 / 4.17 ms, 8.3 / 1.21 / 1.28, 11.9 / 0.96 / 0.97.
constexpr double kCgStop = 0.1;

// The scalars of an iteration from r.z, z.Az and r.r (the same in every thread).
struct CgScalars {
  float alpha = 0.f, beta = 0.f, rr_stop, pap = 0.f;
  FloatPair rz_old;
  bool first = true;
  __device__ CgScalars(FloatPair rz, FloatPair rr, double tol2)
      : rr_stop((float)(kCgStop * tol2 * ((double)rr.hi + (double)rr.lo))), rz_old(rz) {}
  // false: converged (or r.r is no number)
  __device__ __forceinline__ bool direction(FloatPair rz, FloatPair zaz, FloatPair rr) {
    if (!(rr.hi > rr_stop)) return false;
    // p = z + beta p_old is conjugate to p_old: p.Ap = z.Az - beta^2 p_old.Ap_old
    beta = first ? 0.f : pair_ratio(rz, rz_old);
    first = false;
    pap = (zaz.hi - beta * beta * pap) + zaz.lo;
    if (!(pap > 1e-4f * zaz.hi)) {  // rounding has eaten the difference: a new start from z
      beta = 0.f;
      pap = zaz.hi;
    }
    alpha = pair_ratio(rz, {pap, 0.f});
    rz_old = rz;
    return true;
  }
};

// floats of shared memory a CTA of `rows` rows needs: A r of the halo rows (even and odd) and their s, r with its two
// halo rows (a guard element at each end), the couplings
__host__ __device__ inline size_t cg_floats(int rows, int w) {
  return 6 * (size_t)w + (size_t)(rows + 2) * w + 2 + (size_t)(rows + 1) * w + 1 + (size_t)rows * w;
}

template <int K>
__global__ void __launch_bounds__(cg_threads(K), 1) k_cg_cluster(const CgBox B) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float wsum[2][32];                // the warps' sums of r.r and r.Ar
  __shared__ float part[2][2][kCgMaxCluster];  // the CTAs', for even and odd iterations
  const int tid = (int)threadIdx.x, nthr = (int)blockDim.x;
  const uint32_t rank = cluster_rank();
  const int nc = (int)gridDim.x;  // one cluster
  const int r0 = (int)((long long)B.rows * rank / nc), r1 = (int)((long long)B.rows * (rank + 1) / nc);
  const int rows = r1 - r0, w = B.w, cells = rows * w;
  float* wh = sm;                                // A r of the row below and of the row above, even and odd: 2 x 2 x w
  float* sh = wh + 4 * w;                        // their s
  float* x = sh + 2 * w + 1;                     // r, (rows + 2) x w
  float* cr = x + (size_t)(rows + 2) * w + 1;    // coupling of row k - 1 to row k, k = 0 .. rows
  float* ct = cr + (size_t)(rows + 1) * w + 1;   // coupling to the next column, one guard element before
  auto grid_cell = [&](int row, int col) { return (size_t)(B.i0 + r0 + row) * B.nt + B.j0 + col; };

  for (int i = tid; i < 6 * w; i += nthr) wh[i] = 0.f;  // (and sh)
  for (int i = tid; i < (rows + 1) * w; i += nthr) {
    const int row = i / w - 1, col = i - (row + 1) * w;
    cr[i] = r0 + row >= 0 && r0 + row + 1 < B.rows ? B.ar[grid_cell(row, col)] : 0.f;
  }
  for (int i = tid; i < cells; i += nthr) {
    const int row = i / w, col = i - row * w;
    ct[i] = col + 1 < w ? B.at[grid_cell(row, col)] : 0.f;
  }
  if (tid == 0) ct[-1] = x[-1] = x[(size_t)(rows + 2) * w] = 0.f;
  for (int i = tid; i < (rows + 2) * w; i += nthr) {
    const int row = i / w - 1, col = i - (row + 1) * w;
    x[i] = r0 + row >= 0 && r0 + row < B.rows ? (float)(B.rs[grid_cell(row, col)] * B.inv_scale) : 0.f;
  }
  __syncthreads();
  float r[K], y[K], p[K], s[K], ax[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int c = tid + k * nthr;
    r[k] = c < cells ? x[w + c] : 0.f;
    y[k] = p[k] = s[k] = ax[k] = 0.f;
  }
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

  FloatPair sum[2];  // r.r, r.Ar
  auto step = [&](int odd) {
    float v[2] = {0.f, 0.f};
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int c = tid + k * nthr;
      if (c < cells) {
        const float* q = x + w + c;
        float a;
        if constexpr (kRegs) a = r[k] + cd[k] * q[-w] + cu[k] * q[w] + cl[k] * q[-1] + ch[k] * q[1];
        else a = r[k] + cr[c] * q[-w] + cr[c + w] * q[w] + ct[c - 1] * q[-1] + ct[c] * q[1];
        ax[k] = a;
        v[0] += r[k] * r[k];
        v[1] += r[k] * a;
        if (nc > 1) {
          if (rank > 0 && c < w) peer_store(peer_addr(wh + (2 * odd + 1) * w + c, rank - 1), a);
          if ((int)rank + 1 < nc && c >= cells - w) peer_store(peer_addr(wh + 2 * odd * w + c - (cells - w), rank + 1), a);
        }
      }
    }
    cluster_sums<2>(v, sum, wsum, part[odd], nc, rank);
  };

  step(0);
  CgScalars g(sum[0], sum[0], B.tol2);
  int it = 0;
  for (; it < B.max_iter && g.direction(sum[0], sum[1], sum[0]); ++it) {
    const float alpha = g.alpha, beta = g.beta;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int c = tid + k * nthr;
      p[k] = r[k] + beta * p[k];
      s[k] = ax[k] + beta * s[k];
      y[k] += alpha * p[k];
      r[k] -= alpha * s[k];
      if (c < cells) x[w + c] = r[k];
    }
    for (int i = tid; i < 2 * w; i += nthr) {
      const float si = wh[2 * (it & 1) * w + i] + beta * sh[i];
      sh[i] = si;
      x[i < w ? i : (size_t)rows * w + i] -= alpha * si;  // (i - w into row rows + 1)
    }
    __syncthreads();
    step((it + 1) & 1);
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

// The same with a line preconditioner: M = the couplings along theta (and the unit diagonal), solved exactly for every
// row in each iteration. Towards the midplane cells are much thinner in theta than in r (couplings 10 to 270 times
// stronger), where plain CG crawls along theta: iterations to 1e-5 on PDA bands of 400x200 and 60x142 grids
// 473 -> 167, 182 -> 19, 159 -> 6; with equal couplings 84 -> 59 (38x38), 281 -> 199 (198x118).
//
// A warp owns whole rows, a lane E consecutive columns of each, in registers. A row's tridiagonal solve is two linear
// recurrences (the L D L^T factors, made once per launch): E steps within the lane, a five-step scan of the
// lanes' affine maps by shuffle (their multipliers are constants, kept in shared memory), E more to add the carry;
// no barrier. The two neighbour rows are solved here too. Odd E keeps the lanes' shared-memory accesses free of bank
// conflicts (E = 2: two-way). An iteration costs 2.9 us against 2.1; whole solves, diagonal -> line: PDA of the 400x200
// disk 5.25 -> 3.97 ms (at the full residual, kCgStop = 1, as the others), of a 200x120 disk 1.19 -> 0.75, equal
// couplings 98x58 0.89 -> 0.85, 198x118 2.06 -> 1.83,
// 98x278 3.12 -> 2.44, 22x18 0.31 -> 0.33, 298x10 0.47 -> 0.53 (iterations of the diagonal one on strong couplings pay
// for those two many times over).
constexpr int kScan = 10;  // scan multipliers per row and lane: five steps forward, five backward

__host__ __device__ inline size_t pcg_floats(int rows, int W) {
  const size_t e = rows + 2;  // rows with the neighbours' two
  return 4 * (size_t)W + e * W + 2 + (e - 1) * W + e * W + 1 + 4 * e * W + e * kScan * 32;
}

// threads of a CTA at most when each carries E x Q cells
__host__ __device__ constexpr int pcg_threads(int cells) { return cells <= 4 ? 1024 : cells <= 7 ? 768 : 512; }

template <int E, int Q>
__global__ void __launch_bounds__(pcg_threads(E * Q), 1) k_pcg_lines(const CgBox B) {
  constexpr int W = 32 * E;  // columns of a row here (those past the box stay zero)
  extern __shared__ __align__(16) float sm[];
  __shared__ float wsum[3][32];                // the warps' sums of r.z, r.r and z.Az
  __shared__ float part[2][3][kCgMaxCluster];  // the CTAs', for even and odd iterations
  const unsigned full = 0xffffffffu;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = (int)blockDim.x, nw = nthr >> 5;
  const uint32_t rank = cluster_rank();
  const int nc = (int)gridDim.x;  // one cluster
  const int r0 = (int)((long long)B.rows * rank / nc), r1 = (int)((long long)B.rows * (rank + 1) / nc);
  const int rows = r1 - r0, er = rows + 2, w = B.w;  // row e of the er here is row r0 + e - 1 of the box
  float* wh = sm;                            // A z of row 0 and of row rows + 1, even and odd: 2 x 2 x W
  float* zs = wh + 4 * W + 1;                // er x W, a guard element at each end
  float* cr = zs + (size_t)er * W + 1;       // coupling of row e to row e + 1
  float* ct = cr + (size_t)(er - 1) * W + 1;  // coupling to the next column, one guard element before
  float* fm = ct + (size_t)er * W;           // factors: multiplier of the column before, 1 / d, products of multipliers
  float* fd = fm + (size_t)er * W;           // from the lane's first column and down from its last one
  float* qf = fd + (size_t)er * W;
  float* qb = qf + (size_t)er * W;
  float* scan = qb + (size_t)er * W;         // er x kScan x 32
  auto inside = [&](int e) { return r0 + e - 1 >= 0 && r0 + e - 1 < B.rows; };
  auto grid_cell = [&](int e, int col) { return (size_t)(B.i0 + r0 + e - 1) * B.nt + B.j0 + col; };

  for (int i = tid; i < 4 * W + er * W + 2; i += nthr) wh[i] = 0.f;  // (and zs)
  for (int i = tid; i < (er - 1) * W; i += nthr) {
    const int e = i / W, col = i % W;
    cr[i] = col < w && inside(e) && inside(e + 1) ? B.ar[grid_cell(e, col)] : 0.f;
  }
  for (int i = tid; i < er * W; i += nthr) {
    const int e = i / W, col = i % W;
    ct[i] = col + 1 < w && inside(e) ? B.at[grid_cell(e, col)] : 0.f;
  }
  if (tid == 0) ct[-1] = 0.f;
  __syncthreads();
  // L D L^T of each row's tridiagonal matrix (1 on the diagonal, ct beside it): d_j = 1 - ct_{j-1}^2 / d_{j-1},
  // multiplier m_j = -ct_{j-1} / d_{j-1}
  for (int e = tid; e < er; e += nthr) {
    float m = 0.f, id = 1.f;
    for (int j = 0; j < W; ++j) {
      fm[e * W + j] = m;
      fd[e * W + j] = id;
      const float c = ct[e * W + j];
      m = -c * id;
      id = 1.f / fmaxf(1.f + c * m, 1e-6f);  // (positive despite rounding: M stays positive definite)
    }
  }
  __syncthreads();
  for (int row = warp; row < er; row += nw) {
    const float* m = fm + row * W + lane * E;
    float f = 1.f, b = lane < 31 ? m[E] : 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      f *= m[e];
      qf[row * W + lane * E + e] = f;
    }
#pragma unroll
    for (int e = E - 1; e >= 0; --e) {
      qb[row * W + lane * E + e] = b;
      if (e > 0) b *= m[e];
    }
    float* s = scan + row * kScan * 32 + lane;
#pragma unroll
    for (int k = 0; k < 5; ++k) {  // the multiplier of the partner's value, zero without a partner
      const int o = 1 << k;
      s[k * 32] = lane >= o ? f : 0.f;
      s[(5 + k) * 32] = lane + o < 32 ? b : 0.f;
      const float fu = __shfl_up_sync(full, f, o), bd = __shfl_down_sync(full, b, o);
      f = lane >= o ? f * fu : 0.f;
      b = lane + o < 32 ? b * bd : 0.f;
    }
  }
  float r[Q][E], z[Q][E], y[Q][E], p[Q][E], s[Q][E], az[Q][E];
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int row = warp + q * nw, col = lane * E + e;
      r[q][e] = row < er && col < w && inside(row) ? (float)(B.rs[grid_cell(row, col)] * B.inv_scale) : 0.f;
      z[q][e] = y[q][e] = p[q][e] = s[q][e] = az[q][e] = 0.f;
    }
  __syncthreads();
  if (nc > 1) cluster_barrier();  // every CTA of the cluster runs: its shared memory may be written

  FloatPair sum[3];  // r.z, r.r, z.Az
  // z = M^-1 r of all rows, A z of the own ones, its first and last row to the neighbour CTAs, the three sums
  auto step = [&](int odd) {
    float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int row = warp + q * nw;
      if (row >= er) break;  // warp-uniform
      const int at = row * W + lane * E;
      const float* m = scan + row * kScan * 32 + lane;
      float g[E];
      g[0] = r[q][0];
#pragma unroll
      for (int e = 1; e < E; ++e) g[e] = r[q][e] + fm[at + e] * g[e - 1];
      float b = g[E - 1];
#pragma unroll
      for (int k = 0; k < 5; ++k) b += m[k * 32] * __shfl_up_sync(full, b, 1 << k);
      b = __shfl_up_sync(full, b, 1);
      if (lane == 0) b = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) g[e] = (g[e] + qf[at + e] * b) * fd[at + e];
#pragma unroll
      for (int e = E - 2; e >= 0; --e) g[e] += fm[at + e + 1] * g[e + 1];
      b = g[0];
#pragma unroll
      for (int k = 0; k < 5; ++k) b += m[(5 + k) * 32] * __shfl_down_sync(full, b, 1 << k);
      b = __shfl_down_sync(full, b, 1);
      if (lane == 31) b = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) zs[at + e] = z[q][e] = g[e] + qb[at + e] * b;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int row = warp + q * nw;
      if (row >= 1 && row <= rows) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int c = row * W + lane * E + e;
          const float* x = zs + c;
          const float a = z[q][e] + cr[c - W] * x[-W] + cr[c] * x[W] + ct[c - 1] * x[-1] + ct[c] * x[1];
          az[q][e] = a;
          v[0] += r[q][e] * z[q][e];
          v[1] += r[q][e] * r[q][e];
          v[2] += z[q][e] * a;
          if (row == 1 && rank > 0) peer_store(peer_addr(wh + (2 * odd + 1) * W + lane * E + e, rank - 1), a);
          if (row == rows && (int)rank + 1 < nc) peer_store(peer_addr(wh + 2 * odd * W + lane * E + e, rank + 1), a);
        }
      }
    }
    cluster_sums<3>(v, sum, wsum, part[odd], nc, rank);
  };

  step(0);
  CgScalars g(sum[0], sum[1], B.tol2);
  int it = 0;
  for (; it < B.max_iter && g.direction(sum[0], sum[2], sum[1]); ++it) {
    const float alpha = g.alpha, beta = g.beta;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int row = warp + q * nw;
      const bool halo = row == 0 || row == er - 1;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if (halo) az[q][e] = wh[(2 * (it & 1) + (row != 0)) * W + lane * E + e];
        p[q][e] = z[q][e] + beta * p[q][e];
        s[q][e] = az[q][e] + beta * s[q][e];
        y[q][e] += alpha * p[q][e];
        r[q][e] -= alpha * s[q][e];
      }
    }
    step((it + 1) & 1);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int row = warp + q * nw;
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (row >= 1 && row <= rows && lane * E + e < w) B.y[grid_cell(row, lane * E + e)] = y[q][e];
  }
  if (rank == 0 && tid == 0) *B.iters = it;
}

// CTAs of the cluster, kernel and threads for a box. nc = 0: it does not fit (the tile kernels take it).
struct CgPlan {
  int nc = 0, threads = 0;
  void (*kernel)(CgBox) = nullptr;
  size_t smem = 0;
};

// cells of a box at most (the largest of k_cg_cluster's; k_pcg_lines's boxes are smaller)
constexpr long long kCgMaxCells = 8192ll * kCgMaxCluster;

// Rows [0, 1) and columns [2, 3) of the smallest box around the cells with mask 2 (none: all zero). A box of more than
// kCgMaxCells, for which there is no plan, may come out smaller: no more of the mask is read then (8192 x 8192 cells, a wide
// region in the middle: 0.3 ms of host time, 60 for every cell of the mask in turn; 400 x 200 cells 12 us and 72).
inline void cg_box(const signed char* mask, int nr, int nt, int* box) {
  box[0] = box[1] = box[3] = 0;
  box[2] = nt;
  for (int i = 0; i < nr; ++i) {
    const signed char* row = mask + (size_t)i * nt;
    const void* hit = std::memchr(row, 2, nt);
    if (!hit) continue;
    if (box[1] == 0) box[0] = i;
    box[1] = i + 1;
    box[2] = std::min(box[2], (int)((const signed char*)hit - row));
    int last = nt;  // past the row's last cell, if it lies past the box
    while (last > box[3] && row[last - 1] != 2) --last;
    box[3] = last;
    if ((long long)(box[1] - box[0]) * (box[3] - box[2]) > kCgMaxCells) return;
  }
  if (box[1] == 0) box[2] = 0;
}

// dynamic shared memory of a plan's kernel at most (227 KB less the kernel's own few hundred bytes)
constexpr int kCgSmem = 220 * 1024;

// the plan's launch on a stream; check: whether the device can hold its cluster, nothing launched. (A kernel's limit belongs
// to the process, and threads plan and launch boxes of different sizes: it is always set to the same value, never to
// the plan's own size, which would take it from another thread between its plan and its launch.)
inline cudaError_t cg_launch(const CgPlan& L, const CgBox* B, cudaStream_t st, bool check) {
  cudaError_t e = cudaFuncSetAttribute(L.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCgSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(L.kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
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
  if (check) {
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, L.kernel, &cfg);
    return e != cudaSuccess ? e : (n >= 1 ? cudaSuccess : cudaErrorInvalidConfiguration);
  }
  return cudaLaunchKernelEx(&cfg, L.kernel, *B);
}
inline bool cg_resident(const CgPlan& L) {
  if (L.smem <= kCgSmem && cg_launch(L, nullptr, nullptr, true) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

// The line-preconditioned kernel for `per` rows of w columns in a CTA: the fewest columns per lane, the fewest rows
// per warp.
struct PcgShape {
  int E, Q;
  void (*kernel)(CgBox);
};
inline bool pcg_shape(int per, int w, CgPlan& L) {
  static const PcgShape all[] = {{1, 1, k_pcg_lines<1, 1>}, {1, 2, k_pcg_lines<1, 2>}, {1, 4, k_pcg_lines<1, 4>},
                                 {2, 1, k_pcg_lines<2, 1>}, {2, 2, k_pcg_lines<2, 2>},
                                 {3, 1, k_pcg_lines<3, 1>}, {3, 2, k_pcg_lines<3, 2>},
                                 {5, 1, k_pcg_lines<5, 1>}, {5, 2, k_pcg_lines<5, 2>}, {7, 1, k_pcg_lines<7, 1>},
                                 {9, 1, k_pcg_lines<9, 1>}};
  for (const PcgShape& s : all) {
    const int warps = (per + 2 + s.Q - 1) / s.Q;
    if (w > 32 * s.E || warps > pcg_threads(s.E * s.Q) / 32) continue;
    L.kernel = s.kernel;
    L.threads = 32 * warps;
    L.smem = pcg_floats(per, 32 * s.E) * sizeof(float);
    return true;
  }
  return false;
}

// The fewest CTAs with at most 8 rows each (whole solves of 38x38, 98x58, 198x118 boxes with equal couplings: 4 / 8 / 16 CTAs
// 0.52 / 0.49 / 0.52, 1.10 / 0.86 / 0.85, - / 2.21 / 1.83 ms).
inline CgPlan cg_plan(int rows, int w, int max_iter) {
  if (rows < 1 || w < 1 || max_iter > kCgMaxIter) return CgPlan();
  for (int nc = 1; nc <= kCgMaxCluster && nc <= rows; nc *= 2) {
    const int per = (rows + nc - 1) / nc;  // rows of the largest CTA
    const bool last = 2 * nc > kCgMaxCluster || 2 * nc > rows;
    CgPlan L;
    L.nc = nc;
    if ((last || per <= 8) && pcg_shape(per, w, L) && cg_resident(L)) return L;
  }
  // wide or large boxes: diagonal preconditioner, any columns
  if ((long long)rows * w > kCgMaxCells) return CgPlan();
  for (int nc = 1; nc <= kCgMaxCluster && nc <= rows; nc *= 2) {
    const int per = (rows + nc - 1) / nc;
    const long long cells = (long long)per * w;
    const bool last = 2 * nc > kCgMaxCluster || 2 * nc > rows;
    if (!last && cells > 1024) continue;
    for (int k = 2; k <= 16; k *= 2) {
      if (cells > (long long)k * cg_threads(k)) continue;
      CgPlan L;
      L.nc = nc;
      L.kernel = k == 2 ? k_cg_cluster<2> : k == 4 ? k_cg_cluster<4> : k == 8 ? k_cg_cluster<8> : k_cg_cluster<16>;
      L.threads = (int)(((cells + k - 1) / k + 31) / 32 * 32);
      L.smem = cg_floats(per, w) * sizeof(float);
      if (cg_resident(L)) return L;
    }
  }
  return CgPlan();
}

inline cudaError_t cg_solve(const CgBox& B, const CgPlan& L, cudaStream_t st) { return cg_launch(L, &B, st, false); }

}  // namespace mcrt
