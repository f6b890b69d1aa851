// raytrace.cu -- ray-traced observables: images, the SED and interferometric visibilities, by integrating
// the source function along straight rays through the (r, theta) grid with the Monte Carlo temperatures
// (Sect. 2.3: observables from the computed source function, free of Monte Carlo noise; Sect. 4.1: SED at
// 45 degrees, N-band visibilities at a 100 m baseline).
//
// Readings: the source function of a cell in bin b is S_b = kappa_b Bbar_b(T) / chi_b with chi = kappa +
// sigma (thermal emission over the total extinction; scattering takes light out of a ray and adds none);
// S and the extinction are constant in a cell, so a segment of optical depth dtau updates the intensity
// carried towards the observer exactly: I <- S + (I - S) exp(-dtau). The star is a point source at the
// origin, dimmed along the radial line towards the observer, and occults no ray.
//
// Layout: the rays are marched by a lane each (raymarch.cuh: closed-form crossings, one square root or one quadratic
// per cell) and integrated by a warp each, lanes over the wavelength bins. Consecutive lanes take rays that are
// neighbours on the sky (Morton order of the sky positions, built by mcrt_set_rays), whose paths cross the same cells.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

#include "internal.h"
#include "planck.cuh"
#include "raymarch.cuh"
#include "source.cuh"

namespace mcrt {

struct RayState {
  DBuf p, q, w;   // rays: sky-plane coordinates (cm) and areas (cm^2), FP64
  DBuf order;     // the rays in Morton order of their sky positions (int32): neighbours share warps
  long long n = 0;
  double incl = 0, dist = 0;
  DBuf S;         // cells x nlam source table of the last trace (float or double)
  int S_prec = 0, S_which = -1;
  unsigned long long S_epoch = ~0ull;
  DBuf img;       // n x nlam image of the last trace
  int img_prec = 0;
  bool have_img = false;
  DBuf part, F, Fs, cnt;  // SED partial sums, disk + star flux, star flux, counters
  DBuf vis_par;           // per visibility: bin, fu, fv
  DBuf vis_out;
};

void ray_free(RayState* r) { delete r; }

namespace {

constexpr int kRayBlock = 128;
template <class R>
constexpr int kRaySegs = sizeof(R) == 8 ? 8 : 16;  // segments of a ray taken at once
constexpr int kSedBlock = 128;

// One segment of optical depth x through a cell of source function s: I <- I e^-x + s (1 - e^-x).
// 1 - e^-x is not formed as a difference where x is small (optically thin segments, where the FP32
// exponential's absolute error of ~2e-7 would be a large part of it): below 0.1 it is the series
// x (1 - x/2 + x^2/6 - x^3/24), whose truncation is below 1e-6 of it; in FP64, expm1.
// thin / thick: x is known to be below 0.1 / not to be (the same result with half the arithmetic).
template <class R>
__device__ __forceinline__ R segment(R I, R s, R x, bool thin, bool thick);
template <>
__device__ __forceinline__ float segment<float>(float I, float s, float x, bool thin, bool thick) {
  const float e = thin ? 0.f : __expf(-x);
  const float ser = thick ? 0.f : x * (1.f - x * (0.5f - x * (1.f / 6.f - x * (1.f / 24.f))));
  const bool small = thin || (!thick && x < 0.1f);
  const float om = small ? ser : 1.f - e;
  return (small ? 1.f - ser : e) * I + om * s;
}
template <>
__device__ __forceinline__ double segment<double>(double I, double s, double x, bool, bool) {
  return exp(-x) * I - expm1(-x) * s;
}

// A warp takes `rw` rays, neighbours on the sky: its lanes march a ray each (raymarch.cuh) until each has kRaySegs segments
// with dust or has left the grid, then the warp goes through the rays with its lanes over the bins (NB per lane, b = lane +
// 32 k): the segments (cell, optical depth per unit chi) from shared memory, the intensities from and to the image; and so
// on until every ray is out. So a ray is marched once and a segment's row of the source table is a contiguous load of the
// warp. (A thread per ray and 25 bins marched each ray four times and read the rows scattered over the lanes.)
// Instruction issue bounds it, 60 % busy at 18 warps per SM: 1.8 ms for 104,448 rays through 200x120 cells, 100 bins, 18 million
// segments (3.4 before). kRaySegs = 8 / 16 / 32: 1.9 / 1.8 / 2.0 ms.
// cnt[0] += segments with dust, cnt[1] |= 1 when a ray took more events than the bound.
template <class R>
struct RaySeg {
  R a;  // optical depth per unit chi
  int c;
};
template <class R, int NB>
__global__ void __launch_bounds__(kRayBlock, sizeof(R) == 8 ? 3 : NB <= 4 ? 6 : 4)
    k_raytrace(const DevModel<R> M, const R* __restrict__ chi, const R* __restrict__ S, long long n, int rw,
               const int* __restrict__ order, const double* __restrict__ p, const double* __restrict__ q, double inv_l,
               R si, R ci, int max_events, R* __restrict__ img, unsigned long long* __restrict__ cnt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RaySeg<R>* seg = reinterpret_cast<RaySeg<R>*>(smem_raw);  // warps x kRaySegs x 32
  FaceCoef<R>* face = reinterpret_cast<FaceCoef<R>*>(seg + kRayBlock * kRaySegs<R>);  // nt+1 entries for this inclination
  const unsigned full = 0xffffffffu;
  const int lane = (int)threadIdx.x & 31, nlam = M.nlam, nt = M.nt;
  seg += (threadIdx.x >> 5) * (kRaySegs<R> * 32);
  for (int j = threadIdx.x; j <= nt; j += blockDim.x) face[j] = face_coef<R>(M.c2[j], M.s2[j], M.fk[j], si, ci);
  __syncthreads();
  const long long base = ((long long)blockIdx.x * (kRayBlock / 32) + (threadIdx.x >> 5)) * rw;
  if (base >= n) return;
  const int rays = n - base < rw ? (int)(n - base) : rw;
  R ch[NB], cmin = (R)INFINITY, cmax = (R)0;
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    const int b = lane + 32 * k;
    ch[k] = b < nlam ? chi[b] : (R)0;
    if (b < nlam) {
      cmin = ch[k] < cmin ? ch[k] : cmin;
      cmax = ch[k] > cmax ? ch[k] : cmax;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const R x = __shfl_xor_sync(full, cmin, o), y = __shfl_xor_sync(full, cmax, o);
    cmin = x < cmin ? x : cmin;
    cmax = y > cmax ? y : cmax;
  }
  const RayGrid<R> G{M.nr, M.nt, M.rf2, M.cf, face};
  int ray = 0, events = 0;
  bool live = false, err = false;
  RayMarch<R> m;
  if (lane < rays) {
    ray = order[base + lane];
    live = m.begin(G, (R)(p[ray] * inv_l), (R)(q[ray] * inv_l), si, ci);
  }
  unsigned long long segs = 0;
  for (bool first = true;; first = false) {
    int got = 0;
    while (live && got < kRaySegs<R>) {
      live = m.step(G, [&](int ir, int it, R L) {
        const int c = ir * nt + it;
        const R a = M.rho[c] * L;
        if (a > (R)0) seg[got++ * 32 + lane] = {a, c};
      });
      if (live && ++events >= max_events) {
        live = false;
        err = true;
      }
    }
    segs += got;
    const bool more = __any_sync(full, live);
    __syncwarp();
    for (int r = 0; r < rays; ++r) {
      const int ns = __shfl_sync(full, got, r);
      if (ns == 0 && !first) continue;
      R* o = img + (size_t)__shfl_sync(full, ray, r) * nlam + lane;
      R I[NB];
#pragma unroll
      for (int k = 0; k < NB; ++k) I[k] = !first && lane + 32 * k < nlam ? o[32 * k] : (R)0;
#pragma unroll 4
      for (int j = 0; j < ns; ++j) {
        const RaySeg<R> g = seg[j * 32 + r];
        const R* Sc = S + (size_t)g.c * nlam + lane;
        R s[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) s[k] = lane + 32 * k < nlam ? Sc[32 * k] : (R)0;
        // (the same in the whole warp)
        if (g.a * cmax < (R)0.1) {
#pragma unroll
          for (int k = 0; k < NB; ++k) I[k] = segment<R>(I[k], s[k], g.a * ch[k], true, false);
        } else if (g.a * cmin >= (R)0.1) {
#pragma unroll
          for (int k = 0; k < NB; ++k) I[k] = segment<R>(I[k], s[k], g.a * ch[k], false, true);
        } else {
#pragma unroll
          for (int k = 0; k < NB; ++k) I[k] = segment<R>(I[k], s[k], g.a * ch[k], false, false);
        }
      }
#pragma unroll
      for (int k = 0; k < NB; ++k)
        if (lane + 32 * k < nlam) o[32 * k] = I[k];
    }
    __syncwarp();
    if (!more) break;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) segs += __shfl_xor_sync(full, segs, o);
  const bool any_err = __any_sync(full, err);
  if (lane == 0) {
    if (segs) atomicAdd(cnt, segs);
    if (any_err) atomicOr(cnt + 1, 1ull);
  }
}

// Weighted image sums per bin over a contiguous range of rays (one block per range, threads over bins,
// so each ray's row is read contiguously).
template <class R>
__global__ void k_sed_part(long long n, int nlam, long long per_blk, const R* __restrict__ img,
                           const double* __restrict__ w, double* __restrict__ part) {
  const long long r0 = (long long)blockIdx.x * per_blk;
  const long long r1 = r0 + per_blk < n ? r0 + per_blk : n;
  for (int b = threadIdx.x; b < nlam; b += blockDim.x) {
    double s = 0.0;
    for (long long r = r0; r < r1; ++r) s += w[r] * (double)img[r * nlam + b];
    part[(size_t)blockIdx.x * nlam + b] = s;
  }
}

// Sum over the block (kSedBlock threads), in every thread.
__device__ __forceinline__ double sed_block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  v = 0.0;
#pragma unroll
  for (int k = 0; k < kSedBlock / 32; ++k) v += sh[k];
  __syncthreads();
  return v;
}

// The flux of a bin, a block each: F_b = sum of the partial sums (fixed order) / d^2 + star. The star at distance d:
// pi R*^2 Bbar_b(T*) / d^2, dimmed by chi_b times the column sum rho dr of polar row `it` (the row that holds the
// line of sight). Latency bounds it: both sums by one thread per bin took 139 us on a 200-shell grid.
__global__ void k_sed_final(int nr, int nt, int it, int nlam, const double* __restrict__ rho_l,
                            const double* __restrict__ rf_l, const double* __restrict__ lam_e,
                            const double* __restrict__ chi, double Tstar, double Rstar, double dist, int nblk,
                            const double* __restrict__ part, double* __restrict__ Fs, double* __restrict__ F) {
  __shared__ double sh[kSedBlock / 32];
  const int b = blockIdx.x;
  double s = 0.0, col = 0.0;
  for (int j = threadIdx.x; j < nblk; j += kSedBlock) s += part[(size_t)j * nlam + b];
  for (int ir = threadIdx.x; ir < nr; ir += kSedBlock) col += rho_l[ir * nt + it] * (rf_l[ir + 1] - rf_l[ir]);
  s = sed_block_sum(s, sh);
  col = sed_block_sum(col, sh);
  if (threadIdx.x != 0) return;
  const double k4 = kKB * kKB * kKB * kKB;
  const double pref3 = 2.0 * k4 * Tstar * Tstar * Tstar * Tstar / (kH * kH * kH * kC * kC);
  const double g_short = b > 0 ? tail3(kH * kC / (lam_e[b] * 1e-4 * kKB * Tstar)) : 0.0;
  const double g_long = tail3(b + 1 == nlam ? 0.0 : kH * kC / (lam_e[b + 1] * 1e-4 * kKB * Tstar));
  const double B = pref3 * (g_long - g_short);
  const double star = 3.14159265358979323846 * Rstar * Rstar * B / (dist * dist) * exp(-col * chi[b]);
  Fs[b] = star;
  F[b] = s * (1.0 / (dist * dist)) + star;
}

// Sums over the rays of w I exp(-2 pi i t), t = fu p + fv q in turns (fu, fv: spatial frequency over distance, cycles
// per cm at the source), reduced to its fractional part in FP64 before the sine and cosine. Block (j, y) takes part y
// of the rays of visibility j: few visibilities alone would leave most of the chip idle (5 of 104,448 rays: a block each
// 0.41 ms with the copies of the call, now 0.08).
template <class R>
__global__ void k_vis_part(long long n, int nlam, const R* __restrict__ img, const double* __restrict__ p,
                           const double* __restrict__ q, const double* __restrict__ w, const double* __restrict__ par,
                           double* __restrict__ part) {
  const int j = blockIdx.x;
  const int b = (int)par[3 * j];
  const double fu = par[3 * j + 1], fv = par[3 * j + 2];
  double re = 0.0, im = 0.0, tot = 0.0;
#pragma unroll 2
  for (long long r = (long long)blockIdx.y * blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.y * blockDim.x) {
    const double f = w[r] * (double)img[r * nlam + b];
    double t = fu * p[r] + fv * q[r];
    t -= rint(t);
    double sn, cs;
    if (sizeof(R) == 8) {
      sincospi(2.0 * t, &sn, &cs);
    } else {
      float s32, c32;
      sincospif(2.0f * (float)t, &s32, &c32);
      sn = s32;
      cs = c32;
    }
    re += f * cs;
    im -= f * sn;
    tot += f;
  }
  __shared__ double sh[3][32];
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
    tot += __shfl_down_sync(0xffffffffu, tot, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    sh[0][wid] = re;
    sh[1][wid] = im;
    sh[2][wid] = tot;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double a = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) a += sh[threadIdx.x][k];
    part[3 * ((size_t)j * gridDim.y + blockIdx.y) + threadIdx.x] = a;
  }
}

// |V| of each visibility from its parts (a warp each, fixed order).
__global__ void k_vis(int n_vis, int parts, const double* __restrict__ part, const double* __restrict__ par,
                      const double* __restrict__ Fs, int with_star, double inv_d2, double* __restrict__ out) {
  const int j = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = (int)(threadIdx.x & 31u);
  if (j >= n_vis) return;
  double a = 0.0, c = 0.0, t = 0.0;
  for (int k = lane; k < parts; k += 32) {
    const double* x = part + 3 * ((size_t)j * parts + k);
    a += x[0];
    c += x[1];
    t += x[2];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
    t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  if (lane != 0) return;
  const double fs = with_star ? Fs[(int)par[3 * j]] : 0.0;
  a = a * inv_d2 + fs;
  c = c * inv_d2;
  t = t * inv_d2 + fs;
  out[j] = t > 0.0 ? sqrt(a * a + c * c) / t : 0.0;
}

int sm_count(int device) {
  int v = 0;
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device);
  return v > 0 ? v : 1;
}

constexpr size_t kRayFaces = 200 * 1024;  // bytes of the face table (and a value per bin) at most
constexpr int kRaySmem = (int)kRayFaces + 16 * 1024;  // with the segments: a launch's shared memory at most

template <class R>
size_t ray_smem(int nt) {
  static_assert(kRayBlock * kRaySegs<R> * sizeof(RaySeg<R>) <= 16 * 1024, "kRaySmem");
  return (size_t)kRayBlock * kRaySegs<R> * sizeof(RaySeg<R>) + (size_t)(nt + 1) * sizeof(FaceCoef<R>);
}

template <class R, int NB>
cudaError_t launch_trace_nb(mcrt_disk* d, RayState* rs, const DevModel<R>& M, const R* chi, int sms) {
  const R si = (R)std::sin(rs->incl), ci = (R)std::cos(rs->incl);
  const int max_events = 4 * (d->nr + d->nt) + 64;
  const double inv_l = 1.0 / d->l_unit;
  const size_t smem = ray_smem<R>(d->nt);
  if (smem > 48 * 1024) {  // (the limit belongs to the process: one value, which no thread's launch lowers for another's)
    cudaError_t e = cudaFuncSetAttribute(k_raytrace<R, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRaySmem);
    if (e != cudaSuccess) return e;
  }
  // rays per warp: 32, fewer until 16 warps per SM have some (26,112 rays: 8 per warp 0.68 ms, 32 per warp 1.4)
  int rw = 32;
  while (rw > 1 && rs->n < (long long)rw * sms * 16) rw /= 2;
  const long long warps = (rs->n + rw - 1) / rw;
  const int grid = (int)((warps + kRayBlock / 32 - 1) / (kRayBlock / 32));
  k_raytrace<R, NB><<<grid, kRayBlock, smem, d->stream>>>(M, chi, rs->S.as<R>(), rs->n, rw, rs->order.as<int>(),
                                                          rs->p.as<double>(), rs->q.as<double>(), inv_l, si, ci,
                                                          max_events, rs->img.as<R>(),
                                                          rs->cnt.as<unsigned long long>());
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_trace(mcrt_disk* d, RayState* rs, const DevModel<R>& M, const R* chi, int sms) {
  switch ((d->nlam + 31) / 32) {
    case 1: return launch_trace_nb<R, 1>(d, rs, M, chi, sms);
    case 2: return launch_trace_nb<R, 2>(d, rs, M, chi, sms);
    case 3: return launch_trace_nb<R, 3>(d, rs, M, chi, sms);
    case 4: return launch_trace_nb<R, 4>(d, rs, M, chi, sms);
    case 5: return launch_trace_nb<R, 5>(d, rs, M, chi, sms);
    case 6: return launch_trace_nb<R, 6>(d, rs, M, chi, sms);
    case 7: return launch_trace_nb<R, 7>(d, rs, M, chi, sms);
    default: return launch_trace_nb<R, 8>(d, rs, M, chi, sms);
  }
}

}  // namespace
}  // namespace mcrt

using namespace mcrt;

#define CK(call, what)                                    \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return cuda_fail(d, e_, what); \
  } while (0)

namespace {

template <class R>
DevModel<R> model_of(const mcrt_disk* d);
template <>
DevModel<float> model_of<float>(const mcrt_disk* d) { return d->model32(); }
template <>
DevModel<double> model_of<double>(const mcrt_disk* d) { return d->model64(); }
template <class R>
const R* chi_of(const mcrt_disk* d) { return static_cast<const R*>(sizeof(R) == 8 ? d->chi64.p : d->chi32.p); }

static double j_factor(const mcrt_disk* d) {
  return j_factor_of(d->Lpkt(), d->n_total, d->l_unit, d->packets_done);
}

template <class R>
mcrt_status trace_impl(mcrt_disk* d, int which) {
  RayState* rs = d->rays;
  const size_t nc = (size_t)d->nr * d->nt;
  const int nlam = d->nlam;
  const bool scat = (which & MCRT_WITH_SCATTERING) != 0;
  const double* T = (which & ~MCRT_WITH_SCATTERING) == MCRT_T_PDA ? d->T_pda.as<double>() : d->T_mc.as<double>();
  const int prec = sizeof(R) == 8 ? 64 : 32;
  if (rs->S_epoch != d->T_epoch || rs->S_which != which || rs->S_prec != prec || !rs->S.p) {
    if (rs->S.n < nc * nlam * sizeof(R)) CK(rs->S.alloc(nc * nlam * sizeof(R)), "cudaMalloc");
    const int blocks = (int)((nc * 32 + 255) / 256);
    k_source<R><<<blocks, 256, 0, d->stream>>>((int)nc, nlam, T, d->lam_e_d.as<double>(), d->kabs_d.as<double>(),
                                               d->chi64.as<double>(), rs->S.as<R>(),
                                               scat ? d->jlen.as<double>() : nullptr, j_factor(d),
                                               d->alb64.as<double>(), d->rf64.as<double>(), d->cf64.as<double>(),
                                               d->nt);
    d->launches++;
    CK(cudaGetLastError(), "source kernel");
    rs->S_epoch = d->T_epoch;
    rs->S_which = which;
    rs->S_prec = prec;
  }
  const size_t img_bytes = (size_t)rs->n * nlam * sizeof(R);
  if (rs->img.n < img_bytes) CK(rs->img.alloc(img_bytes), "cudaMalloc");
  CK(cudaMemsetAsync(rs->cnt.p, 0, 2 * sizeof(unsigned long long), d->stream), "memset");
  const int sms = sm_count(d->device);
  if ((size_t)(d->nt + 1) * sizeof(FaceCoef<R>) + (size_t)nlam * sizeof(R) > kRayFaces)
    return set_error(d, MCRT_EINVAL, "too many polar cells for the ray-tracing face table");
  CK(launch_trace<R>(d, rs, model_of<R>(d), chi_of<R>(d), sms), "ray-trace kernel");
  d->launches++;
  rs->img_prec = prec;
  rs->have_img = true;
  // star, then the SED from the image
  int it = 0;
  while (it + 1 < d->nt && d->tf[it + 1] <= rs->incl) ++it;
  const int nblk = (int)std::min<long long>(rs->n, (long long)sms * 4);
  const long long per_blk = (rs->n + nblk - 1) / nblk;
  if (rs->part.n < (size_t)nblk * nlam * 8) CK(rs->part.alloc((size_t)nblk * nlam * 8), "cudaMalloc");
  k_sed_part<R><<<nblk, kSedBlock, 0, d->stream>>>(rs->n, nlam, per_blk, rs->img.as<R>(), rs->w.as<double>(),
                                                  rs->part.as<double>());
  k_sed_final<<<nlam, kSedBlock, 0, d->stream>>>(d->nr, d->nt, it, nlam, d->rho64.as<double>(), d->rf64.as<double>(),
                                                 d->lam_e_d.as<double>(), d->chi64.as<double>(), d->Tstar, d->Rstar,
                                                 rs->dist, nblk, rs->part.as<double>(), rs->Fs.as<double>(),
                                                 rs->F.as<double>());
  d->launches += 2;
  CK(cudaGetLastError(), "SED kernels");
  return MCRT_OK;
}

}  // namespace

extern "C" {

mcrt_status mcrt_set_rays(mcrt_disk* d, double incl_rad, double dist_cm, int64_t n, const double* p_cm,
                          const double* q_cm, const double* w_cm2) {
  if (!d) return set_error(nullptr, MCRT_EINVAL, "disk is NULL");
  if (!d->has_opacity) return set_error(d, MCRT_ESTATE, "mcrt_set_opacity must come first");
  if (!(incl_rad >= 0.0 && incl_rad <= 3.14159265358979323846))
    return set_error(d, MCRT_EINVAL, "inclination must lie in [0, pi]");
  if (!(dist_cm > 0.0) || !std::isfinite(dist_cm)) return set_error(d, MCRT_EINVAL, "distance must be > 0");
  if (n < 1 || n > (int64_t)1 << 27) return set_error(d, MCRT_EINVAL, "rays: 1 .. 2^27");
  if (!p_cm || !q_cm || !w_cm2) return set_error(d, MCRT_EINVAL, "p, q, w must not be NULL");
  if (d->nlam > 256) return set_error(d, MCRT_EINVAL, "ray tracing takes at most 256 wavelength bins");
  for (int64_t k = 0; k < n; ++k)
    if (!std::isfinite(p_cm[k]) || !std::isfinite(q_cm[k]) || !(w_cm2[k] >= 0.0) || !std::isfinite(w_cm2[k]))
      return set_error(d, MCRT_EINVAL, "rays: p, q finite and w >= 0");
  CK(cudaSetDevice(d->device), "cudaSetDevice");
  if (!d->rays) d->rays = new RayState();
  RayState* rs = d->rays;
  const size_t bytes = (size_t)n * 8;
  if (rs->p.n < bytes) CK(rs->p.alloc(bytes), "cudaMalloc");
  if (rs->q.n < bytes) CK(rs->q.alloc(bytes), "cudaMalloc");
  if (rs->w.n < bytes) CK(rs->w.alloc(bytes), "cudaMalloc");
  if (!rs->F.p) CK(rs->F.alloc(256 * 8), "cudaMalloc");
  if (!rs->Fs.p) CK(rs->Fs.alloc(256 * 8), "cudaMalloc");
  if (!rs->cnt.p) CK(rs->cnt.alloc(2 * 8), "cudaMalloc");
  // Morton order of the sky positions (16 bits per axis over the square of side 2 r_out): consecutive
  // threads take neighbouring rays, whose paths cross the same cells
  std::vector<std::pair<uint32_t, int>> key((size_t)n);
  const double rmax = d->rf[d->nr];
  for (int64_t k = 0; k < n; ++k) {
    auto quant = [&](double x) {
      const double t = std::min(std::max((x / rmax + 1.0) * 0.5, 0.0), 1.0);
      return (uint32_t)std::min(65535.0, std::floor(t * 65536.0));
    };
    uint32_t x = quant(p_cm[k]), y = quant(q_cm[k]), m = 0;
    for (int bit = 0; bit < 16; ++bit) m |= ((x >> bit) & 1u) << (2 * bit) | ((y >> bit) & 1u) << (2 * bit + 1);
    key[(size_t)k] = {m, (int)k};
  }
  std::stable_sort(key.begin(), key.end(), [](const auto& u, const auto& v) { return u.first < v.first; });
  std::vector<int> order((size_t)n);
  for (int64_t k = 0; k < n; ++k) order[(size_t)k] = key[(size_t)k].second;
  if (rs->order.n < (size_t)n * 4) CK(rs->order.alloc((size_t)n * 4), "cudaMalloc");
  CK(cudaMemcpyAsync(rs->order.p, order.data(), (size_t)n * 4, cudaMemcpyHostToDevice, d->stream), "copy");
  CK(cudaMemcpyAsync(rs->p.p, p_cm, bytes, cudaMemcpyHostToDevice, d->stream), "copy");
  CK(cudaMemcpyAsync(rs->q.p, q_cm, bytes, cudaMemcpyHostToDevice, d->stream), "copy");
  CK(cudaMemcpyAsync(rs->w.p, w_cm2, bytes, cudaMemcpyHostToDevice, d->stream), "copy");
  CK(cudaStreamSynchronize(d->stream), "synchronize");
  rs->n = n;
  rs->incl = incl_rad;
  rs->dist = dist_cm;
  rs->have_img = false;
  return MCRT_OK;
}

mcrt_status mcrt_mean_intensity(mcrt_disk* d, double* J_out) {
  if (!d) return set_error(nullptr, MCRT_EINVAL, "disk is NULL");
  if (!J_out) return set_error(d, MCRT_EINVAL, "J_out must not be NULL");
  if (!d->keep_j) return set_error(d, MCRT_ESTATE, "mcrt_keep_mean_intensity must come first");
  CK(cudaSetDevice(d->device), "cudaSetDevice");
  const size_t nc = (size_t)d->nr * d->nt, n = nc * d->nlam;
  DBuf J;
  CK(J.alloc(n * 8), "cudaMalloc");
  const int blocks = (int)std::min<size_t>((n + 255) / 256, (size_t)sm_count(d->device) * 8);
  k_mean_intensity<<<blocks, 256, 0, d->stream>>>((int)nc, d->nt, d->nlam, d->rf64.as<double>(), d->cf64.as<double>(),
                                                  d->jlen.as<double>(), j_factor(d), J.as<double>());
  d->launches++;
  CK(cudaGetLastError(), "mean-intensity kernel");
  CK(cudaMemcpyAsync(J_out, J.p, n * 8, cudaMemcpyDeviceToHost, d->stream), "copy");
  CK(cudaStreamSynchronize(d->stream), "synchronize");
  return MCRT_OK;
}

mcrt_status mcrt_raytrace(mcrt_disk* d, int which, int precision, double* F_out, double* F_star_out, double* I_out,
                          uint64_t* n_segments) {
  if (!d) return set_error(nullptr, MCRT_EINVAL, "disk is NULL");
  if (!d->rays || d->rays->n < 1) return set_error(d, MCRT_ESTATE, "mcrt_set_rays must come first");
  const int base = which & ~MCRT_WITH_SCATTERING;
  if (base != MCRT_T_MC && base != MCRT_T_PDA) return set_error(d, MCRT_EINVAL, "which");
  if (precision != 0 && precision != 32 && precision != 64) return set_error(d, MCRT_EINVAL, "precision: 32 or 64");
  if (base == MCRT_T_PDA && !d->have_pda) return set_error(d, MCRT_ESTATE, "no PDA solution");
  if ((which & MCRT_WITH_SCATTERING) && !d->keep_j)
    return set_error(d, MCRT_ESTATE, "scattered light needs the mean-intensity tally (mcrt_keep_mean_intensity)");
  if (d->nlam > 256) return set_error(d, MCRT_EINVAL, "ray tracing takes at most 256 wavelength bins");
  CK(cudaSetDevice(d->device), "cudaSetDevice");
  if (!d->have_T) {
    mcrt_status s = compute_temperatures(d);
    if (s != MCRT_OK) return s;
  }
  RayState* rs = d->rays;
  mcrt_status s = precision == 64 ? trace_impl<double>(d, which) : trace_impl<float>(d, which);
  if (s != MCRT_OK) return s;
  unsigned long long c[2];
  CK(cudaMemcpyAsync(c, rs->cnt.p, sizeof(c), cudaMemcpyDeviceToHost, d->stream), "copy");
  if (F_out) CK(cudaMemcpyAsync(F_out, rs->F.p, (size_t)d->nlam * 8, cudaMemcpyDeviceToHost, d->stream), "copy");
  if (F_star_out)
    CK(cudaMemcpyAsync(F_star_out, rs->Fs.p, (size_t)d->nlam * 8, cudaMemcpyDeviceToHost, d->stream), "copy");
  CK(cudaStreamSynchronize(d->stream), "synchronize");
  if (I_out) {
    const size_t m = (size_t)rs->n * d->nlam;
    if (rs->img_prec == 64) {
      CK(cudaMemcpy(I_out, rs->img.p, m * 8, cudaMemcpyDeviceToHost), "copy");
    } else {
      std::vector<float> tmp(m);
      CK(cudaMemcpy(tmp.data(), rs->img.p, m * 4, cudaMemcpyDeviceToHost), "copy");
      for (size_t k = 0; k < m; ++k) I_out[k] = tmp[k];
    }
  }
  if (n_segments) *n_segments = c[0];
  if (c[1]) return set_error(d, MCRT_ETIMEOUT, "a ray took more than 4 (nr + ntheta) + 64 events");
  return MCRT_OK;
}

mcrt_status mcrt_visibilities(mcrt_disk* d, int n_vis, const int* bins, const double* baseline_cm,
                              const double* pa_rad, int with_star, double* vis_out) {
  if (!d) return set_error(nullptr, MCRT_EINVAL, "disk is NULL");
  if (!d->rays || !d->rays->have_img) return set_error(d, MCRT_ESTATE, "mcrt_raytrace must come first");
  if (n_vis < 1 || n_vis > (1 << 20) || !bins || !baseline_cm || !pa_rad || !vis_out)
    return set_error(d, MCRT_EINVAL, "bad arguments");
  RayState* rs = d->rays;
  std::vector<double> par((size_t)3 * n_vis);
  for (int j = 0; j < n_vis; ++j) {
    if (bins[j] < 0 || bins[j] >= d->nlam) return set_error(d, MCRT_EINVAL, "bin out of range");
    if (!(baseline_cm[j] >= 0.0) || !std::isfinite(baseline_cm[j]) || !std::isfinite(pa_rad[j]))
      return set_error(d, MCRT_EINVAL, "baselines: finite, >= 0");
    // bin centre lambda = sqrt(lambda_lo lambda_hi); frequency over distance in cycles per cm at the source
    const double lam_cm = std::sqrt(d->lam_e[bins[j]] * d->lam_e[bins[j] + 1]) * 1e-4;
    const double f = baseline_cm[j] / (lam_cm * rs->dist);
    par[3 * j] = bins[j];
    par[3 * j + 1] = f * std::cos(pa_rad[j]);
    par[3 * j + 2] = f * std::sin(pa_rad[j]);
  }
  CK(cudaSetDevice(d->device), "cudaSetDevice");
  if (rs->vis_par.n < par.size() * 8) CK(rs->vis_par.alloc(par.size() * 8), "cudaMalloc");
  // blocks per visibility: four per SM in all, at least 256 rays each
  const long long most = std::min<long long>((rs->n + 255) / 256, (long long)sm_count(d->device) * 4 / n_vis);
  const int parts = (int)std::max<long long>(most, 1);
  const size_t out_bytes = (size_t)n_vis * 8, part_bytes = (size_t)n_vis * parts * 24;
  if (rs->vis_out.n < out_bytes + part_bytes) CK(rs->vis_out.alloc(out_bytes + part_bytes), "cudaMalloc");
  double* part = rs->vis_out.as<double>() + n_vis;
  CK(cudaMemcpyAsync(rs->vis_par.p, par.data(), par.size() * 8, cudaMemcpyHostToDevice, d->stream), "copy");
  const dim3 grid((unsigned)n_vis, (unsigned)parts);
  if (rs->img_prec == 64)
    k_vis_part<double><<<grid, 256, 0, d->stream>>>(rs->n, d->nlam, rs->img.as<double>(), rs->p.as<double>(),
                                                    rs->q.as<double>(), rs->w.as<double>(), rs->vis_par.as<double>(), part);
  else
    k_vis_part<float><<<grid, 256, 0, d->stream>>>(rs->n, d->nlam, rs->img.as<float>(), rs->p.as<double>(),
                                                   rs->q.as<double>(), rs->w.as<double>(), rs->vis_par.as<double>(), part);
  k_vis<<<(n_vis + 3) / 4, 128, 0, d->stream>>>(n_vis, parts, part, rs->vis_par.as<double>(), rs->Fs.as<double>(),
                                                    with_star, 1.0 / (rs->dist * rs->dist), rs->vis_out.as<double>());
  d->launches += 2;
  CK(cudaGetLastError(), "visibility kernel");
  CK(cudaMemcpyAsync(vis_out, rs->vis_out.p, (size_t)n_vis * 8, cudaMemcpyDeviceToHost, d->stream), "copy");
  CK(cudaStreamSynchronize(d->stream), "synchronize");
  return MCRT_OK;
}

}  // extern "C"
