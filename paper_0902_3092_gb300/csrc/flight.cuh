// flight.cuh -- a packet's straight flight through many cells at once, its 32 lanes each taking one of the
// next cells (FP32, one packet per warp).
//
// What bounds a packet that has a warp to itself is the latency of its serial chain, and most of its steps
// are face crossings (107 of 115 per packet on the 100x60 non-gray disk of midplane optical depth 1e5):
// one crossing after another costs four dependent face distances, a density load and a compare each,
// 0.8 us. But along a straight line the crossings need no order: lane k computes the k-th next crossing of
// the spheres (inward ones while the ray approaches the star, then outward ones) and the k-th next crossing
// of the cones (on the side the polar angle moves to, then back after its one turning point), both in
// closed form from the flight's start. The two sorted lists are merged by rank (each lane finds its place
// on the merge path in five steps of two shuffles), so lane m knows the m-th cell of the flight, loads its
// density, and a prefix sum of the optical depths tells where the flight ends: about the latency of two
// crossings for up to 32 of them.
//
// Host and device code (the per-lane functions); the tests run it lane by lane on the CPU.
#pragma once
#include "common.cuh"

namespace mcrt {

// One ray from point p (cell ir, it; ir = -1: the inner cavity) along the unit vector u.
struct RayCuts {
  float b, r2;           // p.u, |p|^2
  float w2, wz2, d2;     // squares of the horizontal and vertical parts of p x u, their sum: the squared impact parameter
  float px, py, pz, ux, uy, uz;
  float se;              // where the polar angle turns (infinity: not ahead)
  float mu1, mu2;        // cos(theta) that the ray reaches before and after the turn
  int ir, it;
  bool down;             // the polar angle falls first
};

__host__ __device__ __forceinline__ RayCuts ray_cuts(int ir, int it, float px, float py, float pz, float ux, float uy,
                                                     float uz) {
  RayCuts q;
  q.ir = ir;
  q.it = it;
  q.px = px;
  q.py = py;
  q.pz = pz;
  q.ux = ux;
  q.uy = uy;
  q.uz = uz;
  q.b = px * ux + py * uy + pz * uz;
  q.r2 = px * px + py * py + pz * pz;
  // p x u: |.|^2 is the impact parameter's square without the cancellation of r^2 - b^2
  const float wx = py * uz - pz * uy, wy = pz * ux - px * uz, wz = px * uy - py * ux;
  q.w2 = wx * wx + wy * wy;
  q.wz2 = wz * wz;
  q.d2 = q.w2 + q.wz2;
  // d cos(theta)/ds has the sign of g0 + g1 s: one turning point. (g0 and g1 from the same p x u: on a
  // radial ray, where it is rounding noise, they agree in sign and the angle does not turn)
  const float g0 = wx * py - wy * px, g1 = wx * uy - wy * ux;
  q.down = g0 > 0.f || (g0 == 0.f && g1 > 0.f);
  const bool turns = q.d2 > 0.f && ((g0 > 0.f && g1 < 0.f) || (g0 < 0.f && g1 > 0.f));
  q.se = turns ? -g0 / g1 : inf_<float>();
  const float m = sqrtf(q.w2 / q.d2);  // |cos theta| where the great circle of the ray turns
  q.mu2 = uz;
  q.mu1 = turns ? (q.down ? m : -m) : uz;
  return q;
}

// Square of half the chord inside sphere f: b^2 - (r^2 - r_f^2) as sphere_near and sphere_far form it (in the
// rim the mean free path is a few roundings of the position, and this form's landing error on a face is
// the rounding of r^2 alone), and r_f^2 minus the impact parameter's square for a sphere far below, where the
// first form cancels.
__host__ __device__ __forceinline__ float half_chord2(const DevModel<float>& M, const RayCuts& q, int f) {
  const float rf2 = M.rf2[f];
  return 4.f * rf2 < q.r2 ? rf2 - q.d2 : q.b * q.b - (q.r2 - rf2);
}

// The k-th next inward sphere crossing exists (face ir - k, hit before the closest approach).
__host__ __device__ __forceinline__ bool inner_hit(const DevModel<float>& M, const RayCuts& q, int k) {
  const int f = q.ir - k;
  return f >= 0 && q.b < 0.f && half_chord2(M, q, f) > 0.f;
}

// Inward crossings beyond the first count only down to a quarter of the start's radius: the position's
// rounding (6e-8 of it) stays far below the cells there, and the next pass starts closer.
__host__ __device__ __forceinline__ bool inner_precise(const DevModel<float>& M, const RayCuts& q, int k) {
  return k == 0 || 16.f * M.rf2[q.ir - k] >= q.r2;
}

// Face of the k-th sphere crossing, n_in of them inward
__host__ __device__ __forceinline__ int sphere_face(const RayCuts& q, int n_in, int k) {
  return k < n_in ? q.ir - k : q.ir - n_in + 1 + (k - n_in);
}

// Path length to the k-th sphere crossing, n_in of them inward (infinity past the outer radius).
__host__ __device__ __forceinline__ float sphere_cut(const DevModel<float>& M, const RayCuts& q, int n_in, int k) {
  const bool inward = k < n_in;
  const int f = sphere_face(q, n_in, k);
  if (f > M.nr) return inf_<float>();
  // s = -b -+ h without cancellation: near a face its distance comes from r^2 - r_f^2
  const float h = sqrtf(fmaxf(half_chord2(M, q, f), 0.f));
  const float c = q.r2 - M.rf2[f];
  const float s = inward ? c / (h - q.b) : (q.b > 0.f ? -c / (h + q.b) : h - q.b);
  return fmaxf(s, 0.f);
}

// cos(theta) of a polar face (the midplane's exactly 0, so a ray in a plane z = const never reaches it)
__host__ __device__ __forceinline__ float face_mu(const DevModel<float>& M, int f) {
  return M.fk[f] == 0 ? 0.f : M.cf[f];
}

// Face of the k-th cone crossing, n1 of them before the turn
__host__ __device__ __forceinline__ int cone_face(const RayCuts& q, int n1, int k) {
  if (k < n1) return q.down ? q.it - k : q.it + 1 + k;
  return q.down ? q.it - n1 + 1 + (k - n1) : q.it + n1 - (k - n1);
}

// The k-th cone crossing before the turn exists.
__host__ __device__ __forceinline__ bool cone_hit(const DevModel<float>& M, const RayCuts& q, int k) {
  const int f = cone_face(q, 32, k);
  return f >= 1 && f < M.nt && (q.down ? face_mu(M, f) < q.mu1 : face_mu(M, f) > q.mu1);
}

// Quarter of the discriminant of A s^2 + 2 B s + C, B^2 - A C = cos^2 (sin^2 (p x u)_h^2 - cos^2 (p x u)_z^2): the
// same at every point of the ray, and without the cancellation of the two products (the two roots of a
// cone next to the midplane lie within 1e-3 of each other)
__host__ __device__ __forceinline__ float cone_disc(const RayCuts& q, float cc, float ss) {
  return fmaxf(cc * (ss * q.w2 - cc * q.wz2), 0.f);
}

// Whether the ray crosses any cone (none before the turn, but perhaps some after it)
__host__ __device__ __forceinline__ bool meets_cones(const RayCuts& q, int n1) { return n1 > 0 || q.se < inf_<float>(); }

// Path length to the k-th cone crossing, n1 of them before the turn (infinity: there is none).
__host__ __device__ __forceinline__ float cone_cut(const DevModel<float>& M, const RayCuts& q, int n1, int k) {
  const bool back = k >= n1;
  bool down = q.down;
  const int f = cone_face(q, n1, k);
  if (back) {
    if (!(q.se < inf_<float>())) return inf_<float>();
    down = !down;
    if (f < 1 || f >= M.nt || !(down ? face_mu(M, f) < q.mu2 : face_mu(M, f) > q.mu2)) return inf_<float>();
  }
  float s;
  const int kind = M.fk[f];
  if (kind == 0) {
    s = -q.pz / q.uz;
  } else {
    // the root where the ray crosses the cone in its direction of motion (as cone_exit)
    const float sig = (float)kind, cc = M.c2[f], ss = M.s2[f];
    const float A = sig * (cc * (q.ux * q.ux + q.uy * q.uy) - ss * q.uz * q.uz);
    const float B = sig * (cc * (q.px * q.ux + q.py * q.uy) - ss * q.pz * q.uz);
    const float C = sig * (cc * (q.px * q.px + q.py * q.py) - ss * q.pz * q.pz);
    const float h = -(B + copysignf(sqrtf(cone_disc(q, cc, ss)), B));
    s = down == !signbit(B) ? h / A : C / h;
  }
  // (fmin / fmax drop a NaN: a ray along the face turns there)
  s = back ? fmaxf(s, q.se) : fminf(s, q.se);
  return fmaxf(s, 0.f);
}

// Cell after i sphere and j cone crossings.
__host__ __device__ __forceinline__ void cut_cell(const RayCuts& q, int n_in, int n1, int i, int j, int& ir, int& it) {
  ir = i <= n_in ? q.ir - i : q.ir - n_in + (i - n_in);
  const int net = j <= n1 ? j : n1 - (j - n1);
  it = q.down ? q.it - net : q.it + net;
}

// The point where the ray enters the cell after i sphere and j cone crossings, the last of them at path
// length s: p + s u carries the rounding of s (6e-8 of a path that may be many times the radius there, against
// mean free paths of 1e-6 of the radius in the rim), so the face's own root near that point corrects it. Returns
// the correction, a path length in the cell before.
__host__ __device__ __forceinline__ float entry_point(const DevModel<float>& M, const RayCuts& q, int n_in, int n1, int i,
                                                      int j, bool radial, float s, float& x, float& y, float& z) {
  x = q.px + s * q.ux;
  y = q.py + s * q.uy;
  z = q.pz + s * q.uz;
  // (a lane past the flight's last crossing, s infinite, has no face: its number lies outside the tables)
  if (i + j == 0 || !(s < inf_<float>())) return 0.f;
  float d;
  if (radial) {
    const float c = x * x + y * y + z * z - M.rf2[sphere_face(q, n_in, i - 1)], b = x * q.ux + y * q.uy + z * q.uz;
    const float h = sqrtf(fmaxf(b * b - c, 0.f));
    d = i <= n_in ? c / (h - b) : -c / (h + b);
  } else {
    const int f = cone_face(q, n1, j - 1);
    if (M.fk[f] == 0) {
      d = -z / q.uz;
    } else {
      const float cc = M.c2[f], ss = M.s2[f];
      const float B = cc * (x * q.ux + y * q.uy) - ss * z * q.uz, C = cc * (x * x + y * y) - ss * z * z;
      d = -C / (B + copysignf(sqrtf(cone_disc(q, cc, ss)), B));  // (not taken where it is no number)
    }
  }
  // a correction beyond the roundings' size is a grazing root's: not taken
  if (!(fabsf(d) <= 4e-6f * (sqrtf(q.r2) + s))) return 0.f;
  x += d * q.ux;
  y += d * q.uy;
  z += d * q.uz;
  return d;
}

}  // namespace mcrt
