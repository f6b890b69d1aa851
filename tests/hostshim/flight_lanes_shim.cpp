// Host build of what every lane of a flight's pass evaluates (flight.cuh), also the lanes past the flight's
// end: with face tables that lie between two pads, so that a read outside of them shows in the results.
#include "cuda_host_stubs.h"
#include "tables.h"
#include "flight.cuh"

using namespace mcrt;

// out: per ray and lane the entry point, the correction to it and the path length there
extern "C" void host_flight_lanes(int nr, int nt, const double* rf_cm, const double* tf, int n, const float* p,
                                  const float* u, const int* cell0, float pad, int pad_kind, float* out) {
  constexpr int kPad = 64;
  GeomArrays g;
  geometry_arrays(nr, nt, rf_cm, tf, g);
  auto padded = [&](const std::vector<double>& v) {
    std::vector<float> t(v.size() + 2 * kPad, pad);
    for (size_t k = 0; k < v.size(); ++k) t[kPad + k] = (float)v[k];
    return t;
  };
  const std::vector<float> rf = padded(g.rf), rf2 = padded(g.rf2), c2 = padded(g.c2), s2 = padded(g.s2),
                           cf = padded(g.cf), sf = padded(g.sf);
  std::vector<signed char> fk(g.fk.size() + 2 * kPad, (signed char)pad_kind);
  for (size_t k = 0; k < g.fk.size(); ++k) fk[kPad + k] = g.fk[k];
  DevModel<float> M;
  std::memset(&M, 0, sizeof(M));
  M.nr = nr;
  M.nt = nt;
  M.rf = rf.data() + kPad;
  M.rf2 = rf2.data() + kPad;
  M.c2 = c2.data() + kPad;
  M.s2 = s2.data() + kPad;
  M.cf = cf.data() + kPad;
  M.sf = sf.data() + kPad;
  M.fk = fk.data() + kPad;
  for (int r = 0; r < n; ++r) {
    const RayCuts q = ray_cuts(cell0[2 * r], cell0[2 * r + 1], p[3 * r], p[3 * r + 1], p[3 * r + 2], u[3 * r],
                               u[3 * r + 1], u[3 * r + 2]);
    int n_in = 0, n1 = 0;
    for (int k = 0; k < 32; ++k) {
      n_in += inner_hit(M, q, k);
      n1 += cone_hit(M, q, k);
    }
    float sr[32], st[32];
    const bool cones = meets_cones(q, n1);
    for (int k = 0; k < 32; ++k) {
      sr[k] = sphere_cut(M, q, n_in, k);
      st[k] = cones ? cone_cut(M, q, n1, k) : inf_<float>();
    }
    for (int m = 0; m < 32; ++m) {
      int i = cones ? 0 : m, hi = m;  // the lane's place on the merge path
      while (i < hi) {
        const int mid = (i + hi) >> 1;
        if (sr[mid] < st[m - 1 - mid]) i = mid + 1;
        else hi = mid;
      }
      const int j = m - i;
      const float a = i > 0 ? sr[i - 1] : 0.f, c = j > 0 ? st[j - 1] : 0.f;
      float* o = out + ((size_t)r * 32 + m) * 5;
      o[3] = entry_point(M, q, n_in, n1, i, j, j == 0 || (i > 0 && a >= c), std::fmax(a, c), o[0], o[1], o[2]);
      o[4] = std::fmax(a, c);
    }
  }
}
