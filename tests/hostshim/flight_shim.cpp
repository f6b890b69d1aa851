// Host build of a packet's flight through 32 cells at a time (flight.cuh), the warp's lanes run one after
// another: path length and entries per cell of straight rays through the grid.
#include "cuda_host_stubs.h"
#include "tables.h"
#include "flight.cuh"

using namespace mcrt;

namespace {

struct Grid {
  std::vector<float> rf, rf2, c2, s2, cf, sf;
  GeomArrays g;
  DevModel<float> M;
  Grid(int nr, int nt, const double* rf_cm, const double* tf) {
    geometry_arrays(nr, nt, rf_cm, tf, g);
    auto f32 = [](const std::vector<double>& v) { return std::vector<float>(v.begin(), v.end()); };
    rf = f32(g.rf);
    rf2 = f32(g.rf2);
    c2 = f32(g.c2);
    s2 = f32(g.s2);
    cf = f32(g.cf);
    sf = f32(g.sf);
    std::memset(&M, 0, sizeof(M));
    M.nr = nr;
    M.nt = nt;
    M.rf = rf.data();
    M.rf2 = rf2.data();
    M.c2 = c2.data();
    M.s2 = s2.data();
    M.cf = cf.data();
    M.sf = sf.data();
    M.fk = g.fk.data();
  }
};

}  // namespace

extern "C" int host_flights(int nr, int nt, const double* rf_cm, const double* tf, int n, const float* p, const float* u,
                            const int* cell0, double* len, long long* entries, int* passes, double* off) {
  // off: how far a pass's end lies outside the cell it was given (internal units, over the position's radius)
  const Grid grid(nr, nt, rf_cm, tf);
  const DevModel<float>& M = grid.M;
  for (int r = 0; r < n; ++r) {
    float x = p[3 * r], y = p[3 * r + 1], z = p[3 * r + 2];
    const float ux = u[3 * r], uy = u[3 * r + 1], uz = u[3 * r + 2];
    int ir = cell0[2 * r], it = cell0[2 * r + 1];
    double* L = len + (size_t)r * nr * nt;
    long long* E = entries + (size_t)r * nr * nt;
    passes[r] = 0;
    while (ir < nr) {
      if (++passes[r] > 4 * (nr + nt)) return 1 + r;
      const RayCuts q = ray_cuts(ir, it, x, y, z, ux, uy, uz);
      int n_in = 0, n_ok = 32, n1 = 0;
      for (int k = 0; k < 32; ++k) n_in += inner_hit(M, q, k);
      for (int k = n_in - 1; k >= 0; --k)
        if (!inner_precise(M, q, k)) n_ok = k;
      for (int k = 0; k < 32; ++k) n1 += cone_hit(M, q, k);
      for (int k = 0; k < n_in; ++k)
        if (!inner_hit(M, q, k)) return -1 - r;  // (a lane's crossings are consecutive)
      for (int k = 0; k < n1; ++k)
        if (!cone_hit(M, q, k)) return -1 - r;
      float sr[32], st[32];
      for (int k = 0; k < 32; ++k) {
        sr[k] = sphere_cut(M, q, n_in, k);
        st[k] = meets_cones(q, n1) ? cone_cut(M, q, n1, k) : inf_<float>();
      }
      int lr = -1, lt = 0;  // the pass's last cell
      for (int m = 0;; ++m) {
        int i = 0, hi = m;  // the lane's place on the merge path
        while (i < hi) {
          const int mid = (i + hi) >> 1;
          if (sr[mid] < st[m - 1 - mid]) i = mid + 1;
          else hi = mid;
        }
        const int j = m - i;
        const float a = i > 0 ? sr[i - 1] : 0.f, c = j > 0 ? st[j - 1] : 0.f;
        const bool radial = j == 0 || (i > 0 && a >= c);
        const float start = std::fmax(a, c), end = std::fmin(sr[i], st[j]);
        int cr, ct;
        cut_cell(q, n_in, n1, i, j, cr, ct);
        if (ct < 0 || ct >= nt || cr < -1) return -1 - r;
        if (m > 0 && cr >= 0 && cr < nr) E[(size_t)cr * nt + ct]++;
        if (cr >= nr || i >= n_ok || m == 31) {  // the pass ends here
          ir = cr;
          it = ct;
          const float d = entry_point(M, q, n_in, n1, i, j, radial, start, x, y, z);
          if (m > 0 && lr >= 0) L[(size_t)lr * nt + lt] += d;
          break;
        }
        if (cr >= 0) L[(size_t)cr * nt + ct] += std::fmax(end - start, 0.f);
        lr = cr;
        lt = ct;
      }
      if (ir >= 0 && ir < nr) {
        const double X = x, Y = y, Z = z, rc = std::sqrt(X * X + Y * Y), rr = std::sqrt(rc * rc + Z * Z);
        double o = std::fmax(M.rf[ir] - rr, rr - M.rf[ir + 1]);
        if (it > 0) o = std::fmax(o, (double)M.sf[it] * Z - (double)M.cf[it] * rc);
        if (it + 1 < nt) o = std::fmax(o, (double)M.cf[it + 1] * rc - (double)M.sf[it + 1] * Z);
        off[r] = std::fmax(off[r], o / rr);
      }
    }
  }
  return 0;
}
