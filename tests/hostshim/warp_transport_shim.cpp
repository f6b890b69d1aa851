// Host build of the transport with one packet per warp (transport.cuh: launch_packet and run_packet_warp by 32
// lanes), FP32, packets one after another, over a model built by the library's own host builders (tables.h).
#include "warp_host_stubs.h"
#include "tables.h"
#include "transport.cuh"

using namespace mcrt;

namespace {

std::vector<float> f32(const std::vector<double>& v) { return std::vector<float>(v.begin(), v.end()); }

template <bool POL, bool JT, bool FLY>
bool run_packets(const KParams<float>& P, const DevModel<float>* M, uint64_t n, Acc& acc) {
  for (uint64_t k = 0; k < n; ++k) {
    const bool ok = host_warp.run([&](int lane) {
      Acc mine;
      std::memset(&mine, 0, sizeof(mine));
      Pkt<float> s;
      std::memset(&s, 0, sizeof(s));
      WarpRng rng{{(uint32_t)P.seed, (uint32_t)(P.seed >> 32)}, 0u - 32u, make_uint4(0u, 0u, 0u, 0u)};
      launch_packet<float, false, false, POL, JT>(P, rng, M[lane], s, k, -1, mine);
      run_packet_warp<float, false, POL, JT, FLY>(P, rng, M[lane], s, mine);
      if (lane == 0) {
        acc.packets += mine.packets;
        acc.abs += mine.abs;
        acc.sca += mine.sca;
        acc.cross += mine.cross;
        acc.mrw += mine.mrw;
        acc.capped += mine.capped;
        acc.escaped += mine.escaped;
        acc.err |= mine.err;
      }
    });
    if (!ok) return false;
  }
  return true;
}

}  // namespace

// Packets 0 .. n-1 (cgs inputs, as mcrt_disk_create and mcrt_set_opacity take them), polarized with a Mueller
// matrix [nlam][4][nmu], with internal sources Lsrc per cell, with path lengths when jlen is given (each may be NULL). late:
// NULL, or the tallies that the loads of lanes 1 .. 31 find in place of lane 0's. 0, or 1 if the lanes of a packet parted.
extern "C" int host_warp_transport(int nr, int nt, const double* rf_cm, const double* tf, const double* rho_in, int nlam,
                                   const double* lam_e, const double* kabs, const double* ksca, const double* g,
                                   double Tstar, double Rstar, uint64_t n, uint64_t seed, int mrw, double gamma, int nmin,
                                   int exit_dir, int nmu, const double* mueller, const double* Lsrc, uint64_t* late,
                                   uint64_t* tally, uint64_t* visits, uint64_t* nabs, uint64_t* sed, double* jlen,
                                   uint64_t* counters) {
  GeomArrays geo;
  geometry_arrays(nr, nt, rf_cm, tf, geo);
  DensityArrays den;
  density_arrays(nr, nt, rf_cm, tf, rho_in, den);
  DustArrays dust;
  dust_arrays(nlam, lam_e, kabs, ksca, g, Tstar, dust);
  const int nT = 1024;
  TGridTables tt;
  build_T_tables(nlam, lam_e, kabs, dust.chip.data(), nT, 1.0, std::max(1e4, 2.0 * Tstar), tt);
  std::vector<float> mtab(2 * kMrwTab);
  build_mrw_table(mtab.data());
  bool gray = true;
  for (int b = 1; b < nlam; ++b)
    if (kabs[b] != kabs[0] || ksca[b] != ksca[0] || g[b] != g[0]) gray = false;
  std::vector<unsigned long long> cnt(C_NCNT, 0ull);
  const size_t ncell = (size_t)nr * nt;
  std::vector<double> src_cum(ncell + 1, 0.0), mc;
  if (Lsrc)
    for (size_t c = 0; c < ncell; ++c) src_cum[c + 1] = src_cum[c] + Lsrc[c];
  const double Ls = src_cum[ncell], Lstar = 4.0 * kPi * Rstar * Rstar * MCRT_SIGMA * std::pow(Tstar, 4);
  std::vector<float> mt;
  if (mueller) {
    mt.assign(mueller, mueller + (size_t)nlam * 4 * nmu);
    mc.resize((size_t)nlam * nmu);
    for (int b = 0; b < nlam; ++b) mueller_cdf(mueller + (size_t)b * 4 * nmu, nmu, mc.data() + (size_t)b * nmu);
  }
  const std::vector<float> rf = f32(geo.rf), rf2 = f32(geo.rf2), c2 = f32(geo.c2), s2 = f32(geo.s2), cf = f32(geo.cf),
                           sf = f32(geo.sf), rho = f32(den.rhol), chi = f32(dust.chi), alb = f32(dust.alb),
                           gq(g, g + nlam), star = f32(dust.star), mcf = f32(mc);
  std::vector<uint64_t> sq((size_t)nlam * kNInc), su((size_t)nlam * kNInc);
  DevModel<float> M;
  std::memset(&M, 0, sizeof(M));
  M.nr = nr;
  M.nt = nt;
  M.nlam = nlam;
  M.nT = nT;
  M.gray = gray ? 1 : 0;
  M.rf = rf.data();
  M.rf2 = rf2.data();
  M.c2 = c2.data();
  M.s2 = s2.data();
  M.cf = cf.data();
  M.sf = sf.data();
  M.fk = geo.fk.data();
  M.rho = rho.data();
  M.chi = chi.data();
  M.alb = alb.data();
  M.gq = gq.data();
  M.star_cum = star.data();
  M.chi0 = (float)(kabs[0] + ksca[0]);
  M.alb0 = (float)(ksca[0] / (kabs[0] + ksca[0]));
  M.g0 = (float)g[0];
  M.chiR0 = (float)(kabs[0] + (1.0 - g[0]) * ksca[0]);
  M.kbar0 = (float)kabs[0];
  M.lQk = tt.lQk.data();
  M.cbw = tt.cbw.data();
  M.cexit = tt.cexit.data();
  M.chiR = tt.chiRk.data();
  M.kbar = tt.kbark.data();
  M.lqm = den.lqm.data();
  M.lq_run = (float)std::log((Lstar + Ls) / ((double)n * (double)kEUnit));
  M.src_cum = Ls > 0 ? src_cum.data() : nullptr;
  M.src_Lstar = Lstar;
  M.src_Ltot = Lstar + Ls;
  M.n_src = Ls > 0 ? (int)ncell : 0;
  M.mtab = mueller ? mt.data() : nullptr;
  M.mcdf = mueller ? mcf.data() : nullptr;
  M.nmu = mueller ? nmu : 0;
  M.sed_q = (unsigned long long*)sq.data();
  M.sed_u = (unsigned long long*)su.data();
  M.jlen = jlen;
  M.jw = tt.jw.data();
  M.tally = (unsigned long long*)tally;
  M.visits = (unsigned long long*)visits;
  M.nabs = (unsigned long long*)nabs;
  M.sed = (unsigned long long*)sed;
  M.cnt = cnt.data();
  M.n_packets = n;
  DevModel<float> lanes[32];
  for (int l = 0; l < 32; ++l) {
    lanes[l] = M;
    if (late && l > 0) lanes[l].tally = (unsigned long long*)late;
  }
  KParams<float> P;
  std::memset(&P, 0, sizeof(P));
  P.m0 = M;
  P.mrw = mrw ? 1 : 0;
  P.nmin = nmin;
  P.exit_dir = exit_dir;
  P.want_lam = 1;
  P.refill = 4;
  P.defer = 8;
  P.gamma = (float)gamma;
  P.seed = seed;
  P.max_events = 1ull << 31;
  P.max_steps = 4000000000ull;
  P.mrw_tab = mtab.data();
  P.mrw_t0 = mrw_table_t0();
  P.mrw_dt = mrw_table_dt();
  P.nmodels = 1;
  Acc acc;
  std::memset(&acc, 0, sizeof(acc));
  const bool ok = mueller ? run_packets<true, false, false>(P, lanes, n, acc)
                  : jlen  ? run_packets<false, true, true>(P, lanes, n, acc)
                          : run_packets<false, false, true>(P, lanes, n, acc);
  const unsigned long long c[8] = {acc.packets, acc.abs, acc.sca, acc.cross, acc.mrw, acc.capped, acc.escaped, acc.err};
  for (int i = 0; i < 8; ++i) counters[i] = c[i];
  return ok ? 0 : 1;
}

// The run counters (C_NCNT values) after `times` packets of the given counts, kept as the kernel keeps them (and flushed at its end).
extern "C" void host_counters(int times, unsigned cross, unsigned sca, unsigned abs, unsigned mrw, uint64_t* cnt) {
  DevModel<float> M;
  std::memset(&M, 0, sizeof(M));
  M.cnt = (unsigned long long*)cnt;
  Acc acc;
  std::memset(&acc, 0, sizeof(acc));
  for (int k = 0; k < times; ++k) {
    acc.cross += cross;
    acc.sca += sca;
    acc.abs += abs;
    acc.mrw += mrw;
    acc.packets++;
    flush_if_full(M, acc);
  }
  flush(M, acc, false);
}
extern "C" void host_counter_places(int* at) {
  const int p[5] = {C_PACKETS, C_CROSS, C_SCA, C_ABS, C_MRW};
  for (int i = 0; i < 5; ++i) at[i] = p[i];
}
