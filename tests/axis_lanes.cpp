// The axis chains of csrc/ecmc_axis.cuh on the lanes of warp_lanes.h: frames,
// candidates and chains of the active cells of one colour phase.  Prints the
// cells' counters and a hash of the members' coordinates, which have to be the
// same in whatever order the lanes run.
//   axis_lanes k eta cells ell n_m boundary list_mode start precision downwards
// k^2 disks; start 0: square lattice, displaced; 1: rows staggered by sigma / 2
// (cells without static candidates).
#include "warp_lanes.h"

namespace ecmc {
inline double sqrt_rn(double x) { return std::sqrt(x); }
}  // namespace ecmc

#include "ecmc_device.cuh"
#include "ecmc_internal.cuh"
// comparisons of the FP64 search for candidates
static long n_exact;
static bool counted_dlt(double a, double b) {
  __atomic_fetch_add(&n_exact, 1, __ATOMIC_RELAXED);
  return ecmc::dlt(a, b);
}
#define dlt counted_dlt
#include "ecmc_axis.cuh"
#undef dlt

#include <cstdio>
#include <cstdlib>
#include <vector>

using namespace ecmc;

#ifndef LANES
#define LANES 8
#endif

int main(int argc, char** argv) {
  if (argc != 11) return 2;
  constexpr int TPC = LANES, CPW = 32 / TPC;
  const int k = std::atoi(argv[1]), cells = std::atoi(argv[3]), N = k * k;
  const double eta = std::atof(argv[2]), L = std::sqrt(N * M_PI / (4.0 * eta));
  const int reject = std::atoi(argv[6]), start = std::atoi(argv[8]);
  Geom g;
  std::memset(&g, 0, sizeof g);
  g.N = N;
  g.L = L;
  g.sigma = g.sig2 = 1.0;
  g.w = g.h = L / cells;
  g.inv_w = g.inv_h = 1.0 / g.w;
  g.ell = std::atof(argv[4]);
  g.cells_x = g.cells_y = cells;
  g.ncell = cells * cells;
  g.n_m = std::atoi(argv[5]);
  g.list_mode = std::atoi(argv[7]);
  g.boundary = reject;
  g.precision = std::atoi(argv[9]);
  g.seed = 1;
  double M = 1.0;
  while (M < g.w + 1.01) M *= 2.0;
  g.eps_d = (float)(6.5 * std::ldexp(1.0, -24) * M);
  g.sigf = 1.0f;
  g.inv_bin_w = 2.0f;
  g.nbin = (int)std::ceil((g.w + 2.0) / 0.5) + 1;
  g.cap_mem = (int)((g.w + 1) * (g.h + 1) / (M_PI / 4.0)) + 2;
  g.cap_obj = (int)((g.w + 3) * (g.h + 3) / (M_PI / 4.0)) + 2;
  const int cap = g.cap_mem;
  std::vector<UndoEntry> undo((size_t)g.ncell * cap);
  g.undo = undo.data();
  g.undo_stride = cap;

  SweepState st;
  std::memset(&st, 0, sizeof st);
  st.sx = 0.37 * g.w;
  st.sy = 0.61 * g.h;
  st.axis = start == 1 ? 1 : 0;
  std::vector<double> px((size_t)g.ncell * cap), py(px.size());
  std::vector<int> pid(px.size()), cnt(g.ncell);
  std::vector<float2> rel(px.size());
  for (int i = 0; i < N; ++i) {
    const int r = i / k, c = i % k;
    const double a = L / k;
    double x, y;
    if (start == 1) {
      x = 1.02 * c + 0.5 * (r % 2);
      y = 1.02 * (r + 0.25);
    } else {
      x = (c + 0.5 + 0.04 * std::sin(2.1 * i)) * a;
      y = (r + 0.5 + 0.04 * std::cos(3.7 * i)) * a;
    }
    double ux = x - st.sx, uy = y - st.sy;
    ux += ux < 0.0 ? L : 0.0;
    uy += uy < 0.0 ? L : 0.0;
    const int cx = std::min(cells - 1, (int)(ux * g.inv_w));
    const int cy = std::min(cells - 1, (int)(uy * g.inv_h));
    const int cell = cy * cells + cx, s = cell * cap + cnt[cell]++;
    px[s] = x;
    py[s] = y;
    pid[s] = i;
    rel[s] = make_float2((float)(ux - cx * g.w), (float)(uy - cy * g.h));
  }

  AxisShape shp;
  shp.cpw = CPW;
  shp.nbin = g.nbin;
  shp.co_h = shp.co_s = g.cap_obj;
  shp.mp_h = cap;
  shp.mp_s = CPW * cap;
  std::vector<double> smem(axis_smem_bytes(shp, 0) / 8 + 8);
  unsigned char* const sm = (unsigned char*)smem.data();
  std::vector<CellStats> cs(g.ncell);
  std::vector<unsigned long long> hash(CPW), irr(CPW);
  int err = 0;
  const int n_active = (cells / 2) * (cells / 2);
  auto lane_main = [&](int l) {
    const int gi = l / TPC, sub = l % TPC;
    const bool valid = gi < n_active;
    const int la = valid ? gi : 0, cx = 2 * (la % (cells / 2)), cy = 2 * (la / (cells / 2));
    const int c = cy * cells + cx, nc = valid ? cnt[c] : 0;
    const AxisPass pass = axis_pass(shp, CPW, shp.co_s, shp.mp_s, true);
    AxisHead& h = *(AxisHead*)(sm + gi * kAxisHead);
    unsigned char* const obj = sm + pass.obj_off + gi * axis_obj_bytes(pass.co);
    unsigned char* const work = sm + pass.work_off + gi * axis_work_bytes(pass.co, shp.nbin);
    const int mb = gi * cap;
    AxisFrame f;
    f.a = (double*)obj;
    f.b = f.a + pass.co + 2;
    f.key = (int*)(f.b + pass.co);
    f.list = (AxisEntry*)(sm + pass.memb_off) + 2 * mb;
    f.last = (int*)(sm + pass.flag_off) + mb;
    f.rank = (unsigned short*)(sm + pass.flag_off + 4 * shp.mp_s) + mb;
    f.starts = (unsigned short*)((unsigned char*)&h + sizeof(AxisHead));
    f.leg = (AxisLeg*)work;
    axis_build<TPC>(f, h, work, pass, shp.nbin, g, &st, cx, cy, c, cap, nc, valid, false,
                    px.data(), py.data(), pid.data(), rel.data(), cnt.data());
    const bool go = valid && h.ovf == 0;
    if (reject)
      axis_chains<TPC, true>(f, g, 3, c, c, go, go && h.irr != 0, cs.data(), nullptr, 1, 1, &err);
    else
      axis_chains<TPC, false>(f, g, 3, c, c, go, go && h.irr != 0, cs.data(), nullptr, 1, 1,
                              &err);
    if (sub == 0 && go) {
      irr[gi] = (unsigned long long)(h.irr & 1);
      for (int q = 0; q < nc; ++q)
        hash[gi] = (hash[gi] ^ (unsigned long long)dbits(f.a[q]) ^ (f.last[q] != 0 ? 1u : 0u)) *
                   1099511628211ull;
    }
  };
  const bool fine = warp::run(lane_main, 32, std::atoi(argv[10]) != 0);
  for (int gi = 0; gi < CPW && gi < n_active; ++gi) {
    const CellStats& s = cs[2 * (gi % (cells / 2)) + 2 * (gi / (cells / 2)) * cells];
    std::printf("cell %d irregular %llu: chains %d events %d lifts %d frozen %d walls %d replayed %d "
                "rejected %d sum_b %.17g hash %016llx\n", gi, irr[gi], s.chains, s.events, s.lifts,
                s.frozen, s.walls, s.replayed, s.rejected, s.sum_b, hash[gi]);
  }
  int members = 0;
  for (int gi = 0; gi < CPW && gi < n_active; ++gi)
    members += cs[2 * (gi % (cells / 2)) + 2 * (gi / (cells / 2)) * cells].n_mem;
  std::printf("members %d fp64 comparisons %ld\n", members, n_exact);
  return fine && err == 0 ? 0 : 3;
}
