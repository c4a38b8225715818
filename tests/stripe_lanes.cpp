// The stripes of csrc/ecmc_stripes.cu (its device part, as STRIPES) on the
// threads of warp_lanes.h: the sorted-frame kernel on every stripe of one
// colour.  Prints the stripes' counters and a hash of their coordinates.
//   stripe_lanes columns rows L stripes ell n_m reject list_mode downwards
// Staggered rows less than sigma apart, disks displaced.
#include "warp_lanes.h"

namespace ecmc {
inline double sqrt_rn(double x) { return std::sqrt(x); }
}  // namespace ecmc
struct {
  int x;
} blockIdx, blockDim;

#include STRIPES

#include <cstdlib>

using namespace ecmcs;

alignas(16) unsigned char ecmcs::ssm[232448];

int main(int argc, char** argv) {
  if (argc != 10) return 2;
  const int cols = std::atoi(argv[1]), rows = std::atoi(argv[2]), N = cols * rows;
  const double L = std::atof(argv[3]);
  const int S = std::atoi(argv[4]);
  GeomS g;
  std::memset(&g, 0, sizeof g);
  g.N = N;
  g.L = L;
  g.sigma = g.sig2 = 1.0;
  g.w = L / S;
  g.inv_w = 1.0 / g.w;
  g.ell = std::atof(argv[5]);
  g.S = S;
  g.n_m = std::atoi(argv[6]);
  g.reject = std::atoi(argv[7]);
  g.list_mode = std::atoi(argv[8]);
  g.seed = 1;
  g.cap_obj = (int)((g.w + 3.0) * (L + 1.0) / (M_PI / 4.0)) + 2;
  g.cap_mem = (int)((g.w + 1.0) * (L + 1.0) / (M_PI / 4.0)) + 2;
  g.sw = 0.5 * (1.0 + std::ldexp(1.0, -30));
  g.inv_sw = 1.0 / g.sw;
  g.nstrip = (int)std::ceil((g.w + 2.0) / g.sw) + 2;
  g.near = 1;
  if (sorted_smem_bytes(g.cap_obj, g.cap_mem, g.nstrip) > sizeof ssm) return 2;
  StateS st;
  std::memset(&st, 0, sizeof st);
  st.shift = 0.37 * g.w;
  std::vector<double> px(N), py(N);
  std::vector<int> stripe(N), fid((size_t)S * g.cap_obj), flist(fid.size());
  std::vector<double> fU(fid.size()), fV(fid.size()), fU0(fid.size());
  std::vector<long long> fkey(fid.size());
  std::vector<StripeS> stats(S);
  for (int i = 0; i < N; ++i) {
    const int r = i / cols;
    px[i] = (i % cols + 0.5 * (r % 2) + 0.25 + 0.04 * std::sin(2.1 * i)) * (L / cols);
    py[i] = (r + 0.5 + 0.02 * std::cos(3.7 * i)) * (L / rows);
    stripe[i] = cell_1d(py[i], st.shift, L, g.inv_w, S);
  }
  int err = 0;
  bool fine = true;
  for (blockIdx.x = 0; blockIdx.x < S / 2; ++blockIdx.x)
    fine = fine && warp::run(
                       [&](int) {
                         ks_phase_sorted(g, &st, 0, px.data(), py.data(), stripe.data(), fU.data(),
                                         fV.data(), fkey.data(), fid.data(), fU0.data(),
                                         flist.data(), stats.data(), nullptr, &err);
                       },
                       kSortThreads, std::atoi(argv[9]) != 0);
  unsigned long long hash = 0;
  for (int i = 0; i < N; ++i)
    hash = (hash ^ (unsigned long long)__double_as_longlong(px[i])) * 1099511628211ull;
  for (int q = 0; q < S; q += 2)
    std::printf("stripe %d: members %d chains %d accepted %d events %lld lifts %lld frozen %lld "
                "rejected %lld sum_b %.17g\n", q, stats[q].n_mem, stats[q].chains,
                stats[q].accepted, stats[q].events, stats[q].lifts, stats[q].frozen,
                stats[q].rejected, stats[q].sum_b);
  std::printf("hash %016llx\n", hash);
  return fine && err == 0 ? 0 : 3;
}
