// The spheres of csrc/ecmc3.cu (its device part, as SPHERES) on the lanes of
// warp_lanes.h: frames, candidate lists and chains of the active cells of one
// colour.  Prints the counters and a hash of the coordinates.
//   sphere_lanes k eta cells ell n_m rel shortest downwards
// k^3 spheres on a displaced cubic lattice; rel 0: frames without the FP32
// screen; shortest 1: room for one candidate list only.
#include "warp_lanes.h"

inline unsigned atomicAdd(unsigned* p, unsigned v) {
  return __atomic_fetch_add(p, v, __ATOMIC_RELAXED);
}
inline unsigned atomicExch(unsigned* p, unsigned v) {
  return __atomic_exchange_n(p, v, __ATOMIC_RELAXED);
}
inline unsigned long long atomicMin(unsigned long long* p, unsigned long long v) {
  const unsigned long long old = *p;
  if (v < old) *p = v;
  return old;
}
inline void __threadfence() {}
inline void __nanosleep(unsigned) {}
inline long long __double2ll_rd(double v) { return (long long)std::floor(v); }

namespace ecmc {
inline double sqrt_rn(double x) { return std::sqrt(x); }
}  // namespace ecmc
struct {
  int x;
} blockIdx, blockDim;

#include SPHERES

#include <cstdlib>

using namespace ecmc3;

alignas(16) unsigned char ecmc3::smem[232448];

int main(int argc, char** argv) {
  if (argc != 9) return 2;
  const int k = std::atoi(argv[1]), N = k * k * k, cells = std::atoi(argv[3]);
  const double L = std::cbrt(N * M_PI / (6.0 * std::atof(argv[2])));
  Geom3 g;
  std::memset(&g, 0, sizeof g);
  g.N = N;
  g.L = L;
  g.sigma = g.sig2 = 1.0;
  g.cells = cells;
  g.ncell = cells * cells * cells;
  g.nact = g.ncell / 8;
  g.w = L / cells;
  g.inv_w = 1.0 / g.w;
  g.ell = std::atof(argv[4]);
  g.n_m = std::atoi(argv[5]);
  g.replay = 1;
  g.seed = 1;
  const double ext = g.w + 2.0;
  g.scr_c2 = (float)(1.0 + 64.0 * std::ldexp(1.0, -24) * ext * ext);
  g.single_image = L >= 2.0 * (g.w + 1.0) ? 1 : 0;
  g.nbin = (int)std::floor(ext / (1.0 + std::ldexp(1.0, -12)));
  g.inv_hb = (float)(g.nbin / ext);
  g.use_bins = g.nbin > 4 ? 1 : 0;
  const auto bound = [](double w) { return (int)(std::pow(w + 1.0, 3) / (M_PI / 6.0)) + 2; };
  g.cap_mem = std::min(bound(g.w), N);
  g.cap_obj = bound(ext);
  const int one = (int)std::floor(10.01 * (g.w + 3.0)) + 4;
  g.cap_list = std::min(std::atoi(argv[7]) ? one : std::max(one, g.cap_obj / 2 + 8), g.cap_obj);
  g.near_lo = (float)(g.w - 1.0 - 1e-6 * ext);
  g.near_hi = (float)(1.0 + 1e-6 * ext);
  State3 st;
  std::memset(&st, 0, sizeof st);
  for (int i = 0; i < 8; ++i) st.perm[i] = i;
  for (int a = 0; a < 3; ++a) st.s[a] = (0.3 + 0.2 * a) * g.w;

  std::vector<double> p[3];
  for (auto& v : p) v.resize(N);
  std::vector<int> cnt(g.ncell), ids((size_t)g.ncell * g.cap_mem);
  std::vector<float4> rel(ids.size());
  std::vector<Cell3> cs(g.ncell);
  for (int i = 0; i < N; ++i) {
    const int at[3] = {i % k, i / k % k, i / k / k};
    int c = 0, n = 1;
    float f[3];
    for (int a = 0; a < 3; ++a) {
      p[a][i] = (at[a] + 0.5 + 0.03 * std::sin((2.1 + a) * i + a)) * (L / k);
      double u = p[a][i] - st.s[a];
      u += u < 0.0 ? L : 0.0;
      const int q = std::min(cells - 1, (int)(u * g.inv_w));
      f[a] = (float)(u - q * g.w);
      c += n * q;
      n *= cells;
    }
    const size_t slot = (size_t)c * g.cap_mem + cnt[c]++;
    ids[slot] = i;
    rel[slot] = make_float4(f[0], f[1], f[2], __int_as_float(i));
  }
  int err = 0;
  bool fine = true;
  for (int a = 0; a < std::min(8, g.nact); ++a)
    fine = fine && warp::run(
                       [&](int) {
                         cell3<false>(g, st, 0, a, smem, p[0].data(), p[1].data(), p[2].data(),
                                      cnt.data(), ids.data(),
                                      std::atoi(argv[6]) ? rel.data() : nullptr, cs.data(),
                                      nullptr, &err);
                       },
                       32, std::atoi(argv[8]) != 0);
  unsigned long long hash = 0;
  for (double x : p[0])
    hash = (hash ^ (unsigned long long)__double_as_longlong(x)) * 1099511628211ull;
  long events = 0, lifts = 0, frozen = 0, walls = 0, replayed = 0;
  for (const Cell3& c : cs) {
    events += c.events;
    lifts += c.lifts;
    frozen += c.frozen;
    walls += c.walls;
    replayed += c.replayed;
  }
  std::printf("bins %d events %ld lifts %ld frozen %ld walls %ld replayed %ld hash %016llx\n",
              g.use_bins, events, lifts, frozen, walls, replayed, hash);
  return fine && err == 0 ? 0 : 3;
}
