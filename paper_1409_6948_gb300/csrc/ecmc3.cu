// ecmc3.cu -- the parallel event-chain sweep for hard spheres in three
// dimensions (the generalisation of Sec. 3.4 to cubic cells in 2x2x2 blocks;
// interface and readings in ecmc3.h).
//
// Per sweep: k3_begin (draws), k3_bin (bucket every sphere by cell), the
// eight colour phases -- one persistent k3_sweep launch by default, or eight
// k3_phase launches -- and k3_end (deterministic sums).  Either way one warp
// processes one active cell (cell3): it sorts the cell's members by id,
// gathers the members and every periodic image of the 26 neighbour cells'
// spheres within sigma of the cell into a shared-memory frame, and runs the
// cell's n_m chains.
//
// Members move along the sweep's axis only, so an object is a candidate for
// a member's contacts (c^2 < sigma^2 across the axis) for the whole phase or
// not at all, and the square root in the contact distance is fixed as well.
// Both are found when a member first becomes active -- an FP32 screen of the
// frame with a rigorous margin (or of the nine bins across the axis round it,
// where a frame has more than 4 x 4 of them), then the oracle's FP64
// expressions (no contraction: the library is built with -fmad=false) -- and
// kept as a list in shared memory.  An event is then one pass over some 20
// list entries: b, b - root, and a minimum over the warp.  Lists share a room
// of fixed size; when it is full they are dropped and found again.
//
// What bounds it: 16 to 20 warps a SM (registers, frames of 10 KB) that wait
// for fixed latencies, shared memory and instruction fetch (1.4 instructions
// a cycle), and the FP64 pipe, half busy: one warp instruction holds it for
// 14 cycles of the SM however few lanes take part.  Hence comparisons of FP64
// values and the square root run on the integer pipes (bit-pattern orders,
// the correctly rounded sqrt_rn), a replayed leg takes one FP64 addition, and
// the neighbours' spheres pass an FP32 test of their positions within their
// cells (rel) before their coordinates are fetched.  N = 64^3, eta = 0.45,
// 32^3 cells, ell = 2, n_m = 1, GB300: 525 us a sweep, 758 with a search of
// the bins at every event and FP64 tests of all 26 neighbours; frames alone
// 279 / 403; 8^3 cells, n_m = 32: 12.3 / 18.7 ms; 16^3 spheres in 4^3 cells:
// 1.16 / 1.75 ms.  Positions live in sphere-id order; a cell reads its frozen
// neighbours' positions, which no warp writes while it runs (later colours
// wait for it, earlier ones have finished).
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <climits>
#include <vector>

#include "ecmc.h"
#include "ecmc3.h"
#include "ecmc_device.cuh"
#include "ecmc_internal.cuh"

namespace ecmc3 {

using ecmc::U64x4;
using ecmc::below_n;
using ecmc::cell_1d;
using ecmc::clamp0;
using ecmc::dbits;
using ecmc::dlt;
using ecmc::flip_if;
using ecmc::le_nn;
using ecmc::lt_nn;
using ecmc::philox;
using ecmc::plus_zero;
using ecmc::sqrt_rn;
using ecmc::to_float_trunc;
using ecmc::unit_double;
using ecmc::wrap_half;
using ecmc::wrap_half_i;

constexpr int kOk = 0, kCapacity = 1, kChainCap = 2, kWaitTimeout = 4;
constexpr int kWarpsMax = 4;
constexpr int kHistoryCap = 1 << 20;  // sweeps of pressure history kept

struct Geom3 {
  int64_t N;
  double L, sigma, sig2, w, inv_w, ell;
  int cells, ncell, nact, n_m;
  uint64_t seed, replica;
  int cap_mem, cap_obj;  // bucket slots per cell; frame objects per cell
  int cap_list;          // entries of the members' candidate lists, together
  int warp_bytes;        // shared memory of one warp's frame
  // FP32 screen: frame coordinates lie in (-sigma, w + sigma) and are
  // truncated to FP32 (integer pipes) with error < 2^-23 M (M >= w + sigma),
  // so FP32 differences (two truncations and one FP32 rounding of at most
  // 2^-24 2M) are within d = 8 2^-24 M of the FP64 ones; c^2 < sigma^2 then
  // has c2_32 < sigma^2 + 4 d sigma + 2 d^2 + FP32 rounding; the threshold
  // below is twice that bound
  float scr_c2;          // pass iff c2_32 < scr_c2
  // L >= 2 (w + sigma): a periodic image X0 +- L of a wrapped coordinate
  // X0 in [-L/2, L/2) lies outside (-sigma, w + sigma), so only the
  // unshifted image can enter a frame
  int single_image;
  // candidate bins across the chain axis: the frame's extent w + 2 sigma
  // along each perpendicular axis is cut into nbin bins of side
  // >= sigma (1 + 2^-12); a sphere the mover can hit (|dp|, |dq| < sigma)
  // then lies in the mover's bin or a neighbour on both axes, also after
  // the FP32 rounding of the coordinates the bin index is computed from
  int nbin;
  float inv_hb;          // 1 / bin side
  int use_bins;          // the search for a member's candidates goes by bins
  // a neighbour cell's sphere, by its FP32 position in that cell, can lie
  // within sigma of this cell: above near_lo (cell below), below near_hi
  float near_lo, near_hi;
  int replay;            // replay periodic rattles (results unchanged)
};

struct State3 {
  int64_t t;
  int axis;
  int perm[8];
  double s[3];
};

struct Cell3 {
  double sum_b;
  int events, lifts, frozen, walls, chains, n_mem, replayed;
};

struct Totals3 {
  double sum_b, sum_disp, sum_b_w, sum_disp_w;
  long long sweeps, chains, events, lifts, frozen, walls, replayed;
};

// Legs of the current chain kept for the replay of periodic rattles (a
// power of two: the ring index is the leg number's low bits)
constexpr int kHist3 = 16;

// ---- kernels ----------------------------------------------------------------

__global__ void k3_begin(Geom3 g, State3* st, unsigned* sched) {
  if (threadIdx.x != 0) return;
  // persistent sweep: the work list from the start, a new epoch, no abort
  sched[0] = 0u;
  sched[1] += 1u;
  sched[2] = 0u;
  sched[3] = 0u;  // blocks of k3_end that have finished
  State3 s = *st;
  const U64x4 u = philox((uint64_t)s.t, ecmc::kPurposeSweep, 0, 0, g.seed, g.replica);
  for (int a = 0; a < 3; ++a) s.s[a] = unit_double(u.v[a]) * g.w;
  // colour order: permutation number floor(u3 * 8! / 2^64) of 0..7 in
  // lexicographic order, decoded from its factorial-base digits
  int code = (int)below_n(u.v[3], 40320);
  int pool[8] = {0, 1, 2, 3, 4, 5, 6, 7};
  const int radix[8] = {5040, 720, 120, 24, 6, 2, 1, 1};
  int left = 8;
  for (int i = 0; i < 8; ++i) {
    const int d = code / radix[i];
    code -= d * radix[i];
    s.perm[i] = pool[d];
    for (int j = d; j < left - 1; ++j) pool[j] = pool[j + 1];
    --left;
  }
  s.axis = (int)(s.t % 3);
  *st = s;
}

__global__ void k3_bin(Geom3 g, const State3* __restrict__ st, const double* __restrict__ px,
                       const double* __restrict__ py, const double* __restrict__ pz,
                       int* __restrict__ cnt, int* __restrict__ ids, int* __restrict__ cell_of,
                       float4* __restrict__ rel, int* err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  const State3 s = *st;
  const double x = px[i], y = py[i], z = pz[i];
  const int cx = cell_1d(x, s.s[0], g.L, g.inv_w, g.cells);
  const int cy = cell_1d(y, s.s[1], g.L, g.inv_w, g.cells);
  const int cz = cell_1d(z, s.s[2], g.L, g.inv_w, g.cells);
  const int c = (cz * g.cells + cy) * g.cells + cx;
  cell_of[i] = c;
  const int slot = atomicAdd(&cnt[c], 1);
  if (slot >= g.cap_mem) {
    atomicCAS(err, kOk, kCapacity);
    return;
  }
  ids[(int64_t)c * g.cap_mem + slot] = (int)i;
  if (rel != nullptr) {  // the position within the cell, and the id
    const double hL = 0.5 * g.L;
    rel[(int64_t)c * g.cap_mem + slot] = make_float4(
        to_float_trunc(wrap_half_i(x - (s.s[0] + (double)cx * g.w), g.L, hL)),
        to_float_trunc(wrap_half_i(y - (s.s[1] + (double)cy * g.w), g.L, hL)),
        to_float_trunc(wrap_half_i(z - (s.s[2] + (double)cz * g.w), g.L, hL)),
        __int_as_float((int)i));
  }
}

// Cold paths of cell3, kept out of line so that the hot loop's code stays
// small.  Every periodic image of the offset (x0, x1, x2) whose centre lies
// in the open slab (lo, hi)^3 (boxes below the single-image size): bit
// img = (kx+1)*9 + (ky+1)*3 + (kz+1).
__device__ __noinline__ unsigned images_mask3(double x0, double x1, double x2, double L,
                                              double lo, double hi) {
  unsigned mask = 0u;
  for (int kx = -1; kx <= 1; ++kx) {
    const double X = x0 + (double)kx * L;
    if (!(X > lo && X < hi)) continue;
    for (int ky = -1; ky <= 1; ++ky) {
      const double Y = x1 + (double)ky * L;
      if (!(Y > lo && Y < hi)) continue;
      for (int kz = -1; kz <= 1; ++kz) {
        const double Z = x2 + (double)kz * L;
        if (!(Z > lo && Z < hi)) continue;
        mask |= 1u << ((kx + 1) * 9 + (ky + 1) * 3 + (kz + 1));
      }
    }
  }
  return mask;
}

// The lane of set `at` (the lanes whose hit distances are equal) with the
// smallest key.
__device__ __noinline__ int first_key3(unsigned at, long long key) {
  int win = __ffs(at) - 1;
  for (unsigned left = at & (at - 1); left != 0u; left &= left - 1u) {
    const int l = __ffs(left) - 1;
    if (__shfl_sync(0xffffffffu, key, l) < __shfl_sync(0xffffffffu, key, win)) win = l;
  }
  return win;
}

// The distinct neighbour cells with two cells per side, where the cells at
// offsets -1 and +1 coincide (lane 0 only).
__device__ __noinline__ void neighbour_list_small(int* nbl, int cx, int cy, int cz, int nc, int c) {
  int n = 0;
  for (int dz = -1; dz <= 1; ++dz)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx) {
        const int qx = (cx + dx + nc) % nc, qy = (cy + dy + nc) % nc, qz = (cz + dz + nc) % nc;
        const int q = (qz * nc + qy) * nc + qx;
        if (q == c) continue;
        bool dup = false;
        for (int e = 0; e < n; ++e) dup |= nbl[e] == q;
        if (!dup) nbl[n++] = q;
      }
  nbl[26] = n;
}

// wrap_box0 with the comparisons on the integer pipes
__device__ __forceinline__ double wrap_box_i(double v, double L) {
  if (ecmc::dkey(v) < 0) v += L;
  if (!dlt(v, L)) v -= L;
  return v;
}

// Position loads: through L1 in the per-phase kernels (the writers finished
// in an earlier launch), from L2 in the persistent kernel (the writers may
// be warps of other SMs in the same launch).
template <bool CG>
__device__ __forceinline__ double ldpos(const double* p) {
  if constexpr (CG) return __ldcg(p);
  else return *p;
}

// One active cell of colour phase colour_index, by one warp: frame, chains,
// write-back, cell statistics.  base: the warp's shared memory.
template <bool CG>
__device__ __forceinline__ void cell3(const Geom3& g, const State3& st, int colour_index, int a,
                                      unsigned char* base, double* __restrict__ px,
                                      double* __restrict__ py, double* __restrict__ pz,
                                      const int* __restrict__ cnt, const int* __restrict__ ids,
                                      float4* __restrict__ rel, Cell3* __restrict__ cs,
                                      int* __restrict__ recs, int* err) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int colour = st.perm[colour_index];
  const int hx = g.cells >> 1, nc = g.cells;
  const int cx = 2 * (a % hx) + (colour & 1);
  const int cy = 2 * ((a / hx) % hx) + ((colour >> 1) & 1);
  const int cz = 2 * (a / (hx * hx)) + (colour >> 2);
  const int c = (cz * nc + cy) * nc + cx;
  const double L = g.L, w = g.w;
  const double o[3] = {st.s[0] + (double)cx * w, st.s[1] + (double)cy * w,
                       st.s[2] + (double)cz * w};

  // the order of alignment; warp_bytes3 adds up the same sizes
  double* C[3];
  C[0] = reinterpret_cast<double*>(base);
  C[1] = C[0] + g.cap_obj;
  C[2] = C[1] + g.cap_obj;
  double* lroot = C[2] + g.cap_obj;  // candidate lists: sqrt(sigma^2 - c^2) ...
  // the chain's last kHist3 legs: start and end coordinate of the active
  // sphere along the axis, length, contact term bb - bs
  double* hP = lroot + g.cap_list;
  double* hE = hP + kHist3;
  double* hS = hE + kHist3;
  double* hT = hS + kHist3;
  // FP32 roundings of the two coordinates across the axis (fixed)
  float2* F = reinterpret_cast<float2*>(hT + kHist3);
  int* oid = reinterpret_cast<int*>(F + g.cap_obj);     // sphere id of an object
  int* sid = oid + g.cap_obj;                           // members sorted by id
  int* lst = sid + g.cap_mem;  // a member's list (start << 16 | length) or -1
  int* raw = lst;              // before: members as bucketed
  int* nbl = lst + g.cap_mem;                           // 26 neighbour cells + count
  int* npre = nbl + 28;                                 // their bucket sizes, prefix sums
  int* hM = npre + 28;    // legs: active sphere, direction, kind (0 lift, 1 frozen, 2 wall)
  int* hSg = hM + kHist3;
  int* hK = hSg + kHist3;
  const int nb = g.nbin, nb2 = g.use_bins ? nb * nb : 0;
  int* bst = hK + kHist3;                               // bin starts, nb2 + 1
  int* cur = bst + nb2 + 1;                             // scatter cursors, nb2
  unsigned short* lidx = reinterpret_cast<unsigned short*>(cur + nb2);  // ... and objects
  unsigned short* ord = lidx + g.cap_list;              // objects sorted by bin
  // bucket slot of a member; the top bit: it has been active
  unsigned short* mslot = ord + (g.use_bins ? g.cap_obj : 0);
  unsigned char* oimg = reinterpret_cast<unsigned char*>(mslot + g.cap_mem);  // image 0..26
  const int ax = st.axis, axp = ax == 0 ? 1 : 0, axq = ax == 2 ? 1 : 2;

  const int nmem = min(cnt[c], g.cap_mem);
  for (int k = lane; k < nmem; k += 32) raw[k] = ids[(int64_t)c * g.cap_mem + k];
  if (nc >= 3) {
    // 26 distinct neighbour cells: lane e takes offset e of the 3x3x3 block
    // in (dz, dy, dx) order, the centre skipped
    if (lane < 26) {
      const int e = lane < 13 ? lane : lane + 1;
      int qx = cx + e % 3 - 1, qy = cy + (e / 3) % 3 - 1, qz = cz + e / 9 - 1;
      qx = qx < 0 ? qx + nc : (qx >= nc ? qx - nc : qx);
      qy = qy < 0 ? qy + nc : (qy >= nc ? qy - nc : qy);
      qz = qz < 0 ? qz + nc : (qz >= nc ? qz - nc : qz);
      nbl[lane] = (qz * nc + qy) * nc + qx;
    }
    if (lane == 0) nbl[26] = 26;
  } else if (lane == 0) {
    neighbour_list_small(nbl, cx, cy, cz, nc, c);
  }
  __syncwarp();
  // the neighbours' objects as one list: npre[e] = sum of the bucket sizes
  // of neighbours 0 .. e-1
  const int nnb = nbl[26];
  const bool screen = g.single_image && rel != nullptr;  // (26 distinct neighbours)
  {
    const int nq = lane < nnb ? min(cnt[nbl[lane]], g.cap_mem) : 0;
    int incl = nq;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(FULL, incl, off);
      if (lane >= off) incl += v;
    }
    if (lane == 0) npre[0] = 0;
    if (lane < nnb) npre[lane + 1] = incl;
  }
  // members in ascending id (the rank of each is the number of smaller
  // ids); the positions are loaded before the rank is counted
  const double hL = 0.5 * L;
  for (int k0 = 0; k0 < nmem; k0 += 32) {
    const int k = k0 + lane;
    if (k >= nmem) continue;
    const int v = raw[k];
    const double mx = ldpos<CG>(px + v), my = ldpos<CG>(py + v), mz = ldpos<CG>(pz + v);
    int r = 0;
    for (int j = 0; j < nmem; ++j) r += raw[j] < v ? 1 : 0;
    sid[r] = v;
    mslot[r] = (unsigned short)k;
    C[0][r] = wrap_half_i(mx - o[0], L, hL);
    C[1][r] = wrap_half_i(my - o[1], L, hL);
    C[2][r] = wrap_half_i(mz - o[2], L, hL);
    oid[r] = v;
    oimg[r] = 13;
  }
  __syncwarp();
  for (int k = lane; k < nmem; k += 32) lst[k] = -1;  // (raw has been read)
  // frozen images, appended in the order (neighbour, bucket slot, image):
  // 32 entries of the neighbours' joint list per round, warp prefix sums
  int nobj = nmem;
  const double lo = -g.sigma, hi = w + g.sigma;
  const int ntot = npre[nnb];
  // the bucket slot of entry t of the joint list (t < ntot)
  auto slot_of = [&](int t) {  // (and the neighbour)
    int el = 0, eh = nnb;  // the neighbour e with npre[e] <= t < npre[e + 1]
    while (eh - el > 1) {
      const int mid = (el + eh) >> 1;
      if (npre[mid] <= t) el = mid;
      else eh = mid;
    }
    return make_int2(nbl[el] * g.cap_mem + (t - npre[el]), el);
  };
  // one round: the entries of 32 lanes (valid where in) with their box
  // positions p, appended as frame objects in lane order
  auto append = [&](bool in, int id, const double* p) {
    double X0[3] = {0.0, 0.0, 0.0};
    unsigned mask = 0u;  // bit img = (kx+1)*9 + (ky+1)*3 + (kz+1)
    if (in) {
      X0[0] = wrap_half_i(p[0] - o[0], L, hL);
      X0[1] = wrap_half_i(p[1] - o[1], L, hL);
      X0[2] = wrap_half_i(p[2] - o[2], L, hL);
      if (g.single_image) {
        if (dlt(lo, X0[0]) && dlt(X0[0], hi) && dlt(lo, X0[1]) && dlt(X0[1], hi) &&
            dlt(lo, X0[2]) && dlt(X0[2], hi))
          mask = 1u << 13;
      } else {
        mask = images_mask3(X0[0], X0[1], X0[2], L, lo, hi);
      }
    }
    const int nimg = __popc(mask);
    int incl = nimg;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(FULL, incl, off);
      if (lane >= off) incl += v;
    }
    int slot = nobj + incl - nimg;
    while (mask) {
      const int img = __ffs(mask) - 1;
      mask &= mask - 1;
      if (slot < g.cap_obj) {
        // X0 + k L for k in {-1, 0, 1}: (double)k * L is -L, +0.0 or L
        // exactly, and adding +0.0 only turns -0.0 into +0.0
        const int kx = img / 9 - 1, ky = (img / 3) % 3 - 1, kz = img % 3 - 1;
        C[0][slot] = kx == 0 ? plus_zero(X0[0]) : X0[0] + (kx > 0 ? L : -L);
        C[1][slot] = ky == 0 ? plus_zero(X0[1]) : X0[1] + (ky > 0 ? L : -L);
        C[2][slot] = kz == 0 ? plus_zero(X0[2]) : X0[2] + (kz > 0 ? L : -L);
        oid[slot] = id;
        oimg[slot] = (unsigned char)img;
      }
      ++slot;
    }
    nobj += __shfl_sync(FULL, incl, 31);
  };
  // Ids of the spheres to append.  With one image a sphere's FP32 position in
  // its cell (rel) decides for all but a margin whether it comes near this
  // cell: a neighbour's at offset -1 must lie above near_lo, at +1 below
  // near_hi.  Of some 200 spheres in the 26 neighbours about 50 are left for
  // the FP64 test.  Otherwise every sphere is tested.
  int* const app = reinterpret_cast<int*>(lroot);  // (the lists come later)
  const int cap_app = 2 * g.cap_list;
  int n_app = 0;
  if (screen) {
#pragma unroll 1
    for (int t0 = 0; t0 < ntot; t0 += 64) {
      bool near[2];
      int id[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int t = t0 + 32 * h + lane;
        near[h] = t < ntot;
        id[h] = 0;
        if (near[h]) {
          const int2 q = slot_of(t);
          const float4 f = __ldcg(rel + q.x);
          const int e = q.y < 13 ? q.y : q.y + 1;
          const int ez = e / 9, ey = (e - 9 * ez) / 3, ex = e - 9 * ez - 3 * ey;
          near[h] = (ex == 1 || (ex == 0 ? f.x > g.near_lo : f.x < g.near_hi)) &&
                    (ey == 1 || (ey == 0 ? f.y > g.near_lo : f.y < g.near_hi)) &&
                    (ez == 1 || (ez == 0 ? f.z > g.near_lo : f.z < g.near_hi));
          id[h] = __float_as_int(f.w);
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned nbm = __ballot_sync(FULL, near[h]);
        const int at = n_app + __popc(nbm & ((1u << lane) - 1u));
        if (near[h] && at < cap_app) app[at] = id[h];
        n_app += __popc(nbm);
      }
    }
    __syncwarp();
  } else {
    n_app = ntot;
  }
#pragma unroll 1
  for (int t0 = 0; t0 < n_app; t0 += 32) {
    const int t = t0 + lane;
    const bool in = t < n_app && (!screen || t < cap_app);
    const int id = in ? (screen ? app[t] : ids[slot_of(t).x]) : 0;
    double q[3] = {0.0, 0.0, 0.0};
    if (in) {
      q[0] = ldpos<CG>(px + id);
      q[1] = ldpos<CG>(py + id);
      q[2] = ldpos<CG>(pz + id);
    }
    append(in, id, q);
  }
  const bool ok = nobj <= g.cap_obj && !(screen && n_app > cap_app);
  if (!ok && lane == 0) atomicCAS(err, kOk, kCapacity);
  __syncwarp();

  // the coordinates across the sweep's axis, which members move along: these
  // hold for the whole phase, and so do bins across it (counting sort of the
  // objects, q-major)
  const float sigf = (float)g.sigma;
  auto bin_of = [&](float v) {
    const int b = (int)((v + sigf) * g.inv_hb);
    return b < 0 ? 0 : (b >= nb ? nb - 1 : b);
  };
  const int nobj_ok = ok ? nobj : 0;
  for (int o2 = lane; o2 < nobj_ok; o2 += 32)
    F[o2] = make_float2(to_float_trunc(C[axp][o2]), to_float_trunc(C[axq][o2]));
  __syncwarp();
  if (g.use_bins) {
    for (int i = lane; i <= nb2; i += 32) bst[i] = 0;
    __syncwarp();
    for (int o2 = lane; o2 < nobj_ok; o2 += 32)
      atomicAdd(&bst[1 + bin_of(F[o2].y) * nb + bin_of(F[o2].x)], 1);
    __syncwarp();
    int acc = 0;
    for (int i0 = 0; i0 <= nb2; i0 += 32) {  // starts (bst[0] = 0)
      int v = i0 + lane <= nb2 ? bst[i0 + lane] : 0;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int u = __shfl_up_sync(FULL, v, off);
        if (lane >= off) v += u;
      }
      if (i0 + lane <= nb2) bst[i0 + lane] = acc + v;
      acc += __shfl_sync(FULL, v, 31);
    }
    __syncwarp();
    for (int i = lane; i < nb2; i += 32) cur[i] = bst[i];
    __syncwarp();
    for (int o2 = lane; o2 < nobj_ok; o2 += 32)
      ord[atomicAdd(&cur[bin_of(F[o2].y) * nb + bin_of(F[o2].x)], 1)] = (unsigned short)o2;
    __syncwarp();
  }

  auto key_of = [&](int j) { return (long long)oid[j] * 27 + oimg[j]; };
  // the cell's chains
  double* CA = C[ax];
  double* CP = C[axp];
  double* CQ = C[axq];
  const double INF = __longlong_as_double(0x7ff0000000000000ll);
  int n_list = 0;  // entries of the candidate lists in use
  double sum_b = 0.0;
  int n_ev = 0, n_li = 0, n_fr = 0, n_wa = 0, n_ch = 0, n_rep = 0;
  for (int k = 0; k < g.n_m; ++k) {
    int* rec = recs != nullptr ? recs + 4 * ((int64_t)c * g.n_m + k) : nullptr;
    if (!ok || nmem == 0) {
      if (rec != nullptr && lane == 0) {
        rec[0] = -1;
        rec[1] = -1;
        rec[2] = 0;
        rec[3] = 0;
      }
      continue;
    }
    const U64x4 v = philox((uint64_t)st.t, ecmc::kPurposeChain, (uint64_t)c, (uint64_t)k,
                           g.seed, g.replica);
    int m = (int)below_n(v.v[0], (uint64_t)nmem);
    int sg = (v.v[1] >> 63) ? -1 : 1;
    const int start_id = sid[m];
    double r = g.ell;
    int ch_ev = 0, ch_wa = 0;
    int n_leg = 0;        // legs recorded in the history
    int64_t ch_rep = 0;   // legs of this chain replayed
    if (lane == 0) mslot[m] |= 0x8000;
    ++n_ch;
    for (int64_t iter = 0;; ++iter) {
      if (iter + ch_rep >= ecmc::kMaxEventsPerChain) {
        if (lane == 0) atomicCAS(err, kOk, kChainCap);
        break;
      }
      __syncwarp();
      const double P = CA[m];
      const double sw = clamp0(sg > 0 ? w - P : P);
      // The candidates of m: objects less than sigma away across the axis,
      // c^2 < sigma^2.  Neither they nor sqrt(sigma^2 - c^2) change during
      // the phase, so both are found when m first becomes active.
      int list = lst[m];
      if (list < 0) {
        const double Pp = CP[m], Pq = CQ[m];
        const float2 f = F[m];
        int rs[3] = {0, 0, 0}, rl[3] = {nobj, 0, 0};
        if (g.use_bins) {
          // the three rows of bins around m, each a contiguous run of ord[]
          const int bpm = bin_of(f.x), bqm = bin_of(f.y);
          const int plo = bpm > 0 ? bpm - 1 : 0, phi = bpm < nb - 1 ? bpm + 1 : nb - 1;
#pragma unroll
          for (int k3 = 0; k3 < 3; ++k3) {
            const int row = bqm - 1 + k3;
            const bool in = row >= 0 && row < nb;
            rs[k3] = in ? bst[row * nb + plo] : 0;
            rl[k3] = in ? bst[row * nb + phi + 1] - rs[k3] : 0;
          }
        }
        const int n_c = rl[0] + rl[1] + rl[2];
        int nl = 0;
#pragma unroll 1
        for (int t0 = 0; t0 < n_c; t0 += 32) {  // FP32 screen
          const int t = t0 + lane;
          bool pass = false;
          int j = t;
          if (t < n_c) {
            if (g.use_bins)
              j = ord[t < rl[0] ? rs[0] + t
                                : (t < rl[0] + rl[1] ? rs[1] + t - rl[0]
                                                     : rs[2] + t - rl[0] - rl[1])];
            const float2 fj = F[j];
            const float dp32 = fj.x - f.x, dq32 = fj.y - f.y;
            pass = j != m && dp32 * dp32 + dq32 * dq32 < g.scr_c2;
          }
          const unsigned bal = __ballot_sync(FULL, pass);
          const int np = __popc(bal);
          if (n_list + nl + np > g.cap_list) {
            if (n_list == 0) {  // (a list is shorter than that: cap_list)
              if (lane == 0) atomicCAS(err, kOk, kCapacity);
              break;
            }
            // no room: drop the lists and start this one over
            __syncwarp();  // (every lane has read lst[m]; votes order no memory)
            for (int q = lane; q < nmem; q += 32) lst[q] = -1;
            n_list = 0;
            nl = 0;
            t0 = -32;
            continue;
          }
          if (pass)
            lidx[n_list + nl + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)j;
          nl += np;
        }
        __syncwarp();
        for (int t = lane; t < nl; t += 32) {
          const int j = lidx[n_list + t];
          const double dp = CP[j] - Pp;
          const double dq = CQ[j] - Pq;
          const double c2 = dp * dp + dq * dq;
          // sigma^2 - c^2 is a positive normal number here (sigma in
          // [2^-40, 2^40]), as sqrt_rn requires; an object that the screen
          // let through is never hit: s = b + inf
          lroot[n_list + t] = lt_nn(c2, g.sig2) ? sqrt_rn(g.sig2 - c2) : -INF;
        }
        list = n_list << 16 | nl;
        if (lane == 0) lst[m] = list;
        n_list += nl;
        __syncwarp();
      }
      double bs = INF, bb = 0.0;
      int bj = -1;
      const int l0 = list >> 16, nl = list & 0xffff;
      for (int t = lane; t < nl; t += 32) {
        const int j = lidx[l0 + t];
        const double b = flip_if(CA[j] - P, sg < 0);
        if (dbits(b) <= 0) continue;  // b > 0
        const double s = clamp0(b - lroot[l0 + t]);
        if (lt_nn(s, bs) || (dbits(s) == dbits(bs) && bj >= 0 && key_of(j) < key_of(bj))) {
          bs = s;
          bb = b;
          bj = j;
        }
      }
      {
        // the first hit by (s, key): s >= +0 (or +inf) orders as its bit
        // pattern, compared high word, then low word; keys break exact ties
        const unsigned long long sb = (unsigned long long)dbits(bs);
        const unsigned hi = (unsigned)(sb >> 32), lo = (unsigned)sb;
        const unsigned mhi = __reduce_min_sync(FULL, hi);
        unsigned at = __ballot_sync(FULL, hi == mhi);
        if (at & (at - 1)) {
          const unsigned mlo = __reduce_min_sync(FULL, hi == mhi ? lo : 0xffffffffu);
          at = __ballot_sync(FULL, hi == mhi && lo == mlo);
          if ((at & (at - 1)) && mhi != 0x7ff00000u) at = 1u << first_key3(at, bj < 0 ? LLONG_MAX : key_of(bj));
        }
        const int win = __ffs(at) - 1;
        bs = __shfl_sync(FULL, bs, win);
        bb = __shfl_sync(FULL, bb, win);
        bj = __shfl_sync(FULL, bj, win);
      }
      __syncwarp();
      if (le_nn(r, bs) && le_nn(r, sw)) {  // budget used up
        if (lane == 0) CA[m] = P + (sg > 0 ? r : -r);
        break;
      }
      const int hi = n_leg & (kHist3 - 1);
      int kind;
      if (le_nn(bs, sw)) {  // contact
        // one FP64 addition gives three results: lane 0 the mover's new
        // coordinate P +- bs, lane 2 the contact term bb - bs (summed on
        // lane 2), every other lane the budget left, r - bs; x - y is by
        // definition x + (-y), so each equals its separate expression
        const double z = (lane == 0 ? P : (lane == 2 ? bb : r)) +
                         flip_if(bs, lane == 0 ? sg < 0 : true);
        kind = bj < nmem ? 0 : 1;
        if (lane == 0) {
          CA[m] = z;
          hP[hi] = P;
          hE[hi] = z;
          hS[hi] = bs;
          hM[hi] = m;
          hSg[hi] = sg;
          hK[hi] = kind;
        }
        if (lane == 2) {
          sum_b += z;
          hT[hi] = z;
        }
        r = __shfl_sync(FULL, z, 1);
        ++n_ev;
        ++ch_ev;
        if (kind == 0) {  // lift
          ++n_li;
          m = bj;
          if (lane == 0) mslot[m] |= 0x8000;
        } else {  // frozen sphere: back along the axis
          sg = -sg;
          ++n_fr;
        }
      } else {  // wall: onto the wall, back along the axis
        kind = 2;
        if (lane == 0) {
          CA[m] = sg > 0 ? w : 0.0;
          hP[hi] = P;
          hE[hi] = CA[m];
          hS[hi] = sw;
          hT[hi] = 0.0;
          hM[hi] = m;
          hSg[hi] = sg;
          hK[hi] = 2;
        }
        r = r - sw;
        sg = -sg;
        ++n_wa;
        ++ch_wa;
      }
      ++n_leg;
      if (g.replay && kind != 0 && n_leg >= 2) {
        // Replay of a periodic rattle.  After a turn-back, lane l tests the
        // period K = 2 (l + 1) <= n_leg: the next leg starts from the state
        // (active sphere, direction, coordinate bit for bit) that leg
        // n_leg - K started from, and every sphere active in those K legs
        // is back at its coordinate at the start of its first of them.  Frozen spheres
        // and walls do not move, so the whole frame is then as it was K
        // legs ago and, the dynamics being deterministic with the budget
        // entering a leg only through its end, the following legs repeat
        // the recorded ones for as long as the budget exceeds their length.
        __syncwarp();
        bool per = false;
        if (lane < kHist3 / 2 && 2 * (lane + 1) <= n_leg) {
          const int K = 2 * (lane + 1);
          const int i0 = (n_leg - K) & (kHist3 - 1);
          if (hM[i0] == m && hSg[i0] == sg && dbits(hP[i0]) == dbits(CA[m])) {
            per = true;
            for (int j = 1; j < K; ++j) {
              const int ij = (n_leg - K + j) & (kHist3 - 1);
              const int d = hM[ij];
              bool first = true;
              for (int i = 0; i < j; ++i) first = first && hM[(n_leg - K + i) & (kHist3 - 1)] != d;
              if (first && dbits(CA[d]) != dbits(hP[ij])) per = false;
            }
          }
        }
        const unsigned pb = __ballot_sync(FULL, per);
        if (pb != 0u) {
          __syncwarp();  // the search for K has read what lane 0 writes below
          const int K = 2 * __ffs(pb), b0 = n_leg - K;
          // whole legs while the budget exceeds them (a wall's contact term
          // is +0: it leaves the sum as it is)
          const int64_t n_max = ecmc::kMaxEventsPerChain - 1 - iter - ch_rep;
          // (one FP64 addition a leg: lane 2 the sum, the others the budget)
          const double* const hx = lane == 2 ? hT : hS;
          double z = lane == 2 ? sum_b : r;
          const int n_cap = n_max > INT_MAX ? INT_MAX : (int)n_max;
          int n = 0;
          int j = 0;
#pragma unroll 1
          for (; n < n_cap; ++n) {
            const double x = hx[(b0 + j) & (kHist3 - 1)];
            if (__ballot_sync(FULL, le_nn(z, x)) & 1u) break;
            z = z + flip_if(x, lane != 2);
            j = j + 1 == K ? 0 : j + 1;
          }
          if (lane == 2) sum_b = z;
          r = __shfl_sync(FULL, z, 0);
          if (n > 0) {
            const int kd = lane < K ? hK[(b0 + lane) & (kHist3 - 1)] : -1;
            const unsigned part = (1u << j) - 1u;
            const unsigned li = __ballot_sync(FULL, kd == 0), fr = __ballot_sync(FULL, kd == 1);
            const unsigned wa = __ballot_sync(FULL, kd == 2);
            const int whole = n / K;
            const int d_li = whole * __popc(li) + __popc(li & part);
            const int d_fr = whole * __popc(fr) + __popc(fr & part);
            const int d_wa = whole * __popc(wa) + __popc(wa & part);
            n_li += d_li;
            n_fr += d_fr;
            n_wa += d_wa;
            ch_wa += d_wa;
            n_ev += d_li + d_fr;
            ch_ev += d_li + d_fr;
            ch_rep += n;
            n_rep += n;
          }
          // the frame is as at the start of leg b0 (and of every K legs
          // after it); the recorded legs b0 .. b0 + j - 1 bring it to the
          // start of the leg in which the budget runs out, which the full
          // search then takes
          if (lane == 0)
            for (int i = 0; i < j; ++i) {
              const int ii = (b0 + i) & (kHist3 - 1);
              CA[hM[ii]] = hE[ii];
            }
          m = hM[(b0 + j) & (kHist3 - 1)];
          sg = hSg[(b0 + j) & (kHist3 - 1)];
          n_leg = 0;
        }
      }
    }
    __syncwarp();
    if (rec != nullptr && lane == 0) {
      rec[0] = start_id;
      rec[1] = sid[m];
      rec[2] = ch_ev;
      rec[3] = ch_wa;
    }
  }
  __syncwarp();
  // members that moved, back in box coordinates
  for (int q = lane; q < nmem; q += 32) {
    if (!(mslot[q] & 0x8000)) continue;
    const int i = sid[q];
    px[i] = wrap_box_i(C[0][q] + o[0], L);
    py[i] = wrap_box_i(C[1][q] + o[1], L);
    pz[i] = wrap_box_i(C[2][q] + o[2], L);
    if (rel != nullptr)
      rel[(int64_t)c * g.cap_mem + (mslot[q] & 0x7fff)] =
          make_float4(to_float_trunc(C[0][q]), to_float_trunc(C[1][q]), to_float_trunc(C[2][q]),
                      __int_as_float(i));
  }
  sum_b = __shfl_sync(FULL, sum_b, 2);  // the contact sum is kept on lane 2
  if (lane == 0) {
    Cell3 s;
    s.sum_b = sum_b;
    s.events = n_ev;
    s.lifts = n_li;
    s.frozen = n_fr;
    s.walls = n_wa;
    s.chains = n_ch;
    s.n_mem = nmem;
    s.replayed = n_rep;
    cs[c] = s;
  }
}

__global__ void __launch_bounds__(32 * kWarpsMax) k3_phase(
    Geom3 g, const State3* __restrict__ stp, int colour_index, double* __restrict__ px,
    double* __restrict__ py, double* __restrict__ pz, const int* __restrict__ cnt,
    const int* __restrict__ ids, float4* __restrict__ rel, Cell3* __restrict__ cs,
    int* __restrict__ recs, int* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5;
  const int a = blockIdx.x * (blockDim.x >> 5) + warp;
  if (a >= g.nact) return;  // warp-uniform
  const State3 st = *stp;
  cell3<false>(g, st, colour_index, a, smem + (size_t)warp * g.warp_bytes, px, py, pz, cnt, ids,
               rel, cs, recs, err);
}

__device__ __forceinline__ unsigned long long global_ns3() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned load_volatile3(const unsigned* p) {
  return *(const volatile unsigned*)p;
}

// The persistent sweep: all eight colour phases in one launch.  Work item
// i = ci * nact + a (colour phase ci, active cell a) is taken from a device
// counter; the warp waits until each of the cell's 26 neighbours whose colour
// comes earlier in this sweep's order has finished (done[] holds the sweep's
// epoch), then processes the cell and publishes it.  A cell of a later
// colour has not moved yet and waits for this one in turn, so the result is
// that of the per-phase launches bit for bit.  Progress: an item waits only
// for smaller items, taken earlier by running warps that wait only for still
// smaller ones.  Every wait is bounded (global timer): on timeout the kernel
// raises kWaitTimeout and an abort flag that makes every warp leave.
// (five blocks: 95 registers instead of 121 and no spills, 541 us against 563
// at N = 64^3; six spill: 615)
__global__ void __launch_bounds__(32 * kWarpsMax, 5) k3_sweep(
    Geom3 g, const State3* __restrict__ stp, double* __restrict__ px, double* __restrict__ py,
    double* __restrict__ pz, const int* __restrict__ cnt, const int* __restrict__ ids,
    float4* __restrict__ rel, Cell3* __restrict__ cs, int* __restrict__ recs, unsigned* sched,
    unsigned* done,
    unsigned long long wait_ns, int wait_test, int* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned FULL = 0xffffffffu;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* base = smem + (size_t)warp * g.warp_bytes;
  const State3 st = *stp;
  const unsigned epoch = load_volatile3(&sched[1]);
  // the failure test waits for a value nobody writes
  const unsigned want = wait_test ? (epoch ^ 0x80000000u) : epoch;
  int phase_of[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) phase_of[st.perm[k]] = k;
  const int n_items = 8 * g.nact, hx = g.cells >> 1, nc = g.cells;
  for (;;) {
    int item = 0;
    if (lane == 0) item = (int)atomicAdd(&sched[0], 1u);
    item = __shfl_sync(FULL, item, 0);
    if (item >= n_items || load_volatile3(&sched[2]) != 0u) break;
    const int ci = item / g.nact, a = item - ci * g.nact;
    const int colour = st.perm[ci];
    const int cx = 2 * (a % hx) + (colour & 1);
    const int cy = 2 * ((a / hx) % hx) + ((colour >> 1) & 1);
    const int cz = 2 * (a / (hx * hx)) + (colour >> 2);
    bool ok = true;
    if (ci > 0 && lane < 26) {
      // lane d waits for neighbour d of the 3x3x3 block (the centre skipped)
      const int e = lane < 13 ? lane : lane + 1;
      const int dx = e % 3 - 1, dy = (e / 3) % 3 - 1, dz = e / 9 - 1;
      const int ncol = colour ^ (dx != 0 ? 1 : 0) ^ (dy != 0 ? 2 : 0) ^ (dz != 0 ? 4 : 0);
      if (phase_of[ncol] < ci) {
        const int q = (((cz + dz + nc) % nc) * nc + (cy + dy + nc) % nc) * nc + (cx + dx + nc) % nc;
        if (load_volatile3(&done[q]) != want) {
          const unsigned long long t0 = global_ns3();
          while (load_volatile3(&done[q]) != want) {
            if (load_volatile3(&sched[2]) != 0u) {
              ok = false;
              break;
            }
            if (global_ns3() - t0 > wait_ns) {
              atomicCAS(err, kOk, kWaitTimeout);
              atomicExch(&sched[2], 1u);
              ok = false;
              break;
            }
            __nanosleep(256);
          }
        }
      }
    }
    if (!__all_sync(FULL, ok)) break;
    __threadfence();  // the finished neighbours' positions are visible from here on
    cell3<true>(g, st, ci, a, base, px, py, pz, cnt, ids, rel, cs, recs, err);
    __syncwarp();
    if (lane == 0) {
      __threadfence();
      *(volatile unsigned*)&done[(cz * nc + cy) * nc + cx] = epoch;
    }
    __syncwarp();
  }
}

// End of sweep: the cells' sums in a fixed order (256 strided threads, trees
// over their warps, the eight warps in turn), the running totals, the sweep's
// member-weighted pressure sums, t + 1.  Each of the eight warps is a block of
// its own, the last to finish adds them up: with 32^3 cells the FP64 pipe of
// one SM set the pace, 541 us a sweep against
// 525 now.
struct Part3 {
  double b, bw;
  long long v[6];
};
constexpr int kEndWarps = 8;

__global__ void __launch_bounds__(32) k3_end(Geom3 g, State3* st, const Cell3* __restrict__ cs,
                                             unsigned* sched, Part3* part, Totals3* tot,
                                             double* history, int64_t* hist_len) {
  const int lane = threadIdx.x, tid = 32 * blockIdx.x + lane;
  double b = 0.0, bw = 0.0;
  long long v[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 8
  for (int c = tid; c < g.ncell; c += 32 * kEndWarps) {
    const Cell3 s = cs[c];
    b += s.sum_b;
    bw += (double)s.n_mem * s.sum_b;
    v[0] += s.events;
    v[1] += s.lifts;
    v[2] += s.frozen;
    v[3] += s.walls;
    v[4] += s.chains;
    v[5] += s.replayed;
  }
  for (int off = 16; off > 0; off >>= 1) {
    b += __shfl_down_sync(0xffffffffu, b, off);
    bw += __shfl_down_sync(0xffffffffu, bw, off);
    for (int q = 0; q < 6; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], off);
  }
  if (lane != 0) return;
  volatile Part3* mine = part + blockIdx.x;
  mine->b = b;
  mine->bw = bw;
  for (int q = 0; q < 6; ++q) mine->v[q] = v[q];
  __threadfence();
  if (atomicAdd(&sched[3], 1u) != kEndWarps - 1) return;
  __threadfence();
  const volatile Part3* all = part;
  double B = 0.0, BW = 0.0;
  long long V[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int wv = 0; wv < kEndWarps; ++wv) {
    B += all[wv].b;
    BW += all[wv].bw;
    for (int q = 0; q < 6; ++q) V[q] += all[wv].v[q];
  }
  const double dw = (double)g.N * (double)g.n_m * g.ell;
  Totals3& T = *tot;
  T.sum_b += B;
  T.sum_b_w += BW;
  T.sum_disp += (double)V[4] * g.ell;
  T.sum_disp_w += dw;
  T.events += V[0];
  T.lifts += V[1];
  T.frozen += V[2];
  T.walls += V[3];
  T.chains += V[4];
  T.replayed += V[5];
  T.sweeps += 1;
  const int64_t n = *hist_len;
  if (n < kHistoryCap) {
    history[2 * n] = BW;
    history[2 * n + 1] = dw;
  }
  *hist_len = n + 1;
  st->t += 1;
}

// interleaved [x0, y0, z0, ...] <-> three arrays
__global__ void k3_split(const double* __restrict__ xyz, int64_t N, double* __restrict__ px,
                         double* __restrict__ py, double* __restrict__ pz) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  px[i] = xyz[3 * i];
  py[i] = xyz[3 * i + 1];
  pz[i] = xyz[3 * i + 2];
}

__global__ void k3_join(const double* __restrict__ px, const double* __restrict__ py,
                        const double* __restrict__ pz, int64_t N, double* __restrict__ xyz) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  xyz[3 * i] = px[i];
  xyz[3 * i + 1] = py[i];
  xyz[3 * i + 2] = pz[i];
}

// Smallest squared minimum-image distance below rcut^2 over the pairs of the
// last binning's 27-cell neighbourhoods (FP64, the oracle's formula), as the
// bits of a non-negative double (their order is the order of the values).
__global__ void k3_min_dist(Geom3 g, const double* __restrict__ px, const double* __restrict__ py,
                            const double* __restrict__ pz, const int* __restrict__ cnt,
                            const int* __restrict__ ids, const int* __restrict__ cell_of,
                            unsigned long long r2_bits, unsigned long long* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long best = r2_bits;
  if (i < g.N) {
    const int c = cell_of[i], nc = g.cells;
    const int cx = c % nc, cy = (c / nc) % nc, cz = c / (nc * nc);
    const double xi = px[i], yi = py[i], zi = pz[i];
    for (int dz = -1; dz <= 1; ++dz)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) {
          const int q = (((cz + dz + nc) % nc) * nc + (cy + dy + nc) % nc) * nc +
                        (cx + dx + nc) % nc;
          const int nq = min(cnt[q], g.cap_mem);
          for (int k = 0; k < nq; ++k) {
            const int j = ids[(int64_t)q * g.cap_mem + k];
            if (j == i) continue;
            const double ex = wrap_half(px[j] - xi, g.L);
            const double ey = wrap_half(py[j] - yi, g.L);
            const double ez = wrap_half(pz[j] - zi, g.L);
            const double d2 = ex * ex + ey * ey + ez * ez;
            const unsigned long long bits = __double_as_longlong(d2);
            best = bits < best ? bits : best;
          }
        }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o2 = __shfl_xor_sync(0xffffffffu, best, off);
    best = o2 < best ? o2 : best;
  }
  if ((threadIdx.x & 31) == 0 && best < r2_bits) atomicMin(out, best);
}

// The same minimum on fixed-point positions, as in two dimensions
// (ecmc_measure.cu, k_min_dist_fixed, which derives the method): coordinates as
// 32-bit fractions of the box side, squared distances D in FP32, one FP64
// evaluation per lane unless its two smallest D are too close to call, and then
// the window that holds every candidate.  Three dimensions change the bounds:
// |D - D*| <= 2 sqrt(3) e sqrt(D) + 9 e^2 with e = 1 + 2^-16, and the FP64
// formula adds less than 2^-18 sqrt(3 D) + 2^-50 D, below Bt(D) = 4.2 sqrt(D) +
// 16 + D / 2^40; the FP32 value of D (two roundings per square, two sums) stays
// within 2^-21 of D.  Pairs are visited once: the own cell with kk > k, then the
// 13 neighbours of the half stencil, so boxes need four cells per side and
// rcut < L / 4 (the FP64 scan takes the others).
//
// The FP64 scan was bound by the FP64 pipe, 27 x 8 candidates of three wraps
// each per sphere: 2.1 ms at N = 64^3 in 32^3 cells.  One warp per cell; cells
// of up to 8 (16) members split the stencil over four (two) groups of lanes.
__global__ void k3_fixed_point(Geom3 g, double scale, const double* __restrict__ px,
                               const double* __restrict__ py, const double* __restrict__ pz,
                               const int* __restrict__ cnt, const int* __restrict__ ids,
                               uint4* __restrict__ fq) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)g.ncell * g.cap_mem) return;
  const int c = (int)(i / g.cap_mem);
  if ((int)(i - (int64_t)c * g.cap_mem) >= min(cnt[c], g.cap_mem)) return;
  const int id = ids[i];
  fq[i] = make_uint4((unsigned)__double2ll_rd(px[id] * scale),
                     (unsigned)__double2ll_rd(py[id] * scale),
                     (unsigned)__double2ll_rd(pz[id] * scale), (unsigned)id);
}

__device__ __forceinline__ float bt_bound3(float x) {
  return 4.2f * sqrtf(x) + 16.0f + x * 0x1p-40f;
}

__global__ void __launch_bounds__(256) k3_min_dist_fixed(
    Geom3 g, const double* __restrict__ px, const double* __restrict__ py,
    const double* __restrict__ pz, const int* __restrict__ cnt, const uint4* __restrict__ fq,
    float t_skip, unsigned long long r2_bits, unsigned long long* __restrict__ out) {
  constexpr unsigned FULL = 0xffffffffu;
  const float kInf = __int_as_float(0x7f800000);
  const int c = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (c >= g.ncell) return;  // warp-uniform
  const int lane = threadIdx.x & 31, nc = g.cells;
  const int cx = c % nc, cy = (c / nc) % nc, cz = c / (nc * nc);
  const int nmem = min(cnt[c], g.cap_mem);
  const int gsz = nmem <= 8 ? 8 : (nmem <= 16 ? 16 : 32);
  unsigned long long best = r2_bits;
  for (int m0 = 0; m0 < nmem; m0 += gsz) {
    const int k = m0 + (lane & (gsz - 1));
    const bool act = k < nmem;
    const uint4 pi = fq[(int64_t)c * g.cap_mem + (act ? k : 0)];
    // cells of the half stencil: 0 the own one (kk > k), then offsets 14 .. 26
    // of the 3x3x3 block
    auto scan = [&](auto&& visit) {
      for (int e = lane / gsz; e < 14; e += 32 / gsz) {
        int q = c;
        if (e > 0) {
          const int f = 13 + e;
          int qx = cx + f % 3 - 1, qy = cy + (f / 3) % 3 - 1, qz = cz + f / 9 - 1;
          qx = qx < 0 ? qx + nc : (qx >= nc ? qx - nc : qx);
          qy = qy < 0 ? qy + nc : (qy >= nc ? qy - nc : qy);
          qz = qz < 0 ? qz + nc : (qz >= nc ? qz - nc : qz);
          q = (qz * nc + qy) * nc + qx;
        }
        const int nq = min(cnt[q], g.cap_mem);
        const uint4* const f = fq + (int64_t)q * g.cap_mem;
        const int kmin = e == 0 ? k : -1;
#pragma unroll 4
        for (int kk = 0; kk < nq; ++kk) {
          const uint4 pj = f[kk];
          const float dx = (float)(int)(pj.x - pi.x), dy = (float)(int)(pj.y - pi.y),
                      dz = (float)(int)(pj.z - pi.z);
          const float D = dx * dx + dy * dy + dz * dz;
          visit(kk > kmin ? D : kInf, (int)pj.w);
        }
      }
    };
    auto exact = [&](int j) {
      const int i = (int)pi.w;
      const double ex = wrap_half(px[j] - px[i], g.L);
      const double ey = wrap_half(py[j] - py[i], g.L);
      const double ez = wrap_half(pz[j] - pz[i], g.L);
      const unsigned long long bits =
          (unsigned long long)__double_as_longlong(ex * ex + ey * ey + ez * ez);
      best = bits < best ? bits : best;
    };
    float m1 = kInf, m2 = kInf;
    int j1 = 0;
    if (act)
      scan([&](float D, int j) {
        const bool lt1 = D < m1;
        m2 = lt1 ? m1 : fminf(m2, D);
        j1 = lt1 ? j : j1;
        m1 = lt1 ? D : m1;
      });
    if (act && m1 <= t_skip) {
      if (m2 - m1 > bt_bound3(m1) + bt_bound3(m2) + m2 * 0x1p-20f) {
        exact(j1);
      } else {
        const float win = (m1 + 4.0f * bt_bound3(m1) + 64.0f) * (1.0f + 0x1p-19f);
        scan([&](float D, int j) {
          if (D <= win) exact(j);
        });
      }
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o2 = __shfl_xor_sync(FULL, best, off);
    best = o2 < best ? o2 : best;
  }
  if (lane == 0 && best < r2_bits) atomicMin(out, best);
}

}  // namespace ecmc3

// ---- host side ----------------------------------------------------------------

using namespace ecmc3;

struct ecmc3_ctx {
  Geom3 g;
  cudaStream_t stream = nullptr, own = nullptr;
  double *px = nullptr, *py = nullptr, *pz = nullptr, *xyz_tmp = nullptr;
  int *cnt = nullptr, *ids = nullptr, *cell_of = nullptr, *err = nullptr, *recs = nullptr;
  // persistent sweep: work counter, epoch, abort; k3_end: blocks finished, their sums
  unsigned *sched = nullptr, *done = nullptr;
  int persistent = 1, fused_blocks = 0;
  unsigned long long wait_ns = 5000000000ull;
  int wait_test = 0;
  Cell3* cs = nullptr;
  State3* st = nullptr;
  Totals3* tot = nullptr;
  double* history = nullptr;
  int64_t* hist_len = nullptr;
  unsigned long long* u64 = nullptr;
  // by bucket slot: fixed-point positions (overlap check) or FP32 positions
  // within cells (sweeps); optional
  uint4* fq = nullptr;
  int warps = 1;
  int64_t t_host = 0;
  bool valid = false;
};

namespace {

int fail3(int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  return ecmc::report_error(code, buf);
}

#define CK3(call)                                                                         \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return fail3(e_ == cudaErrorMemoryAllocation ? ECMC_ERR_OOM : ECMC_ERR_CUDA,        \
                   "%s failed: %s", #call, cudaGetErrorString(e_));                       \
  } while (0)

// spheres of diameter sigma whose centres lie in a cube of side s: they sit
// inside the cube of side s + sigma, and no packing of spheres is denser
// than pi / (3 sqrt 2), so there are at most sqrt(2) (s + sigma)^3 / sigma^3
int sphere_bound(double s, double sigma) {
  const double q = (s + sigma) / sigma;
  return (int)std::floor(std::sqrt(2.0) * q * q * q) + 2;
}

int check3(ecmc3_ctx* h) {
  int e = 0;
  CK3(cudaMemcpyAsync(&e, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  CK3(cudaStreamSynchronize(h->stream));
  if (e == kCapacity) {
    h->valid = false;
    return fail3(ECMC_ERR_CAPACITY, "a cell bucket or frame exceeded its packing bound");
  }
  if (e == kChainCap) {
    h->valid = false;
    return fail3(ECMC_ERR_CHAIN_CAP, "a chain reached the per-chain event cap");
  }
  if (e == kWaitTimeout) {
    h->valid = false;
    CK3(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
    return fail3(ECMC_ERR_TIMEOUT, "a dependency wait of the persistent sweep exceeded %.0f ms; "
                 "the sweep was abandoned (positions must be set again)",
                 (double)h->wait_ns * 1e-6);
  }
  return ECMC_OK;
}

// Positions within cells by bucket slot, rewritten by every binning: in the
// buffer of the overlap check, which keeps nothing there between calls.
float4* rel3(const ecmc3_ctx* h) { return reinterpret_cast<float4*>(h->fq); }

int enqueue_sweep(ecmc3_ctx* h, bool records) {
  const Geom3& g = h->g;
  CK3(cudaMemsetAsync(h->cnt, 0, sizeof(int) * (size_t)g.ncell, h->stream));
  k3_begin<<<1, 32, 0, h->stream>>>(g, h->st, h->sched);
  k3_bin<<<(unsigned)((g.N + 255) / 256), 256, 0, h->stream>>>(g, h->st, h->px, h->py, h->pz,
                                                               h->cnt, h->ids, h->cell_of,
                                                               rel3(h), h->err);
  const int wpb = h->warps;
  const size_t sm = (size_t)wpb * g.warp_bytes;
  if (h->persistent && h->fused_blocks > 0) {
    k3_sweep<<<(unsigned)h->fused_blocks, 32 * wpb, sm, h->stream>>>(
        g, h->st, h->px, h->py, h->pz, h->cnt, h->ids, rel3(h), h->cs,
        records ? h->recs : nullptr,
        h->sched, h->done, h->wait_ns, h->wait_test, h->err);
  } else {
    const unsigned blocks = (unsigned)((g.nact + wpb - 1) / wpb);
    for (int ci = 0; ci < 8; ++ci)
      k3_phase<<<blocks, 32 * wpb, sm, h->stream>>>(g, h->st, ci, h->px, h->py, h->pz, h->cnt,
                                                    h->ids, rel3(h), h->cs,
                                                    records ? h->recs : nullptr, h->err);
  }
  k3_end<<<kEndWarps, 32, 0, h->stream>>>(g, h->st, h->cs, h->sched,
                                          reinterpret_cast<Part3*>(h->sched + 4), h->tot,
                                          h->history, h->hist_len);
  CK3(cudaGetLastError());
  return ECMC_OK;
}

int bin_now(ecmc3_ctx* h) {
  const Geom3& g = h->g;
  CK3(cudaMemsetAsync(h->cnt, 0, sizeof(int) * (size_t)g.ncell, h->stream));
  k3_begin<<<1, 32, 0, h->stream>>>(g, h->st, h->sched);
  k3_bin<<<(unsigned)((g.N + 255) / 256), 256, 0, h->stream>>>(g, h->st, h->px, h->py, h->pz,
                                                               h->cnt, h->ids, h->cell_of,
                                                               rel3(h), h->err);
  CK3(cudaGetLastError());
  return ECMC_OK;
}

double rcut3(const Geom3& g) { return std::fmin(2.0 * g.sigma, g.w); }

int min_dist2_3(ecmc3_ctx* h, double* d2) {
  const Geom3& g = h->g;
  const double rc = rcut3(g), r2 = rc * rc;
  unsigned long long bits = 0;
  std::memcpy(&bits, &r2, sizeof(r2));
  CK3(cudaMemcpyAsync(h->u64, &bits, sizeof(bits), cudaMemcpyHostToDevice, h->stream));
  const int64_t slots = (int64_t)g.ncell * g.cap_mem;
  bool fixed = rc < 0.25 * g.L && g.cells >= 4;
  if (fixed && !h->fq && cudaMalloc(&h->fq, sizeof(uint4) * (size_t)slots) != cudaSuccess) {
    cudaGetLastError();  // no room: the FP64 scan needs none
    h->fq = nullptr;
    fixed = false;
  }
  if (fixed) {
    const double scale = 4294967296.0 / g.L;
    const double R = (rc * scale) * (rc * scale);
    const double skip = (R + 4.2 * std::sqrt(R) + 17.0 + R * std::ldexp(1.0, -40)) *
                        (1.0 + std::ldexp(1.0, -19));
    k3_fixed_point<<<(unsigned)((slots + 255) / 256), 256, 0, h->stream>>>(
        g, scale, h->px, h->py, h->pz, h->cnt, h->ids, h->fq);
    k3_min_dist_fixed<<<(unsigned)(((int64_t)g.ncell * 32 + 255) / 256), 256, 0, h->stream>>>(
        g, h->px, h->py, h->pz, h->cnt, h->fq, std::nextafter((float)skip, 3.0e38f), bits,
        h->u64);
  } else {
    k3_min_dist<<<(unsigned)((g.N + 255) / 256), 256, 0, h->stream>>>(
        g, h->px, h->py, h->pz, h->cnt, h->ids, h->cell_of, bits, h->u64);
  }
  CK3(cudaGetLastError());
  CK3(cudaMemcpyAsync(&bits, h->u64, sizeof(bits), cudaMemcpyDeviceToHost, h->stream));
  const int rc2 = check3(h);
  if (rc2) return rc2;
  std::memcpy(d2, &bits, sizeof(*d2));
  return ECMC_OK;
}

int load_dev(ecmc3_ctx* h, const double* xyz_dev, int64_t t0) {
  const Geom3& g = h->g;
  k3_split<<<(unsigned)((g.N + 255) / 256), 256, 0, h->stream>>>(xyz_dev, g.N, h->px, h->py,
                                                                 h->pz);
  State3 s;
  std::memset(&s, 0, sizeof(s));
  s.t = t0;
  CK3(cudaMemcpyAsync(h->st, &s, sizeof(s), cudaMemcpyHostToDevice, h->stream));
  CK3(cudaMemsetAsync(h->tot, 0, sizeof(Totals3), h->stream));
  CK3(cudaMemsetAsync(h->hist_len, 0, sizeof(int64_t), h->stream));
  CK3(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
  h->t_host = t0;
  h->valid = true;
  int rc = bin_now(h);
  if (rc) return rc;
  rc = check3(h);
  if (rc) return rc;
  double d2 = 0.0;
  rc = min_dist2_3(h, &d2);
  if (rc) return rc;
  if (d2 < g.sig2 * (1.0 - 1e-9)) {
    h->valid = false;
    return fail3(ECMC_ERR_OVERLAP, "positions overlap: smallest distance %.17g < sigma",
                 std::sqrt(d2));
  }
  return ECMC_OK;
}

void free3(ecmc3_ctx* h) {
  cudaFree(h->px);
  cudaFree(h->py);
  cudaFree(h->pz);
  cudaFree(h->xyz_tmp);
  cudaFree(h->cnt);
  cudaFree(h->ids);
  cudaFree(h->cell_of);
  cudaFree(h->err);
  cudaFree(h->recs);
  cudaFree(h->cs);
  cudaFree(h->st);
  cudaFree(h->tot);
  cudaFree(h->history);
  cudaFree(h->hist_len);
  cudaFree(h->u64);
  cudaFree(h->fq);
  cudaFree(h->sched);
  cudaFree(h->done);
  if (h->own) cudaStreamDestroy(h->own);
}

// shared memory of one warp's frame, and the launch's warps per block
int layout3(ecmc3_ctx* h) {
  Geom3& g = h->g;
  const size_t nb2 = g.use_bins ? (size_t)g.nbin * g.nbin : 0;
  g.warp_bytes = (int)(((size_t)g.cap_obj * (3 * sizeof(double) + sizeof(float2) + sizeof(int) +
                                             (g.use_bins ? sizeof(short) : 0) + 1) +
                        (size_t)g.cap_list * (sizeof(double) + sizeof(short)) +
                        (2 * nb2 + 1) * sizeof(int) +
                        (size_t)g.cap_mem * (2 * sizeof(int) + sizeof(short)) +
                        56 * sizeof(int) +
                        (size_t)kHist3 * (4 * sizeof(double) + 3 * sizeof(int)) + 15) &
                       ~(size_t)15);
  int dev = 0, optin = 0, n_sm = 0;
  CK3(cudaGetDevice(&dev));
  CK3(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  CK3(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
  if ((size_t)g.warp_bytes > (size_t)optin)
    return fail3(ECMC_ERR_UNSUPPORTED, "a cell's frame (%d bytes) exceeds shared memory",
                 g.warp_bytes);
  // The attribute is per kernel for the whole process: request the most the
  // kernels can have, so that a handle with small frames never lowers the
  // limit a handle with larger frames launches with.
  cudaFuncAttributes fa;
  CK3(cudaFuncGetAttributes(&fa, k3_phase));
  CK3(cudaFuncSetAttribute(k3_phase, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           optin - (int)fa.sharedSizeBytes));
  CK3(cudaFuncGetAttributes(&fa, k3_sweep));
  CK3(cudaFuncSetAttribute(k3_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           optin - (int)fa.sharedSizeBytes));
  // block shape: the warps per block (one cell each) that keep the most
  // cells resident per SM; larger blocks on ties
  int wpb = 1, per_sm = 0, best = -1;
  for (int w = 1; w <= kWarpsMax; ++w) {
    const size_t smw = (size_t)w * g.warp_bytes;
    if (smw > (size_t)optin) break;
    int nb = 0;
    CK3(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k3_sweep, 32 * w, smw));
    if (nb * w >= best) {
      best = nb * w;
      wpb = w;
      per_sm = nb;
    }
  }
  h->warps = wpb;
  // the persistent grid: as many blocks as are resident at once, at most one
  // warp per work item
  const long long items = 8LL * g.nact;
  long long blocks = (long long)per_sm * n_sm;
  if (blocks > (items + wpb - 1) / wpb) blocks = (items + wpb - 1) / wpb;
  h->fused_blocks = per_sm > 0 ? (int)blocks : 0;
  return ECMC_OK;
}

}  // namespace

extern "C" {

int ecmc3_create(ecmc3_t* out, int64_t N, double L, double sigma, int cells, double ell,
                 uint64_t seed) {
  if (!out) return fail3(ECMC_ERR_ARG, "NULL output handle");
  *out = nullptr;
  if (N < 1 || N >= (int64_t(1) << 30)) return fail3(ECMC_ERR_ARG, "N out of range");
  int64_t k = (int64_t)std::llround(std::cbrt((double)N));
  while (k * k * k > N) --k;
  while ((k + 1) * (k + 1) * (k + 1) <= N) ++k;
  if (k * k * k != N) return fail3(ECMC_ERR_ARG, "N must be a perfect cube (lattice start)");
  if (!(L > 0.0) || !(sigma > 0.0) || !std::isfinite(L) || !std::isfinite(sigma))
    return fail3(ECMC_ERR_ARG, "L and sigma must be positive");
  if (!(sigma >= std::ldexp(1.0, -40) && sigma <= std::ldexp(1.0, 40) &&
        L < std::ldexp(sigma, 40)))
    return fail3(ECMC_ERR_ARG, "sigma must lie in [2^-40, 2^40] and L below 2^40 sigma");
  if (cells < 2 || (cells & 1) || cells > 1024)
    return fail3(ECMC_ERR_ARG, "cells per side must be even, >= 2 and <= 1024");
  if (!(L / (double)cells > sigma)) return fail3(ECMC_ERR_ARG, "cell side must exceed sigma");
  if (!(L / (double)k > sigma)) return fail3(ECMC_ERR_ARG, "cubic lattice would overlap");
  if (!(ell >= 0.0) || !std::isfinite(ell)) return fail3(ECMC_ERR_ARG, "ell must be >= 0");
  ecmc3_ctx* h = new ecmc3_ctx();
  Geom3& g = h->g;
  std::memset(&g, 0, sizeof(g));
  g.N = N;
  g.L = L;
  g.sigma = sigma;
  g.sig2 = sigma * sigma;
  g.cells = cells;
  g.ncell = cells * cells * cells;
  g.nact = g.ncell / 8;
  g.w = L / (double)cells;
  g.inv_w = 1.0 / g.w;
  g.ell = ell;
  g.n_m = 1;
  g.replay = 1;
  g.seed = seed;
  g.replica = 0;
  {
    const double M = g.w + 2.0 * sigma;
    const double d = 8.0 * std::ldexp(1.0, -24) * M;
    const double c2 = sigma * sigma + 4.0 * d * sigma + 2.0 * d * d +
                      4.0 * std::ldexp(1.0, -24) * (sigma * sigma + 4.0 * M * M);
    g.scr_c2 = std::nextafter((float)(sigma * sigma + 2.0 * (c2 - sigma * sigma)), 1e30f);
  }
  g.single_image = L >= 2.0 * (g.w + sigma) ? 1 : 0;
  {
    const double ext = g.w + 2.0 * sigma;
    int nb = (int)std::floor(ext / (sigma * (1.0 + std::ldexp(1.0, -12))));
    if (nb < 1) nb = 1;
    if (nb > 64) nb = 64;
    g.nbin = nb;
    g.inv_hb = (float)((double)nb / ext);
  }
  g.cap_mem = sphere_bound(g.w, sigma);
  g.cap_obj = sphere_bound(g.w + 2.0 * sigma, sigma);
  if ((int64_t)g.cap_mem > N) g.cap_mem = (int)N;
  {
    // spheres with centres within sigma of a line of length w + 2 sigma: they
    // lie in a cylinder of radius 1.5 sigma and length w + 3 sigma, none
    // denser than pi / (3 sqrt 2); a list of candidates (the FP32 screen adds
    // a skin of 2^-18 sigma) always fits, several usually do
    const int one = (int)std::floor(10.01 * (g.w + 3.0 * sigma) / sigma) + 4;
    int cap = g.cap_obj / 2 + 8 > 96 ? g.cap_obj / 2 + 8 : 96;
    cap = cap > one ? cap : one;
    g.cap_list = cap < g.cap_obj ? cap : g.cap_obj;
    // up to four bins a side a member's three rows and columns are most of the
    // frame, and the counting sort costs more than it spares
    g.use_bins = g.nbin > 4 ? 1 : 0;
    const double eps = 1e-6 * (g.w + sigma) + 1e-12 * L;
    g.near_lo = (float)(g.w - sigma - eps);
    g.near_hi = (float)(sigma + eps);
  }
  if ((double)g.ncell * g.cap_mem > 2.0e9) {
    delete h;
    return fail3(ECMC_ERR_ARG, "too many cells");
  }
  int rc = layout3(h);
  if (rc) {
    delete h;
    return rc;
  }
  if (cudaStreamCreateWithFlags(&h->own, cudaStreamNonBlocking) != cudaSuccess) {
    delete h;
    return fail3(ECMC_ERR_CUDA, "stream creation failed");
  }
  h->stream = h->own;
  const size_t nn = (size_t)N;
  if (cudaMalloc(&h->px, sizeof(double) * nn) != cudaSuccess ||
      cudaMalloc(&h->py, sizeof(double) * nn) != cudaSuccess ||
      cudaMalloc(&h->pz, sizeof(double) * nn) != cudaSuccess ||
      cudaMalloc(&h->xyz_tmp, sizeof(double) * 3 * nn) != cudaSuccess ||
      cudaMalloc(&h->cnt, sizeof(int) * (size_t)g.ncell) != cudaSuccess ||
      cudaMalloc(&h->ids, sizeof(int) * (size_t)g.ncell * g.cap_mem) != cudaSuccess ||
      cudaMalloc(&h->cell_of, sizeof(int) * nn) != cudaSuccess ||
      cudaMalloc(&h->err, sizeof(int)) != cudaSuccess ||
      cudaMalloc(&h->cs, sizeof(Cell3) * (size_t)g.ncell) != cudaSuccess ||
      cudaMalloc(&h->st, sizeof(State3)) != cudaSuccess ||
      cudaMalloc(&h->tot, sizeof(Totals3)) != cudaSuccess ||
      cudaMalloc(&h->history, sizeof(double) * 2 * kHistoryCap) != cudaSuccess ||
      cudaMalloc(&h->hist_len, sizeof(int64_t)) != cudaSuccess ||
      cudaMalloc(&h->u64, sizeof(unsigned long long)) != cudaSuccess ||
      cudaMalloc(&h->sched, sizeof(unsigned) * 4 + sizeof(Part3) * kEndWarps) != cudaSuccess ||
      cudaMalloc(&h->done, sizeof(unsigned) * (size_t)g.ncell) != cudaSuccess) {
    cudaGetLastError();
    free3(h);
    delete h;
    return fail3(ECMC_ERR_OOM, "device allocation failed");
  }
  cudaMemsetAsync(h->sched, 0, sizeof(unsigned) * 4, h->stream);
  cudaMemsetAsync(h->done, 0, sizeof(unsigned) * (size_t)g.ncell, h->stream);
  // the cubic lattice start
  std::vector<double> xyz(3 * nn);
  const double a = L / (double)k;
  for (int64_t i = 0; i < N; ++i) {
    xyz[3 * i] = ((double)(i % k) + 0.5) * a;
    xyz[3 * i + 1] = ((double)((i / k) % k) + 0.5) * a;
    xyz[3 * i + 2] = ((double)(i / (k * k)) + 0.5) * a;
  }
  rc = ecmc3_set_positions(h, xyz.data(), 0, 0);
  if (rc) {
    free3(h);
    delete h;
    return rc;
  }
  *out = h;
  return ECMC_OK;
}

int ecmc3_destroy(ecmc3_t h) {
  if (!h) return ECMC_OK;  // like ecmc_destroy: nothing to release
  if (h->stream) cudaStreamSynchronize(h->stream);
  free3(h);
  delete h;
  return ECMC_OK;
}

int ecmc3_set_param(ecmc3_t h, int key, double v) {
  if (!h) return fail3(ECMC_ERR_ARG, "NULL handle");
  switch (key) {
    case ECMC3_PARAM_N_CHAINS: {
      const int n = (int)v;
      if ((double)n != v || n < 1 || n > (1 << 20)) return fail3(ECMC_ERR_ARG, "n_m");
      if (n != h->g.n_m) {
        h->g.n_m = n;
        cudaFree(h->recs);
        h->recs = nullptr;
      }
      return ECMC_OK;
    }
    case ECMC3_PARAM_REPLICA:
      if (!(v >= 0.0) || v != std::floor(v) || v > 9.0e15) return fail3(ECMC_ERR_ARG, "replica");
      h->g.replica = (uint64_t)v;
      return ECMC_OK;
    case ECMC3_PARAM_PERSISTENT:
      if (v != 0.0 && v != 1.0) return fail3(ECMC_ERR_ARG, "persistent must be 0 or 1");
      h->persistent = (int)v;
      return ECMC_OK;
    case ECMC3_PARAM_WAIT_LIMIT_MS:
      if (!(v >= 1.0 && v <= 600000.0)) return fail3(ECMC_ERR_ARG, "wait limit in [1, 600000] ms");
      h->wait_ns = (unsigned long long)(v * 1e6);
      return ECMC_OK;
    case ECMC3_PARAM_WAIT_TEST:
      if (v != 0.0 && v != 1.0) return fail3(ECMC_ERR_ARG, "wait test must be 0 or 1");
      h->wait_test = (int)v;
      return ECMC_OK;
    case ECMC3_PARAM_REPLAY:
      if (v != 0.0 && v != 1.0) return fail3(ECMC_ERR_ARG, "replay must be 0 or 1");
      h->g.replay = (int)v;
      return ECMC_OK;
    default:
      return fail3(ECMC_ERR_ARG, "unknown parameter %d", key);
  }
}

int ecmc3_get_param(ecmc3_t h, int key, double* v) {
  if (!h || !v) return fail3(ECMC_ERR_ARG, "NULL argument");
  switch (key) {
    case ECMC3_PARAM_N_CHAINS: *v = h->g.n_m; return ECMC_OK;
    case ECMC3_PARAM_REPLICA: *v = (double)h->g.replica; return ECMC_OK;
    case ECMC3_PARAM_PERSISTENT: *v = (h->persistent && h->fused_blocks > 0) ? 1.0 : 0.0;
      return ECMC_OK;
    case ECMC3_PARAM_WAIT_LIMIT_MS: *v = (double)h->wait_ns * 1e-6; return ECMC_OK;
    case ECMC3_PARAM_WAIT_TEST: *v = h->wait_test; return ECMC_OK;
    case ECMC3_PARAM_REPLAY: *v = h->g.replay; return ECMC_OK;
    default: return fail3(ECMC_ERR_ARG, "unknown parameter %d", key);
  }
}

int ecmc3_set_stream(ecmc3_t h, void* stream) {
  if (!h) return fail3(ECMC_ERR_ARG, "NULL handle");
  CK3(cudaStreamSynchronize(h->stream));
  h->stream = stream ? (cudaStream_t)stream : h->own;
  return ECMC_OK;
}

int ecmc3_set_positions(ecmc3_t h, const double* xyz, int on_device, int64_t t0) {
  if (!h || !xyz) return fail3(ECMC_ERR_ARG, "NULL argument");
  if (t0 < 0) return fail3(ECMC_ERR_ARG, "t0 must be >= 0");
  const double* src = xyz;
  if (!on_device) {
    CK3(cudaMemcpyAsync(h->xyz_tmp, xyz, sizeof(double) * 3 * (size_t)h->g.N,
                        cudaMemcpyHostToDevice, h->stream));
    src = h->xyz_tmp;
  }
  return load_dev(h, src, t0);
}

int ecmc3_positions(ecmc3_t h, double* xyz, int on_device) {
  if (!h || !xyz) return fail3(ECMC_ERR_ARG, "NULL argument");
  if (!h->valid) return fail3(ECMC_ERR_STATE, "state invalid after an earlier error");
  const Geom3& g = h->g;
  double* dst = on_device ? xyz : h->xyz_tmp;
  k3_join<<<(unsigned)((g.N + 255) / 256), 256, 0, h->stream>>>(h->px, h->py, h->pz, g.N, dst);
  CK3(cudaGetLastError());
  if (!on_device)
    CK3(cudaMemcpyAsync(xyz, h->xyz_tmp, sizeof(double) * 3 * (size_t)g.N,
                        cudaMemcpyDeviceToHost, h->stream));
  return check3(h);
}

int ecmc3_sweep(ecmc3_t h, int64_t n) {
  if (!h) return fail3(ECMC_ERR_ARG, "NULL handle");
  if (n < 0) return fail3(ECMC_ERR_ARG, "negative sweep count");
  if (!h->valid) return fail3(ECMC_ERR_STATE, "state invalid after an earlier error");
  const bool rec = n > 0;
  if (rec && !h->recs) {
    CK3(cudaMalloc(&h->recs, sizeof(int) * 4 * (size_t)h->g.ncell * h->g.n_m));
  }
  for (int64_t s = 0; s < n; ++s) {
    const int rc = enqueue_sweep(h, s == n - 1);
    if (rc) return rc;
  }
  h->t_host += n;
  return ECMC_OK;
}

int ecmc3_synchronize(ecmc3_t h) {
  if (!h) return fail3(ECMC_ERR_ARG, "NULL handle");
  return check3(h);
}

int ecmc3_sweep_index(ecmc3_t h, int64_t* t) {
  if (!h || !t) return fail3(ECMC_ERR_ARG, "NULL argument");
  *t = h->t_host;
  return ECMC_OK;
}

int ecmc3_counters(ecmc3_t h, ecmc_counters_t* out) {
  if (!h || !out) return fail3(ECMC_ERR_ARG, "NULL argument");
  Totals3 t;
  CK3(cudaMemcpyAsync(&t, h->tot, sizeof(t), cudaMemcpyDeviceToHost, h->stream));
  const int rc = check3(h);
  if (rc) return rc;
  std::memset(out, 0, sizeof(*out));
  out->sweeps = t.sweeps;
  out->chains = t.chains;
  out->events = t.events;
  out->lifts = t.lifts;
  out->frozen_hits = t.frozen;
  out->wall_hits = t.walls;
  out->replayed_legs = t.replayed;
  out->sum_b = t.sum_b;
  out->sum_disp = t.sum_disp;
  return ECMC_OK;
}

int ecmc3_pressure(ecmc3_t h, double* betaP, double* se) {
  if (!h || !betaP) return fail3(ECMC_ERR_ARG, "NULL argument");
  Totals3 t;
  int64_t n = 0;
  CK3(cudaMemcpyAsync(&t, h->tot, sizeof(t), cudaMemcpyDeviceToHost, h->stream));
  CK3(cudaMemcpyAsync(&n, h->hist_len, sizeof(n), cudaMemcpyDeviceToHost, h->stream));
  int rc = check3(h);
  if (rc) return rc;
  if (n < 1 || !(t.sum_disp_w > 0.0)) return fail3(ECMC_ERR_STATE, "no sweep since the last reset");
  const Geom3& g = h->g;
  const double rho_s3 = (double)g.N / (g.L * g.L * g.L) * g.sig2 * g.sigma;
  *betaP = rho_s3 * (1.0 + t.sum_b_w / t.sum_disp_w);
  if (se) {
    *se = 0.0;
    const int64_t m = n < kHistoryCap ? n : kHistoryCap;
    const int64_t nb = m >= 20 ? 20 : m;
    if (nb >= 2) {
      std::vector<double> hist(2 * (size_t)m);
      CK3(cudaMemcpyAsync(hist.data(), h->history, sizeof(double) * 2 * (size_t)m,
                          cudaMemcpyDeviceToHost, h->stream));
      CK3(cudaStreamSynchronize(h->stream));
      std::vector<double> vals;
      for (int64_t b = 0; b < nb; ++b) {
        const int64_t lo = b * m / nb, hi = (b + 1) * m / nb;
        double sb = 0.0, sd = 0.0;
        for (int64_t i = lo; i < hi; ++i) {
          sb += hist[2 * i];
          sd += hist[2 * i + 1];
        }
        vals.push_back(rho_s3 * (1.0 + sb / sd));
      }
      double mean = 0.0;
      for (double v : vals) mean += v;
      mean /= (double)nb;
      double var = 0.0;
      for (double v : vals) var += (v - mean) * (v - mean);
      *se = std::sqrt(var / (double)(nb - 1) / (double)nb);
    }
  }
  return ECMC_OK;
}

int ecmc3_reset_stats(ecmc3_t h) {
  if (!h) return fail3(ECMC_ERR_ARG, "NULL handle");
  CK3(cudaMemsetAsync(h->tot, 0, sizeof(Totals3), h->stream));
  CK3(cudaMemsetAsync(h->hist_len, 0, sizeof(int64_t), h->stream));
  return ECMC_OK;
}

int ecmc3_min_distance(ecmc3_t h, double* dmin) {
  if (!h || !dmin) return fail3(ECMC_ERR_ARG, "NULL argument");
  double d2 = 0.0;
  const int rc = min_dist2_3(h, &d2);
  if (rc) return rc;
  *dmin = std::sqrt(d2);
  return ECMC_OK;
}

int ecmc3_last_cells(ecmc3_t h, int32_t* cell_of_id) {
  if (!h || !cell_of_id) return fail3(ECMC_ERR_ARG, "NULL argument");
  CK3(cudaMemcpyAsync(cell_of_id, h->cell_of, sizeof(int32_t) * (size_t)h->g.N,
                      cudaMemcpyDeviceToHost, h->stream));
  return check3(h);
}

int ecmc3_chain_records(ecmc3_t h, int32_t* out) {
  if (!h || !out) return fail3(ECMC_ERR_ARG, "NULL argument");
  if (!h->recs) return fail3(ECMC_ERR_STATE, "no sweep has run");
  CK3(cudaMemcpyAsync(out, h->recs, sizeof(int32_t) * 4 * (size_t)h->g.ncell * h->g.n_m,
                      cudaMemcpyDeviceToHost, h->stream));
  return check3(h);
}

}  // extern "C"
