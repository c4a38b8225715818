// ecmc_axis.cuh -- axis chains in cells small enough for shared memory: the
// frame of a group of cells, the static hit candidates of its members, and
// the event-chain loop that follows them.
//
// A chain moves disks along one axis only, so during a colour phase the
// coordinate b across the axis of every object of a frame (members and frozen
// images) is fixed, and two objects less than sigma apart across the axis can
// never pass each other along it.  Round a member j, divide the band
// |b_o - b_j| < sigma into three windows:
//   0: -sigma < db <= -sigma/2,   1: |db| < sigma/2,   2: sigma/2 <= db < sigma.
// Two objects of one window are less than sigma apart across (window 1) or at
// most sigma/2 (windows 0, 2), so they keep their order along the axis, and
// so does each against j: the first object ahead of j in a window, and the
// first behind, are the same for the whole phase.  That first object o1 is
// also hit before any other object o2 of its window.  With c = db / sigma,
// distances in sigma and o1, o2 not overlapping,
//   s2 - s1 >= sqrt(1 - (c1 - c2)^2) + sqrt(1 - c1^2) - sqrt(1 - c2^2) > 0
// in each window (at its corners the bound goes to 0, see below).  So a
// member's next contact in either direction lies among three objects that are
// found once per phase, and since c is fixed the square root of the hit
// distance s = max(0, b - sqrt(sigma^2 - c^2)) is found once per phase too.
// An event is then three loads, two dependent FP64 subtractions and a
// minimum, with the results of a search through the whole frame bit for bit:
// the same operands enter the same rounded operations.
//
// Rounding.  Frame coordinates are below 2^16 sigma here (frames fit in
// shared memory), so the dynamics places centres to within 2^-36 sigma, and
// loaded configurations may overlap by 5e-10 sigma (the overlap check).
//   - Pairs with c^2 < sigma^2 have sqrt(sigma^2 - c^2) >= 2^-27 sigma: a
//     mover stops well before it could pass its contact, and the sign of the
//     separation never changes.  Only a pair at exactly equal coordinates
//     along the axis is ahead in neither direction.
//   - The window bound: at the corner of a side window (|c1| = 1 - e, |c2| =
//     1/2 + g) it is sqrt(2 e) + 1.15 g > 1.4e-8 (e >= 2^-53); opposite
//     corners of window 1 (|c| = 1/2 - g) leave 2 sqrt(g).  With g >= 2^-24
//     both exceed the overlap and the rounding, also after s is clamped at 0.
// A member with an object at | |db| - sigma/2 | <= 2^-24 sigma, or at equal
// coordinates along the axis in one of its windows, searches the whole frame
// at every event instead.  (Crystals aligned with the axes; otherwise a few
// cells in 10^5 of 18 members hold such a pair, but one in 400 of 750 members,
// where a search takes four times a leg: with every member of the cell
// searching, a sweep over 384 cells of 28.6 sigma that held one took 22 ms
// instead of 6.9.)
//
// What bounds it: a chain is a serial dependence and the kernel's time is that
// of its instructions -- about 22,000 warp instructions per group of four cells
// of 18 disks, half of them in the build, at 1.5 per cycle and SM (waits for
// fixed latencies, shared memory and instruction fetch); the FP64 pipe is 43 %
// busy, HBM 1 %.  Measured on GB300, us per sweep, this kernel against the
// one that searched strips of candidates at every event (ecmc_chain.cuh):
//   N = 2^20, eta = 0.72,  240^2 cells, ell = 1.04, n_m = 2:   679 / 1140
//   N = 2^22, eta = 0.716, 484^2 cells, ell = 1.05, n_m = 2:  2577 / 6135
//   N = 2^16, eta = 0.708, 32^2 cells,  ell = 8,    n_m = 1:   319 / 1217
//   N = 256,  eta = 0.70,  2^2 cells,   ell = 4,    n_m = 2:   302 / 642
// It loses where few legs follow in a large cell: the rule is axis_pays in
// ecmc_api.cu.
#pragma once
#include <climits>

#include "ecmc_device.cuh"
#include "ecmc_internal.cuh"

namespace ecmc {

// Legs of the current chain kept for cycle detection (a power of two).
constexpr int kLegs = 32;
// Start draws made at a time (Philox runs on all lanes of a cell at once).
constexpr int kStarts = 16;
constexpr int kAxisHead = 160;      // bytes per cell: neighbours, counters, start draws
constexpr int kAxisHist = kLegs * 32;

__host__ __device__ inline int axis_al16(int v) { return (v + 15) & ~15; }
// objects of a cell: coordinates along the axis (and the two walls'), across
// it, keys
__host__ __device__ inline int axis_obj_bytes(int co) { return axis_al16(co * 20 + 16); }
// the builder's staging area of a cell, later its leg history
__host__ __device__ inline int axis_work_bytes(int co, int nbin) {
  const int st = axis_al16(co * 10 + 4 * (nbin + 1));
  return st > kAxisHist ? st : axis_al16(kAxisHist);
}
// candidate lists of mp members: 32 bytes per member and direction
__host__ __device__ inline int axis_list_bytes(int mp) { return mp * 64; }
__host__ __device__ inline int axis_flag_bytes(int mp) { return axis_al16(mp * 6); }

__host__ __device__ inline size_t axis_pass_bytes(const AxisShape& s, int cells, int co, int mp,
                                                  int fm) {
  return (size_t)kAxisHead * s.cpw + (size_t)cells * (axis_obj_bytes(co) + axis_work_bytes(co, s.nbin)) +
         (fm == 1 ? 0 : (size_t)axis_list_bytes(mp)) + axis_flag_bytes(mp);
}

// Shared memory of a warp: all its cells at their usual sizes, or one cell at
// its largest.
__host__ __device__ inline size_t axis_smem_bytes(const AxisShape& s, int fm) {
  const size_t a = axis_pass_bytes(s, s.cpw, s.co_s, s.mp_s, fm);
  const size_t b = axis_pass_bytes(s, 1, s.co_h, s.mp_h, fm);
  return a > b ? a : b;
}
// fm 1: the candidate lists live in a per-warp scratch area of global memory
__host__ __device__ inline size_t axis_scratch_bytes(const AxisShape& s) {
  return (size_t)axis_list_bytes(s.mp_s > s.mp_h ? s.mp_s : s.mp_h);
}

// Candidates of one member in one direction: sqrt(sigma^2 - c^2) of the first
// object of each window (-inf: nobody there), the three objects and, as a
// fourth, the wall (object co for +, co + 1 for -).
struct AxisEntry {
  double sq[3];
  unsigned short nb[4];
};
static_assert(sizeof(AxisEntry) == 32, "two entries are 64 bytes");

// One leg of the current chain, for the detection of cycles.
struct AxisLeg {
  double P, S;  // start along the axis, length
  double B;     // contact term (0 at a wall)
  int M;        // member * 2 + direction | how it ended | legs since the disk's last one
  int pad;
};
static_assert(sizeof(AxisLeg) == 32, "two 16-byte stores");
constexpr int kLegEntry = (1 << 20) - 1, kLegFrozen = 1 << 20, kLegWall = 1 << 21;
constexpr int kLegGap = 22, kLegGapMax = 63;

struct AxisFrame {
  double* a;                // along the axis; objects 0 .. nmem-1 are the members in
  double* b;                // bucket order, the frozen images follow; a[co], a[co+1]: walls
  int* key;                 // disk id * 16 + image (of members 4, 12: searches the frame)
  AxisEntry* list;          // [member * 2 + direction]
  int* last;                // 1 + number of the member's latest leg; 0: never in a chain
  unsigned short* rank;     // members in id order
  const int* zero;          // {0, 0}
  int* irr;                 // 1 if a member searches the frame, plus 2 for every search
  unsigned short* starts;   // start draws: [kStarts] member ranks, [kStarts] signs
  AxisLeg* leg;             // history, leg n at n mod kLegs
  int nmem, nobj, co;
};

// The kernel runs at the rate its instructions arrive: with every path inlined
// it has 160 KB of code and loses a third of its speed, so what runs rarely
// is kept out of line.

// Whole-frame search of a cell without static candidates, by the lanes of its
// group: the first contact of the mover at (P, Q) as the general search of
// ecmc_chain.cuh finds it.  Returns the object (-1: none) with its distance
// and square root on every lane.
struct AxisStop {
  double s, q;
  int j;
};
template <int TPC>
__device__ __noinline__ AxisStop axis_search(const double* a, const double* b, const int* key,
                                             int nobj, int m, double P, int dir, double sig2,
                                             int sub, unsigned gmask) {
  AxisStop best;
  best.s = __longlong_as_double(0x7ff0000000000000ll);
  best.q = 0.0;
  best.j = -1;
  const double Q = b[m];
#pragma unroll 1
  for (int j = sub; j < nobj; j += TPC) {
    if (j == m) continue;
    const double d = flip_if(a[j] - P, dir != 0), db = b[j] - Q;
    const double c2 = db * db;
    if (!(dbits(d) > 0 && lt_nn(c2, sig2))) continue;
    const double q = sqrt_rn(sig2 - c2);
    const double s = clamp0(d - q);
    if (best.j < 0 || lt_nn(s, best.s) ||
        (dbits(s) == dbits(best.s) && key[j] < key[best.j])) {
      best.s = s;
      best.q = q;
      best.j = j;
    }
  }
#pragma unroll 1
  for (int o = 1; o < TPC; o <<= 1) {
    const double os = __shfl_xor_sync(gmask, best.s, o), oq = __shfl_xor_sync(gmask, best.q, o);
    const int oj = __shfl_xor_sync(gmask, best.j, o);
    if (oj < 0) continue;
    if (best.j < 0 || lt_nn(os, best.s) ||
        (dbits(os) == dbits(best.s) && key[oj] < key[best.j])) {
      best.s = os;
      best.q = oq;
      best.j = oj;
    }
  }
  return best;
}

// The lane of the quad whose candidate comes first by exact distance (equal
// distances: the smaller key; the wall, lane 3, last).
__device__ __noinline__ int axis_tie(double s, int key, unsigned gmask) {
  int w = (int)(threadIdx.x & 3);
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    const double os = __shfl_xor_sync(gmask, s, o);
    const int ok = __shfl_xor_sync(gmask, key, o), ow = __shfl_xor_sync(gmask, w, o);
    if (lt_nn(os, s) || (dbits(os) == dbits(s) && ok < key)) {
      s = os;
      key = ok;
      w = ow;
    }
  }
  return w;
}

__device__ __noinline__ U64x4 axis_philox(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                          uint64_t k0, uint64_t k1) {
  return philox(c0, c1, c2, c3, k0, k1);
}

// The draws of chains k .. k + kStarts - 1 of a cell, by the lanes of its group.
template <int TPC>
__device__ __noinline__ void axis_draws(unsigned short* starts, int k, int n_m, int nmem,
                                        int dir_mode, int64_t t, int lc, uint64_t seed,
                                        uint64_t replica, int sub) {
#pragma unroll 1
  for (int i = sub; i < kStarts && k + i < n_m; i += TPC) {
    const U64x4 v = axis_philox((uint64_t)t, kPurposeChain, (uint64_t)lc, (uint64_t)(k + i), seed,
                                replica);
    starts[i] = (unsigned short)below_n(v.v[0], (uint64_t)nmem);
    starts[kStarts + i] = dir_mode == 1 ? 0 : (unsigned short)(v.v[1] >> 63);
  }
}

// Cycle replay (the argument is in ecmc_chain.cuh, replay_cycle): if after a
// turn-back the configuration equals the one K legs earlier, the next legs
// repeat those K legs until the budget runs out.  K is the distance to one of
// the last TPC turn-backs, after which the mover, its direction and its
// position were the same bit for bit (each lane of the group compares one of
// them, kept in its registers); the lanes then share the check that every
// other disk moved in those legs is back where its first leg among them
// started.  n_tot numbers the legs of the cell; the last kLegs of them are in
// the history.
template <int TPC>
__device__ __forceinline__ bool axis_cycle_holds(const AxisFrame& f, int sub, int n_tot, int K,
                                                 int m) {
  bool same = true;  // as far as this lane's legs go
#pragma unroll 1
  for (int i = sub; i < K; i += TPC) {
    const AxisLeg& l = f.leg[(n_tot - K + i) & (kLegs - 1)];
    const int D = (l.M & kLegEntry) >> 1;
    if (D != m && (l.M >> kLegGap) > i) same &= dbits(f.a[D]) == dbits(l.P);
  }
  return same;
}

// Whole cycles at once.  While r stays in one binade [2^e, 2^(e+1)), with
// G = 2^(e-52) its unit in the last place, the rounded subtraction r - s takes
// exactly S = s / G rounded to an integer off r / G, unless s / G lies half way
// between two integers or the result leaves the binade.  So c cycles of K legs
// take c sum(S) off as long as more than 2^52 is left.  c is an FP32 estimate
// from below, checked in integers.  Returns the budget after them in .s and c
// in .j.  The lanes of the group share the legs.
template <int TPC>
__device__ __noinline__ AxisStop axis_jump(const AxisLeg* leg, unsigned gmask, int gshift, int sub,
                                           int base, int K, int legs_left, double r) {
  constexpr unsigned long long kOne = 1ull << 52;
  const unsigned long long rb = (unsigned long long)dbits(r);
  const int er = (int)(rb >> 52);
  const unsigned long long R = rb & (kOne - 1);  // r / G - 2^52
  unsigned long long sum = 0;
  bool good = er > 0 && er < 0x7ff;
#pragma unroll 1
  for (int i = sub; i < K; i += TPC) {
    const unsigned long long u = (unsigned long long)dbits(leg[(base + i) & (kLegs - 1)].S);
    const int es = (int)(u >> 52);
    const unsigned long long M = (u & (kOne - 1)) | kOne;
    const int sh = er - es;
    if (es == 0 || sh >= 54) continue;  // below half a unit of r
    if (sh <= 0) {
      good = false;  // s as long as r: no whole cycle fits
    } else {
      const unsigned long long rem = M & ((1ull << sh) - 1), half = 1ull << (sh - 1);
      good &= rem != half;
      sum += (M >> sh) + (rem > half ? 1 : 0);
    }
  }
  // lanes from K on hold nothing: sum the first ones and spread the result
#pragma unroll 1
  for (int o = 1; o < TPC && o < K; o <<= 1) sum += __shfl_xor_sync(gmask, sum, o);
  if (TPC > 1) sum = __shfl_sync(gmask, sum, gshift);
  good = __all_sync(gmask, good);
  AxisStop res;
  res.s = r;
  res.q = 0.0;
  res.j = 0;
  if (good && sum > 0) {
    // one cycle less than fits, so that every result stays above 2^52
    const float est = __ull2float_rz(R) / __ull2float_rz(sum) * (1.0f - 0x1p-20f) - 1.5f;
    const int most = legs_left / K - 1;
    int c = est < (float)most ? (int)est : most;
    if (c > 0 && (unsigned long long)c * sum < R) {
      res.s = __longlong_as_double((long long)(rb - (unsigned long long)c * sum));
      res.j = c;
    }
  }
  return res;
}

// len: the length of one cycle; cyc_walls, cyc_frozen: its turn-backs.
template <int TPC>
__device__ __forceinline__ void axis_replay(const AxisFrame& f, unsigned gmask, int gshift,
                                            int sub, int Kf, float len, int cyc_walls,
                                            int cyc_frozen, int tot0, int& n_tot, int& em,
                                            double& P, double& r, double& sum_b, int& n_frozen,
                                            int& n_walls, int& n_replayed) {
  const int base = n_tot - Kf;
  const int legs_left = (int)kMaxEventsPerChain - (n_tot - tot0);
  // a jump costs about as much as eight legs, one per binade of r
  const float worth = 24.0f * len / (float)Kf;
  int binade = -1, o = 0, cycles = 0, n = 0;
  const AxisLeg* l = &f.leg[base & (kLegs - 1)];
  double sl = l->S, ab = l->B;
#pragma unroll 1
  for (;;) {
    if (o == 0) {
      const int e = __double2hiint(r) >> 20;
      if (e != binade && to_float_trunc(r) > worth) {
        binade = e;
        const AxisStop js =
            axis_jump<TPC>(f.leg, gmask, gshift, sub, base, Kf, legs_left - n, r);
        if (js.j > 0) {
          r = js.s;
          cycles += js.j;
          n += js.j * Kf;
          double cyc_b = 0.0;
#pragma unroll 1
          for (int i = 0; i < Kf; ++i) cyc_b += f.leg[(base + i) & (kLegs - 1)].B;
          sum_b += (double)js.j * cyc_b;
        }
      }
    }
    if (le_nn(r, sl) || n >= legs_left) break;
    r = r - sl;
    sum_b += ab;
    ++n;
    if (++o == Kf) {
      o = 0;
      ++cycles;
    }
    l = &f.leg[(base + o) & (kLegs - 1)];
    sl = l->S;
    ab = l->B;
  }
  n_tot += n;
  n_replayed += n;
  n_walls += cycles * cyc_walls;
  n_frozen += cycles * cyc_frozen;
  em = l->M & kLegEntry;
  P = l->P;
  // the first o legs were run once more: their turn-backs, and the disks that
  // stopped stand where they left them (written in the order of the legs; the
  // lanes form the ends of TPC legs together)
  int turns = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < o; i0 += TPC) {
    const int i = i0 + sub;
    const AxisLeg& q = f.leg[(base + (i < o ? i : 0)) & (kLegs - 1)];
    const int M = i < o ? q.M : kLegEntry;
    const double end = q.P + flip_if(q.S, (M & 1) != 0);
    const int D = i < o && (M & (kLegWall | kLegFrozen)) == 0 ? (M & kLegEntry) >> 1 : -1;
    turns += i < o ? ((M & kLegWall) ? 1 : 0) + ((M & kLegFrozen) ? 0x10000 : 0) : 0;
#pragma unroll 1
    for (int k = 0; k < TPC && i0 + k < o; ++k) {
      if (k == sub && D >= 0) f.a[D] = end;
      __syncwarp(gmask);
    }
  }
#pragma unroll 1
  for (int k = 1; k < TPC && k < o; k <<= 1) turns += __shfl_xor_sync(gmask, turns, k);
  if (TPC > 1 && o > 0) turns = __shfl_sync(gmask, turns, gshift);
  n_walls += turns & 0xffff;
  n_frozen += turns >> 16;
}

// The start list without replacement (the negative control of Sec. 3.4), as
// shuffled_list in ecmc_chain.cuh: entry 0 the member drawn for chain 0, then
// the others shuffled by Fisher-Yates from the top.
__device__ __noinline__ void axis_shuffled_list(int* pl, int n, int first, int64_t t, int lc,
                                                uint64_t seed, uint64_t replica) {
  int q = 0;
  pl[0] = first;
#pragma unroll 1
  for (int i = 0; i < n; ++i)
    if (i != first) pl[++q] = i;
  U64x4 u;
  int cur = -1;
#pragma unroll 1
  for (int i = n - 1; i >= 2; --i) {
    if ((i >> 2) != cur) {
      cur = i >> 2;
      u = axis_philox((uint64_t)t, kPurposeShuffle, (uint64_t)lc, (uint64_t)cur, seed, replica);
    }
    const int j = 1 + (int)below_n(u.v[i & 3], (uint64_t)i);
    const int a = pl[i];
    pl[i] = pl[j];
    pl[j] = a;
  }
}

// The chains of the warp's cells (Sec. 3.4 steps 5-6) and their statistics.
// run: this lane group has a cell in this pass; irregular: some of its members
// search their whole frame.
//
// One turn of the loop is one leg of every running chain of the warp.  Its
// length is a chain of dependent operations: two loads, two FP64 additions,
// the minimum over the candidates; so with four lanes or more per cell each
// lane of a quad takes one candidate (three objects and the wall), the
// minimum compares the high words of the four distances (two shuffle rounds;
// an exact comparison only when the two smallest agree in 29 bits), and one
// FP64 addition forms the mover's end, the budget left and the contact sum on
// three lanes.  An FP64 instruction of a warp takes its scheduler's unit for
// 57 cycles, whatever the number of lanes.  The lanes of one group hold the
// same chain state, but the contact sum is kept on lane 2 of each quad, and
// what a group keeps in memory (coordinates, latest legs, history, undo log)
// is written by its first lane.  Votes and shuffles order no memory: a
// __syncwarp stands wherever other lanes read or write the same words.
template <int TPC, bool REJECT>
__device__ __forceinline__ void axis_chains(const AxisFrame& f, const Geom& g, int64_t t,
                                            int lc, int c, bool run, bool irregular,
                                            CellStats* __restrict__ cs,
                                            ChainRec* __restrict__ recs, int rec_stride,
                                            int replay, int* err) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool QUAD = TPC >= 4;
  const int lane = threadIdx.x & 31;
  const int sub = lane & (TPC - 1), gi = lane / TPC;
  const int q4 = lane & 3, quad0 = lane & ~3;
  constexpr unsigned GM = TPC == 32 ? FULL : (1u << (TPC & 31)) - 1u;
  const int gshift = gi * TPC;
  const unsigned gmask = GM << gshift;
  const double INF = __longlong_as_double(0x7ff0000000000000ll);
  const int nmem = run ? f.nmem : 0;
  const int n_m = g.n_m;
  const bool shuffled = g.list_mode == 1;
  const bool keep_legs = replay && !REJECT && !shuffled;
  const double sig2 = g.sig2, ell = g.ell;

  // the candidate of this lane: lane 3 takes the wall, with 0 for the square
  // root (a[co + 1] is 0)
  const unsigned char* const list = (const unsigned char*)f.list;
  const unsigned char* const sq_base =
      QUAD && q4 == 3 ? (const unsigned char*)(f.a + f.co + 1) : list + (QUAD ? q4 * 8 : 0);
  const int sq_stride = QUAD && q4 == 3 ? 0 : 32;
  // a group without chains reads index 0
  const unsigned char* const nb_base =
      nmem > 0 ? list + 24 + (QUAD ? q4 * 2 : 0) : (const unsigned char*)f.zero;

  double sum_b = 0.0, ch_b = 0.0;  // QUAD: on lane 2 of each quad
  int n_tot = 0, n_frozen = 0, n_walls = 0, n_chains = 0, n_replayed = 0;
  int n_undo = 0, n_rejected = 0;
  int k = 0;
  bool active = false;
  int em = 0, tot0 = 0, start_key = 0, wall0 = 0;
  double P = 0.0, r = 0.0, z = 0.0;
  int moved = -1;  // QUAD: the disk the last leg stopped, its end still in z
  // the state after one of the chain's last TPC turn-backs (one per lane)
  int t_em = -1, t_tot = 0, t_walls = 0, t_frozen = 0, n_turn = 0;
  double t_P = 0.0;
  float t_r = 0.0f;
  int gap = 0;  // legs since the mover's previous one (first lane)

  // Everything that needs the lanes of a group to work together is done by
  // the whole warp, for all the groups it concerns: collectives on part of a
  // warp would make its groups run one after the other.
  bool need = nmem > 0, starting = true;  // a group wants its next chain; any does
  const bool any_irregular = __any_sync(FULL, irregular);
#pragma unroll 1
  for (;;) {
    if (starting) {
      __syncwarp();
      if (!REJECT) {
        if (need && active && sub == 0) f.a[em >> 1] = P;  // where the last chain ended
        __syncwarp();
      }
      const bool go = need && k < n_m;
      const bool refill = go && (k & (kStarts - 1)) == 0;
      if (__any_sync(FULL, refill)) {
        if (refill)
          axis_draws<TPC>(f.starts, k, n_m, nmem, g.dir_mode, t, lc, g.seed, g.replica, sub);
        __syncwarp();
        // the list takes the room of the leg history
        if (refill && shuffled && k == 0 && sub == 0)
          axis_shuffled_list((int*)f.leg, nmem, f.starts[0], t, lc, g.seed, g.replica);
        __syncwarp();
      }
      if (need) active = go;
      need = false;
      if (go) {
        int idx = f.starts[k & (kStarts - 1)];
        if (shuffled) idx = ((const int*)f.leg)[k % nmem];
        const int m = f.rank[idx];
        em = m * 2 + f.starts[kStarts + (k & (kStarts - 1))];
        P = f.a[m];
        r = ell;
        if (REJECT) {
          if (sub == 0) {
            UndoEntry& u = g.undo[(int64_t)c * g.undo_stride];
            u.a = P;
            u.m = m;
            u.touched = f.last[m];
          }
          n_undo = 1;
          ch_b = 0.0;
        }
        gap = kLegGapMax;
        if (sub == 0) f.last[m] = n_tot + 1;
        start_key = f.key[m];
        tot0 = n_tot;
        wall0 = n_walls;
        t_em = -1;
        ++k;
        ++n_chains;
      }
      if (!__any_sync(FULL, active)) break;
      starting = false;
    }
    __syncwarp();  // lanes read what others of their group wrote
    const int dir = em & 1;
    // the first stop ahead: at distance s object bj at aw (the wall: bj >= co),
    // contact term bq
    double s, aw, bq;
    int bj;
    bool tie;
    if (QUAD) {
      const int j = *(const unsigned short*)(nb_base + em * 32);
      const double q = *(const double*)(sq_base + em * sq_stride);
      const double A = f.a[j];
      const double b = flip_if(A - P, dir != 0);
      const double d = b - q;
      // the previous leg's results, if it passed the chain on: they were
      // still on their way when this one's loads were issued (its candidates
      // lie ahead, so the stopped disk is not among them)
      const double rz = __shfl_sync(FULL, z, quad0 + 1);
      if (any_irregular) __syncwarp();  // (there it may be: the search decides)
      if (moved >= 0) {
        r = rz;
        if (sub == 0) f.a[moved] = z;
        moved = -1;
      }
      const bool neg = dbits(d) < 0;
      const double sl = neg ? 0.0 : d;
      const double bl = neg ? b : q;  // b - s
      const unsigned v = ((unsigned)__double2hiint(sl) & ~3u) | (unsigned)q4;
      const unsigned v1 = __shfl_xor_sync(FULL, v, 1);
      const unsigned lo = v < v1 ? v : v1, hi = v < v1 ? v1 : v;
      const unsigned lo2 = __shfl_xor_sync(FULL, lo, 2), hi2 = __shfl_xor_sync(FULL, hi, 2);
      const unsigned first = lo < lo2 ? lo : lo2;
      const unsigned up = lo < lo2 ? lo2 : lo, hm = hi < hi2 ? hi : hi2;
      const unsigned second = up < hm ? up : hm;
      tie = (first ^ second) < 4u;
      int src = quad0 | (int)(first & 3u);
      if (tie) {
        src = quad0 | axis_tie(sl, q4 == 3 ? INT_MAX : f.key[j], gmask);
      }
      s = __shfl_sync(FULL, sl, src);
      aw = __shfl_sync(FULL, A, src);
      bq = __shfl_sync(FULL, bl, src);
      bj = __shfl_sync(FULL, j, src);
    } else {
      // all four candidates on every lane
      s = INF;
      aw = bq = 0.0;
      bj = f.co + dir;
      int bk = INT_MAX;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int j = *(const unsigned short*)(nb_base + em * 32 + 2 * w);
        const double q = w == 3 ? 0.0 : *(const double*)(sq_base + em * 32 + 8 * w);
        const double A = f.a[j];
        const double b = flip_if(A - P, dir != 0);
        const double d = b - q;
        const bool neg = dbits(d) < 0;
        const double sl = neg ? 0.0 : d;
        bool take = lt_nn(sl, s);
        if (dbits(sl) == dbits(s) && w < 3 && dbits(s) != dbits(INF)) take = f.key[j] < bk;
        if (take) {
          s = sl;
          bq = neg ? b : q;
          aw = A;
          bj = j;
          bk = w < 3 ? f.key[j] : INT_MAX;
        }
      }
    }
    if (any_irregular) __syncwarp();
    if (irregular && active && (f.key[em >> 1] & 8)) {
      if (sub == 0) *f.irr += 2;
      const AxisStop st = axis_search<TPC>(f.a, f.b, f.key, f.nobj, em >> 1, P, dir, sig2, sub,
                                           gmask);
      const double wall = f.a[f.co + dir];
      s = clamp0(flip_if(wall - P, dir != 0));
      aw = wall;
      bj = f.co + dir;
      bq = 0.0;
      if (st.j >= 0 && le_nn(st.s, s)) {
        s = st.s;
        aw = f.a[st.j];
        bj = st.j;
        bq = dbits(s) == 0 ? flip_if(aw - P, dir != 0) : st.q;
      }
    }
    // event decision: the budget's end before a contact before the wall
    const bool is_end = le_nn(r, s);
    const bool is_wall = bj >= f.co;
    const bool is_lift = !is_end && bj < nmem;
    const double step = is_end ? r : s;
    const double addb = (is_end || is_wall) ? 0.0 : bq;
    double Pnew, rnew;
    if (QUAD) {
      // P +- step, r - step and the contact sum with one FP64 addition
      const double x = q4 == 0 ? P : (q4 == 1 ? r : (REJECT ? ch_b : sum_b));
      const double y = q4 == 0 ? flip_if(step, dir != 0)
                               : (q4 == 1 ? flip_if(step, true) : (active ? addb : 0.0));
      z = x + y;
      if (REJECT) ch_b = z;
      else sum_b = z;
    } else {
      Pnew = P + flip_if(step, dir != 0);
      rnew = r - step;
      if (active) {
        if (REJECT) ch_b += addb;
        else sum_b += addb;
      }
    }
    const int m = em >> 1;
    if (TPC == 2) __syncwarp();  // both lanes have read the mover's coordinate
    if (active && keep_legs && !is_end && sub == 0) {
      AxisLeg q;
      q.P = P;
      q.S = step;
      q.B = addb;
      q.M = em | (is_lift ? 0 : (is_wall ? kLegWall : kLegFrozen)) | (gap << kLegGap);
      q.pad = 0;
      int4* const at = (int4*)&f.leg[n_tot & (kLegs - 1)];
      at[0] = ((const int4*)&q)[0];
      at[1] = ((const int4*)&q)[1];
    }
    const bool slow = active && !is_lift;
    if (active && is_lift) {
      // the hit member carries on with the rest of the budget
      ++n_tot;
      if (QUAD) {
        moved = m;
      } else {
        if (sub == 0) f.a[m] = Pnew;
        r = rnew;
      }
      em = bj * 2 + dir;
      P = aw;
      int latest = 0;
      if (sub == 0) latest = f.last[bj];
      if (REJECT) {
        if (sub == 0) {
          if (n_undo < g.cap_mem) {
            UndoEntry& u = g.undo[(int64_t)c * g.undo_stride + n_undo];
            u.a = P;
            u.m = bj;
            u.touched = latest;
          } else {
            atomicCAS(err, DEV_OK, DEV_CAPACITY);
          }
        }
        ++n_undo;
      }
      const int back = n_tot + 1 - latest;  // n_tot + 1 if it never moved
      gap = back < kLegGapMax ? back : kLegGapMax;
      if (sub == 0) f.last[bj] = n_tot + 1;
    }
    if (!__any_sync(FULL, slow)) continue;

    // turn-backs and chain ends
    if (REJECT) __syncwarp();
    if (QUAD) {
      Pnew = __shfl_sync(FULL, z, quad0);
      rnew = __shfl_sync(FULL, z, quad0 + 1);
    }
    bool turned = false;
    if (slow) {
      r = rnew;
      P = is_wall && !is_end ? aw : Pnew;
      need = is_end;
      if (is_end) {
        if (REJECT && sub == 0) f.a[m] = P;
        if (REJECT) sum_b += ch_b;
      } else {
        ++n_tot;
        n_walls += is_wall ? 1 : 0;
        n_frozen += is_wall ? 0 : 1;
        if (REJECT) {
          // every disk the chain moved returns to its position at the start
          // (a straight chain moves each disk once, in any order)
          const int n = n_undo < g.cap_mem ? n_undo : g.cap_mem;
#pragma unroll 1
          for (int e = sub; e < n; e += TPC) {
            const UndoEntry& u = g.undo[(int64_t)c * g.undo_stride + e];
            f.a[u.m] = u.a;
            f.last[u.m] = u.touched;
          }
          ++n_rejected;
          need = true;
        } else {
          // frozen disk or wall: the chain turns back along its axis
          em ^= 1;
          turned = keep_legs;
          gap = 1;
          if (sub == 0) f.last[m] = n_tot + 1;
        }
      }
    }
    if (!REJECT) {
      const unsigned match =
          __ballot_sync(FULL, turned && t_em == em && dbits(t_P) == dbits(P) &&
                                  n_tot - t_tot <= kLegs);
      if (match) {
        __syncwarp();
        unsigned mine = (match >> gshift) & GM;
        bool cyc = mine != 0;
        // the latest of the matching turn-backs: turn n lives on lane n mod TPC
        const int s0 = n_turn & (TPC - 1);
        mine = (mine << ((TPC - s0) & 31) | mine >> s0) & GM;
        const int l = cyc ? (31 - __clz((int)mine) + s0) & (TPC - 1) : 0;
        const int K = n_tot - __shfl_sync(FULL, t_tot, gshift + l);
        const float len = __shfl_sync(FULL, t_r, gshift + l) - to_float_trunc(r);
        const int cw = n_walls - __shfl_sync(FULL, t_walls, gshift + l);
        const int cf = n_frozen - __shfl_sync(FULL, t_frozen, gshift + l);
        const bool same = !cyc || axis_cycle_holds<TPC>(f, sub, n_tot, K, em >> 1);
        const unsigned differ = __ballot_sync(FULL, !same);
        cyc = cyc && ((differ >> gshift) & GM) == 0;
        __syncwarp();  // the comparison has read what the replay writes
        if (cyc) {
          axis_replay<TPC>(f, gmask, gshift, sub, K, len, cw, cf, tot0, n_tot, em, P, r, sum_b,
                           n_frozen, n_walls, n_replayed);
          t_em = -1;
          // the legs before the jump are no longer in the history
          gap = kLegGapMax;
        }
      }
      if (turned) {
        if ((n_turn & (TPC - 1)) == sub) {
          t_em = em;
          t_P = P;
          t_r = to_float_trunc(r);
          t_tot = n_tot;
          t_walls = n_walls;
          t_frozen = n_frozen;
        }
        ++n_turn;
      }
    }
    if (slow && n_tot - tot0 >= (int)kMaxEventsPerChain) {
      atomicCAS(err, DEV_OK, DEV_CHAIN_CAP);
      if (REJECT && !need && sub == 0) f.a[em >> 1] = P;
      need = true;
    }
    if (need && recs != nullptr && sub == 0) {
      ChainRec rc;
      rc.start_id = start_key >> 4;
      rc.end_id = f.key[em >> 1] >> 4;
      rc.walls = n_walls - wall0;
      rc.events = n_tot - tot0 - rc.walls;
      recs[(int64_t)c * rec_stride + (k - 1)] = rc;
    }
    starting = __any_sync(FULL, need);
  }
  __syncwarp();
  if (QUAD) sum_b = __shfl_sync(FULL, sum_b, quad0 + 2);
  if (run && sub == 0) {
    CellStats s;
    s.sum_b = sum_b;
    s.events = n_tot - n_walls;
    s.lifts = n_tot - n_walls - n_frozen;
    s.frozen = n_frozen;
    s.walls = n_walls;
    // for every leg that was not replayed, the last legs of the chains among
    // them: the three windows' candidates (whether or not an object is there),
    // and every other object of the frame where that was searched
    const long long legs = (long long)n_tot - n_replayed + n_chains - n_rejected;
    s.fp64_evals = 3 * legs + (long long)(*f.irr >> 1) * (f.nobj - 1);
    s.chains = n_chains;
    s.n_mem = nmem;
    s.replayed = n_replayed;
    s.rejected = n_rejected;
    cs[c] = s;
  }
}

// One warp's memory for a pass over `cells` of its cells, frames of up to co
// objects each and mp members in all.
struct AxisPass {
  int obj_off, work_off, memb_off, flag_off, co;
};
__device__ __forceinline__ AxisPass axis_pass(const AxisShape& s, int cells, int co, int mp,
                                              bool lists_in_smem) {
  AxisPass p;
  p.co = co;
  p.obj_off = kAxisHead * s.cpw;
  p.work_off = p.obj_off + cells * axis_obj_bytes(co);
  p.memb_off = p.work_off + cells * axis_work_bytes(co, s.nbin);
  p.flag_off = p.memb_off + (lists_in_smem ? axis_list_bytes(mp) : 0);
  return p;
}

struct AxisHead {
  int nq[9];    // neighbour cells of the 3x3 block
  int pre[10];  // prefix sums of their disk counts (the centre and repeats count 0)
  int cnt;      // objects of the frame
  int ovf;      // more of them than this pass allows
  int irr;      // AxisFrame::irr
  int zero[2];
};
static_assert(sizeof(AxisHead) + 4 * kStarts <= kAxisHead, "head of a cell");

__device__ __forceinline__ unsigned long long abs_bits(double v) {
  return (unsigned long long)dbits(v) & 0x7fffffffffffffffull;
}

// v - o in the cell's frame: the periodic wrap into [-L/2, L/2), one FP64
// addition unless it wraps
__device__ __forceinline__ double axis_diff(double v, double o, double L, double hL) {
  double r = v - o;
  if (abs_bits(r) >= abs_bits(hL)) {  // outside (-L/2, L/2)
    if (dbits(r) >= 0) r = r - L;
    else if (abs_bits(r) != abs_bits(hL)) r = r + L;
  }
  return r;
}

// -sigma < v < top (top > 0)
__device__ __forceinline__ bool axis_within(double v, double sigma, double top) {
  return abs_bits(v) < abs_bits(dbits(v) < 0 ? sigma : top);
}

// Screens off the usual path: boxes of two or four cells per side on box
// coordinates (wide), and the FP64 placement itself (exact).
__device__ __noinline__ bool axis_screen(double x, double y, double ox, double oy, const Geom& g,
                                         bool exact) {
  const double L = g.L, hL = 0.5 * L, sigma = g.sigma, wl = g.w + g.sigma, hl = g.h + g.sigma;
  bool kx = false, ky = false;
  if (exact) {
    const double X = axis_diff(x, ox, L, hL), Y = axis_diff(y, oy, L, hL);
#pragma unroll 1
    for (int m = -1; m <= 1; ++m) {
      const double Xk = m == 0 ? X : X + flip_if(L, m < 0);
      const double Yk = m == 0 ? Y : Y + flip_if(L, m < 0);
      kx |= axis_within(Xk, sigma, wl);
      ky |= axis_within(Yk, sigma, hl);
    }
    return kx && ky;
  }
  // |error| < 4 * 2^-23 L
  const float Lf = (float)L, mf = 0x1p-20f * Lf;
  const float X = to_float_trunc(x) - to_float_trunc(ox);
  const float Y = to_float_trunc(y) - to_float_trunc(oy);
  const float lo = -(float)sigma * 1.0000002f - mf;
  const float xhi = (float)wl * 1.0000002f + mf, yhi = (float)hl * 1.0000002f + mf;
#pragma unroll 1
  for (int m = -1; m <= 1; ++m) {
    kx |= X + m * Lf > lo && X + m * Lf < xhi;
    ky |= Y + m * Lf > lo && Y + m * Lf < yhi;
  }
  return kx && ky;
}

// The images of object i (boxes of two or four cells per side): object i
// becomes the first one that lies in the frame, or moves out of reach; the
// others are appended.
constexpr double kAxisFar = 1e30;
__device__ __noinline__ void axis_images(double* a, double* b, int* key, int* cnt, int* ovf, int i,
                                         int co, int axis, const Geom& g) {
  const double L = g.L, sigma = g.sigma, wl = g.w + g.sigma, hl = g.h + g.sigma;
  const double X0 = axis == 0 ? a[i] : b[i], Y0 = axis == 0 ? b[i] : a[i];
  const int id16 = key[i] & ~15;
  double X = kAxisFar, Y = kAxisFar;
  bool first = true;
#pragma unroll 1
  for (int k = 0; k < 9; ++k) {
    const int kx = k / 3 - 1, ky = k % 3 - 1;
    const double Xk = kx == 0 ? X0 : X0 + flip_if(L, kx < 0);
    const double Yk = ky == 0 ? Y0 : Y0 + flip_if(L, ky < 0);
    if (!axis_within(Xk, sigma, wl) || !axis_within(Yk, sigma, hl)) continue;
    if (first) {
      X = Xk;
      Y = Yk;
      key[i] = id16 + k;
      first = false;
      continue;
    }
    const int j = atomicAdd(cnt, 1);
    if (j >= co) {
      *ovf = 1;
      continue;
    }
    a[j] = axis == 0 ? Xk : Yk;
    b[j] = axis == 0 ? Yk : Xk;
    key[j] = id16 + k;
  }
  a[i] = axis == 0 ? X : Y;
  b[i] = axis == 0 ? Y : X;
}

// The first objects ahead of and behind member j in its window w, decided in
// FP64, among the sorted objects p0 .. p1 - 1: the first | the second << 16
// (j: nobody), and bit 31 when j has no static candidates.
__device__ __noinline__ unsigned axis_scan_exact(const double* a, const double* b,
                                                 const unsigned short* si, int p0, int p1, int j,
                                                 int w, double sigma, double sig2) {
  unsigned none = 0;
  const double half = 0.5 * sigma, guard = 0x1p-24 * sigma;
  const double aj = a[j], bj = b[j];
  int jp = j, jm = j;
#pragma unroll 1
  for (int p = p0; p < p1; ++p) {
    const int o = si[p];
    if (o == j) continue;
    const double d = b[o] - bj, d1 = fabs(d), ao = a[o];
    if (dlt(fabs(d1 - half), guard)) none = 0x80000000u;
    const bool in = w == 1 ? dlt(d1, half)
                           : (!dlt(d1, half) && lt_nn(d * d, sig2) && (dbits(d) >= 0) == (w == 2));
    if (!in) continue;
    if (dlt(aj, ao)) {
      if (jp == j || dlt(ao, a[jp])) jp = o;
    } else if (dlt(ao, aj)) {
      if (jm == j || dlt(a[jm], ao)) jm = o;
    } else {
      none = 0x80000000u;
    }
  }
  return (unsigned)jp | (unsigned)jm << 16 | none;
}

// Build the frames of the warp's cells of one pass: each lane group of TPC
// lanes places its own cell (act: it has one), all groups in step.  exact:
// screen with the FP64 placement itself (a frame near its capacity must count
// true images only).  On return h.ovf / h.irr are set and f.nmem, f.nobj
// filled in.  Positions are read through L2: other SMs move disks meanwhile.
//
// A frame holds the members and the disks of the eight neighbour cells within
// sigma of the cell.  The screen reads the disks' FP32 coordinates relative
// to their own cell (rel; written by the binning and kept up by the
// write-back): the neighbour's offset makes them relative to this one, with
// no wrap.  Four rounds of its loads are in flight at once, as are those of
// the placements: a build waits for few L2 round trips.  Boxes of
// two or four cells per side, where a disk may have several images, screen
// the box coordinates instead.
template <int TPC>
__device__ __forceinline__ void axis_build(AxisFrame& f, AxisHead& h, unsigned char* stage,
                                           const AxisPass& pass, int nbin, const Geom& g,
                                           const SweepState* __restrict__ st, int cx, int cy,
                                           int c, int cap, int nc, bool act, bool exact,
                                           const double* __restrict__ px,
                                           const double* __restrict__ py,
                                           const int* __restrict__ pid,
                                           const float2* __restrict__ rel,
                                           const int* __restrict__ cnt) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr unsigned GM = TPC == 32 ? FULL : (1u << (TPC & 31)) - 1u;
  const int lane = threadIdx.x & 31;
  const int sub = lane & (TPC - 1), gshift = lane & ~(TPC - 1);
  const int co = pass.co;
  const int axis = st->axis;
  const double L = g.L, sigma = g.sigma, hL = 0.5 * L;
  const double ox = st->sx + (double)cx * g.w;
  const double oy = st->sy + (double)cy * g.h;
  const double wl = g.w + sigma, hl = g.h + sigma;
  const bool wide = g.cells_x < 6 || g.cells_y < 6;

  // the neighbour cells and the prefix sums of their disk counts: their disks
  // are visited as one index range
  const bool fits = act && nc <= co;
#pragma unroll 1
  for (int e = sub; e < 9; e += TPC) {
    const int dx = e % 3 - 1, dy = e / 3 - 1;
    int qx = cx + dx, qy = cy + dy;
    qx += qx < 0 ? g.cells_x : (qx >= g.cells_x ? -g.cells_x : 0);
    qy += qy < 0 ? g.cells_y : (qy >= g.cells_y ? -g.cells_y : 0);
    const int q = g.cell_off + qy * g.cells_x + qx;
    int n = fits && e != 4 ? min(cnt[q], cap) : 0;
    // two cells per side: the left and the right neighbour are one cell
    if ((dx == 1 && g.cells_x == 2) || (dy == 1 && g.cells_y == 2)) n = 0;
    h.nq[e] = q;
    h.pre[e] = n;
  }
  if (sub == 0) {
    h.zero[0] = h.zero[1] = 0;
    h.ovf = act && nc > co ? 1 : 0;
    h.irr = 0;
  }
  f.zero = h.zero;
  f.irr = &h.irr;
  __syncwarp();
  int T = 0;
  {
    int n[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) n[e] = h.pre[e];
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      if ((e & (TPC - 1)) == sub) h.pre[e] = T;
      T += n[e];
    }
    if (sub == 0) h.pre[9] = T;
  }
  __syncwarp();

  // screen; the margin is above the FP32 error: 2^-21 (L + w) of rel (see the
  // binning) and its sum.  Survivors leave their bucket slots in key[].
  int ns = fits ? nc : 0;
  {
    const float Lf = (float)L, wf = (float)g.w, hf = (float)g.h;
    const float mx = 0x1p-20f * (Lf + wf), my = 0x1p-20f * (Lf + hf);
    const float xlo = -(float)sigma * 1.0000002f - mx, xhi = (float)wl * 1.0000002f + mx;
    const float ylo = -(float)sigma * 1.0000002f - my, yhi = (float)hl * 1.0000002f + my;
    const bool slow = wide || exact;
    constexpr int U = 4;
    int e = 0;
#pragma unroll 1
    for (int base = 0; __any_sync(FULL, base < T); base += TPC * U) {
      float2 v[U];
      int qs[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = base + u * TPC + sub;
        qs[u] = -1;
        v[u] = make_float2(0.0f, 0.0f);
        if (idx < T) {
#pragma unroll 1
          while (h.pre[e + 1] <= idx) ++e;
          const int dy = e / 3;
          v[u].x = (float)(e - 3 * dy - 1) * wf;
          v[u].y = (float)(dy - 1) * hf;
          qs[u] = h.nq[e] * cap + (idx - h.pre[e]);
        }
      }
      float2 r[U];
#pragma unroll
      for (int u = 0; u < U; ++u) r[u] = qs[u] >= 0 ? __ldcg(rel + qs[u]) : v[u];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float X = r[u].x + v[u].x, Y = r[u].y + v[u].y;
        bool keep = qs[u] >= 0 && X > xlo && X < xhi && Y > ylo && Y < yhi;
        if (slow && qs[u] >= 0)
          keep = axis_screen(__ldcg(px + qs[u]), __ldcg(py + qs[u]), ox, oy, g, exact);
        const unsigned kept = (__ballot_sync(FULL, keep) >> gshift) & GM;
        const int i = ns + __popc(kept & ((1u << sub) - 1u));
        if (keep && i < co) f.key[i] = qs[u];
        ns += __popc(kept);
      }
    }
  }
  if (act && ns > co && sub == 0) h.ovf = 1;
  ns = min(ns, co);
  if (act && sub == 0) h.cnt = ns;
  __syncwarp();
  // FP64 placement of the members (objects 0 .. nc - 1, in bucket order) and
  // the survivors: box coordinates first, then, on the same lanes, the frame's;
  // one that no image brings into the frame is moved out of reach
  constexpr int U = 4;
#pragma unroll 1
  for (int i0 = sub; i0 < ns; i0 += TPC * U) {
    double x[U], y[U];
    int id[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * TPC;
      if (i < ns) {
        const int slot = i < nc ? c * cap + i : f.key[i];
        x[u] = __ldcg(px + slot);
        y[u] = __ldcg(py + slot);
        id[u] = pid[slot];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * TPC;
      if (i < ns) {
        f.a[i] = x[u];
        f.b[i] = y[u];
        f.key[i] = id[u] * 16 + 4;
      }
    }
  }
#pragma unroll 1
  for (int i = sub; i < ns; i += TPC) {
    double X = axis_diff(f.a[i], ox, L, hL), Y = axis_diff(f.b[i], oy, L, hL);
    if (i < nc) {
      f.last[i] = 0;
    } else if (!wide && !(axis_within(X, sigma, wl) && axis_within(Y, sigma, hl))) {
      X = Y = kAxisFar;
    }
    f.a[i] = axis == 0 ? X : Y;
    f.b[i] = axis == 0 ? Y : X;
    if (wide && i >= nc) axis_images(f.a, f.b, f.key, &h.cnt, &h.ovf, i, co, axis, g);
  }
  __syncwarp();
  const bool ok = act && h.ovf == 0;
  const int nobj = ok ? h.cnt : 0;
  f.nobj = nobj;
  f.nmem = nc;
  f.co = co;
  if (act && sub == 0) {
    f.a[co] = axis == 0 ? g.w : g.h;
    f.a[co + 1] = 0.0;
  }

  // staging: objects sorted into strips across the axis, with the coordinate
  // along it in fixed point (p_bits are left for the sorted position)
  int2* const sab = (int2*)stage;
  int* const bins = (int*)(sab + co);  // nbin + 1
  unsigned short* const si = (unsigned short*)(bins + nbin + 1);
#pragma unroll 1
  for (int k = sub; k <= nbin && ok; k += TPC) bins[k] = 0;
  const int p_bits = 32 - __clz(nobj | 1);
  const float ext = fmaxf((float)g.w, (float)g.h) + 2.0f * g.sigf;
  const float fix = __int_as_float((127 + 29 - p_bits) << 23) / ext;
  __syncwarp();
  const float sigf = g.sigf, inv_bw = g.inv_bin_w;
  auto bin_of = [&](float b32) {
    const int kb = (int)((b32 + sigf) * inv_bw);
    return kb < 0 ? 0 : (kb >= nbin ? nbin - 1 : kb);
  };
#pragma unroll 1
  for (int i = sub; i < nobj; i += TPC) atomicAdd(&bins[bin_of(to_float_trunc(f.b[i]))], 1);
  __syncwarp();
  {
    // exclusive prefix sums of the strip counts, TPC strips at a time
    int carry = 0;
#pragma unroll 1
    for (int k0 = 0; k0 < nbin; k0 += TPC) {
      const int k = k0 + sub;
      const int v = ok && k < nbin ? bins[k] : 0;
      int incl = v;
#pragma unroll
      for (int o = 1; o < TPC; o <<= 1) {
        const int u = __shfl_up_sync(FULL, incl, o, TPC);
        if (sub >= o) incl += u;
      }
      if (ok && k < nbin) bins[k] = carry + incl - v;
      carry += __shfl_sync(FULL, incl, TPC - 1, TPC);
    }
  }
  __syncwarp();
#pragma unroll 1
  for (int i = sub; i < nobj; i += TPC) {
    const float b32 = to_float_trunc(f.b[i]);
    const int p = atomicAdd(&bins[bin_of(b32)], 1);  // afterwards: the strip's end
    const float a32 = to_float_trunc(f.a[i]);
    // out of reach: beyond every window, the coordinate does not matter
    const int afix = b32 < ext ? (int)(a32 * fix) : 0;
    sab[p] = make_int2(afix, __float_as_int(b32));
    si[p] = (unsigned short)i;
  }
  // members ranked by disk id (start disks are drawn by rank), four keys a load
#pragma unroll 1
  for (int i = sub; i < nc && ok; i += TPC) {
    const int ki = f.key[i];
    int r = 0, k = 0;
#pragma unroll 2
    for (; k + 4 <= nc; k += 4) {
      const int4 q = *(const int4*)(f.key + k);
      r += (q.x < ki) + (q.y < ki) + (q.z < ki) + (q.w < ki);
    }
#pragma unroll 1
    for (; k < nc; ++k) r += (f.key[k] < ki);
    f.rank[r] = (unsigned short)i;
  }
  __syncwarp();

  // static candidates: one (member, window) per lane and step, both
  // directions.  An object whose window FP32 can tell is at least sqrt(2 ew)
  // ahead or behind, and two of one window are 2 sqrt(2^-24) sigma = 5e-4 sigma
  // apart along the axis (header): fixed point to ext 2^(p_bits - 29) and the
  // FP32 error ew settle the order, as long as their sum is below 2e-4 sigma.
  // The nearest ahead is the smallest positive (difference, position) word,
  // the nearest behind the largest negative one: as unsigned words, a minimum
  // and a maximum.  Objects near |db| = sigma (many pairs that met in sweeps
  // along the other axis lie there) are decided in FP64 after the loop over 32
  // objects; objects near sigma / 2 and frames too large for these precisions
  // send the lane to the FP64 search, and so does the caller who asks for every
  // candidate in FP64 (N = 2^18, 120^2 cells, four sweeps and a load: 1550 us,
  // 1270 with FP32 selection).
  const double sig2 = g.sig2;
  const float halff = 0.5f * sigf;
  const float ew = 2.0f * g.eps_d + 4e-7f * sigf;
  const bool coarse = g.precision == 0 || ew + 1.0f / fix > 2e-4f * sigf;
  const int near_fix = (int)(1e-3f * sigf * fix) + 1;  // ahead or behind beyond doubt
  const double NONE = __longlong_as_double((long long)0xfff0000000000000ull);
  const int items = ok ? 3 * nc : 0;
  constexpr unsigned kNobody = 0x7fffffffu;
#pragma unroll 1
  for (int it = sub; it < items; it += TPC) {
    const int j = it / 3, w = it - 3 * j;
    const double bj = f.b[j];
    const int ajf = (int)(to_float_trunc(f.a[j]) * fix);
    // the window as an interval of b: centre and half width
    const float mid =
        to_float_trunc(bj) + (w == 1 ? 0.0f : (w == 0 ? -1.5f * halff : 1.5f * halff));
    const float hw = w == 1 ? halff : 0.5f * halff;
    const float hin = hw - ew, hout = hw + ew;
    const int klo = bin_of(mid - hout), khi = bin_of(mid + hout);
    const int p0 = klo > 0 ? bins[klo - 1] : 0, p1 = bins[khi];
    unsigned up = kNobody, down = kNobody;
    bool amb = coarse;
#pragma unroll 1
    for (int pb = coarse ? p1 : p0; pb < p1; pb += 32) {
      unsigned edges = 0;  // objects near an edge of the window
      const int n = min(32, p1 - pb);
#pragma unroll 4
      for (int i = 0; i < n; ++i) {
        const int2 ab = sab[pb + i];
        const float t = fabsf(__int_as_float(ab.y) - mid);
        const int da = ab.x - ajf;
        const bool inside = t < hin;
        edges |= (!inside & (t <= hout) ? 1u : 0u) << i;
        const unsigned v =
            inside & (da != 0) ? ((unsigned)da << p_bits) | (unsigned)(pb + i) : kNobody;
        up = min(up, v);
        down = max(down, v);
      }
      amb |= edges != 0 && w == 1;
#pragma unroll 1
      while (edges && !amb) {
        const int p = pb + __ffs((int)edges) - 1;
        edges &= edges - 1;
        const double d = f.b[si[p]] - bj;
        const int da = sab[p].x - ajf;
        amb = abs(da) <= near_fix || abs_bits(d) < abs_bits(0.75 * sigma);
        if ((dbits(d) >= 0) == (w == 2) && lt_nn(d * d, sig2)) {
          const unsigned v = ((unsigned)da << p_bits) | (unsigned)p;
          up = min(up, v);
          down = max(down, v);
        }
      }
    }
    int jp = j, jm = j;  // first ahead, first behind
    const unsigned pm = (1u << p_bits) - 1u;
    if (up != kNobody) jp = si[up & pm];
    if (down != kNobody) jm = si[down & pm];
    if (amb) {
      const unsigned res = axis_scan_exact(f.a, f.b, si, p0, p1, j, w, sigma, sig2);
      jp = (int)(res & 0xffffu);
      jm = (int)(res >> 16 & 0x7fffu);
      if (res >> 31) {
        atomicOr(&f.key[j], 8);
        atomicOr(&h.irr, 1);
      }
    }
    // square roots of both (of a placeholder where nobody is there)
    const double dP = f.b[jp] - bj, dM = f.b[jm] - bj;
    const double xP = sig2 - dP * dP, xM = sig2 - dM * dM;
    const double qP = sqrt_rn(xP), qM = sqrt_rn(xM);
    AxisEntry* const e = f.list + 2 * j;
    e[0].sq[w] = jp == j ? NONE : qP;
    e[1].sq[w] = jm == j ? NONE : qM;
    e[0].nb[w] = (unsigned short)jp;
    e[1].nb[w] = (unsigned short)jm;
    if (w == 0) {
      e[0].nb[3] = (unsigned short)co;
      e[1].nb[3] = (unsigned short)(co + 1);
    }
  }
  __syncwarp();
}

}  // namespace ecmc
