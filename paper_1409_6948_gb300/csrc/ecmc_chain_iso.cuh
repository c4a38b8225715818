// ecmc_chain_iso.cuh -- the event-chain loop with isotropic directions.
//
// The variant the paper prefers for its applications (Sec. 3.2-3.4): every
// chain draws its own unit direction d, uniform on the circle; the active
// disk moves along d until the first of
//   - the end of the displacement budget,
//   - a contact with another member (the rest of the budget passes to it,
//     d unchanged),
//   - a contact with a frozen disk: specular reflection about the line of
//     centres at contact, d <- d - 2 (d.n) n / (n.n) (Fig. 1),
//   - a cell wall: the component of d normal to it flips (both at a corner).
// Ties as for axis chains: budget end < contact < wall; equal hit distances
// go to the smaller (disk id, image) key.
//
// The direction of chain k of cell c in sweep t is the first point (u, v) of
// the Philox pairs keyed (seed, replica), counter (t, direction purpose, c,
// k * 2^32 + attempt), uniform on [-1,1)^2, that lies in the unit disc and not
// at its centre, divided by its length: square root and division are IEEE
// operations, so the direction is reproducible to the last bit.
//
// SCREEN = false: every candidate of the frame is tested in FP64 with the
// expressions of the reference arithmetic (no contraction).  SCREEN = true:
// the projections b = D.d and c = D x d of every candidate are first computed
// in FP32 from the frame's FP32 coordinates and bracketed by rigorous error
// bounds, giving an interval for its hit distance; only candidates whose lower
// bound reaches the smallest certain upper bound (or the budget and wall
// distance) are tested in FP64, so the first hit and the new position are
// those of the full FP64 search.  Either way trajectories are bit-identical to
// the reference.  Frames are built with axis 0 (frame coordinates a = x, b = y).
//
// What bounds it: the chain's serial dependence and the FP64 pipe, which one
// warp instruction holds for some 57 cycles of its scheduler however few lanes
// take part.  So a vector's components are shared out between two lanes (one
// FP64 instruction for both), comparisons run on the integer pipes, the wall
// distances are bounded in FP32 and divided exactly only where a wall can come
// first (one division for both axes instead of one per axis and sign), and the
// one candidate that the screen leaves in most events is tested by the whole
// group, without a reduction.  About 45 FP64 instructions an event where there
// were 130.  GB300, us per sweep at eta = 0.708, ell = 1.06, n_m = 2:
//   N = 2^20, 240^2 cells: 2457 / 4522,  2^18, 120^2: 964 / 2281,
//   2^16, 60^2: 619 / 1345,  2^12, 14^2: 470 / 953;
//   2^16, 32^2 cells, ell = 8, n_m = 1: 1470 / 3091
// against every lane doing all of an event's scalar work (with the lanes per
// cell that were then the best).
#pragma once

#include "ecmc_chain.cuh"

namespace ecmc {

constexpr uint64_t kPurposeDirection = 3;

__device__ __forceinline__ void iso_direction(int64_t t, int lc, int k, uint64_t seed,
                                              uint64_t replica, double& dx, double& dy) {
  for (uint64_t attempt = 0; attempt < 4096; ++attempt) {
    const U64x4 q = philox((uint64_t)t, kPurposeDirection, (uint64_t)lc,
                           ((uint64_t)k << 32) | attempt, seed, replica);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double u = 2.0 * unit_double(q.v[2 * h]) - 1.0;
      const double v = 2.0 * unit_double(q.v[2 * h + 1]) - 1.0;
      const double n2 = u * u + v * v;
      if (n2 > 0.0 && n2 <= 1.0) {
        const double n = sqrt(n2);
        dx = u / n;
        dy = v / n;
        return;
      }
    }
  }
  // unreachable in practice (each attempt succeeds with probability
  // 1 - (1 - pi/4)^2 > 0.95); a fixed direction keeps the loop bounded
  dx = 1.0;
  dy = 0.0;
}

// `better` for distances >= +0 (or +inf), on the integer pipes
__device__ __forceinline__ bool better_nn(double s, int key, double bs, int bkey) {
  return lt_nn(s, bs) || (dbits(s) == dbits(bs) && key < bkey);
}

// FP64 hit test of candidate j along d, the reference expressions
__device__ __forceinline__ bool iso_hit(const Frame& f, int j, int CPW, int gi, double X, double Y,
                                        double dx, double dy, double sig2, double& s, double& b) {
  const double ddx = f.a64[j * CPW + gi] - X;
  const double ddy = f.b64[j * CPW + gi] - Y;
  b = ddx * dx + ddy * dy;
  if (dbits(b) <= 0) return false;
  const double cc = ddx * dy - ddy * dx;
  const double c2 = cc * cc;
  if (!lt_nn(c2, sig2)) return false;
  s = clamp0(b - sqrt_rn(sig2 - c2));
  return true;
}

__device__ __forceinline__ float iso_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// FP32 bracket [lo, hi] of the hit distance of candidate j (certain: j hits
// for sure, so hi bounds the first hit); false when j certainly misses
__device__ __forceinline__ bool iso_bracket(const Frame& f, const Geom& g, int j, int CPW, int gi,
                                            float X32, float Y32, float dx32, float dy32,
                                            float& lo, float& hi, bool& certain) {
  const float ex = __fsub_rn(f.a32[j * CPW + gi], X32);
  const float ey = __fsub_rn(f.b32[j * CPW + gi], Y32);
  const float b32 = __fadd_rn(__fmul_rn(ex, dx32), __fmul_rn(ey, dy32));
  const float e = g.iso_e;
  if (!(b32 > -e)) return false;
  const float c32 = __fsub_rn(__fmul_rn(ex, dy32), __fmul_rn(ey, dx32));
  const float ac = fabsf(c32);
  if (!(ac < __fadd_rn(g.iso_sig_hi, e))) return false;
  const float cl = fmaxf(__fsub_rn(ac, e), 0.0f), ch = __fadd_rn(ac, e);
  const float xhi = fmaxf(__fsub_rn(g.sig2f, __fmul_rn(cl, cl)), 0.0f);
  const float xlo = fmaxf(__fsub_rn(g.sig2f, __fmul_rn(ch, ch)), 0.0f);
  // (iso_sq leaves 2^-14 sigma for the SFU root's error of 2^-23 sigma)
  const float sq_hi = __fadd_rn(iso_sqrt(xhi), g.iso_sq);
  const float sq_lo = fmaxf(__fsub_rn(iso_sqrt(xlo), g.iso_sq), 0.0f);
  lo = __fsub_rn(__fsub_rn(__fsub_rn(b32, e), sq_hi), g.iso_r);
  hi = fmaxf(__fadd_rn(__fsub_rn(__fadd_rn(b32, e), sq_lo), g.iso_r), 0.0f);
  certain = __fsub_rn(b32, e) > 0.0f && __fadd_rn(ch, e) < g.iso_sig_lo;
  return true;
}

template <int TPC, bool SCREEN>
__device__ __forceinline__ void run_group_iso(const Frame& f, const int* hdr, void* hl,
                                              const Geom* __restrict__ rg,
                                              const SweepState* __restrict__ sts, int rep, int a,
                                              bool valid, int colour_index,
                                              double* __restrict__ px, double* __restrict__ py,
                                              CellStats* __restrict__ cs,
                                              ChainRec* __restrict__ recs, int rec_stride,
                                              int* err) {
  constexpr int CPW = 32 / TPC;
  const int lane = threadIdx.x & 31;
  const int gi = lane / TPC, sub = lane - gi * TPC;
  const Geom& g = rg[rep];
  const SweepState* st = sts + rep;
  const int colour = st->perm[colour_index];
  const int hx = g.cells_x >> 1;
  const int la = a - g.act_off;
  const int cx = 2 * (la % hx) + (colour & 1);
  const int cy = 2 * (la / hx) + (colour >> 1);
  const int lc = cy * g.cells_x + cx;
  const int c = g.cell_off + lc;
  const int64_t t = st->t;
  const double W = g.w, H = g.h, sig2 = g.sig2;
  const int nmem = valid ? hdr[CPW + gi] : 0;
  const int nobj = valid ? hdr[gi] : 0;
  const double INF = __longlong_as_double(0x7ff0000000000000ll);
  const unsigned FULL = 0xffffffffu;

  double sum_b = 0.0;
  int n_events = 0, n_lifts = 0, n_frozen = 0, n_walls = 0, n_fp64 = 0, n_chains = 0;
  int k = 0;
  bool active = false;
  int m = 0;
  double X = 0.0, Y = 0.0, dx = 1.0, dy = 0.0, r = 0.0;
  float dx32 = 1.0f, dy32 = 0.0f;  // the direction rounded to FP32
  // Two lanes share the work on the two components of a vector: `own` picks
  // this lane's component, `both` hands each lane the pair.
  constexpr int NC = TPC >= 2 ? 1 : 2;
  const int par = sub & 1;
  auto own = [&](double x, double y, int q) { return (NC == 1 ? par : q) ? y : x; };
  auto both = [&](const double* v, double& x, double& y) {
    if constexpr (NC == 1) {
      const double o = __shfl_xor_sync(FULL, v[0], 1);
      x = par ? o : v[0];
      y = par ? v[0] : o;
    } else {
      x = v[0];
      y = v[NC - 1];
    }
  };
  const float Wf = to_float_trunc(W), Hf = to_float_trunc(H);
  int64_t n_iter = 0;
  int ch_events = 0, ch_walls = 0, start_key = 0;
  bool done = (!valid) || nmem == 0;

  for (;;) {
    if (!done && !active) {
      if (k >= g.n_m) {
        done = true;
      } else {
        const U64x4 v = philox((uint64_t)t, kPurposeChain, (uint64_t)lc, (uint64_t)k, g.seed,
                               g.replica);
        int idx = (int)below_n(v.v[0], (uint64_t)nmem);
        if (g.list_mode == 1) {
          int* pl = (int*)hl;
          if (k == 0) shuffled_list(pl, CPW, gi, nmem, idx, t, lc, g.seed, g.replica);
          idx = pl[(k % nmem) * CPW + gi];
        }
        m = f.mrank[idx * CPW + gi];
        iso_direction(t, lc, k, g.seed, g.replica, dx, dy);
        dx32 = __double2float_rn(dx);
        dy32 = __double2float_rn(dy);
        X = f.a64[m * CPW + gi];
        Y = f.b64[m * CPW + gi];
        r = g.ell;
        f.touched[m * CPW + gi] = 1;
        start_key = f.key[m * CPW + gi];
        n_iter = 0;
        ch_events = 0;
        ch_walls = 0;
        active = true;
        ++k;
        ++n_chains;
      }
    }
    if (__all_sync(FULL, done)) break;
    const bool live = !done;
    const bool capped = live && (n_iter >= kMaxEventsPerChain);
    if (capped) atomicCAS(err, DEV_OK, DEV_CHAIN_CAP);
    const bool go = live && !capped;

    // FP32 bounds of the distance to the walls along d
    const float X32 = to_float_trunc(X), Y32 = to_float_trunc(Y);
    float wall_lo, wall_hi;
    {
      const float ax = fabsf(dx32), ay = fabsf(dy32);
      float nx = dx32 > 0.0f ? Wf - X32 : X32, ny = dy32 > 0.0f ? Hf - Y32 : Y32;
      if (ax < 0x1p-20f) nx = fminf(X32, Wf - X32);  // (its sign may be lost)
      if (ay < 0x1p-20f) ny = fminf(Y32, Hf - Y32);
      // numerators within iso_e; FP32 direction within 2^-24, quotients within
      // the factors
      const float qx = __fdividef(fmaxf(nx - g.iso_e, 0.0f), ax + 0x1p-20f);
      const float qy = __fdividef(fmaxf(ny - g.iso_e, 0.0f), ay + 0x1p-20f);
      wall_lo = fminf(qx, qy) * (1.0f - 0x1p-19f);
      const float INF32 = __int_as_float(0x7f800000);
      const float hx = ax > 0x1p-8f ? __fdividef(nx + g.iso_e, ax) : INF32;
      const float hy = ay > 0x1p-8f ? __fdividef(ny + g.iso_e, ay) : INF32;
      wall_hi = fminf(hx, hy) * (1.0f + 0x1p-12f);
    }

    // first contact along d
    double best_s = INF, best_b = 0.0;
    int best_key = INT_MAX, best_j = m;
    int nev = 0;     // FP64 evaluations (summed over the cell's lanes)
    bool multi = go;  // the exact tests run over all the lanes
    auto consider = [&](int j) {
      double s, b;
      ++nev;
      if (iso_hit(f, j, CPW, gi, X, Y, dx, dy, sig2, s, b)) {
        const int kj = f.key[j * CPW + gi];
        if (better_nn(s, kj, best_s, best_key)) {
          best_s = s;
          best_b = b;
          best_key = kj;
          best_j = j;
        }
      }
    };
    if (SCREEN) {
      // FP32 brackets; the candidates that can be the first hit go to FP64
      float U = __int_as_float(0x7f800000), L1 = U, L2 = U;
      int j1 = m;
      if (go) {
        for (int j = sub; j < nobj; j += TPC) {
          if (j == m) continue;
          float lo, hi;
          bool certain;
          if (!iso_bracket(f, g, j, CPW, gi, X32, Y32, dx32, dy32, lo, hi, certain)) continue;
          if (lo < L1) {
            L2 = L1;
            L1 = lo;
            j1 = j;
          } else if (lo < L2) {
            L2 = lo;
          }
          if (certain) U = fminf(U, hi);
        }
      }
      if (TPC > 1) {
#pragma unroll
        for (int o = 1; o < TPC; o <<= 1) {
          const float oU = __shfl_xor_sync(FULL, U, o);
          const float oL1 = __shfl_xor_sync(FULL, L1, o);
          const float oL2 = __shfl_xor_sync(FULL, L2, o);
          const int oj1 = __shfl_xor_sync(FULL, j1, o);
          U = fminf(U, oU);
          const float nL2 = fminf(fmaxf(L1, oL1), fminf(L2, oL2));
          if (oL1 < L1 || (oL1 == L1 && oj1 < j1)) {
            L1 = oL1;
            j1 = oj1;
          }
          L2 = nL2;
        }
      }
      const float Lam = fminf(U, fminf(to_float_up_nn(r), wall_hi));
      const bool need = go && (L1 <= Lam);
      multi = need && (L2 <= Lam);
      // one candidate: iso_hit, a component a lane
      const bool one = need && !multi;
      const int jc = one ? j1 : m;
      double v[NC], w2[NC], vx, vy;
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const double dd = own(f.a64[jc * CPW + gi], f.b64[jc * CPW + gi], q) - own(X, Y, q);
        v[q] = dd * own(dx, dy, q);
        w2[q] = dd * own(dy, dx, q);
      }
      both(v, vx, vy);
      const double b = vx + vy;
      both(w2, vx, vy);
      const double cc = vx - vy;
      const double c2 = cc * cc;
      if (one && dbits(b) > 0 && lt_nn(c2, sig2)) {
        best_s = clamp0(b - sqrt_rn(sig2 - c2));
        best_b = b;
        best_key = f.key[jc * CPW + gi];
        best_j = jc;
      }
      nev = one && sub == 0 ? 1 : 0;
      if (multi) {
        for (int j = sub; j < nobj; j += TPC) {
          if (j == m) continue;
          float lo, hi;
          bool certain;
          if (!iso_bracket(f, g, j, CPW, gi, X32, Y32, dx32, dy32, lo, hi, certain)) continue;
          if (lo <= Lam) consider(j);
        }
      }
    } else if (go) {
      for (int j = sub; j < nobj; j += TPC)
        if (j != m) consider(j);
    }
    if (TPC > 1 && __any_sync(FULL, multi)) {
#pragma unroll
      for (int o = 1; o < TPC; o <<= 1) {
        const double os = __shfl_xor_sync(FULL, best_s, o);
        const double ob = __shfl_xor_sync(FULL, best_b, o);
        const int ok = __shfl_xor_sync(FULL, best_key, o);
        const int oj = __shfl_xor_sync(FULL, best_j, o);
        nev += __shfl_xor_sync(FULL, nev, o);
        if (better_nn(os, ok, best_s, best_key)) {
          best_s = os;
          best_b = ob;
          best_key = ok;
          best_j = oj;
        }
      }
    }
    n_fp64 += go ? nev : 0;

    // Exact wall distances, unless the bounds leave no doubt: one division a
    // lane, for a component each.  Without doubt they count as infinite.
    const double q0 = min_nn(r, best_s);
    const bool need_wall = go && !(to_float_up_nn(q0) < wall_lo);
    double swx = INF, swy = INF;
    if (__any_sync(FULL, need_wall)) {
      double sw[NC];
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const double P = own(X, Y, q), D = own(dx, dy, q);
        const long long kD = dkey(D);
        const double up = own(W, H, q) - P;
        const double num = kD > 0 ? up : P;
        const double den = kD == 0 ? 1.0 : flip_if(D, kD < 0);
        sw[q] = kD == 0 ? INF : clamp0(num / den);
      }
      both(sw, swx, swy);
      swx = need_wall ? swx : INF;
      swy = need_wall ? swy : INF;
    }
    const double swall = min_nn(swx, swy);

    const bool is_end = go && le_nn(r, best_s) && le_nn(r, swall);  // budget used up
    const bool is_hit = go && !is_end && le_nn(best_s, swall);
    const bool is_wall = go && !is_end && !is_hit;
    const bool flip_x = is_wall && dbits(swx) == dbits(swall);
    const bool flip_y = is_wall && dbits(swy) == dbits(swall);
    const double s = is_end ? r : (is_hit ? best_s : (is_wall ? swall : 0.0));
    double v[NC], u[NC], nX, nY, r1, db;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const double D = own(dx, dy, q);
      v[q] = own(X, Y, q) + s * D;
      // onto the wall
      if ((NC == 1 ? par : q) ? flip_y : flip_x) v[q] = dkey(D) > 0 ? own(W, H, q) : 0.0;
      u[q] = own(r, best_b, q) - s;
    }
    both(v, nX, nY);
    both(u, r1, db);
    bool end_chain = capped || is_end;
    bool frozen = false;
    if (is_hit) {
      r = r1;
      sum_b += db;
      ++n_events;
      ++ch_events;
      ++n_iter;
      frozen = f.info[best_j * CPW + gi] < 0;
    } else if (is_wall) {  // the normal component(s) flip
      r = r1;
      if (flip_x) {
        dx = -dx;
        dx32 = -dx32;
      }
      if (flip_y) {
        dy = -dy;
        dy32 = -dy32;
      }
      ++n_walls;
      ++ch_walls;
      ++n_iter;
    }
    if (__any_sync(FULL, frozen)) {
      // frozen disk: specular reflection about the line of centres
      double n1[NC], n2[NC], n3[NC], vx, vy;
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        n1[q] = own(f.a64[best_j * CPW + gi], f.b64[best_j * CPW + gi], q) - own(nX, nY, q);
        n2[q] = n1[q] * n1[q];
        n3[q] = own(dx, dy, q) * n1[q];
      }
      both(n2, vx, vy);
      const double nn = vx + vy;
      both(n3, vx, vy);
      const double dot = vx + vy;
      const double kk = 2.0 * dot / (frozen ? nn : 1.0);
#pragma unroll
      for (int q = 0; q < NC; ++q) n1[q] = own(dx, dy, q) - kk * n1[q];
      both(n1, vx, vy);
      if (frozen) {
        ++n_frozen;
        dx = vx;
        dy = vy;
        dx32 = __double2float_rn(dx);
        dy32 = __double2float_rn(dy);
      }
    }
    if (is_hit && !frozen) {
      // lift: the hit member moves on along d
      ++n_lifts;
      // the stopped disk, in FP64 and in the FP32 copy the screen reads
      f.a64[m * CPW + gi] = nX;
      f.b64[m * CPW + gi] = nY;
      f.a32[m * CPW + gi] = to_float_trunc(nX);
      f.b32[m * CPW + gi] = to_float_trunc(nY);
      m = best_j;
      X = f.a64[m * CPW + gi];
      Y = f.b64[m * CPW + gi];
      f.touched[m * CPW + gi] = 1;
    } else if (go) {
      X = nX;
      Y = nY;
    }
    if (end_chain) {
      f.a64[m * CPW + gi] = X;
      f.b64[m * CPW + gi] = Y;
      f.a32[m * CPW + gi] = to_float_trunc(X);
      f.b32[m * CPW + gi] = to_float_trunc(Y);
      if (recs != nullptr && sub == 0) {
        ChainRec rc;
        rc.start_id = start_key >> 4;
        rc.end_id = f.key[m * CPW + gi] >> 4;
        rc.events = ch_events;
        rc.walls = ch_walls;
        recs[(int64_t)c * rec_stride + (k - 1)] = rc;
      }
      active = false;
    }
  }

  __syncwarp();
  if (!valid) return;
  const double ox = st->sx + (double)cx * g.w;
  const double oy = st->sy + (double)cy * g.h;
  for (int q = sub; q < nmem; q += TPC) {
    const int j = f.mrank[q * CPW + gi];
    if (!f.touched[j * CPW + gi]) continue;
    const int slot = f.mslot[q * CPW + gi];
    px[slot] = wrap_box0(f.a64[j * CPW + gi] + ox, g.L);
    py[slot] = wrap_box0(f.b64[j * CPW + gi] + oy, g.L);
  }
  if (sub == 0) {
    CellStats s;
    s.sum_b = sum_b;
    s.events = n_events;
    s.lifts = n_lifts;
    s.frozen = n_frozen;
    s.walls = n_walls;
    s.fp64_evals = n_fp64;
    s.chains = n_chains;
    s.n_mem = nmem;
    s.replayed = 0;
    s.rejected = 0;
    cs[c] = s;
  }
}

}  // namespace ecmc
