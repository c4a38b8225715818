// ecmc_sweep.cu -- the persistent sweep kernel: all four colour phases of a
// sweep (Sec. 3.4 steps 4-6) in one launch.
//
// Work list: item i = (colour phase ci, group G) in the order of i = ci * groups + G;
// a group is the cpw = 32/TPC consecutive active cells one warp serves.  Each
// warp takes the next item from a device counter, waits until every
// neighbour cell of an earlier colour phase of the same sweep has finished,
// builds the group's frames in its shared memory, runs the chains (axis
// chains: ecmc_axis.cuh; isotropic ones: ecmc_chain_iso.cuh) and publishes the
// cells as finished.  Frozen disks of a later
// colour have not moved yet, and a later cell waits for this one in turn, so
// every cell sees exactly the configuration of the phase-by-phase schedule,
// and the results are those of the per-phase launches bit for bit.  The tail of
// one colour phase overlaps the start of the next.
//
// Progress: an item only waits for items with a smaller index, which were
// taken earlier by running warps and never wait for later items; the
// smallest unfinished item therefore always progresses, whatever the number of
// resident warps.  Every wait is bounded nonetheless (global timer): on
// timeout the kernel raises DEV_WAIT_TIMEOUT and an abort flag that makes
// every warp leave at its next item or wait.
#include "ecmc_axis.cuh"
#include "ecmc_build.cuh"
#include "ecmc_chain.cuh"
#include "ecmc_chain_iso.cuh"

namespace ecmc {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned load_volatile(const unsigned* p) {
  return *(const volatile unsigned*)p;
}

// Wait for the neighbours of cell (cx, cy) whose colour phase comes before
// phase ci (the TPC lanes of the group share the eight directions); false if
// a wait ran into its limit or the sweep was abandoned.
template <int TPC>
__device__ __forceinline__ bool wait_for_neighbours(const Geom& g, const SweepState* st, int cx,
                                                    int cy, int colour, int ci, bool valid,
                                                    int sub, unsigned* sched,
                                                    const unsigned* done, unsigned want,
                                                    unsigned long long wait_ns, int* err) {
  if (!valid || ci == 0) return true;
  int phase_of[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) phase_of[st->perm[k]] = k;
  for (int d = sub; d < 8; d += TPC) {
    const int e = d < 4 ? d : d + 1;  // skip the centre of the 3x3 block
    const int ddx = e % 3 - 1, ddy = e / 3 - 1;
    const int ncol = colour ^ (ddx != 0 ? 1 : 0) ^ (ddy != 0 ? 2 : 0);
    if (phase_of[ncol] >= ci) continue;
    int qx = cx + ddx, qy = cy + ddy;
    qx += qx < 0 ? g.cells_x : 0;
    qx -= qx >= g.cells_x ? g.cells_x : 0;
    qy += qy < 0 ? g.cells_y : 0;
    qy -= qy >= g.cells_y ? g.cells_y : 0;
    const int q = g.cell_off + qy * g.cells_x + qx;
    if (load_volatile(&done[q]) == want) continue;
    const unsigned long long t0 = global_ns();
    while (load_volatile(&done[q]) != want) {
      if (load_volatile(&sched[2]) != 0u) return false;
      if (global_ns() - t0 > wait_ns) {
        atomicCAS(err, DEV_OK, DEV_WAIT_TIMEOUT);
        atomicExch(&sched[2], 1u);
        return false;
      }
      __nanosleep(256);
    }
  }
  return true;
}

// Shared memory of one warp: the frame record of its group, the touched
// flags, the leg histories (which also serve as the builder's staging area,
// used before the chains start) and the builder's scratch.
__host__ __device__ inline size_t fused_touch_bytes(const RecLayout& lay) {
  return align16((size_t)lay.cap_obj * lay.cpw);
}
__host__ __device__ inline size_t fused_hist_bytes(const RecLayout& lay) {
  const size_t h = kHistLegBytes * kHist * (size_t)lay.cpw;
  const size_t s = build_stage_bytes(lay);
  return h > s ? h : s;
}
__host__ __device__ inline size_t fused_warp_bytes(const RecLayout& lay) {
  return lay.bytes + fused_touch_bytes(lay) + fused_hist_bytes(lay) + build_aux_bytes(32);
}

// Isotropic chains: frames by build_frame, whole records in shared memory.
template <int TPC, bool SCREEN>
__global__ void __launch_bounds__(32, 16) k_sweep_iso(
    const Geom* __restrict__ rg, const SweepState* __restrict__ sts,
    const int* __restrict__ act_rep, int n_active, int cap, double* __restrict__ px,
    double* __restrict__ py, const int* __restrict__ pid, const int* __restrict__ cnt,
    RecLayout lay, CellStats* __restrict__ cs, ChainRec* __restrict__ recs, int rec_stride,
    unsigned* sched, unsigned* done, unsigned long long wait_ns, int wait_test, int* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int CPW = 32 / TPC;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned char* const rec = smem;
  unsigned char* const tbase = rec + lay.bytes;
  double* const a64 = (double*)(rec + lay.off_a64);
  double* const b64 = (double*)(rec + lay.off_b64);
  unsigned char* const hbase = tbase + fused_touch_bytes(lay);
  unsigned char* const aux = hbase + fused_hist_bytes(lay);

  Frame f;
  f.cpw = CPW;
  f.bst = (const int*)(rec + lay.off_bstart);
  f.mrank = (const int*)(rec + lay.off_mrank);
  f.mslot = (const int*)(rec + lay.off_mslot);
  f.a32 = (float*)(rec + lay.off_a32);
  f.b32 = (float*)(rec + lay.off_b32);
  f.a64 = a64;
  f.b64 = b64;
  f.key = (const int*)(rec + lay.off_key);
  f.info = (const int*)(rec + lay.off_info);
  f.touched = tbase;
  const int* hdr = (const int*)(rec + lay.off_hdr);
  // the sweep's epoch: cells finished in this sweep carry it in done[]; the
  // failure test waits for a value nobody writes
  const unsigned epoch = load_volatile(&sched[1]);
  const unsigned want = wait_test ? (epoch ^ 0x80000000u) : epoch;
  const int n_groups = (n_active + CPW - 1) / CPW;
  const int n_items = 4 * n_groups;
  const int gi = lane / TPC, sub = lane - gi * TPC;

  for (;;) {
    int item = 0;
    if (lane == 0) item = (int)atomicAdd(&sched[0], 1u);
    item = __shfl_sync(FULL, item, 0);
    if (item >= n_items || load_volatile(&sched[2]) != 0u) break;
    const int ci = item / n_groups, G = item - ci * n_groups;

    // this lane group's cell
    const int a = G * CPW + gi;
    const bool valid = a < n_active;
    const int rep = valid ? act_rep[a] : act_rep[n_active - 1];
    const Geom& g = rg[rep];
    const SweepState* st = sts + rep;
    const int colour = st->perm[ci];
    const int hx = g.cells_x >> 1;
    const int la = a - g.act_off;
    const int cx = 2 * (la % hx) + (colour & 1);
    const int cy = 2 * (la / hx) + (colour >> 1);

    const bool ok = wait_for_neighbours<TPC>(g, st, cx, cy, colour, ci, valid, sub, sched, done,
                                             want, wait_ns, err);
    if (!__all_sync(FULL, ok)) break;
    __threadfence();  // the finished neighbours' positions are visible from here on

    // the group's frames, one cell after another, by the whole warp
    for (int g2 = 0; g2 < CPW; ++g2) {
      const int a2 = G * CPW + g2;
      if (a2 >= n_active) break;
      const int rep2 = act_rep[a2];
      const Geom& gg = rg[rep2];
      const SweepState* st2 = sts + rep2;
      const int col2 = st2->perm[ci];
      const int hx2 = gg.cells_x >> 1;
      const int la2 = a2 - gg.act_off;
      BuildArgs A;
      A.g = &gg;
      A.st = st2;
      A.cx = 2 * (la2 % hx2) + (col2 & 1);
      A.cy = 2 * (la2 / hx2) + (col2 >> 1);
      A.c = gg.cell_off + A.cy * gg.cells_x + A.cx;
      A.cap = cap;
      A.px = px;
      A.py = py;
      A.pid = pid;
      A.cnt = cnt;
      A.aux = aux;
      A.stage = hbase;
      A.rec = rec;
      A.a64 = a64;
      A.b64 = b64;
      A.lay = lay;
      A.gi = g2;
      A.err = err;
      build_frame<true, true>(A);
    }
    {
      int4* tz = reinterpret_cast<int4*>(tbase);
      const int4 z = make_int4(0, 0, 0, 0);
      for (int i = lane; i < (int)(fused_touch_bytes(lay) / 16); i += 32) tz[i] = z;
    }
    __syncwarp();
    run_group_iso<TPC, SCREEN>(f, hdr, (double*)hbase, rg, sts, rep, a, valid, ci, px, py, cs,
                               recs, rec_stride, err);

    // publish: every lane's write-back is visible before the cell is marked
    __threadfence();
    __syncwarp();
    if (valid && sub == 0) {
      const int c = g.cell_off + cy * g.cells_x + cx;
      __threadfence();
      *(volatile unsigned*)&done[c] = epoch;
    }
    __syncwarp();
  }
}

// Axis chains (both boundary rules): frames and static candidates by
// axis_build, chains by axis_chains (ecmc_axis.cuh).  FM 0: all of it in
// shared memory; FM 1: the candidate lists in a per-warp scratch area of
// global memory (cells of many members).  phase < 0: the persistent sweep;
// else one block per item of that colour phase.
template <int TPC, bool REJECT, int FM>
__global__ void __launch_bounds__(32, 16) k_sweep_axis(
    const Geom* __restrict__ rg, const SweepState* __restrict__ sts,
    const int* __restrict__ act_rep, int n_active, int cap, double* __restrict__ px,
    double* __restrict__ py, const int* __restrict__ pid, float2* __restrict__ rel,
    const int* __restrict__ cnt, AxisShape shp, CellStats* __restrict__ cs, ChainRec* __restrict__ recs, int rec_stride,
    int replay, unsigned* sched, unsigned* done, unsigned long long wait_ns, int wait_test,
    unsigned char* __restrict__ scratch, int phase, int* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int CPW = 32 / TPC;
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int gi = lane / TPC, sub = lane & (TPC - 1);
  const unsigned epoch = load_volatile(&sched[1]);
  const unsigned want = wait_test ? (epoch ^ 0x80000000u) : epoch;
  const int n_groups = (n_active + CPW - 1) / CPW;
  const int n_items = 4 * n_groups;
  AxisHead& h = *(AxisHead*)(smem + gi * kAxisHead);
  unsigned char* const lists = FM == 1 ? scratch + (size_t)blockIdx.x * axis_scratch_bytes(shp)
                                       : nullptr;

  for (;;) {
    int item = 0;
    if (phase < 0) {
      if (lane == 0) item = (int)atomicAdd(&sched[0], 1u);
      item = __shfl_sync(FULL, item, 0);
      if (item >= n_items || load_volatile(&sched[2]) != 0u) break;
    } else {
      item = phase * n_groups + blockIdx.x;
    }
    const int ci = (item >= n_groups) + (item >= 2 * n_groups) + (item >= 3 * n_groups);
    const int G = item - ci * n_groups;

    // this lane group's cell
    const int act_cell = G * CPW + gi;
    const bool valid = act_cell < n_active;
    const int rep = act_rep[valid ? act_cell : n_active - 1];
    const Geom& g = rg[rep];
    const SweepState* st = sts + rep;
    const int colour = st->perm[ci];
    const int hx = g.cells_x >> 1;
    const int la = valid ? act_cell - g.act_off : 0;
    const int cx = 2 * (la % hx) + (colour & 1);
    const int cy = 2 * (la / hx) + (colour >> 1);
    const int lc = cy * g.cells_x + cx;
    const int c = g.cell_off + lc;
    if (phase < 0) {
      const bool ok = wait_for_neighbours<TPC>(g, st, cx, cy, colour, ci, valid, sub, sched,
                                               done, want, wait_ns, err);
      if (!__all_sync(FULL, ok)) break;
      __threadfence();  // the finished neighbours' positions are visible from here on
    }
    const int nc = valid ? min(cnt[c], cap) : 0;

    // all cells of the item together; those whose frames outgrow the usual
    // sizes again, one by one with the whole memory of the warp
    bool todo = valid, alone = false;
    while (__any_sync(FULL, todo)) {
      AxisPass pass;
      int mb = 0;
      bool act;
      if (!alone) {
        pass = axis_pass(shp, CPW, shp.co_s, shp.mp_s, FM == 0);
        int incl = nc;
#pragma unroll
        for (int o = TPC; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(FULL, incl, o);
          if (lane >= o) incl += u;
        }
        act = todo && incl <= shp.mp_s;
        mb = act ? incl - nc : 0;
      } else {
        pass = axis_pass(shp, 1, shp.co_h, shp.mp_h, FM == 0);
        act = gi == (__ffs(__ballot_sync(FULL, todo)) - 1) / TPC;
      }
      const int slot = alone ? 0 : gi;
      unsigned char* const obj = smem + pass.obj_off + slot * axis_obj_bytes(pass.co);
      unsigned char* const work =
          smem + pass.work_off + slot * axis_work_bytes(pass.co, shp.nbin);
      const int mp = alone ? shp.mp_h : shp.mp_s;
      AxisFrame f;
      f.a = (double*)obj;
      f.b = f.a + pass.co + 2;
      f.key = (int*)(f.b + pass.co);
      unsigned char* const lb = FM == 1 ? lists : smem + pass.memb_off;
      f.list = (AxisEntry*)lb + 2 * mb;
      f.last = (int*)(smem + pass.flag_off) + mb;
      f.rank = (unsigned short*)(smem + pass.flag_off + 4 * mp) + mb;
      f.starts = (unsigned short*)((unsigned char*)&h + sizeof(AxisHead));
      f.leg = (AxisLeg*)work;
      axis_build<TPC>(f, h, work, pass, shp.nbin, g, st, cx, cy, c, cap, nc, act, alone, px, py,
                      pid, rel, cnt);
      const bool full = act && h.ovf != 0;
      if (full && alone && sub == 0) atomicCAS(err, DEV_OK, DEV_CAPACITY);
      const bool run = act && !full;
      axis_chains<TPC, REJECT>(f, g, st->t, lc, c, run,
                               run && h.irr != 0, cs, recs, rec_stride, replay, err);
      if (run) {
        // the members that were active in a chain, back in box coordinates
        const double ox = st->sx + (double)cx * g.w;
        const double oy = st->sy + (double)cy * g.h;
        const bool along_x = st->axis == 0;
        for (int q = sub; q < nc; q += TPC) {
          if (f.last[q] == 0) continue;
          const double A = f.a[q], B = f.b[q];
          const int64_t at = (int64_t)c * cap + q;
          const double X = along_x ? A : B, Y = along_x ? B : A;
          px[at] = wrap_box0(X + ox, g.L);
          py[at] = wrap_box0(Y + oy, g.L);
          rel[at] = make_float2(to_float_trunc(X), to_float_trunc(Y));
        }
      }
      const bool finished = run || (full && alone);
      // publish: every lane's write-back is visible before the cell is marked
      __threadfence();
      __syncwarp();
      if (finished) {
        if (sub == 0) {
          __threadfence();
          *(volatile unsigned*)&done[c] = epoch;
        }
        todo = false;
      }
      __syncwarp();
      alone = true;
    }
    if (phase >= 0) break;
  }
}

// Dispatch over lanes per cell, boundary rule and list placement: FN is
// called as FN(kernel).
#define ECMC_AXIS_T(T, FN)                                                       case T:                                                                          return reject ? (fm == 1 ? FN((k_sweep_axis<T, true, 1>))                                                 : FN((k_sweep_axis<T, true, 0>)))                                     : (fm == 1 ? FN((k_sweep_axis<T, false, 1>))                                                : FN((k_sweep_axis<T, false, 0>)));
#define ECMC_AXIS(FN)                                                            switch (tpc) {                                                                   ECMC_AXIS_T(1, FN)                                                             ECMC_AXIS_T(2, FN)                                                             ECMC_AXIS_T(4, FN)                                                             ECMC_AXIS_T(8, FN)                                                             ECMC_AXIS_T(16, FN)                                                            ECMC_AXIS_T(32, FN)                                                            default: return -1;                                                          }

size_t axis_smem(const AxisShape& s, int fm) { return axis_smem_bytes(s, fm); }
size_t axis_scratch(const AxisShape& s) { return axis_scratch_bytes(s); }

// The attribute is a per-kernel, per-process maximum: request the largest
// amount the kernel can have, so that a handle with small frames never lowers
// the limit that a handle with larger frames needs.
template <typename K>
static int configure_sweep_kernel(K kernel, size_t sm, int* blocks_per_sm) {
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
          cudaSuccess ||
      cudaFuncGetAttributes(&fa, kernel) != cudaSuccess)
    return -1;
  const int mx = optin - (int)fa.sharedSizeBytes;
  if (sm > (size_t)mx ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, mx) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, 32, sm) !=
          cudaSuccess)
    return -1;
  return *blocks_per_sm > 0 ? 0 : -1;
}

int configure_axis(const AxisShape& s, int tpc, int fm, int reject, int* blocks_per_sm) {
  const size_t sm = axis_smem_bytes(s, fm);
#define ECMC_AXIS_CFG(K) configure_sweep_kernel(K, sm, blocks_per_sm)
  ECMC_AXIS(ECMC_AXIS_CFG)
#undef ECMC_AXIS_CFG
}

template <typename K>
static int launch_axis_t(K kernel, const DevBufs& b, const AxisShape& s, int fm, int blocks,
                         int phase, int records_on, cudaStream_t st) {
  kernel<<<blocks, 32, axis_smem_bytes(s, fm), st>>>(
      b.rg, b.state, b.act_rep, b.A_total, b.cap, b.px[b.cur], b.py[b.cur], b.pid[b.cur], b.rel,
      b.count[b.cur], s, b.cell_stats, records_on ? b.chain_recs : nullptr, b.rec_stride,
      b.replay, b.sched, b.done, b.wait_ns, b.wait_test, b.records, phase, b.err);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_axis(const DevBufs& b, const AxisShape& s, int tpc, int blocks, int phase,
                int records_on, cudaStream_t st) {
  const int reject = b.reject, fm = b.fmode;
#define ECMC_AXIS_RUN(K) launch_axis_t(K, b, s, fm, blocks, phase, records_on, st)
  ECMC_AXIS(ECMC_AXIS_RUN)
#undef ECMC_AXIS_RUN
}
#undef ECMC_AXIS
#undef ECMC_AXIS_T

size_t fused_smem_bytes(const RecLayout& lay) { return fused_warp_bytes(lay); }

#define ECMC_ISO_T(T, FN) \
  case T: return screen ? FN((k_sweep_iso<T, true>)) : FN((k_sweep_iso<T, false>));
#define ECMC_ISO(FN)                                                           \
  switch (tpc) {                                                               \
    ECMC_ISO_T(1, FN)                                                          \
    ECMC_ISO_T(2, FN)                                                          \
    ECMC_ISO_T(4, FN)                                                          \
    ECMC_ISO_T(8, FN)                                                          \
    ECMC_ISO_T(16, FN)                                                         \
    ECMC_ISO_T(32, FN)                                                         \
    default: return -1;                                                        \
  }

static int configure_iso(const RecLayout& lay, int tpc, bool screen, int* blocks_per_sm) {
  const size_t sm = fused_warp_bytes(lay);
#define ECMC_ISO_CFG(K) configure_sweep_kernel(K, sm, blocks_per_sm)
  ECMC_ISO(ECMC_ISO_CFG)
#undef ECMC_ISO_CFG
}

int configure_fused(const RecLayout& lay, int tpc, int* blocks_per_sm) {
  int n0 = 0, n1 = 0;
  if (configure_iso(lay, tpc, false, &n0) || configure_iso(lay, tpc, true, &n1)) return -1;
  *blocks_per_sm = n0 < n1 ? n0 : n1;
  return 0;
}

template <typename K>
static int launch_fused_t(K kernel, const DevBufs& b, const RecLayout& lay, int blocks,
                          int records_on, cudaStream_t s) {
  kernel<<<blocks, 32, fused_warp_bytes(lay), s>>>(
      b.rg, b.state, b.act_rep, b.A_total, b.cap, b.px[b.cur], b.py[b.cur], b.pid[b.cur],
      b.count[b.cur], lay, b.cell_stats, records_on ? b.chain_recs : nullptr, b.rec_stride,
      b.sched, b.done, b.wait_ns, b.wait_test, b.err);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_fused(const DevBufs& b, const RecLayout& lay, int tpc, int blocks, int records_on,
                 int precision, cudaStream_t s) {
  const bool screen = precision == 1;
#define ECMC_ISO_RUN(K) launch_fused_t(K, b, lay, blocks, records_on, s)
  ECMC_ISO(ECMC_ISO_RUN)
#undef ECMC_ISO_RUN
}
#undef ECMC_ISO
#undef ECMC_ISO_T

}  // namespace ecmc
