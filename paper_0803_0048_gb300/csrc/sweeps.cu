// sweeps.cu -- a4: the triangular solve L~U~ y = p applied in every Krylov
// iteration (Eq. triangleSolve), and its transpose.
//
// Forward (Eq. forwardsubA): x_i = p_i - sum_{h<i} f_ih x_h, h ascending.
// Backward: y_i = (x_i - sum_{j>i} f_ij y_j) / f_ii, j descending (the mirror
// image: rows last to first, each row right to left).  Each row's
// subtraction chain keeps the sequential order (one rounding per product, one
// per difference); the division by f_ii runs on the integer pipes from the
// factor's fixed-point reciprocal of f_ii and gives IEEE's quotient
// (div_fin, common.cuh).
//
// Six schedules of the same row task, all bit-identical; the factor handle
// times those that suit the shape of its DAG (the warp-per-row ones at several
// CTA widths) on its first application and keeps the fastest for each direction
// (a one-call solve picks from the shape alone):
//  * WARP_CLUSTER: one warp per row in one 16-CTA thread-block cluster, x in
//    the cluster's distributed shared memory on the producer's SM; the warp
//    subtracts the longest ready prefix of its chain as values arrive, and
//    when only the last entry is missing, the lane that owns it finishes the
//    row alone (poll, multiply, subtract, divide, store).
//    Suits deep, narrow DAGs, where the hand-off latency sets the time.
//  * WARP_CLUSTER_HELP: the same with a second cluster that subtracts the
//    leading entries of long rows ahead of their warps.
//  * WARP_GRID: the same over all SMs with x in global memory (L2 hand-offs);
//    suits wide DAGs, which need many SMs in flight.
//  * FLAGS: 32 rows of one level per warp in lockstep over all SMs (L2
//    hand-offs); packs the FP64 work of 32 rows into each instruction but
//    couples the rows of a warp.
//  * SINGLE_CTA / CLUSTER: the same on one SM or on a small cluster, x handed
//    over through a ring in shared memory; for rows of at most 8 entries
//    (longer ones run as WARP_GRID).  Suits narrow DAGs of short rows.
// Rows are taken in level order (padded to warps for the lockstep kernels);
// every wait is bounded.
//
// The transposed solve (L~U~)^-T p runs the same kernels on an explicit CSR
// transpose T = F^T: forward with division by t_ii (U~^T), then backward with
// unit diagonal (L~^T).
#include <climits>
#include <cstring>
#include <mutex>

#include "internal.h"

namespace iluk {

// Scratch ints kept per factor handle: the numeric phase's row ticket (rows
// hand their results over through the values themselves, so no flags).
size_t sweep_sync_ints(int64_t n) {
  (void)n;
  return 4;
}

constexpr int kCtaThreads = 1024;
constexpr int kGridThreads = 256;

// Sweep outputs double as their own ready flags: an entry holds kPending (a
// signalling NaN, which no arithmetic produces) until its row is final, so a
// row that reads x_c simply polls x_c.  No flag array, no fence, no memset.
constexpr unsigned long long kPending = 0x7FF0DEADBEEFCAFEull;
constexpr unsigned long long kQuietNaN = 0x7FF8000000000000ull;

__device__ __forceinline__ double ld_val(const double *p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ void st_val(double *p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

__device__ __forceinline__ bool pending(double v) {
  return (unsigned long long)__double_as_longlong(v) == kPending;
}

// Wait for *p to leave the pending state; false on time-out or on a failure
// recorded by another thread.
// Rows of a sweep are taken 32 at a time from the level order (a warp's 32
// rows belong to one level, padding slots hold -1), and the warp walks the
// 32 subtraction chains in lockstep, a window of W entries at a time: it
// loads the W values each lane needs, waits (warp-uniformly) until none of
// them is pending, then forms the products and the differences with every
// lane active.  Keeping the FP64 instructions converged matters on GB300,
// where an FP64 warp instruction occupies the pipe for ~20 SM cycles however
// few lanes it serves.  Each chain still runs left to right in its own lane.
// `clear` (may alias `in`) gets kPending at position `row` once in[row] has
// been read, which re-arms the buffer the next sweep writes.
template <bool FORWARD, bool DIVIDE, int W>
__global__ void __launch_bounds__(kGridThreads)
k_sweep(const int32_t *__restrict__ order, int64_t len, const int64_t *__restrict__ rp,
        const int32_t *__restrict__ ci, const int64_t *__restrict__ dg,
        const double *__restrict__ v, const DivPrep *__restrict__ rd, const double *in,
        double *out, double *clear, DevErr *err, int64_t limit_ns) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t slot0 = gw * 32; slot0 < len; slot0 += nw * 32) {
    const int64_t row = order[slot0 + lane];
    // Entry e (0-based, in subtraction order) of this row sits at
    // first + step * e: left to right in the forward sweep, right to left in
    // the backward sweep, so the nearest columns, whose rows finish last, are
    // always subtracted last.
    int64_t first = 0, d = 0;
    int mylen = 0;
    double s = 0.0;
    DivPrep rr{0ull, 1.0};
    if (row >= 0) {
      d = dg[row];
      if (DIVIDE) rr = rd[row];  // u_ii and its reciprocal, fetched off the chain
      if (FORWARD) {
        first = rp[row];
        mylen = (int)(d - first);
      } else {
        first = rp[row + 1] - 1;
        mylen = (int)(first - d);
      }
      s = in[row];
      if (clear) clear[row] = __longlong_as_double((long long)kPending);
    }
    constexpr int64_t step = FORWARD ? 1 : -1;
    const int maxlen = __reduce_max_sync(FULL_MASK, mylen);
    // Chains are right-aligned across the warp: lane entry e runs at lockstep
    // position e + (maxlen - mylen), so every lane's newest dependencies fall
    // in the last windows.
    const int off = maxlen - mylen;
    bool ok = true;
    for (int q0 = 0; q0 < maxlen; q0 += W) {
      int32_t c[W];
      double f[W], x[W];
      bool pend = false;
#pragma unroll
      for (int u = 0; u < W; ++u) {
        const int e = q0 + u - off;
        if (e >= 0 && e < mylen) {
          c[u] = ci[first + step * e];
          f[u] = v[first + step * e];
        }
      }
#pragma unroll
      for (int u = 0; u < W; ++u) {
        const int e = q0 + u - off;
        if (e >= 0 && e < mylen) {
          x[u] = ld_val(&out[c[u]]);
          pend |= pending(x[u]);
        }
      }
      if (__any_sync(FULL_MASK, pend)) {
        // Re-read every still-pending value each round (they may arrive in any
        // order), sleeping briefly between rounds so that waiting warps leave
        // issue slots to the warps that can make progress.
        const uint64_t t0 = globaltimer_ns();
        unsigned backoff = 16;
        for (unsigned it = 0; __any_sync(FULL_MASK, pend); ++it) {
          pend = false;
#pragma unroll
          for (int u = 0; u < W; ++u) {
            const int e = q0 + u - off;
            if (e >= 0 && e < mylen && pending(x[u])) {
              x[u] = ld_val(&out[c[u]]);
              pend |= pending(x[u]);
            }
          }
          // the decision to give up is taken by the whole warp at once
          const bool stop = (it & 15u) == 15u &&
                            (any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns);
          if (__any_sync(FULL_MASK, stop)) {
            ok = false;
            break;
          }
          if (__any_sync(FULL_MASK, pend)) {
            __nanosleep(backoff);
            if (backoff < 256u) backoff <<= 1;
          }
        }
        if (!__all_sync(FULL_MASK, ok)) break;
      }
#pragma unroll
      for (int u = 0; u < W; ++u) {
        const int e = q0 + u - off;
        if (e >= 0 && e < mylen) x[u] = __dmul_rn(f[u], x[u]);
      }
#pragma unroll
      for (int u = 0; u < W; ++u) {
        const int e = q0 + u - off;
        if (e >= 0 && e < mylen) s = __dsub_rn(s, x[u]);
      }
    }
    if (!__all_sync(FULL_MASK, ok)) {
      if (row >= 0) set_err(err, row, ILUK_ETIMEOUT);
      return;
    }
    if (DIVIDE && row >= 0) s = div_fin(s, rr);
    if (row >= 0) {
      if ((unsigned long long)__double_as_longlong(s) == kPending)
        s = __longlong_as_double((long long)kQuietNaN);
      st_val(&out[row], s);
    }
  }
}

// ---------------------------------------------------------------------------
// The ring.  The SINGLE_CTA and CLUSTER sweeps hand x from row to row through
// a ring in shared memory: every CTA of the launch holds a copy, slot p of the
// walked order at entry p mod kRing, and a finished row stores its value into
// all copies, so a waiting row polls its own SM's shared memory (~46 cycles a
// look) and a hand-off costs one store's flight (probe, one warp per SM: ~205
// cycles a hop within an SM, 230-370 pushed to another SM of the cluster,
// 305-430 when the reader polls the other SM's memory, ~900 through L2).
// An entry is the value and the slot it belongs to: two 64-bit words, each
// half of the value beside the 32-bit tag slot + 1, so a reader that finds its
// tag in both words has the whole value whatever the order the words landed
// in, any bit pattern is a valid value, and an entry overwritten by a later
// slot shows a later tag.  A reader then takes the value from the sweep's
// output in global memory, where every row also stores its result (armed with
// kPending on entry), and so does a row whose input lies kRingNear or more
// slots back.  So the ring needs no flow control: it is a cache of the last
// kRing results, and how far one warp runs ahead of another changes nothing
// but speed.
// ---------------------------------------------------------------------------
constexpr int kRing = 8192;
constexpr int kRingNear = kRing - 2048;
constexpr int kLaneMaxThreads = 256;
constexpr int kLaneW = 4;        // most entries of a window
constexpr int kLaneMaxRow = kRingSide;  // and of a row
// the ring, a spare entry of no tag, and spare entries of every thread
constexpr size_t kRingBytes = (size_t)(kRing + 1 + kLaneMaxThreads * kLaneW) * 16;

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// The launch shape a cluster kernel finds, checked against the one its host
// side sized the shared memory for (cluster width, grid, dynamic shared
// memory): a launch that arrives otherwise records an error (row = width << 16
// | grid) and does nothing, rather than index past its shared memory.  The
// decision is the same in every CTA, so no CTA is left at a cluster barrier.
__device__ __forceinline__ bool cluster_launch_ok(unsigned C, int expect_c, int expect_grid,
                                                  uint64_t smem_need, DevErr *err) {
  unsigned dyn;
  asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
  const bool ok = (int)C == expect_c && (int)gridDim.x == expect_grid && smem_need <= dyn;
  if (!ok && threadIdx.x == 0 && blockIdx.x == 0)
    set_err(err, ((int64_t)C << 16) | (int64_t)gridDim.x, ILUK_ECUDA);
  return ok;
}

struct RingCtx {
  unsigned rank, C, base;  // this CTA's rank and ring, the cluster's width
};

// Empty ring (tag 0 belongs to no slot); every CTA's ring is empty when this
// returns.
__device__ __forceinline__ void ring_start(const RingCtx &r, uint4 *ring) {
  for (int j = threadIdx.x; j <= kRing; j += blockDim.x) ring[j] = make_uint4(0u, 0u, 0u, 0u);
  cluster_sync_all();
}

__device__ __forceinline__ RingCtx ring_ctx(const uint4 *ring) {
  RingCtx r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r.rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r.C));
  r.base = (unsigned)__cvta_generic_to_shared(ring);
  return r;
}

// Value x of slot `sl` into the ring of CTA `cta`.
__device__ __forceinline__ void ring_put(unsigned base, unsigned cta, int64_t sl, double x) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(base), "r"(cta));
  a += ((unsigned)sl & (kRing - 1)) << 4;
  const unsigned long long tag = (unsigned long long)((unsigned)sl + 1u) << 32;
  asm volatile("st.relaxed.cluster.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(a),
               "l"(tag | (unsigned)__double2loint(x)), "l"(tag | (unsigned)__double2hiint(x))
               : "memory");
}

__device__ __forceinline__ void ring_put_local(unsigned base, int64_t sl, double x) {
  const unsigned tag = (unsigned)sl + 1u;
  asm volatile("st.volatile.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(
                   base + (((unsigned)sl & (kRing - 1)) << 4)),
               "r"((unsigned)__double2loint(x)), "r"(tag), "r"((unsigned)__double2hiint(x)),
               "r"(tag)
               : "memory");
}

// How often (in polls) a waiting warp looks at the clock, the error word and
// for overwritten entries: that is a round trip to L2, a poll is a shared-
// memory load.
constexpr unsigned kRingPolls = 256;

// ---------------------------------------------------------------------------
// Lockstep sweep on the ring: a warp takes a chunk, 32 rows of one level, a
// row per lane, and the lanes advance their chains together, a window of
// two or four entries at a time (lane_take), so one FP64 warp instruction serves 32 rows.
// An FP64 warp instruction holds its sub-partition's pipe ~76 cycles however
// few lanes it serves, so on short rows this is what a level costs: the
// hand-off, and the products and differences of the entries that arrive last.
// The rows of a chunk are right-aligned, so those are the last window of every
// row.  Where an entry's input sits in the walked order comes from the order's
// plan (LanePlan), its coefficient from F; both are loaded a whole chunk ahead
// of their use, and the rows they belong to one chunk earlier.  Chunk c belongs
// to CTA c mod C: neighbours of a level run on different SMs or
// sub-partitions.
// What bounds it: the latency of that chain, ~590 cycles a level forward.
// 2D 64^2 grid, k = 2 (253 levels): one application 0.335 ms with a warp per
// row on a cluster, 0.177 ms here on one SM; 2D 256^2 (1,021 levels) 1.49 ->
// 0.85 ms; 3D 20^3, k = 1 (115 levels) 0.215 -> 0.150 ms on four SMs.  Rows of
// more than 8 entries ran no faster than a warp per row at any size tried (three
// early windows: 3D 20^3, k = 2 0.37 / 0.30 ms; 64^3 1.51 / 1.52; 27-point grids
// lose by 1.1 to 2 times), so they do not take this.
// Other forms measured slower: windows of up to 16 entries polled together
// with the ready ones multiplied and subtracted as they came (the longer loop
// body costs more than it saves, 1.6 ms on 256^2), and levels separated by
// barriers instead of polled values with the loads of later levels between
// them (2.0 ms: the barrier waits for the slowest warp's bookkeeping).
// ---------------------------------------------------------------------------
constexpr int kLaneThreads1 = 256;  // one CTA: more warps, to load further ahead
constexpr int kLaneThreads = 128;   // a cluster: a warp per sub-partition

struct LaneMeta {
  int64_t first, coff;  // position of the chain's first entry; the chunk's plan rows
  int32_t row, len, w;  // row (-1: padding), chain length, longest chain of the chunk
};

template <int W>
struct LaneWin {
  int sl[W];  // slot of the input; far_code(row): read from global memory; kNoSlot: none
  double f[W];
};
constexpr int kNoSlot = INT_MAX;  // reads the spare entry

// A far input (row 0 .. INT_MAX - 1) in a plan: negative, and its tag, code + 1
// like a slot's, has the top bit set.  No slot's tag has it, nor has the tag 0
// of the entries that no slot has reached, so a far input is never taken for
// one that the ring holds.  (~row is no such code: row 0's tag would be 0.)
__host__ __device__ constexpr int far_code(int row) { return -2 - row; }
__host__ __device__ constexpr int far_row(int code) { return -2 - code; }
static_assert(far_code(0) < 0 && (unsigned)far_code(0) + 1u > (unsigned)INT_MAX &&
                  far_code(INT_MAX - 1) < 0 &&
                  (unsigned)far_code(INT_MAX - 1) + 1u > (unsigned)INT_MAX,
              "far inputs: negative codes, tags of no slot");

__device__ __forceinline__ void lane_meta(LaneMeta &m, const int32_t *__restrict__ order,
                                          const LanePlan &pl, int64_t c, int lane) {
  m.row = -1;
  m.len = m.w = 0;
  m.first = m.coff = 0;
  if (c < pl.nch) {
    const int64_t slot = c * 32 + lane;
    m.row = order[slot];
    m.len = pl.len[slot];
    m.first = pl.first[slot];
    m.coff = pl.coff[c];
    m.w = (int)(pl.coff[c + 1] - m.coff);
  }
}

// Entries q0 .. q0 + W - 1 (those >= 0) of the chunk's right-aligned chains.
template <bool FORWARD, int W>
__device__ __forceinline__ void lane_window(LaneWin<W> &wn, const LaneMeta &m, int q0,
                                            const int32_t *__restrict__ pslot,
                                            const double *__restrict__ v, int lane) {
  const int skip = m.w - m.len;
  const int32_t *ps = pslot + m.coff * 32 + lane;
  const double *pv = v + (FORWARD ? m.first - skip : m.first + skip);
#pragma unroll
  for (int u = 0; u < W; ++u) {
    const int e = q0 + u;
    wn.sl[u] = kNoSlot;
    wn.f[u] = 0.0;
    if (e >= skip && e >= 0) {
      wn.sl[u] = ps[e * 32];
      wn.f[u] = pv[FORWARD ? e : -e];
    }
  }
}

// Waits until every lane has the window's inputs, multiplies and subtracts
// them in order.  What follows the last arrival is on the sweep's critical
// path, so the loop holds nothing but the loads, the tag comparison and a
// vote, and the FP64 instructions come after it, unconditionally: one with
// every lane predicated off would hold the FP64 pipe as long.  An input
// that is not (or no longer) in the ring is copied from global memory into
// this thread's own spare entry, and then looked for there.
template <int W>
__device__ __forceinline__ bool lane_take(const LaneWin<W> &wn, double &s, unsigned base,
                                          unsigned own, const double *out,
                                          const int32_t *__restrict__ order, DevErr *err,
                                          int64_t limit_ns) {
  unsigned a[W], want[W];
  bool far = false;
#pragma unroll
  for (int u = 0; u < W; ++u) {
    // a lane without an entry takes +0.0 from the spare entry of no tag, and
    // subtracts 0 * 0, which changes no value
    const bool none = wn.sl[u] == kNoSlot;
    a[u] = base + ((none ? (unsigned)kRing : (unsigned)wn.sl[u] & (kRing - 1)) << 4);
    want[u] = none ? 0u : (unsigned)wn.sl[u] + 1u;
    far |= wn.sl[u] < 0;
  }
  double x[W];
  uint64_t t0 = 0;
  for (unsigned it = __any_sync(FULL_MASK, far) ? kRingPolls - 1 : 0;; ++it) {
    uint4 r[W];
    bool all = true;
#pragma unroll
    for (int u = 0; u < W; ++u)
      asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(r[u].x), "=r"(r[u].y), "=r"(r[u].z), "=r"(r[u].w)
                   : "r"(a[u]));
#pragma unroll
    for (int u = 0; u < W; ++u) {
      all = all && r[u].y == want[u] && r[u].w == want[u];
      x[u] = __hiloint2double((int)r[u].z, (int)r[u].x);
    }
    if (__all_sync(FULL_MASK, all)) break;
    if ((it & (kRingPolls - 1)) == kRingPolls - 1) {
      if (t0 == 0) t0 = globaltimer_ns();
      const bool stop = any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns;
      if (__any_sync(FULL_MASK, stop)) return false;  // the whole warp gives up together
      bool again = false;
#pragma unroll
      for (int u = 0; u < W; ++u) {
        if (wn.sl[u] == kNoSlot || (r[u].y == want[u] && r[u].w == want[u])) continue;
        const bool is_far = wn.sl[u] < 0;
        if (!is_far && r[u].y <= want[u] && r[u].w <= want[u]) continue;  // not there yet
        const double g = ld_val(&out[is_far ? far_row(wn.sl[u]) : order[wn.sl[u]]]);
        if (pending(g)) {
          again = true;
          continue;
        }
        a[u] = own + u * 16u;
        asm volatile("st.volatile.shared.v4.u32 [%0], {%1, %2, %3, %2};" ::"r"(a[u]),
                     "r"((unsigned)__double2loint(g)), "r"(want[u]),
                     "r"((unsigned)__double2hiint(g)));
      }
      if (__any_sync(FULL_MASK, again)) --it;
    }
  }
#pragma unroll
  for (int u = 0; u < W; ++u) x[u] = __dmul_rn(wn.f[u], x[u]);
#pragma unroll
  for (int u = 0; u < W; ++u) s = __dsub_rn(s, x[u]);
  return true;
}

// A row's entries (at most 2 W) sit right-aligned in two windows, both loaded a
// whole chunk ahead of their use.
template <int W>
struct LaneChunk {
  LaneMeta m;
  LaneWin<W> early, last;
  double s;
};

template <bool FORWARD, int W>
__device__ __forceinline__ void lane_chunk(LaneChunk<W> &ch, const int32_t *__restrict__ pslot,
                                           const double *__restrict__ v, const double *in,
                                           int lane) {
  lane_window<FORWARD, W>(ch.early, ch.m, ch.m.w - 2 * W, pslot, v, lane);
  lane_window<FORWARD, W>(ch.last, ch.m, ch.m.w - W, pslot, v, lane);
  ch.s = ch.m.row >= 0 ? in[ch.m.row] : 0.0;
}

template <bool FORWARD, bool DIVIDE, int W>
__global__ void __launch_bounds__(kLaneMaxThreads, 1)
k_sweep_lane(const int32_t *__restrict__ order, LanePlan pl, const double *__restrict__ v,
             const DivPrep *__restrict__ rd, const double *in, double *out, double *clear,
             DevErr *err, int64_t limit_ns, int expect_c) {
  extern __shared__ __align__(16) uint4 ring[];
  const RingCtx rc = ring_ctx(ring);
  if (!cluster_launch_ok(rc.C, expect_c, expect_c, kRingBytes, err)) return;
  ring_start(rc, ring);
  const int lane = threadIdx.x & 31;
  const unsigned own = rc.base + (unsigned)(kRing + 1 + threadIdx.x * kLaneW) * 16u;
  const int64_t step = (int64_t)rc.C * (blockDim.x >> 5);
  int64_t c = (int64_t)rc.rank + (int64_t)rc.C * (threadIdx.x >> 5);
  auto hand_over = [&](int64_t slot, double s) {
    if (rc.C == 1) {
      ring_put_local(rc.base, slot, s);
    } else {
      for (unsigned k = 1; k <= rc.C; ++k)
        ring_put(rc.base, (rc.rank + k) & (rc.C - 1), slot, s);
    }
  };
  // Level 1 comes first and reads no x.  Without a divisor its rows pass their right-
  // hand side through, and the marker becomes the quiet NaN that the other
  // schedules store.
  for (; c < pl.nch && pl.coff[c + 1] == pl.coff[c]; c += step) {
    const int64_t slot = c * 32 + lane;
    const int32_t row = order[slot];
    double s = row >= 0 ? in[row] : 0.0;
    if (DIVIDE && row >= 0) s = div_fin(s, rd[row]);
    if (pending(s)) s = __longlong_as_double((long long)kQuietNaN);
    if (clear && row >= 0) clear[row] = __longlong_as_double((long long)kPending);
    hand_over(slot, s);
    if (row >= 0) st_val(&out[row], s);
  }
  LaneChunk<W> cur, nxt;
  lane_meta(cur.m, order, pl, c, lane);
  lane_meta(nxt.m, order, pl, c + step, lane);
  lane_chunk<FORWARD, W>(cur, pl.slot, v, in, lane);
  bool ok = true;
  for (; c < pl.nch; c += step) {
    LaneMeta far;  // the rows of the chunk after the next one
    lane_meta(far, order, pl, c + 2 * step, lane);
    lane_chunk<FORWARD, W>(nxt, pl.slot, v, in, lane);
    const int32_t row = cur.m.row;
    DivPrep rr{0ull, 1.0};
    if (DIVIDE && row >= 0) rr = rd[row];
    if (clear && row >= 0) clear[row] = __longlong_as_double((long long)kPending);
    double s = cur.s;
    if (cur.m.w > W) ok = lane_take<W>(cur.early, s, rc.base, own, out, order, err, limit_ns);
    if (ok) ok = lane_take<W>(cur.last, s, rc.base, own, out, order, err, limit_ns);
    if (!ok) {
      if (row >= 0) set_err(err, row, ILUK_ETIMEOUT);
      break;
    }
    // (a padding lane has no divisor)
    if (DIVIDE && row >= 0) s = div_fin(s, rr);
    hand_over(c * 32 + lane, s);
    // (s comes from a subtraction or a division, never the signalling marker)
    if (row >= 0) st_val(&out[row], s);
    cur = nxt;
    nxt.m = far;
  }
  // every CTA arrives here: no shared memory is released while written to
  __syncwarp();
  cluster_sync_all();
}

// Plan of a padded order (LanePlan, internal.h).  Chain entry e of a row is
// its e-th in subtraction order.
template <bool FORWARD>
__global__ void k_lane_rows(const int32_t *__restrict__ order, int64_t nch,
                            const int64_t *__restrict__ rp, const int64_t *__restrict__ dg,
                            int32_t *slot_of, int64_t *first, int32_t *len, int32_t *w,
                            int32_t *maxw) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < nch; c += nw) {
    const int64_t slot = c * 32 + lane;
    const int32_t row = order[slot];
    int64_t f = 0;
    int l = 0;
    if (row >= 0) {
      slot_of[row] = (int32_t)slot;
      const int64_t d = dg[row];
      f = FORWARD ? rp[row] : rp[row + 1] - 1;
      l = (int)(FORWARD ? d - f : f - d);
    }
    first[slot] = f;
    len[slot] = l;
    const int m = __reduce_max_sync(FULL_MASK, l);
    if (lane == 0) {
      w[c] = m;
      atomicMax(maxw, m);
    }
  }
}

template <bool FORWARD>
__global__ void k_lane_slots(LanePlan pl, const int32_t *__restrict__ slot_of,
                             const int32_t *__restrict__ ci, int32_t *pslot,
                             unsigned long long *far) {
  unsigned long long beyond = 0;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < pl.nch; c += nw) {
    const int64_t slot = c * 32 + lane, f = pl.first[slot], off = pl.coff[c];
    const int len = pl.len[slot], w = (int)(pl.coff[c + 1] - off), skip = w - len;
    for (int e = 0; e < w; ++e) {
      int32_t v = 0;
      if (e >= skip) {
        const int32_t col = ci[FORWARD ? f + (e - skip) : f - (e - skip)];
        const int32_t sl = slot_of[col];
        const bool near = slot - sl < kRingNear;
        v = near ? sl : far_code(col);
        beyond += near ? 0 : 1;
      }
      pslot[(off + e) * 32 + lane] = v;
    }
  }
  if (beyond) atomicAdd(far, beyond);
}

// ---------------------------------------------------------------------------
// Warp-per-row schedules.  One warp owns one row (rows taken from the level
// order, so every dependency lies at an earlier position and is owned by a
// warp that is already running).  The lanes load and poll up to 32 entries at
// a time and form their products as soon as their values arrive; the warp
// then subtracts the longest ready prefix of the chain, in order, and goes
// back to polling only if the prefix stopped at a still-pending entry.  A row
// therefore pays, after its last dependency arrives, only for the rest of its
// own chain.  Below: values in the distributed shared memory of one
// thread-block cluster; k_sweep_grid: in global memory, over all SMs.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double ld_dsm(unsigned a) {
  unsigned long long v;
  asm volatile("ld.relaxed.cluster.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return __longlong_as_double((long long)v);
}

__device__ __forceinline__ void st_dsm(unsigned a, double x) {
  asm volatile("st.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(a),
               "l"((unsigned long long)__double_as_longlong(x))
               : "memory");
}

// Prefix helpers (ILUK_SCHED_WARP_CLUSTER_HELP).  The FP64 pipes of the
// cluster's SMs are kept busy by the rows' subtraction chains (one warp
// instruction per entry, however few lanes it serves), and that queueing
// delays the few FP64 operations on the critical path.  A second cluster of
// the same cooperative launch therefore takes most of each chain: its warps
// walk the slots in order, one row per warp, and for slot s, once the row at
// slot s - lag is final, subtract the products of the row's leading entries
// whose x is already final (read from a global copy of x that the row warps
// keep), stopping at the first one that is not, and publish the partial
// difference with the number of entries it covers.  The row's own warp,
// when it takes the row, starts from there.  Same products, same
// differences, same order: the result does not change.  A prefix is tagged
// with the launch's epoch (a device word the last CTA of the launch advances),
// so one left over from an earlier launch is never used; a row whose prefix
// is not published in time is simply done in full by its warp, which never
// waits for a helper.
template <bool FORWARD>
__device__ void sweep_prefixes(const int32_t *__restrict__ order, int64_t len,
                               const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                               const int64_t *__restrict__ dg, const double *__restrict__ v,
                               const double *in, const double *xg, double *pre_s,
                               unsigned long long *pre_k, unsigned epoch, int64_t hid,
                               int64_t hp, int64_t lag, const DevErr *err, int64_t limit_ns,
                               int lane) {
  for (int64_t slot = hid; slot < len; slot += hp) {
    const int64_t ps = slot - lag;
    if (ps >= 0) {  // pace: start once the row at slot ps is final
      bool ok = true;
      if (lane == 0) {
        const double *pa = &xg[order[ps]];
        const uint64_t t0 = globaltimer_ns();
        for (unsigned it = 0;; ++it) {
          if (!pending(ld_val(pa))) break;
          if ((it & 15u) == 15u &&
              (any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns)) {
            ok = false;
            break;
          }
          __nanosleep(128);
        }
      }
      if (!__shfl_sync(FULL_MASK, ok ? 1 : 0, 0)) return;  // stop helping
    }
    const int64_t row = order[slot];
    if (!pending(ld_val(&xg[row]))) continue;  // the row is done already
    const int64_t d = dg[row];
    const int64_t first = FORWARD ? rp[row] : rp[row + 1] - 1;
    const int mylen = (int)(FORWARD ? d - first : first - d);
    constexpr int64_t step = FORWARD ? 1 : -1;
    double s = in[row];
    int covered = 0;
    for (int b = 0; b < mylen; b += 32) {
      const int e = b + lane;
      const int cnt = mylen - b < 32 ? mylen - b : 32;
      double prod = 0.0;
      bool have = e >= mylen;
      if (e < mylen) {
        const double x = ld_val(&xg[ci[first + step * e]]);
        if (!pending(x)) {
          prod = __dmul_rn(v[first + step * e], x);
          have = true;
        }
      }
      const unsigned ready = __ballot_sync(FULL_MASK, have);
      const int run = ready == FULL_MASK ? 32 : __ffs(~ready) - 1;
      const int upto = run < cnt ? run : cnt;
      for (int j = 0; j < upto; ++j) s = __dsub_rn(s, __shfl_sync(FULL_MASK, prod, j));
      covered += upto;
      if (upto < cnt) break;
    }
    if (covered > 0 && lane == 0) {
      pre_s[row] = s;
      __threadfence();  // the difference before the count that publishes it
      asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(pre_k + row),
                   "l"(((unsigned long long)epoch << 32) | (unsigned)covered)
                   : "memory");
    }
    __syncwarp();
  }
}

template <bool FORWARD, bool DIVIDE>
__device__ __forceinline__ void
sweep_wpr_body(const int32_t *__restrict__ order, int64_t len, int64_t n,
               const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
               const int64_t *__restrict__ dg, const double *__restrict__ v,
               const DivPrep *__restrict__ rd, const double *in, double *out, double *clear,
               DevErr *err, int64_t limit_ns, const int32_t *__restrict__ owner, double *pre_s,
               unsigned long long *pre_k, unsigned *aux_words, int64_t lag, int expect_c,
               int expect_grid) {
  // x_i lives in the shared memory of the CTA whose warp computes
  // row i, at slot (k * wpc + warp) for the warp's k-th row; owner[i] holds
  // (rank << 26 | slot), so the producer's store stays on its own SM and only
  // the dependants' polls cross SMs.  With prefix helpers (pre_s non-null) the
  // launch holds a second cluster of helper CTAs (blockIdx.x >= C), and the
  // row warps also keep x in `out` (armed with kPending on entry) for them.
  extern __shared__ __align__(16) double xs[];
  unsigned rank = 0, C = 1, base = 0;
  const int wpc = blockDim.x >> 5;  // warps per CTA
  const bool help = pre_s != nullptr;
  const unsigned epoch = help ? *((volatile unsigned *)aux_words) : 0u;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  const int64_t nw = (int64_t)C * wpc;
  const int64_t slice = (len + nw - 1) / nw * wpc;
  if (!cluster_launch_ok(C, expect_c, expect_grid, (uint64_t)slice * sizeof(double), err)) return;
  for (int64_t j = threadIdx.x; j < slice; j += blockDim.x)
    xs[j] = __longlong_as_double((long long)kPending);
  base = (unsigned)__cvta_generic_to_shared(xs);
  cluster_sync_all();
  const int lane = threadIdx.x & 31;
  const int64_t gw = (int64_t)rank * wpc + (threadIdx.x >> 5);
  unsigned own_slot = 0;  // the slot of this warp's current row
  unsigned own_base = 0;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(own_base) : "r"(base), "r"(rank));
  bool ok = true;
  if (help && blockIdx.x >= C) {  // a helper CTA: no rows of its own
    const int hw = (int)(blockDim.x >> 5);
    sweep_prefixes<FORWARD>(order, len, rp, ci, dg, v, in, out, pre_s, pre_k, epoch,
                            (int64_t)(blockIdx.x - C) * hw + (threadIdx.x >> 5),
                            (int64_t)(gridDim.x - C) * hw, lag, err, limit_ns, lane);
    ok = false;
  }
  for (int64_t slot = gw; slot < len && ok; slot += nw, own_slot += wpc) {
    const int64_t row = order[slot];
    if (row < 0) continue;
    const int64_t d = dg[row];
    DivPrep rr{0ull, 1.0};
    if (DIVIDE) rr = rd[row];  // u_ii and its reciprocal, fetched off the chain
    const int64_t first = FORWARD ? rp[row] : rp[row + 1] - 1;
    const int mylen = (int)(FORWARD ? d - first : first - d);
    constexpr int64_t step = FORWARD ? 1 : -1;
    double s = in[row];
    int k0 = 0;  // leading entries a helper has subtracted already
    if (help) {
      unsigned long long pk = 0;
      if (lane == 0)
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(pk) : "l"(pre_k + row));
      pk = __shfl_sync(FULL_MASK, pk, 0);
      if ((unsigned)(pk >> 32) == epoch) {
        __threadfence();  // the difference was written before the count
        k0 = (int)(pk & 0xffffffffu);
        s = ld_val(&pre_s[row]);
      }
    }
    // where x_row goes: this CTA's slot for the warp's current row
    const unsigned sa = own_base + ((own_slot + (threadIdx.x >> 5)) << 3);
    if (clear && lane == 0) clear[row] = __longlong_as_double((long long)kPending);
    bool stored = false;  // the last-entry path below stored x_row already
    for (int b = k0; b < mylen && ok; b += 32) {
      const int e = b + lane;
      const bool act = e < mylen;
      const int cnt = (mylen - b) < 32 ? mylen - b : 32;
      const bool last_batch = b + 32 >= mylen;
      int32_t c = 0;
      unsigned da = 0;
      double f = 0.0, x = 0.0, prod = 0.0;
      bool have = !act;
      if (act) {
        c = ci[first + step * e];
        f = v[first + step * e];
        const unsigned oc = (unsigned)owner[c];
        unsigned a;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(base), "r"(oc >> 26));
        da = a + ((oc & ((1u << 26) - 1u)) << 3);
        x = ld_dsm(da);
        if (!pending(x)) {
          prod = __dmul_rn(f, x);
          have = true;
        }
      }
      int done = 0;
      const uint64_t t0 = globaltimer_ns();
      for (unsigned it = 0;; ++it) {
        const unsigned ready = __ballot_sync(FULL_MASK, have);
        const unsigned rest = ~(ready >> done);  // first not-ready lane at or after `done`
        const int run = rest == 0u ? 32 - done : __ffs(rest) - 1;
        const int upto = done + run < cnt ? done + run : cnt;
        for (int j = done; j < upto; ++j) s = __dsub_rn(s, __shfl_sync(FULL_MASK, prod, j));
        done = upto;
        if (done >= cnt) break;
        if (last_batch && done == cnt - 1) {
          // Only the row's last entry is missing (most often the one from
          // the row that finished last): the lane that owns it polls alone,
          // then subtracts, divides and stores, with no warp vote or shuffle
          // between the value's arrival and the store.  Same operations,
          // same order.
          bool gave_up = false;
          if (lane == done) {
            for (unsigned jt = 0; !have; ++jt) {
              x = ld_dsm(da);
              if (!pending(x)) {
                prod = __dmul_rn(f, x);
                have = true;
              } else if ((jt & 15u) == 15u &&
                         (any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns)) {
                gave_up = true;
                break;
              }
            }
            if (!gave_up) {
              double r = __dsub_rn(s, prod);
              if (DIVIDE) r = div_fin(r, rr);
              if ((unsigned long long)__double_as_longlong(r) == kPending)
                r = __longlong_as_double((long long)kQuietNaN);
              st_dsm(sa, r);
              if (help) st_val(&out[row], r);  // the helpers' copy
            }
          }
          ok = __shfl_sync(FULL_MASK, gave_up ? 0 : 1, done) != 0;
          stored = ok;
          break;
        }
        const bool stop = (it & 15u) == 15u &&
                          (any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns);
        if (__any_sync(FULL_MASK, stop)) {
          ok = false;
          break;
        }
        // spin: a DSMEM poll is cheap and sleeping measured slower
        if (!have) {
          x = ld_dsm(da);
          if (!pending(x)) {
            prod = __dmul_rn(f, x);
            have = true;
          }
        }
      }
    }
    if (!ok) {
      if (lane == 0) set_err(err, row, ILUK_ETIMEOUT);
      break;
    }
    if (stored) {
      __syncwarp();
      continue;
    }
    if (DIVIDE) s = div_fin(s, rr);
    if ((unsigned long long)__double_as_longlong(s) == kPending)
      s = __longlong_as_double((long long)kQuietNaN);
    if (lane == 0) {
      st_dsm(sa, s);
      if (help) st_val(&out[row], s);  // the helpers' copy
    }
    __syncwarp();
  }
  cluster_sync_all();
  if (!help)  // with helpers every row already wrote its x to out
    for (int64_t j = threadIdx.x; j < slice; j += blockDim.x) {
      const int64_t pos = (j / wpc) * nw + (int64_t)rank * wpc + j % wpc;
      if (pos < len) out[order[pos]] = xs[j];
    }
  if (help) {
    // the last CTA to finish advances the epoch: every CTA read it at its
    // start and published its last prefix before arriving here
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(&aux_words[1], 1u) == gridDim.x - 1) {
        aux_words[1] = 0u;
        __threadfence();
        aux_words[0] = epoch + 1u == 0xffffffffu ? 0u : epoch + 1u;
      }
    }
  }
}

#define ILUK_WPR_PARAMS                                                                     \
  const int32_t *__restrict__ order, int64_t len, int64_t n, const int64_t *__restrict__ rp,  \
      const int32_t *__restrict__ ci, const int64_t *__restrict__ dg,                         \
      const double *__restrict__ v, const DivPrep *__restrict__ rd, const double *in,         \
      double *out, double *clear, DevErr *err, int64_t limit_ns,                              \
      const int32_t *__restrict__ owner, double *pre_s, unsigned long long *pre_k,            \
      unsigned *aux_words, int64_t lag, int expect_c, int expect_grid
#define ILUK_WPR_ARGS                                                                      \
  order, len, n, rp, ci, dg, v, rd, in, out, clear, err, limit_ns, owner, pre_s, pre_k,     \
      aux_words, lag, expect_c, expect_grid

// Warp-per-row sweeps on one cluster whose width the launch gives.
template <bool FORWARD, bool DIVIDE>
__global__ void __launch_bounds__(kCtaThreads, 1) k_sweep_wpr(ILUK_WPR_PARAMS) {
  sweep_wpr_body<FORWARD, DIVIDE>(ILUK_WPR_ARGS);
}

// The helped form: a cooperative launch of two clusters of kHelpCluster CTAs,
// the sweep's and the helpers'.  The cluster width is part of the kernel
// (not an attribute of the launch), so every path that launches it gets it.
constexpr int kHelpCluster = 16;
template <bool FORWARD, bool DIVIDE>
__global__ void __cluster_dims__(kHelpCluster, 1, 1) __launch_bounds__(kCtaThreads, 1)
    k_sweep_wpr_help(ILUK_WPR_PARAMS) {
  sweep_wpr_body<FORWARD, DIVIDE>(ILUK_WPR_ARGS);
}
#undef ILUK_WPR_PARAMS
#undef ILUK_WPR_ARGS

// ---------------------------------------------------------------------------
// Warp-per-row sweep over all SMs (WARP_GRID), x in global memory.  A row costs
// four dependent loads before its first look at x (its index, its position, its
// entries, x), and only a few levels' rows are in flight, so while a warp
// waits for one row's inputs it loads the next row's: index two rows ahead,
// position, right-hand side and divisor one row ahead, the entries once those
// are there.  What bounds it: an L2 hand-off a level (~1,900 cycles a level with
// the rest of the chain), and on the widest DAGs the FP64 unit, one warp
// instruction an entry (27-point 90^3).  One application, without the loads
// ahead -> with them: 3D 64^3 k = 2 1.48 -> 1.35 ms, 72^3 k = 0 0.72 -> 0.50, 27-point
// 90^3 k = 0 2.22 -> 1.88, 50^3 k = 1 1.39 -> 1.32 ms.  Tried and slower or no
// faster: a row per lane (32 rows wait for the slowest of their inputs: 64^3
// 1.75 ms, 90^3 1.90), two rows a warp (64^3 1.48 ms; 90^3 1.69).
// ---------------------------------------------------------------------------
constexpr unsigned kGridSleep = 32u;  // longest pause between looks, ns

struct GridRow {
  int64_t row, first;
  int len;
  double s;
  DivPrep rr;
};

template <bool FORWARD, bool DIVIDE>
__device__ __forceinline__ void grid_row(GridRow &g, int64_t row, const int64_t *__restrict__ rp,
                                         const int64_t *__restrict__ dg,
                                         const DivPrep *__restrict__ rd, const double *in) {
  g.row = row;
  g.first = 0;
  g.len = 0;
  g.s = 0.0;
  g.rr = DivPrep{0ull, 1.0};
  if (row >= 0) {
    const int64_t d = dg[row];
    g.first = FORWARD ? rp[row] : rp[row + 1] - 1;
    g.len = (int)(FORWARD ? d - g.first : g.first - d);
    if (DIVIDE) g.rr = rd[row];
    g.s = in[row];
  }
}

template <bool FORWARD, bool DIVIDE>
__global__ void __launch_bounds__(kCtaThreads, 1)
k_sweep_grid(const int32_t *__restrict__ order, int64_t len, const int64_t *__restrict__ rp,
             const int32_t *__restrict__ ci, const int64_t *__restrict__ dg,
             const double *__restrict__ v, const DivPrep *__restrict__ rd, const double *in,
             double *out, double *clear, DevErr *err, int64_t limit_ns) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  constexpr int64_t step = FORWARD ? 1 : -1;
  auto index = [&](int64_t slot) { return slot < len ? (int64_t)order[slot] : (int64_t)-1; };
  GridRow cur, nxt;
  grid_row<FORWARD, DIVIDE>(cur, index(gw), rp, dg, rd, in);
  int64_t r1 = index(gw + nw);
  int32_t c = 0, cn = 0;
  double f = 0.0, fn = 0.0;
  if (lane < cur.len) {
    c = ci[cur.first + step * lane];
    f = v[cur.first + step * lane];
  }
  for (int64_t slot = gw; slot < len; slot += nw) {
    const int64_t r2 = index(slot + 2 * nw);
    grid_row<FORWARD, DIVIDE>(nxt, r1, rp, dg, rd, in);
    if (clear && lane == 0) clear[cur.row] = __longlong_as_double((long long)kPending);
    double s = cur.s, res = 0.0;
    bool fetched = false;  // the next row's entries are on their way
    auto fetch = [&]() {
      fetched = true;
      if (lane < nxt.len) {
        cn = ci[nxt.first + step * lane];
        fn = v[nxt.first + step * lane];
      }
    };
    bool ok = true, stored = false;
    for (int b = 0; b < cur.len && ok; b += 32) {
      const int e = b + lane;
      const bool act = e < cur.len;
      const int cnt = (cur.len - b) < 32 ? cur.len - b : 32;
      const bool last_batch = b + 32 >= cur.len;
      if (b > 0 && act) {
        c = ci[cur.first + step * e];
        f = v[cur.first + step * e];
      }
      double x = 0.0, prod = 0.0;
      bool have = !act;
      auto look = [&]() {
        x = ld_val(&out[c]);
        if (!pending(x)) {
          prod = __dmul_rn(f, x);
          have = true;
        }
      };
      if (act) look();
      if (!fetched) fetch();
      int done = 0;
      const uint64_t t0 = globaltimer_ns();
      unsigned backoff = 8;
      for (unsigned it = 0;; ++it) {
        const unsigned ready = __ballot_sync(FULL_MASK, have);
        const unsigned rest = ~(ready >> done);  // first not-ready lane at or after `done`
        const int run = rest == 0u ? 32 - done : __ffs(rest) - 1;
        const int upto = done + run < cnt ? done + run : cnt;
        for (int j = done; j < upto; ++j) s = __dsub_rn(s, __shfl_sync(FULL_MASK, prod, j));
        done = upto;
        if (done >= cnt) break;
        if (last_batch && done == cnt - 1) {
          // only the row's last entry is missing: the lane that owns it
          // finishes the row alone, with no vote or shuffle in between
          bool gave_up = false;
          if (lane == done) {
            for (unsigned jt = 0; !have; ++jt) {
              look();
              if (have) break;
              if ((jt & 15u) == 15u &&
                  (any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns)) {
                gave_up = true;
                break;
              }
              __nanosleep(backoff);
              if (backoff < kGridSleep) backoff <<= 1;
            }
            if (!gave_up) {
              res = __dsub_rn(s, prod);
              if (DIVIDE) res = div_fin(res, cur.rr);
              if ((unsigned long long)__double_as_longlong(res) == kPending)
                res = __longlong_as_double((long long)kQuietNaN);
              st_val(&out[cur.row], res);
            }
          }
          ok = __shfl_sync(FULL_MASK, gave_up ? 0 : 1, done) != 0;
          stored = ok;
          break;
        }
        const bool stop = (it & 15u) == 15u &&
                          (any_failed(err) || (int64_t)(globaltimer_ns() - t0) > limit_ns);
        if (__any_sync(FULL_MASK, stop)) {
          ok = false;
          break;
        }
        // back off: L2 polls compete with the stores they wait for
        __nanosleep(backoff);
        if (backoff < kGridSleep) backoff <<= 1;
        if (!have) look();
      }
    }
    if (!ok) {
      if (lane == 0) set_err(err, cur.row, ILUK_ETIMEOUT);
      return;
    }
    if (!fetched) fetch();
    if (!stored) {
      if (DIVIDE) s = div_fin(s, cur.rr);
      if ((unsigned long long)__double_as_longlong(s) == kPending)
        s = __longlong_as_double((long long)kQuietNaN);
      if (lane == 0) st_val(&out[cur.row], s);
    }
    __syncwarp();
    cur = nxt;
    c = cn;
    f = fn;
    r1 = r2;
  }
}

// owner[order[pos]] = (rank << 26 | slot) for the CTA layout above.
__global__ void k_owner_codes(const int32_t *__restrict__ order, int64_t len, int C, int wpc,
                              int32_t *owner) {
  const int64_t nw = (int64_t)C * wpc;
  for (int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; pos < len;
       pos += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = pos % nw;
    const int64_t slot = (pos / nw) * wpc + g % wpc;
    owner[order[pos]] = (int32_t)(((g / wpc) << 26) | slot);
  }
}

// The (cached) owner codes of a level order for one cluster and CTA width.
static std::mutex g_owner_mu;
static const int32_t *owner_codes(const LevelOrder &lo_c, int64_t n, int C, int threads,
                                  cudaStream_t s) {
  LevelOrder &lo = const_cast<LevelOrder &>(lo_c);  // a cache of the order
  std::lock_guard<std::mutex> lk(g_owner_mu);
  for (OwnerCode &oc : lo.owner)
    if (oc.code && oc.C == C && oc.threads == threads) return oc.code;
  OwnerCode *slot = nullptr;
  for (OwnerCode &oc : lo.owner)
    if (!oc.code) {
      slot = &oc;
      break;
    }
  if (!slot) {  // full: reuse the first entry (stream order keeps its users safe)
    slot = &lo.owner[0];
    cudaFreeAsync(slot->code, s);
    slot->code = nullptr;
  }
  if (cudaMallocAsync((void **)&slot->code, (size_t)(n > 0 ? n : 1) * sizeof(int32_t), s) !=
      cudaSuccess) {
    slot->code = nullptr;
    return nullptr;
  }
  int64_t b = (lo.clen + 255) / 256;
  if (b > (int64_t)num_sms() * 8) b = (int64_t)num_sms() * 8;
  if (b < 1) b = 1;
  k_owner_codes<<<(unsigned)b, 256, 0, s>>>(lo.corder, lo.clen, C, threads / 32, slot->code);
  note_launch();
  slot->C = C;
  slot->threads = threads;
  return slot->code;
}

static unsigned row_blocks(int64_t n) {
  int64_t b = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms() * 8;
  return (unsigned)(b > cap ? cap : b < 1 ? 1 : b);
}

// What the ring kernels need beside a level order, built once per order and
// kept with it, in at most an eighth of the free memory (rows in levels of one take
// 512 bytes each, most of them padding); an order that was refused for that stays
// with the other kinds.  (Asking costs 12 us, 0.4 % of a one-call solve on 2D 64^2:
// up to 64 MB it is not done.)  Nothing is built while `s` is being captured.
constexpr size_t kPlanUnasked = 64u << 20;
static std::mutex g_plan_mu;

static bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cs);
  return cs != cudaStreamCaptureStatusNone;
}

template <bool FORWARD>
static bool ensure_lane_plan(const LevelOrder &lo_c, int64_t n, const int64_t *rp,
                             const int32_t *ci, const int64_t *dg, cudaStream_t s) {
  LevelOrder &lo = const_cast<LevelOrder &>(lo_c);  // a cache of the order
  std::lock_guard<std::mutex> lk(g_plan_mu);
  if (lo.plan.slot) return true;
  if (!lo.order || lo.plan.maxw > kLaneMaxRow || lo.plan.refused || capturing(s)) return false;
  if (lo.longest > kLaneMaxRow) {  // not for these sweeps: remembered by maxw
    lo.plan.maxw = lo.longest;
    return false;
  }
  const size_t need = (size_t)lo.len * (12 + 4 * (size_t)lo.longest);
  if (need > kPlanUnasked) {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || need > free_b / 8) {
      cudaGetLastError();
      lo.plan.refused = true;
      return false;
    }
  }
  LanePlan pl;
  pl.nch = lo.len / 32;
  int32_t *slot_of = nullptr, *w = nullptr, *len = nullptr, *pslot = nullptr;
  int64_t *first = nullptr, *coff = nullptr, *scan_tmp = nullptr;
  unsigned long long far = 0;
  auto free_all = [&](bool keep) {
    for (void *p : {(void *)slot_of, (void *)w, (void *)scan_tmp})
      if (p) cudaFreeAsync(p, s);
    if (!keep) {
      for (void *p : {(void *)len, (void *)first, (void *)coff, (void *)pslot})
        if (p) cudaFreeAsync(p, s);
      cudaGetLastError();
    }
    return keep;
  };
  const size_t nch = (size_t)pl.nch;
  if (cudaMallocAsync((void **)&slot_of, (size_t)n * 4, s) != cudaSuccess ||
      cudaMallocAsync((void **)&w, (nch + 1) * 4, s) != cudaSuccess ||
      cudaMemsetAsync(w + nch, 0, 4, s) != cudaSuccess ||
      cudaMallocAsync((void **)&len, nch * 32 * 4, s) != cudaSuccess ||
      cudaMallocAsync((void **)&first, nch * 32 * 8, s) != cudaSuccess ||
      cudaMallocAsync((void **)&coff, (nch + 1) * 8, s) != cudaSuccess ||
      cudaMallocAsync((void **)&scan_tmp, (size_t)scan_tmp_elems(pl.nch) * 8, s) != cudaSuccess)
    return free_all(false);
  k_lane_rows<FORWARD><<<row_blocks(lo.len), 256, 0, s>>>(lo.order, pl.nch, rp, dg, slot_of,
                                                          first, len, w, w + nch);
  note_launch();
  int64_t rows = 0;
  int32_t maxw = 0;
  if (launch_scan_lengths(pl.nch, w, coff, scan_tmp, s) != cudaSuccess ||
      cudaMemcpyAsync(&rows, coff + nch, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&maxw, w + nch, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return free_all(false);
  pl.maxw = maxw;
  if (cudaMallocAsync((void **)&pslot, (size_t)(rows > 0 ? rows : 1) * 32 * 4, s) != cudaSuccess)
    return free_all(false);
  pl.len = len;
  pl.first = first;
  pl.coff = coff;
  // (the scan is done with its scratch)
  unsigned long long *dfar = reinterpret_cast<unsigned long long *>(scan_tmp);
  if (cudaMemsetAsync(dfar, 0, sizeof(far), s) != cudaSuccess) return free_all(false);
  k_lane_slots<FORWARD><<<row_blocks(lo.len), 256, 0, s>>>(pl, slot_of, ci, pslot, dfar);
  note_launch();
  // complete before another stream's sweep may find it
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&far, dfar, sizeof(far), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return free_all(false);
  pl.far = (int64_t)far;
  pl.slot = pslot;
  lo.plan = pl;
  return free_all(true);
}

// An input from beyond the ring costs its chunk a look at the clock, the error word
// and global memory, ~1 us, so a chunk in few may have one: random bands, whose
// rows without inputs all lie in level 1, run 2.5 times slower on the ring than on
// a cluster (n = 40,000, 3 a row, half-width 300: 1.31 / 0.52 ms an application).
bool ring_suits(bool forward, int64_t n, const int64_t *rp, const int32_t *ci, const int64_t *dg,
                const LevelOrder &lo, cudaStream_t s) {
  const bool planned = forward ? ensure_lane_plan<true>(lo, n, rp, ci, dg, s)
                               : ensure_lane_plan<false>(lo, n, rp, ci, dg, s);
  return planned && 100 * lo.plan.far <= lo.entries;
}

__global__ void k_fill_pending(int64_t n, double *x, unsigned long long bits) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = __longlong_as_double((long long)bits);
}

static cudaError_t fill_bits(int64_t n, double *x, unsigned long long bits, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int64_t b = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms() * 8;
  if (b > cap) b = cap;
  k_fill_pending<<<(unsigned)b, 256, 0, s>>>(n, x, bits);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_fill_pending(int64_t n, double *x, cudaStream_t s) {
  return fill_bits(n, x, kPending, s);
}

cudaError_t launch_fill_value(int64_t n, double *x, double v, cudaStream_t s) {
  unsigned long long bits;
  std::memcpy(&bits, &v, sizeof bits);
  return fill_bits(n, x, bits, s);
}

// q_i = a_i / b_i through div_prep + div_fin, the division of the numeric
// phase's multipliers and of the sweeps.
__global__ void k_div_check(int64_t n, const double *__restrict__ a,
                            const double *__restrict__ b, double *__restrict__ q) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    q[i] = div_int(a[i], b[i]);
}

cudaError_t launch_div_check(int64_t n, const double *a, const double *b, double *q,
                             cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int64_t g = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms() * 8;
  if (g > cap) g = cap;
  k_div_check<<<(unsigned)g, 256, 0, s>>>(n, a, b, q);
  note_launch();
  return cudaGetLastError();
}

// Cluster width for n rows: the largest of 16, 8, 4, 2 (at most `widest`)
// whose slices of x, or `fixed` bytes, fit in one CTA's shared memory and that
// the device can schedule (0 when none).
template <typename K>
static int cluster_width(int64_t n, K kern, size_t fixed = 0, int widest = 16) {
  static int cached[64][2] = {};  // per kernel type, as every static of a template
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  const size_t budget = (size_t)max_smem_optin() - 1024;
  for (int C : {16, 8, 4, 2}) {
    if (C > widest) continue;
    const size_t smem = fixed ? fixed : (size_t)((n + C - 1) / C) * sizeof(double);
    if (smem > budget) continue;
    {
      std::lock_guard<std::mutex> lk(mu);
      // schedulable widths do not depend on n beyond the shared memory size
      if (dev < 64 && cached[dev][0] == C && (size_t)cached[dev][1] >= smem) return C;
    }
    if (allow_smem(kern) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3(fixed ? kLaneMaxThreads : kCtaThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters >= 1) {
      std::lock_guard<std::mutex> lk(mu);
      if (dev < 64) {
        cached[dev][0] = C;
        cached[dev][1] = (int)smem;
      }
      return C;
    }
    cudaGetLastError();
  }
  return 0;
}

// Cluster width of the lockstep ring sweep on this device: four SMs, enough for
// the levels it suits (eight or sixteen measured the same or slower: every
// result goes to each CTA's ring), or two (0 when neither can be scheduled).
static int ring_cluster() {
  return cluster_width((int64_t)0, k_sweep_lane<true, false, 4>, kRingBytes, 4);
}

template <typename K, typename... Args>
static cudaError_t launch_on_cluster(K kern, int C, int threads, size_t smem, cudaStream_t s,
                                     Args... args) {
  cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, args...);
  note_launch();
  return e;
}

// The helped sweep: two clusters (width from the kernel), launched
// cooperatively, so every CTA is resident at once or the launch fails: the
// helper CTAs wait on the sweep's.
template <typename K, typename... Args>
static cudaError_t launch_help(K kern, int threads, size_t smem, cudaStream_t s, Args... args) {
  cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * kHelpCluster));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, args...);
  note_launch();
  return e;
}

// Slots beyond the row warps' own span at which a prefix helper starts a row
// (it waits until the row `lag` slots earlier is final): late enough that
// most of the row's leading entries are final, early enough to publish before
// the row's warp takes the row.  Measured on the random band matrix with
// n = 160,000, k = 2: forward best at 384-512, backward at 256.
constexpr int64_t kHelpLagFwd = 448;
constexpr int64_t kHelpLagBwd = 256;

template <bool FORWARD, bool DIVIDE>
static cudaError_t run_sweep(int64_t n, const LevelOrder &lo, const int64_t *rp, const int32_t *ci,
                             const int64_t *dg, const double *v, const DivPrep *rd,
                             const double *in, double *out, double *clear, int sched, DevErr *err,
                             const SweepAux *aux, cudaStream_t s) {
  ProfScope prof_scope(FORWARD ? ILUK_PROF_SWEEP : ILUK_PROF_SWEEP_BWD, s);
  // an empty order: nothing to sweep (n = 0, or a direction the caller skips)
  if (n == 0 || (!lo.order && !lo.corder)) return cudaSuccess;
  int64_t limit = wait_limit();
  const int w = (sched >> 4) & 0xf;  // CTA width / 128 of the warp-per-row kinds
  const int threads = w ? w * 128 : kCtaThreads;
  int kind = sched & 0xf;
  if (kind == ILUK_SCHED_SINGLE_CTA || kind == ILUK_SCHED_CLUSTER) {
    if (!lo.order) return cudaErrorInvalidValue;  // an index order: no levels to walk
    if (ensure_lane_plan<FORWARD>(lo, n, rp, ci, dg, s)) {
      const bool one = kind == ILUK_SCHED_SINGLE_CTA;
      const int C = one ? 1 : ring_cluster();
      const auto kern = lo.plan.maxw <= 4 ? k_sweep_lane<FORWARD, DIVIDE, 2>
                                          : k_sweep_lane<FORWARD, DIVIDE, 4>;
      return launch_on_cluster(kern, C, one ? kLaneThreads1 : kLaneThreads, kRingBytes, s,
                               (const int32_t *)lo.order, lo.plan, v, rd, in, out, clear, err,
                               limit, C);
    }
    // rows too long for a lane, or no plan (a capture before the first use)
    kind = ILUK_SCHED_WARP_GRID;
  }
  if (kind == ILUK_SCHED_WARP_CLUSTER || kind == ILUK_SCHED_WARP_CLUSTER_HELP) {
    if (!lo.corder) return cudaErrorInvalidValue;
    // one warp per row needs no warp-aligned levels: the unpadded order keeps
    // every warp's next row further ahead and wastes no slot loads
    const int32_t *order = lo.corder;
    const int64_t len = lo.clen;
    const int C = cluster_width(n, k_sweep_wpr<FORWARD, DIVIDE>);
    if (C == 0) return cudaErrorInvalidConfiguration;
    const int wpc = threads / 32;
    const int64_t nwc = (int64_t)C * wpc;
    const size_t wsmem = (size_t)((len + nwc - 1) / nwc * wpc) * sizeof(double);
    if (wsmem > (size_t)max_smem_optin()) return cudaErrorInvalidConfiguration;
    const int32_t *owner = owner_codes(lo, n, C, threads, s);
    if (!owner) return cudaErrorMemoryAllocation;
    double *no_ps = nullptr;
    unsigned long long *no_pk = nullptr;
    unsigned *no_words = nullptr;
    // the helped kind needs its scratch; without it, the plain cluster kind
    if (kind == ILUK_SCHED_WARP_CLUSTER_HELP && aux && aux->pre_s && aux->n >= n &&
        C == kHelpCluster) {  // a second cluster of prefix helpers
      const int64_t lag = (FORWARD ? kHelpLagFwd : kHelpLagBwd) + nwc;
      const cudaError_t e =
          launch_help(k_sweep_wpr_help<FORWARD, DIVIDE>, threads, wsmem, s, order, len, n, rp,
                      ci, dg, v, rd, in, out, clear, err, limit, owner, aux->pre_s, aux->pre_k,
                      aux->words, lag, C, 2 * C);
      if (e == cudaSuccess) return e;
      cudaGetLastError();  // cannot hold both clusters at once: the plain kind
    }
    return launch_on_cluster(k_sweep_wpr<FORWARD, DIVIDE>, C, threads, wsmem, s, order, len,
                             n, rp, ci, dg, v, rd, in, out, clear, err, limit, owner, no_ps,
                             no_pk, no_words, (int64_t)0, C, C);
  }
  if (kind == ILUK_SCHED_WARP_GRID) {
    if (!lo.corder) return cudaErrorInvalidValue;
    const int32_t *order = lo.corder;
    int64_t len = lo.clen;
    auto kern = k_sweep_grid<FORWARD, DIVIDE>;
    int bps = 1;  // an explicit width means one CTA of that width per SM
    if (w == 0) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, kCtaThreads, 0);
    if (bps < 1) bps = 1;
    int64_t grid = (int64_t)bps * num_sms();
    const int64_t want = (len + (threads / 32) - 1) / (threads / 32);
    if (grid > want) grid = want;
    void *args[] = {(void *)&order, (void *)&len, (void *)&rp, (void *)&ci, (void *)&dg,
                    (void *)&v, (void *)&rd, (void *)&in, (void *)&out, (void *)&clear,
                    (void *)&err, (void *)&limit};
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid),
                                                dim3((unsigned)threads), args, 0, s);
    note_launch();
    return e;
  }
  // FLAGS.  Multi-SM: every block must be resident (rows wait on rows of
  // other blocks), so the grid is launched cooperatively and sized by
  // occupancy.
  if (!lo.order) return cudaErrorInvalidValue;
  const int32_t *order = lo.order;
  int64_t len = lo.len;
  int bps = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_sweep<FORWARD, DIVIDE, 8>, kGridThreads,
                                                0);
  if (bps > 2) bps = 2;
  if (bps < 1) bps = 1;
  int64_t grid = (int64_t)bps * num_sms();
  const int64_t want = (len + kGridThreads - 1) / kGridThreads;  // one warp per 32 slots
  if (grid > want) grid = want;
  void *args[] = {(void *)&order, (void *)&len, (void *)&rp, (void *)&ci, (void *)&dg,
                  (void *)&v, (void *)&rd, (void *)&in, (void *)&out, (void *)&clear,
                  (void *)&err, (void *)&limit};
  cudaError_t e = cudaLaunchCooperativeKernel((const void *)k_sweep<FORWARD, DIVIDE, 8>,
                                              dim3((unsigned)grid), dim3(kGridThreads), args, 0, s);
  note_launch();
  return e;
}

// One schedule byte made usable for n rows: an unknown kind becomes the
// warp-per-row grid, a cluster kind without a usable cluster likewise, and a
// width only stays with the warp-per-row kinds (256..1024 threads).
static int usable_sched(int64_t n, int sc) {
  int kind = sc & 0xf, w = (sc >> 4) & 0xf;
  if (kind < ILUK_SCHED_FLAGS || kind > ILUK_SCHED_WARP_CLUSTER_HELP) kind = ILUK_SCHED_WARP_GRID;
  if (kind == ILUK_SCHED_CLUSTER && ring_cluster() == 0) kind = ILUK_SCHED_WARP_GRID;
  if ((kind == ILUK_SCHED_WARP_CLUSTER || kind == ILUK_SCHED_WARP_CLUSTER_HELP) &&
      cluster_width(n, k_sweep_wpr<true, false>) == 0)
    kind = ILUK_SCHED_WARP_GRID;
  const bool per_row = kind == ILUK_SCHED_WARP_GRID || kind == ILUK_SCHED_WARP_CLUSTER ||
                       kind == ILUK_SCHED_WARP_CLUSTER_HELP;
  if (!per_row || w < 2 || w > 8) w = 0;
  return kind | (w << 4);
}

cudaError_t launch_apply_backward(int64_t n, const int64_t *rp, const int32_t *ci,
                                  const int64_t *dg, const double *v, const DivPrep *rd,
                                  const LevelOrder &bwd, double *tmp, double *y, int sched,
                                  DevErr *err, const SweepAux *aux, cudaStream_t s) {
  // tmp already holds L^-1 p; y is armed here as the forward sweep would
  // have armed it, and the backward sweep re-arms tmp as usual
  int sb = (sched >> 8) & 0xff;
  if (sb == 0) sb = sched & 0xff;
  cudaError_t e = launch_fill_pending(n, y, s);
  if (e != cudaSuccess) return e;
  return run_sweep<false, true>(n, bwd, rp, ci, dg, v, rd, tmp, y, tmp, usable_sched(n, sb), err,
                                aux, s);
}

cudaError_t launch_apply(int64_t n, const int64_t *rp, const int32_t *ci, const int64_t *dg,
                         const double *v, const DivPrep *rd, const LevelOrder &fwd,
                         const LevelOrder &bwd,
                         const double *p, double *tmp, double *y, int transpose, int sched,
                         DevErr *err, const SweepAux *aux, cudaStream_t s) {
  // sched packs the forward schedule in bits 0-7 and the backward one in 8-15
  // (a single value applies to both).
  int sf = sched & 0xff, sb = (sched >> 8) & 0xff;
  if (sb == 0) sb = sf;
  sf = usable_sched(n, sf);
  sb = usable_sched(n, sb);
  cudaError_t e;
  // tmp is pending on entry (left so by the previous backward sweep); the
  // forward sweep re-arms y, the backward sweep re-arms tmp.
  if (!transpose) {
    e = run_sweep<true, false>(n, fwd, rp, ci, dg, v, rd, p, tmp, y, sf, err, aux, s);
    if (e != cudaSuccess) return e;
    return run_sweep<false, true>(n, bwd, rp, ci, dg, v, rd, tmp, y, tmp, sb, err, aux, s);
  }
  e = run_sweep<true, true>(n, fwd, rp, ci, dg, v, rd, p, tmp, y, sf, err, aux, s);
  if (e != cudaSuccess) return e;
  return run_sweep<false, false>(n, bwd, rp, ci, dg, v, rd, tmp, y, tmp, sb, err, aux, s);
}

// ---------------------------------------------------------------------------
// CSR transpose: count, scan, scatter, then sort every row by source row so
// that row i of T lists column i of F top to bottom.
// ---------------------------------------------------------------------------
__global__ void k_count_cols(int64_t nnz, const int32_t *__restrict__ ci, int32_t *cnt) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz;
       p += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&cnt[ci[p]], 1);
}

__global__ void k_scatter_t(int64_t n, const int64_t *__restrict__ rp,
                            const int32_t *__restrict__ ci, const double *__restrict__ v,
                            const int64_t *__restrict__ trp, int32_t *cursor, int32_t *tci,
                            double *tv) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    for (int64_t p = rp[i]; p < rp[i + 1]; ++p) {
      const int32_t c = ci[p];
      const int64_t dst = trp[c] + atomicAdd(&cursor[c], 1);
      tci[dst] = (int32_t)i;
      tv[dst] = v[p];
    }
  }
}

__global__ void k_sort_rows_t(int64_t n, const int64_t *__restrict__ trp, int32_t *tci,
                              double *tv, int64_t *tdiag) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = trp[r], e = trp[r + 1];
    for (int64_t p = b + 1; p < e; ++p) {  // insertion sort by source row
      const int32_t key = tci[p];
      const double val = tv[p];
      int64_t q = p - 1;
      while (q >= b && tci[q] > key) {
        tci[q + 1] = tci[q];
        tv[q + 1] = tv[q];
        --q;
      }
      tci[q + 1] = key;
      tv[q + 1] = val;
    }
    int64_t dpos = -1;
    for (int64_t p = b; p < e; ++p)
      if (tci[p] == r) dpos = p;
    if (tdiag) tdiag[r] = dpos;
  }
}

cudaError_t launch_transpose(int64_t n, int64_t nnz, const int64_t *rp, const int32_t *ci,
                             const double *v, int64_t *trp, int32_t *tci, double *tv,
                             int64_t *tdiag, int32_t *cursor, int64_t *scan_tmp, cudaStream_t s) {
  ProfScope prof_scope(ILUK_PROF_TRANSPOSE, s);
  if (n == 0) return cudaMemsetAsync(trp, 0, sizeof(int64_t), s);
  int64_t g = (int64_t)num_sms() * 8;
  cudaError_t e = cudaMemsetAsync(cursor, 0, (size_t)n * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  k_count_cols<<<(unsigned)g, 256, 0, s>>>(nnz, ci, cursor);
  note_launch();
  e = launch_scan_lengths(n, cursor, trp, scan_tmp, s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(cursor, 0, (size_t)n * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  k_scatter_t<<<(unsigned)g, 256, 0, s>>>(n, rp, ci, v, trp, cursor, tci, tv);
  note_launch();
  k_sort_rows_t<<<(unsigned)g, 256, 0, s>>>(n, trp, tci, tv, tdiag);
  note_launch();
  return cudaGetLastError();
}

}  // namespace iluk
