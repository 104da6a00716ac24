// levels.cu -- level sets of the two sweep DAGs (the level/backward
// scheduling of the paper's related work: Anderson 1988, Heroux 1991).
//
// depth(i) = 1 + max depth(h) over the rows h that row i reads (h < i in the
// forward sweep, h > i in the backward sweep); rows of equal depth are
// independent.  The sweeps walk rows in level order, with every level
// starting on a warp boundary (short levels are padded with -1), so the 32
// rows of a warp never depend on one another: a warp's lanes only ever wait
// for rows held by other warps.
#include <algorithm>

#include "internal.h"

namespace iluk {

constexpr int kDepthThreads = 512;
constexpr int kWindowRows = 2048;          // about the rows in flight of a numeric phase
constexpr int kDepthBatch = 4;  // inputs a lane looks at together

// One row per lane: a warp claims the next 32 rows in sweep order through a
// global ticket per direction, and its lanes walk their rows' inputs, nearest
// last, kDepthBatch at a time; a lane that finds an input without a depth yet
// looks at it again in the warp's next round, while the others go on.
// depth[] doubles as the ready flag (0 until the row is final), handed over
// through L2.  A warp claims rows only while it runs, and every row it reads
// holds an earlier ticket or belongs to the same warp, so the waits end whether
// or not all CTAs are resident.
// What bounds it: one L2 round trip (~900 cycles) a level.  With a warp per
// row the rows in flight (one per warp) covered only a part of a wide DAG's
// wavefront: 3D 64^3, k = 2 (694 levels) 5.8 -> 1.2 ms for both directions.
// A row deeper than `cap` ends the launch, both directions of it (fail = 2): the
// caller wants no orders for a DAG that deep.
// With g, the warps that complete the first rows decide whether rows in index order
// are worth more than waiting for the orders (fail = 3 ends the launch).  They look
//  * at 1/64 of the rows, if that is 1,024 or more, whether their depth is over 2.05
//    times that of the first half of them: faster than along any line of a grid;
//  * at 1/32, whether it is 1.65 times that of the first 1/64: it grows with the row
//    index (random bands at k >= 1, 1.85 to 3.2), index order nearly is level order;
//  * at the same or at 4,096 rows, by what each way costs.  In index order the rows in
//    flight are about kWindowRows successive ones, so the rows take n / kWindowRows
//    times a window's depth, here the first one's; with the orders first they take
//    the DAG's depth, reckoned from what the last quarter of those rows added, in
//    steps that cost as much, after a depth kernel of that depth and ~0.3 ms.
// Symbolic and numeric phase, orders first / beside the rows (steps in index order,
// levels): 2D 256^2 k = 0 (8,448, 511) 1.87 / 6.0 ms, 128 x 512 k = 0 (4,608, 639) 2.28 /
// 3.36, 64 x 1,024 k = 0 (3,072, 1,087) 3.52 / 2.55, 30 x 3,000 k = 0 (4,312, 3,029) 11.9 /
// 7.3; 3D 30^3 k = 0 (818, 88) 0.94 / 1.07; 27-point 30^3 k = 0 (1,300, 204) 1.29 / 1.53,
// k = 1 (1,850, 378) 2.35 / 2.39; random bands, whose windows add up to their depth, n =
// 160,000 k = 0 2.46 / 1.58, k = 1 7.2 / 5.1, n = 40,000 with 4 a row k = 0 0.94 / 0.65.
// The wrong side costs these differences and no more.
struct DepthGrowth {
  int most[6];  // depths of the first rows looked at (GrowthRows)
  int done[3];  // rows completed of the three looks'
};
struct GrowthRows {
  // the first 1/128, 1/64 and 1/32 of all rows, a window, 3/4 of and all of the last
  // look's; whole warps
  int part128, part64, part32, window, before, all;
};
__device__ __forceinline__ bool index_order_serves(int64_t n, int window, int before, int all,
                                                   const GrowthRows &gr) {
  const int64_t in_index_order = n * window / gr.window;
  const int64_t levels = all + (n - gr.all) * (all - before) / (gr.all - gr.before);
  return in_index_order <= 3 * levels + 200;
}
// Rows t0r .. t0r + 31, of depth m at most, are done: whether the launch should end.
// Not inlined: the rows' loop above all is on the critical path.
__device__ __noinline__ bool growth_look(int64_t n, int64_t t0r, int m, DepthGrowth *g,
                                         GrowthRows gr) {
  if (t0r < gr.part128) atomicMax(&g->most[0], m);
  if (t0r < gr.part64) atomicMax(&g->most[1], m);
  if (t0r < gr.part32) atomicMax(&g->most[2], m);
  if (t0r < gr.window) atomicMax(&g->most[3], m);
  if (t0r < gr.before) atomicMax(&g->most[4], m);
  atomicMax(&g->most[5], m);
  __threadfence();
  const bool look0 = t0r < gr.part64 && atomicAdd(&g->done[0], 32) + 32 == gr.part64;
  const bool look1 = t0r < gr.part32 && atomicAdd(&g->done[1], 32) + 32 == gr.part32;
  const bool look2 = atomicAdd(&g->done[2], 32) + 32 == gr.all;
  if (!look0 && !look1 && !look2) return false;
  __threadfence();
  const volatile int *most = g->most;
  return (look0 && gr.part64 >= 1024 && 20 * (int64_t)most[1] > 41 * (int64_t)most[0]) ||
         (look1 && 20 * (int64_t)most[2] >= 33 * (int64_t)most[1]) ||
         (look2 && index_order_serves(n, most[3], most[4], most[5], gr));
}

template <bool FORWARD>
__device__ void depth_rows(int64_t n, const int64_t *__restrict__ rp,
                           const int32_t *__restrict__ ci, const int64_t *__restrict__ dg,
                           int32_t *depth, int32_t *maxdepth, DevErr *err, int64_t limit_ns,
                           unsigned long long *ticket, int *fail, int *other, int cap,
                           DepthGrowth *g, const GrowthRows &gr) {
  const int lane = threadIdx.x & 31;
  int dmax_local = 0;
  for (;;) {
    unsigned long long tk = 0;
    if (lane == 0) tk = atomicAdd(ticket, 32ull);
    const int64_t t = (int64_t)__shfl_sync(FULL_MASK, tk, 0) + lane;
    if (t - lane >= n) break;
    if (__any_sync(FULL_MASK, *((volatile int *)fail) != 0)) break;
    const bool mine = t < n;
    const int64_t row = FORWARD ? t : n - 1 - t;
    // inputs q = 0 .. len - 1, the nearest row last
    int64_t first = 0;
    int len = 0;
    if (mine) {
      const int64_t d = dg[row];
      first = FORWARD ? rp[row] : rp[row + 1] - 1;
      len = (int)(FORWARD ? d - first : first - d);
    }
    int q = 0, dm = 0;
    bool done = !mine;
    const uint64_t t0 = globaltimer_ns();
    unsigned backoff = 16;
    bool gone = false;
    for (unsigned it = 0;; ++it) {
      bool moved = false;
      if (!done) {
        int v[kDepthBatch];
#pragma unroll
        for (int u = 0; u < kDepthBatch; ++u) {
          v[u] = 1;
          if (q + u < len) {
            const int32_t *src = &depth[ci[FORWARD ? first + q + u : first - q - u]];
            asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v[u]) : "l"(src));
          }
        }
        bool go = true;
        int adv = 0;
#pragma unroll
        for (int u = 0; u < kDepthBatch; ++u) {
          go = go && v[u] != 0;
          if (go && q + u < len) {
            if (v[u] > dm) dm = v[u];
            ++adv;
          }
        }
        q += adv;
        moved = adv > 0;
        if (q >= len) {
          ++dm;
          asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(&depth[row]), "r"(dm)
                       : "memory");
          if (dm > dmax_local) dmax_local = dm;
          if (dm > cap) {
            atomicExch(fail, 2);
            atomicCAS(other, 0, 2);
          }
          done = moved = true;
        }
      }
      if (__all_sync(FULL_MASK, done)) break;
      if ((it & 15u) == 15u) {
        const bool late = (int64_t)(globaltimer_ns() - t0) > limit_ns;
        const bool stop = *((volatile int *)fail) != 0 || late;
        if (__any_sync(FULL_MASK, stop)) {  // the whole warp gives up together
          if (late && !done) {
            atomicCAS(fail, 0, 1);
            set_err(err, t, ILUK_ETIMEOUT);
          }
          gone = true;
          break;
        }
      }
      if (!__any_sync(FULL_MASK, moved)) {
        // far from its inputs: only the first waiting lane looks, at its first
        // missing input, so that the waiting warps leave L2 to the others
        const unsigned waiting = __ballot_sync(FULL_MASK, !done);
        const bool leader = lane == __ffs(waiting) - 1;
        const int32_t *src = nullptr;
        if (leader) src = &depth[ci[FORWARD ? first + q : first - q]];
        for (int k = 0; k < 8; ++k) {
          __nanosleep(backoff);
          int v = 0;
          if (leader) asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(src));
          if (__any_sync(FULL_MASK, v != 0)) break;
        }
        if (backoff < 256u) backoff <<= 1;
      } else {
        backoff = 16;
      }
    }
    if (gone) break;
    const int64_t t0r = t - lane;
    if (g != nullptr && t0r < gr.all) {
      const int m = __reduce_max_sync(FULL_MASK, dm);
      if (lane == 0 && growth_look(n, t0r, m, g, gr)) {
        atomicExch(fail, 3);
        atomicExch(other, 3);
      }
    }
  }
  dmax_local = __reduce_max_sync(FULL_MASK, dmax_local);
  if (lane == 0 && dmax_local) atomicMax(maxdepth, dmax_local);
}

// Even CTAs compute the forward depths, odd CTAs the backward depths (the two
// DAGs are independent).  ctl: two tickets, then two failure flags.
__global__ void __launch_bounds__(kDepthThreads)
k_depth_pair(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
             const int64_t *__restrict__ dg, int32_t *depth_f, int32_t *depth_b, int32_t *mx,
             DevErr *err, unsigned long long *ctl, int64_t limit_ns, int cap, int cap_b,
             DepthGrowth *g, GrowthRows gr) {
  int *fail = reinterpret_cast<int *>(ctl + 2);
  if ((blockIdx.x & 1) == 0)
    depth_rows<true>(n, rp, ci, dg, depth_f, mx, err, limit_ns, ctl, fail, fail + 1, cap, g, gr);
  else
    depth_rows<false>(n, rp, ci, dg, depth_b, mx + 1, err + 1, limit_ns, ctl + 1, fail + 1, fail,
                      cap_b, nullptr, gr);
}

// Rows per level; shape[0], shape[1] (0 before): the entries the sweep reads, and the
// most of a row.
template <bool FORWARD>
__global__ void k_level_count(int64_t n, const int32_t *__restrict__ depth,
                              const int64_t *__restrict__ rp, const int64_t *__restrict__ dg,
                              int32_t *cnt, unsigned long long *shape) {
  __shared__ unsigned long long entries;
  __shared__ int longest;
  if (threadIdx.x == 0) {
    entries = 0;
    longest = 0;
  }
  __syncthreads();
  unsigned long long e = 0;
  int mx = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    atomicAdd(&cnt[depth[i] - 1], 1);
    const int len = (int)(FORWARD ? dg[i] - rp[i] : rp[i + 1] - 1 - dg[i]);
    e += (unsigned long long)len;
    if (len > mx) mx = len;
  }
  mx = __reduce_max_sync(FULL_MASK, mx);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) e += __shfl_xor_sync(FULL_MASK, e, o);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&entries, e);
    atomicMax(&longest, mx);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (entries) atomicAdd(&shape[0], entries);
    if (longest) atomicMax(&shape[1], (unsigned long long)longest);
  }
}

__global__ void k_level_pad(int64_t nlev, int32_t *cnt) {
  for (int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < nlev;
       l += (int64_t)gridDim.x * blockDim.x)
    cnt[l] = (cnt[l] + 31) & ~31;
}

__global__ void k_level_scatter(int64_t n, const int32_t *__restrict__ depth,
                                const int64_t *__restrict__ lstart, int32_t *cursor,
                                int32_t *order) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int l = depth[i] - 1;
    order[lstart[l] + atomicAdd(&cursor[l], 1)] = (int32_t)i;
  }
}

static unsigned grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms() * 8;
  if (b > cap) b = cap;
  return (unsigned)(b < 1 ? 1 : b);
}

// Padded level order from depths, and the same order without padding
// (synchronous).
template <bool FORWARD>
static int order_from_depth(int64_t n, const int32_t *depth, const int64_t *rp, const int64_t *dg,
                            int32_t nlev, LevelOrder *lo, cudaStream_t s) {
  int32_t *cnt = nullptr, *cursor = nullptr;
  int64_t *lstart = nullptr, *scan_tmp = nullptr, *cstart = nullptr;
  auto cleanup = [&]() {
    if (cnt) cudaFreeAsync(cnt, s);
    if (cursor) cudaFreeAsync(cursor, s);
    if (cstart) cudaFreeAsync(cstart, s);
    if (scan_tmp) cudaFreeAsync(scan_tmp, s);
  };
#define CKL(call)                              \
  do {                                         \
    if ((call) != cudaSuccess) {               \
      cleanup();                               \
      if (lstart) cudaFreeAsync(lstart, s);    \
      if (lo->order) cudaFreeAsync(lo->order, s); \
      if (lo->corder) cudaFreeAsync(lo->corder, s); \
      lo->order = lo->corder = nullptr;        \
      return ILUK_ECUDA;                       \
    }                                          \
  } while (0)
  CKL(cudaMallocAsync((void **)&cnt, (size_t)nlev * sizeof(int32_t), s));
  CKL(cudaMallocAsync((void **)&cursor, (size_t)nlev * sizeof(int32_t), s));
  // the level starts, the order's length, and what k_level_count finds
  CKL(cudaMallocAsync((void **)&lstart, ((size_t)nlev + 3) * sizeof(int64_t), s));
  CKL(cudaMemsetAsync(lstart + nlev + 1, 0, 2 * sizeof(int64_t), s));
  CKL(cudaMallocAsync((void **)&scan_tmp, (size_t)scan_tmp_elems(nlev) * sizeof(int64_t), s));
  CKL(cudaMemsetAsync(cnt, 0, (size_t)nlev * sizeof(int32_t), s));
  CKL(cudaMemsetAsync(cursor, 0, (size_t)nlev * sizeof(int32_t), s));
  CKL(cudaMallocAsync((void **)&cstart, ((size_t)nlev + 1) * sizeof(int64_t), s));
  k_level_count<FORWARD><<<grid_for(n), 256, 0, s>>>(
      n, depth, rp, dg, cnt, reinterpret_cast<unsigned long long *>(lstart + nlev + 1));
  note_launch();
  CKL(launch_scan_lengths(nlev, cnt, cstart, scan_tmp, s));  // unpadded level starts
  k_level_pad<<<grid_for(nlev), 256, 0, s>>>(nlev, cnt);
  note_launch();
  CKL(launch_scan_lengths(nlev, cnt, lstart, scan_tmp, s));
  int64_t shape[3] = {0, 0, 0};
  CKL(cudaMemcpyAsync(shape, lstart + nlev, sizeof(shape), cudaMemcpyDeviceToHost, s));
  CKL(cudaStreamSynchronize(s));
  const int64_t len = shape[0];
  CKL(cudaMallocAsync((void **)&lo->order, (size_t)len * sizeof(int32_t), s));
  CKL(cudaMemsetAsync(lo->order, 0xff, (size_t)len * sizeof(int32_t), s));
  k_level_scatter<<<grid_for(n), 256, 0, s>>>(n, depth, lstart, cursor, lo->order);
  note_launch();
  CKL(cudaMallocAsync((void **)&lo->corder, (size_t)n * sizeof(int32_t), s));
  CKL(cudaMemsetAsync(cursor, 0, (size_t)nlev * sizeof(int32_t), s));
  k_level_scatter<<<grid_for(n), 256, 0, s>>>(n, depth, cstart, cursor, lo->corder);
  note_launch();
  CKL(cudaGetLastError());
#undef CKL
  cleanup();
  lo->lstart = lstart;
  lo->len = len;
  lo->nlev = nlev;
  lo->entries = shape[1];
  lo->longest = (int32_t)shape[2];
  lo->clen = n;
  return ILUK_OK;
}

// Synchronous: the depths of both sweep DAGs (one launch), then the two padded
// level orders.  On success fwd->order / bwd->order (and their level starts)
// are new device allocations.  kLevelsTooDeep (and no orders) when the forward
// DAG is deeper than cap or the backward one than cap_b; kLevelsLinear (and none)
// when `growth` asks and rows in index order do not need them: a DAG of fewer than
// kLevelOrderRows rows (3D 20^3 k = 2 1.12 ms with the orders first, 0.79 beside the
// rows), or see index_order_serves.
int build_levels_pair(int64_t n, const int64_t *rp, const int32_t *ci, const int64_t *dg,
                      LevelOrder *fwd, LevelOrder *bwd, int cap, int cap_b, bool growth,
                      cudaStream_t s) {
  ProfScope prof_scope(ILUK_PROF_DEPTH, s);
  *fwd = LevelOrder();
  *bwd = LevelOrder();
  if (n == 0) return ILUK_OK;
  int32_t *depth = nullptr, *mx = nullptr;
  DevErr *err = nullptr;
  unsigned long long *ctl = nullptr;  // two tickets, two failure flags
  if (growth && n < kLevelOrderRows) return kLevelsLinear;
  DepthGrowth *g = nullptr;
  GrowthRows gr = {};
  auto warps = [](int64_t rows) {
    return (int)(std::min<int64_t>(rows, INT32_MAX / 2) / 32 * 32);
  };
  gr.part128 = warps(n / 128);
  gr.part64 = warps(n / 64);
  gr.part32 = warps(n / 32);
  gr.window = kWindowRows;
  gr.all = std::max(gr.part32, 2 * kWindowRows);
  gr.before = warps(gr.all - gr.all / 4);
  auto cleanup = [&]() {
    if (depth) cudaFreeAsync(depth, s);
    if (mx) cudaFreeAsync(mx, s);
    if (err) cudaFreeAsync(err, s);
    if (ctl) cudaFreeAsync(ctl, s);
    if (g) cudaFreeAsync(g, s);
  };
  if (growth && (cudaMallocAsync((void **)&g, sizeof(*g), s) != cudaSuccess ||
                 cudaMemsetAsync(g, 0, sizeof(*g), s) != cudaSuccess)) {
    cleanup();
    return ILUK_ECUDA;
  }
  if (cudaMallocAsync((void **)&depth, 2 * n * sizeof(int32_t), s) != cudaSuccess ||
      cudaMallocAsync((void **)&mx, 2 * sizeof(int32_t), s) != cudaSuccess ||
      cudaMallocAsync((void **)&err, 2 * sizeof(DevErr), s) != cudaSuccess ||
      cudaMallocAsync((void **)&ctl, 3 * sizeof(unsigned long long), s) != cudaSuccess ||
      cudaMemsetAsync(depth, 0, 2 * n * sizeof(int32_t), s) != cudaSuccess ||
      cudaMemsetAsync(mx, 0, 2 * sizeof(int32_t), s) != cudaSuccess ||
      cudaMemsetAsync(ctl, 0, 3 * sizeof(unsigned long long), s) != cudaSuccess ||
      launch_fill_err(err, s) != cudaSuccess || launch_fill_err(err + 1, s) != cudaSuccess) {
    cleanup();
    return ILUK_ECUDA;
  }
  // all the rows in flight that the SMs take: half the CTAs of each direction
  int bps = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_depth_pair, kDepthThreads, 0);
  if (bps < 1) bps = 1;
  int64_t grid = ((int64_t)bps * num_sms() + 1) / 2 * 2;
  const int64_t want = 2 * ((n + kDepthThreads - 1) / kDepthThreads);
  if (grid > want) grid = want;
  if (grid < 2) grid = 2;
  k_depth_pair<<<(unsigned)grid, kDepthThreads, 0, s>>>(n, rp, ci, dg, depth, depth + n, mx, err,
                                                        ctl, wait_limit(), cap, cap_b, g, gr);
  note_launch();
  DevErr herr[2];
  int32_t nlev[2] = {0, 0}, fail[2] = {0, 0};
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(herr, err, sizeof(herr), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(nlev, mx, sizeof(nlev), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(fail, ctl + 2, sizeof(fail), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cleanup();
    return ILUK_ECUDA;
  }
  for (int d = 0; d < 2; ++d)
    if (herr[d].key != kNoErr) {
      cleanup();
      return (int)(herr[d].key & 0xff);
    }
  if (fail[0] == 3 || fail[1] == 3) {
    cleanup();
    return kLevelsLinear;
  }
  if (nlev[0] > cap || nlev[1] > cap_b) {
    cleanup();
    return kLevelsTooDeep;
  }
  int st = order_from_depth<true>(n, depth, rp, dg, nlev[0], fwd, s);
  if (st == ILUK_OK) st = order_from_depth<false>(n, depth + n, rp, dg, nlev[1], bwd, s);
  // the orders are read on other streams than the one they were built on (beside
  // a numeric phase; another caller's), which nothing else makes wait
  if (st == ILUK_OK && cudaStreamSynchronize(s) != cudaSuccess) st = ILUK_ECUDA;
  cleanup();
  return st;
}

// Index orders for the warp-per-row sweeps of a factorization whose level
// orders are not built: rows ascending (forward) and descending (backward),
// valid since every dependency lies at a smaller (forward) or larger
// (backward) index.  Only corder/clen are set.
__global__ void k_index_orders(int64_t n, int32_t *fwd, int32_t *bwd) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    fwd[i] = (int32_t)i;
    bwd[i] = (int32_t)(n - 1 - i);
  }
}

cudaError_t build_index_orders(int64_t n, LevelOrder *fwd, LevelOrder *bwd, cudaStream_t s) {
  *fwd = LevelOrder();
  *bwd = LevelOrder();
  if (n == 0) return cudaSuccess;
  cudaError_t e = cudaMallocAsync((void **)&fwd->corder, (size_t)n * sizeof(int32_t), s);
  if (e == cudaSuccess) e = cudaMallocAsync((void **)&bwd->corder, (size_t)n * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  k_index_orders<<<grid_for(n), 256, 0, s>>>(n, fwd->corder, bwd->corder);
  note_launch();
  fwd->clen = bwd->clen = n;
  return cudaGetLastError();
}

}  // namespace iluk

// LevelOrder is declared at global scope (internal.h), and so is this.
void level_order_free(LevelOrder &lo, cudaStream_t s) {
  if (lo.order) cudaFreeAsync(lo.order, s);
  if (lo.corder) cudaFreeAsync(lo.corder, s);
  if (lo.lstart) cudaFreeAsync(lo.lstart, s);
  for (OwnerCode &oc : lo.owner)
    if (oc.code) cudaFreeAsync(oc.code, s);
  for (const void *p : {(const void *)lo.plan.coff, (const void *)lo.plan.first,
                        (const void *)lo.plan.len, (const void *)lo.plan.slot})
    if (p) cudaFreeAsync(const_cast<void *>(p), s);
  lo = LevelOrder();
}
