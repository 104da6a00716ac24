// fill.cu -- a2: the symbolic phase without waits, one level of fill at a time.
//
// An entry of level p >= 1 is there because of two entries (j, i), (i, t),
// i < min(j, t), whose levels sum to p - 1, so both have levels below p: once
// all entries of levels 0 .. p - 1 are known, every row finds its entries of
// level p on its own (Sec. 3.3 makes this remark for p = 1).  The k passes
// together insert what Algorithm 1's walk inserts, with the same minimal
// levels; an entry found in pass p is in no earlier pass's pattern, so p is
// its minimum.
//
// The columns right of the diagonal are kept level by level (FillBucket), so a
// pivot of level l meets only the partners of level p - 1 - l, and a pair of
// entries is looked at in one pass only, the one whose level it gives.  A pass is
// two launches of k_fill_rows, one warp per row, over the pattern so far (CSR
// with levels): the first counts the row's new columns, a scan gives the new row
// pointers, the second finds them again, in the rows that have any, and writes the
// row and its part of the level's bucket.  The columns are two bitmaps in shared
// memory over the row's window (the pattern's widest reach left and right of the
// diagonal): those present, and those the pass adds.  The candidates of up to 32
// pivots are taken as one list (prefix sums of the partners' counts), 32 at a time,
// so short partner lists fill the lanes and all loads of a step are independent.
// What bounds it: the latency of those loads, hidden by the rows in flight; no
// row waits for another.  The whole call, the walk with waits / these passes when each
// looked at all pairs twice / now: 2D 256^2 k = 2 4.36 / 0.33 / 0.34 ms, 27-point 30^3
// k = 2 2.95 / 0.41 / 0.35, 3D 20^3 k = 8 9.6 / 1.20 / 0.69, band n = 20,000 k = 4 279 /
// 7.8 / 1.3, random n = 1,000 with 5 a row k = 12 3.67 / 17.2 / 2.6, n = 2,000 nine
// tenths full k = 2 48 / 93 / 34.
// Patterns whose window exceeds kMaxFillCols keep the walk of symbolic.cu (clearing
// and scanning such a window for every row would cost more than the waits), and so do
// some at a high k (see fill_window).
#include <utility>
#include <vector>

#include "internal.h"

namespace iluk {

constexpr int kFillThreads = 256;
constexpr int64_t kMaxFillCols = 65536;

// A row's part of a list of columns: where it begins, and how many (a window's at most).
constexpr int kSpanBits = 20;
static_assert(kMaxFillCols < (1 << kSpanBits), "a row's columns fit a span");
__device__ __forceinline__ int64_t span_of(int64_t beg, int64_t cnt) {
  return (beg << kSpanBits) | cnt;
}
__device__ __forceinline__ int64_t span_beg(int64_t s) { return s >> kSpanBits; }
__device__ __forceinline__ int span_cnt(int64_t s) { return (int)(s & ((1 << kSpanBits) - 1)); }

// The columns of one level right of the diagonal, ascending in each row: row i's
// are ci[span up[i]].  up null: the level has no entries.
struct FillBucket {
  const int64_t *up;
  const int32_t *ci;
};

// Without bk, reach[0] and reach[1]: the most columns a row reaches left and right of
// its diagonal.  With bk, the first entry of each row right of the diagonal
// (ustart) and the bucket of A's own entries (up, bk[0]).
__global__ void k_fill_reach(int64_t n, const int64_t *__restrict__ rp,
                             const int32_t *__restrict__ ci, int32_t *reach, int64_t *ustart,
                             int64_t *up, FillBucket *bk) {
  int32_t left = 0, right = 0;
  if (bk && blockIdx.x == 0 && threadIdx.x == 0) bk[0] = FillBucket{up, ci};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = rp[i], e = rp[i + 1];
    if (bk) {
      const int64_t u = lower_bound_l(ci, b, e, (int32_t)(i + 1));
      ustart[i] = u;
      up[i] = span_of(u, e - u);
    } else if (e > b) {
      const int32_t l = (int32_t)i - ci[b], r = ci[e - 1] - (int32_t)i;
      if (l > left) left = l;
      if (r > right) right = r;
    }
  }
  if (bk) return;
  left = __reduce_max_sync(FULL_MASK, left);
  right = __reduce_max_sync(FULL_MASK, right);
  if ((threadIdx.x & 31) == 0) {
    if (left > 0) atomicMax(&reach[0], left);
    if (right > 0) atomicMax(&reach[1], right);
  }
}

// An inclusive prefix sum over the warp.
__device__ __forceinline__ unsigned warp_prefix(unsigned v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(FULL_MASK, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Pass p over the rows of the pattern (rp, ci, lev, ustart), bk: the levels' buckets.
// FIRST: p = 1 on A's rows, all level 0 (no lev, no bk; up0: their spans), without
// the loads that find a pivot's bucket.  WRITE false: row_len[j] = entries after the pass,
// *found (0 before) = new ones of all rows.  WRITE true: the rows into (nrp, nci,
// nlev).  words: window words per warp (32 columns each).
template <bool WRITE, bool FIRST>
__global__ void __launch_bounds__(kFillThreads, FIRST ? 8 : 6)
k_fill_rows(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
            const uint8_t *__restrict__ lev, const int64_t *__restrict__ ustart,
            const int64_t *__restrict__ up0, const FillBucket *__restrict__ bk, int p, int words,
            int32_t *row_len,
            unsigned long long *found, const int64_t *__restrict__ nrp, int32_t *nci,
            uint8_t *nlev) {
  extern __shared__ unsigned bits[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  unsigned *old = bits + (size_t)wib * 2 * words, *add = old + words;
  const int64_t nw = (int64_t)gridDim.x * nwarps;
  unsigned long long all = 0;
  __shared__ unsigned long long cta_all;  // one atomic a CTA: 39,000 warps' cost 10 us
  if (!WRITE) {
    if (threadIdx.x == 0) cta_all = 0;
    __syncthreads();
  }
  for (int64_t row = (int64_t)blockIdx.x * nwarps + wib; row < n; row += nw) {
    const int64_t b0 = rp[row], b1 = rp[row + 1];
    const int m0 = (int)(b1 - b0);
    const int npiv_max = (int)(ustart[row] - b0);  // lower entries, and the diagonal if stored
    const int64_t dst = WRITE ? nrp[row] : 0;
    if (WRITE && nrp[row + 1] - dst == m0) {  // as it was
      for (int q = lane; q < m0; q += 32) {
        nci[dst + q] = ci[b0 + q];
        nlev[dst + q] = FIRST ? (uint8_t)0 : lev[b0 + q];
      }
      continue;
    }
    // every column of the finished row lies at or right of its first one (a
    // fill column t lies right of a pivot that is itself in the row)
    const int32_t c0 = m0 > 0 ? ci[b0] : 0;
    auto make_bitmaps = [&]() {
      for (int w = lane; w < words; w += 32) old[w] = add[w] = 0u;
      __syncwarp();
      for (int t = lane; t < m0; t += 32) {
        const int d = ci[b0 + t] - c0;
        atomicOr(&old[d >> 5], 1u << (d & 31));
      }
      __syncwarp();
    };
    // where the last pass found entries most rows find some in this one; else only
    // rows with candidates need the bitmaps
    bool present = FIRST || bk[p - 1].up != nullptr;
    if (present) make_bitmaps();
    bool hit = false;
    for (int base = 0; base < npiv_max; base += 32) {
      const int q = base + lane;
      int len = 0;
      const int32_t *start = nullptr;  // the partners
      if (q < npiv_max) {
        const int32_t i = ci[b0 + q];
        if (i < row) {
          const FillBucket with = FIRST ? FillBucket{up0, ci} : bk[p - 1 - (int)lev[b0 + q]];
          if (FIRST || with.up) {
            const int64_t sp = with.up[i];
            start = with.ci + span_beg(sp);
            len = span_cnt(sp);
          }
        }
      }
      const int incl = (int)warp_prefix((unsigned)len, lane);
      const int total = __shfl_sync(FULL_MASK, incl, 31);
      const int excl = incl - len;
      if (total > 0 && !present) {
        present = true;
        make_bitmaps();
      }
      for (int t0 = 0; t0 < total; t0 += 32) {
        const int t = t0 + lane;
        // the pivot of candidate t: the last lane with excl <= t (empty pivots
        // share their successor's excl and come before it)
        int s = 0;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
          const int e = __shfl_sync(FULL_MASK, excl, s + o);
          if (e <= t) s += o;
        }
        const int32_t *src = reinterpret_cast<const int32_t *>(__shfl_sync(
                                 FULL_MASK, reinterpret_cast<unsigned long long>(start), s)) +
                             (t - __shfl_sync(FULL_MASK, excl, s));
        if (t < total) {
          const int d = *src - c0;
          const unsigned bit = 1u << (d & 31);
          if (!(old[d >> 5] & bit)) {
            atomicOr(&add[d >> 5], bit);
            hit = true;
          }
        }
      }
    }
    __syncwarp();
    if (!WRITE) {
      int cnt = 0;
      if (__any_sync(FULL_MASK, hit)) {
        for (int w = lane; w < words; w += 32) cnt += __popc(add[w]);
        cnt = __reduce_add_sync(FULL_MASK, cnt);
      }
      if (lane == 0) row_len[row] = m0 + cnt;
      all += (unsigned long long)cnt;
    } else {
      int done = 0, old_done = 0;
      for (int w0 = 0; w0 < words; w0 += 32) {
        const int w = w0 + lane;
        const unsigned o = w < words ? old[w] : 0u;
        unsigned x = o | (w < words ? add[w] : 0u);
        // both counts in one scan: present columns and earlier ones
        const unsigned c = (unsigned)__popc(x) | ((unsigned)__popc(o) << 16);
        if (!__any_sync(FULL_MASK, c != 0u)) continue;
        const unsigned inc = warp_prefix(c, lane);
        const unsigned ex = inc - c;
        int64_t pos = dst + done + (int)(ex & 0xffffu);
        int64_t oq = b0 + old_done + (int)(ex >> 16);
        while (x) {
          const int b = __ffs(x) - 1;
          x &= x - 1u;
          nci[pos] = c0 + w * 32 + b;
          if ((o >> b) & 1u) {
            nlev[pos] = FIRST ? (uint8_t)0 : lev[oq];
            ++oq;
          } else {
            nlev[pos] = (uint8_t)p;
          }
          ++pos;
        }
        const unsigned tot = __shfl_sync(FULL_MASK, inc, 31);
        done += (int)(tot & 0xffffu);
        old_done += (int)(tot >> 16);
      }
    }
    __syncwarp();
  }
  if (!WRITE) {
    if (lane == 0 && all) atomicAdd(&cta_all, all);
    __syncthreads();
    if (threadIdx.x == 0 && cta_all) atomicAdd(found, cta_all);
  }
}

// After pass p, for those that follow: where the columns right of each row's diagonal
// begin in the new pattern, and the bucket of level p (bk[p]): of row j's new
// columns, for which fresh has room from nrp[j] - rp[j] on, those on that side.
// Eight lanes a row: four rows' loads in flight a warp (60 us with a warp a row on
// 3D 64^3, 18 so).
constexpr int kBucketLanes = 8;
__global__ void __launch_bounds__(kFillThreads)
k_fill_bucket(int64_t n, const int64_t *__restrict__ rp, const int64_t *__restrict__ nrp,
              const int32_t *__restrict__ nci, const uint8_t *__restrict__ nlev, int p,
              int64_t *nustart, int32_t *fresh, int64_t *up, FillBucket *bk) {
  const int lane = threadIdx.x & (kBucketLanes - 1);
  const unsigned group = ((1u << kBucketLanes) - 1u) << (threadIdx.x & 31 & ~(kBucketLanes - 1));
  const unsigned before = (1u << (threadIdx.x & 31)) - 1u;
  const int64_t ng = ((int64_t)gridDim.x * blockDim.x) / kBucketLanes;
  if (blockIdx.x == 0 && threadIdx.x == 0) bk[p] = FillBucket{up, fresh};
  for (int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kBucketLanes; row < n;
       row += ng) {
    const int64_t b = nrp[row], e = nrp[row + 1];
    const int64_t f0 = b - rp[row];
    const int64_t u = lower_bound_l(nci, b, e, (int32_t)(row + 1));
    int cnt = 0;
    if (e - rp[row + 1] > f0) {  // the row has new columns
      for (int64_t q0 = u; q0 < e; q0 += kBucketLanes) {
        const int64_t q = q0 + lane;
        const bool mine = q < e && nlev[q] == (uint8_t)p;
        const unsigned m = __ballot_sync(group, mine) & group;
        if (mine) fresh[f0 + cnt + __popc(m & before)] = nci[q];
        cnt += __popc(m);
      }
    }
    if (lane == 0) {
      nustart[row] = u;
      up[row] = span_of(f0, cnt);
    }
  }
}

// The finished pattern's diagonal positions and longest row; a row without its
// diagonal or longer than max_row is an error.
__global__ void k_fill_finish(int64_t n, const int64_t *__restrict__ rp,
                              const int32_t *__restrict__ ci, int64_t *diag, int32_t *maxrow,
                              DevErr *err, int64_t max_row) {
  int32_t mx = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = rp[i], e = rp[i + 1];
    const int64_t d = lower_bound_l(ci, b, e, (int32_t)i);
    diag[i] = d;
    if (e - b > max_row) {
      set_err(err, i, ILUK_ENOMEM);
      atomicMax(&err->need, (unsigned long long)(e - b));
    } else if (d >= e || ci[d] != (int32_t)i) {
      set_err(err, i, ILUK_ENODIAG);
    }
    if (e - b > mx) mx = (int32_t)(e - b);
  }
  mx = __reduce_max_sync(FULL_MASK, mx);
  if ((threadIdx.x & 31) == 0 && mx > 0) atomicMax(maxrow, mx);
}

static unsigned fill_blocks(int64_t threads) {
  int64_t b = (threads + 255) / 256;
  const int64_t cap = (int64_t)num_sms() * 8;
  return (unsigned)(b > cap ? cap : b < 1 ? 1 : b);
}

// Columns of the widest row's window, 0 when the passes do not take it: wider than
// kMaxFillCols, or as wide as the matrix (no band or grid numbering) at a high k,
// where levels of fill are many and the walk waits little.  Walk / passes, random
// patterns: n = 1,000, 5 a row, k = 12 3.67 / 2.6 ms, k = 16 3.79 / 4.08, k = 250
// 3.85 / 8.2; n = 300 0.91 / 1.01, 0.91 / 1.28, 0.92 / 2.1; 3 a row, n = 1,000, k = 3
// 0.278 / 0.285, k = 4 0.289 / 0.334, k = 8 0.469 / 0.551.  Grids and bands gain at every
// k (2D 64^2 k = 40 13.1 / 2.4 ms).  Fill
// never widens it: a row keeps its first column, and a fill column t comes from
// a pivot i < j with t - i at most the pattern's reach.  Synchronous.
int64_t fill_window(int64_t n, int64_t nnz, const int64_t *arp, const int32_t *aci, int k,
                    cudaStream_t s) {
  if (n == 0) return 0;
  int32_t *reach = nullptr, h[2] = {0, 0};
  bool ok = cudaMallocAsync((void **)&reach, sizeof(h), s) == cudaSuccess &&
            cudaMemsetAsync(reach, 0, sizeof(h), s) == cudaSuccess;
  if (ok) {
    k_fill_reach<<<fill_blocks(n), 256, 0, s>>>(n, arp, aci, reach, nullptr, nullptr, nullptr);
    note_launch();
    ok = cudaGetLastError() == cudaSuccess &&
         cudaMemcpyAsync(h, reach, sizeof(h), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
  }
  if (reach) cudaFreeAsync(reach, s);
  if (!ok) {
    cudaGetLastError();
    return 0;
  }
  const int64_t cols = (int64_t)h[0] + h[1] + 1;
  if (cols >= n && (k > 12 || (k >= 4 && nnz < 4 * n))) return 0;
  return cols <= kMaxFillCols ? cols : 0;
}

// Level-of-fill pattern of A (see the top) for a window of `cols` columns
// (fill_window).  On cudaSuccess fp holds the pattern (arrays owned by the
// caller) and err, *maxrow (device words) its checks.  Synchronises `s`.
cudaError_t build_fill_pattern(int64_t n, int64_t nnz, const int64_t *arp, const int32_t *aci,
                               int k, int64_t cols, FillPattern *fp, int32_t *maxrow, DevErr *err,
                               int64_t max_row, cudaStream_t s) {
  bool ok = false;
  *fp = FillPattern();
  ProfScope prof_scope(ILUK_PROF_SYMBOLIC, s);
  int64_t *rp = nullptr, *nrp = nullptr;
  int32_t *ci = nullptr, *nci = nullptr;
  uint8_t *lev = nullptr, *nlev = nullptr;
  unsigned char *fixed = nullptr, *bucket = nullptr;  // scratch of all passes, of one level
  std::vector<void *> kept;  // the levels' buckets, and small old patterns
  cudaError_t e = cudaSuccess;
  auto alloc = [&](auto **p, size_t cnt) {
    if (e == cudaSuccess) e = cudaMallocAsync((void **)p, (cnt ? cnt : 1) * sizeof(**p), s);
  };
  auto drop = [&](auto *&p) {
    if (p) cudaFreeAsync(p, s);
    p = nullptr;
  };
  auto keep = [&](auto *&p) {
    kept.push_back(p);
    p = nullptr;
  };
  // Memory freed before a synchronisation goes back to the driver, and the next pass
  // maps it anew: up to 64 MB of old patterns wait for the end instead.
  size_t held = 0;
  auto retire = [&](auto *&p, int64_t cnt) {
    held += (size_t)cnt * sizeof(*p);
    if (p && held <= (64u << 20)) keep(p);
    drop(p);
  };
  auto leave = [&](cudaError_t r) {
    drop(fixed);
    drop(bucket);
    drop(nrp);
    drop(nci);
    drop(nlev);
    for (void *p : kept) cudaFreeAsync(p, s);
    if (!ok) {
      drop(rp);
      drop(ci);
      drop(lev);
    }
    return r;
  };
  const int words = (int)((cols + 31) / 32);
  int warps = kFillThreads / 32;
  while (warps > 1 && (size_t)words * 8 * warps > (size_t)max_smem_optin() / 2) warps >>= 1;
  const size_t smem = (size_t)words * 8 * warps;  // the bitmaps
  int64_t grid = (n + warps - 1) / warps;
  if (grid > (int64_t)num_sms() * 32) grid = (int64_t)num_sms() * 32;
  int64_t *ustart = nullptr, *nustart = nullptr, *up0 = nullptr, *scan_tmp = nullptr;
  int32_t *row_len = nullptr;
  FillBucket *bk = nullptr;
  unsigned long long *found = nullptr;
  if (k > 0) {
    const size_t N = (size_t)n, scan = (size_t)scan_tmp_elems(n);
    const size_t tables = ((size_t)k + 1) * sizeof(FillBucket) + sizeof(*found);
    alloc(&fixed, tables + (3 * N + scan) * sizeof(int64_t) + N * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemsetAsync(fixed, 0, tables, s);
    for (auto kern : {k_fill_rows<false, true>, k_fill_rows<true, true>, k_fill_rows<false, false>,
                      k_fill_rows<true, false>})
      if (e == cudaSuccess) e = allow_smem(kern, 1024);
    if (e != cudaSuccess) return leave(e);
    bk = reinterpret_cast<FillBucket *>(fixed);
    found = reinterpret_cast<unsigned long long *>(bk + k + 1);
    ustart = reinterpret_cast<int64_t *>(found + 1);
    nustart = ustart + N;
    up0 = nustart + N;
    scan_tmp = up0 + N;
    row_len = reinterpret_cast<int32_t *>(scan_tmp + scan);
    k_fill_reach<<<fill_blocks(n), 256, 0, s>>>(n, arp, aci, nullptr, ustart, up0, bk);
    note_launch();
    e = cudaGetLastError();
  }
  int64_t cur_nnz = nnz;
  int top = 0;  // highest level present
  // levels above 2 top + 1 have no two entries to come from
  for (int p = 1; p <= k && p <= 2 * top + 1 && e == cudaSuccess; ++p) {
    const int64_t *crp = rp ? rp : arp;
    const int32_t *cci = rp ? ci : aci;
    unsigned long long add = 0;
    e = cudaMemsetAsync(found, 0, sizeof(*found), s);
    if (e != cudaSuccess) break;
    const auto count = p == 1 ? k_fill_rows<false, true> : k_fill_rows<false, false>;
    count<<<(unsigned)grid, warps * 32, smem, s>>>(n, crp, cci, lev, ustart, up0, bk, p, words,
                                                   row_len, found, nullptr, nullptr, nullptr);
    note_launch();
    e = cudaGetLastError();
    if (!nrp) alloc(&nrp, n + 1);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&add, found, sizeof(add), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) break;
    if (add == 0) continue;  // no entry of this level
    const int64_t nn = cur_nnz + (int64_t)add;
    e = launch_scan_lengths(n, row_len, nrp, scan_tmp, s);
    alloc(&nci, nn);
    alloc(&nlev, nn);
    if (p < k) alloc(&bucket, (size_t)n * sizeof(int64_t) + (size_t)add * sizeof(int32_t));
    if (e != cudaSuccess) break;
    const auto write = p == 1 ? k_fill_rows<true, true> : k_fill_rows<true, false>;
    write<<<(unsigned)grid, warps * 32, smem, s>>>(n, crp, cci, lev, ustart, up0, bk, p, words,
                                                   nullptr, nullptr, nrp, nci, nlev);
    note_launch();
    if (p < k) {
      int64_t *up = reinterpret_cast<int64_t *>(bucket);
      int32_t *fresh = reinterpret_cast<int32_t *>(up + n);
      k_fill_bucket<<<fill_blocks(n * kBucketLanes), kFillThreads, 0, s>>>(
          n, crp, nrp, nci, nlev, p, nustart, fresh, up, bk);
      note_launch();
      keep(bucket);
    }
    // a launch that was refused has written no pattern for the next pass to read
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    retire(rp, n + 1);
    retire(ci, cur_nnz);
    retire(lev, cur_nnz);
    rp = nrp;
    ci = nci;
    lev = nlev;
    std::swap(ustart, nustart);
    nrp = nullptr;
    nci = nullptr;
    nlev = nullptr;
    cur_nnz = nn;
    top = p;
  }
  if (e == cudaSuccess && !rp) {  // no fill: A's own pattern, all level 0
    alloc(&rp, n + 1);
    alloc(&ci, cur_nnz);
    alloc(&lev, cur_nnz);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(rp, arp, (n + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess && cur_nnz)
      e = cudaMemcpyAsync(ci, aci, cur_nnz * sizeof(int32_t), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess && cur_nnz) e = cudaMemsetAsync(lev, 0, cur_nnz, s);
  }
  int64_t *diag = nullptr;
  alloc(&diag, n);
  if (e != cudaSuccess) {
    drop(diag);
    return leave(e);
  }
  k_fill_finish<<<fill_blocks(n), 256, 0, s>>>(n, rp, ci, diag, maxrow, err, max_row);
  note_launch();
  ok = true;
  fp->nnz = cur_nnz;
  fp->rowptr = rp;
  fp->colind = ci;
  fp->level = lev;
  fp->diag = diag;
  return leave(cudaGetLastError());
}

}  // namespace iluk
