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
// Each pass is two launches of k_fill_rows over the pattern so far (CSR with
// levels), one warp per row: the first counts the row's new columns, a scan
// gives the new row pointers, the second finds them again and writes the row.
// The columns are two bitmaps in shared memory over the row's window (the
// pattern's widest reach left and right of the diagonal): those present, and
// those the pass adds.  The candidates of up to 32 pivots are taken as one list
// (prefix sums of the pivots' upper lengths), 32 at a time, so short pivot rows
// fill the lanes and all loads of a step are independent.
// What bounds it: the latency of those loads, hidden by the rows in flight; no
// row waits for another.  The waiting walk this replaces was a chain over
// index-ordered rows: 3D 64^3, k = 2 9.4 -> 0.78 ms, random band (n = 160,000)
// k = 2 18.7 -> 0.64 ms.
// Patterns whose window exceeds kMaxFillCols keep the walk of symbolic.cu (clearing
// and scanning such a window for every row would cost more than the waits).
#include "internal.h"

namespace iluk {

constexpr int kFillThreads = 256;
constexpr int64_t kMaxFillCols = 65536;

// reach[0], reach[1]: the most columns a row reaches left and right of its
// diagonal; ustart[i]: the first entry of row i right of the diagonal.
__global__ void k_fill_reach(int64_t n, const int64_t *__restrict__ rp,
                             const int32_t *__restrict__ ci, int64_t *ustart, int32_t *reach) {
  int32_t left = 0, right = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = rp[i], e = rp[i + 1];
    ustart[i] = lower_bound_l(ci, b, e, (int32_t)(i + 1));
    if (e > b) {
      const int32_t l = (int32_t)i - ci[b], r = ci[e - 1] - (int32_t)i;
      if (l > left) left = l;
      if (r > right) right = r;
    }
  }
  left = __reduce_max_sync(FULL_MASK, left);
  right = __reduce_max_sync(FULL_MASK, right);
  if ((threadIdx.x & 31) == 0) {
    if (left > 0) atomicMax(&reach[0], left);
    if (right > 0) atomicMax(&reach[1], right);
  }
}

// Pass p over rows of the pattern (rp, ci, lev; lev null: all level 0).
// WRITE false: row_len[j] = entries after the pass.  WRITE true: the rows into
// (nrp, nci, nlev).  words: window words per warp (32 columns each).
template <bool WRITE>
__global__ void __launch_bounds__(kFillThreads)
k_fill_rows(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
            const uint8_t *__restrict__ lev, const int64_t *__restrict__ ustart, int p, int words,
            int32_t *row_len, const int64_t *__restrict__ nrp, int32_t *nci, uint8_t *nlev) {
  extern __shared__ unsigned bits[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  unsigned *old = bits + (size_t)wib * 2 * words, *add = old + words;
  const int64_t nw = (int64_t)gridDim.x * nwarps;
  for (int64_t row = (int64_t)blockIdx.x * nwarps + wib; row < n; row += nw) {
    const int64_t b0 = rp[row], b1 = rp[row + 1];
    const int m0 = (int)(b1 - b0);
    for (int w = lane; w < words; w += 32) old[w] = add[w] = 0u;
    __syncwarp();
    // every column of the finished row lies at or right of its first one (a
    // fill column t lies right of a pivot that is itself in the row)
    const int32_t c0 = m0 > 0 ? ci[b0] : 0;
    const int npiv_max = (int)(ustart[row] - b0);  // lower entries, and the diagonal if stored
    for (int q = lane; q < m0; q += 32) {
      const int d = ci[b0 + q] - c0;
      atomicOr(&old[d >> 5], 1u << (d & 31));
    }
    __syncwarp();
    for (int base = 0; base < npiv_max; base += 32) {
      const int q = base + lane;
      int len = 0, want = -1;  // the level a partner entry must have
      int64_t start = 0;
      if (q < npiv_max) {
        const int32_t i = ci[b0 + q];
        if (i < row) {
          want = p - 1 - (lev ? (int)lev[b0 + q] : 0);
          start = ustart[i];
          if (want >= 0) len = (int)(rp[i + 1] - start);
        }
      }
      int incl = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += y;
      }
      const int total = __shfl_sync(FULL_MASK, incl, 31);
      const int excl = incl - len;
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
        const int64_t src = __shfl_sync(FULL_MASK, start, s) + (t - __shfl_sync(FULL_MASK, excl, s));
        const int wl = __shfl_sync(FULL_MASK, want, s);
        if (t < total) {
          const int l = lev ? (int)lev[src] : 0;
          if (l == wl) {
            const int d = ci[src] - c0;
            const unsigned bit = 1u << (d & 31);
            if (!(old[d >> 5] & bit)) atomicOr(&add[d >> 5], bit);
          }
        }
      }
    }
    __syncwarp();
    if (!WRITE) {
      int cnt = 0;
      for (int w = lane; w < words; w += 32) cnt += __popc(add[w]);
      cnt = __reduce_add_sync(FULL_MASK, cnt);
      if (lane == 0) row_len[row] = m0 + cnt;
    } else {
      const int64_t dst = nrp[row];
      int done = 0, old_done = 0;
      for (int w0 = 0; w0 < words; w0 += 32) {
        const int w = w0 + lane;
        const unsigned o = w < words ? old[w] : 0u;
        unsigned x = o | (w < words ? add[w] : 0u);
        // both counts in one scan: present columns and earlier ones
        const unsigned c = (unsigned)__popc(x) | ((unsigned)__popc(o) << 16);
        if (!__any_sync(FULL_MASK, c != 0u)) continue;
        unsigned inc = c;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
          const unsigned y = __shfl_up_sync(FULL_MASK, inc, s);
          if (lane >= s) inc += y;
        }
        const unsigned ex = inc - c;
        int64_t pos = dst + done + (int)(ex & 0xffffu);
        int64_t oq = b0 + old_done + (int)(ex >> 16);
        while (x) {
          const int b = __ffs(x) - 1;
          x &= x - 1u;
          nci[pos] = c0 + w * 32 + b;
          if ((o >> b) & 1u) {
            nlev[pos] = lev ? lev[oq] : (uint8_t)0;
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

// Columns of the widest row's window, 0 when the passes do not take it.  Fill
// never widens it: a row keeps its first column, and a fill column t comes from
// a pivot i < j with t - i at most the pattern's reach.  Synchronous.
int64_t fill_window(int64_t n, const int64_t *arp, const int32_t *aci, cudaStream_t s) {
  if (n == 0) return 0;
  int64_t *ustart = nullptr;
  int32_t *reach = nullptr, h[2] = {0, 0};
  bool ok = cudaMallocAsync((void **)&reach, sizeof(h), s) == cudaSuccess &&
            cudaMallocAsync((void **)&ustart, (size_t)n * sizeof(int64_t), s) == cudaSuccess &&
            cudaMemsetAsync(reach, 0, sizeof(h), s) == cudaSuccess;
  if (ok) {
    k_fill_reach<<<fill_blocks(n), 256, 0, s>>>(n, arp, aci, ustart, reach);
    note_launch();
    ok = cudaMemcpyAsync(h, reach, sizeof(h), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
  }
  if (reach) cudaFreeAsync(reach, s);
  if (ustart) cudaFreeAsync(ustart, s);
  if (!ok) {
    cudaGetLastError();
    return 0;
  }
  const int64_t cols = (int64_t)h[0] + h[1] + 1;
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
  int64_t *rp = nullptr, *ustart = nullptr, *nrp = nullptr, *scan_tmp = nullptr;
  int32_t *ci = nullptr, *nci = nullptr, *reach = nullptr, *row_len = nullptr;
  uint8_t *lev = nullptr, *nlev = nullptr;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](auto **p, size_t cnt) {
    if (e == cudaSuccess) e = cudaMallocAsync((void **)p, (cnt ? cnt : 1) * sizeof(**p), s);
  };
  auto drop = [&](auto *&p) {
    if (p) cudaFreeAsync(p, s);
    p = nullptr;
  };
  auto leave = [&](cudaError_t r) {
    drop(ustart);
    drop(scan_tmp);
    drop(reach);
    drop(row_len);
    drop(nrp);
    drop(nci);
    drop(nlev);
    if (!ok) {
      drop(rp);
      drop(ci);
      drop(lev);
    }
    return r;
  };
  alloc(&ustart, n);
  alloc(&scan_tmp, scan_tmp_elems(n));
  alloc(&reach, 2);
  alloc(&row_len, n);
  if (e == cudaSuccess) e = cudaMemsetAsync(reach, 0, 2 * sizeof(int32_t), s);
  int64_t cur_nnz = nnz;
  int top = 0;  // highest level present
  // levels above 2 top + 1 have no two entries to come from
  for (int p = 1; p <= k && p <= 2 * top + 1 && e == cudaSuccess; ++p) {
    const int64_t *crp = rp ? rp : arp;
    const int32_t *cci = rp ? ci : aci;
    k_fill_reach<<<fill_blocks(n), 256, 0, s>>>(n, crp, cci, ustart, reach);
    note_launch();
    const int words = (int)((cols + 31) / 32);
    int warps = kFillThreads / 32;
    while (warps > 1 && (size_t)words * 8 * warps > (size_t)max_smem_optin() / 2) warps >>= 1;
    const size_t smem = (size_t)words * 8 * warps;
    e = allow_smem(k_fill_rows<false>);
    if (e == cudaSuccess) e = allow_smem(k_fill_rows<true>);
    if (e != cudaSuccess) break;
    int64_t grid = (n + warps - 1) / warps;
    if (grid > (int64_t)num_sms() * 32) grid = (int64_t)num_sms() * 32;
    k_fill_rows<false><<<(unsigned)grid, warps * 32, smem, s>>>(n, crp, cci, lev, ustart, p, words,
                                                               row_len, nullptr, nullptr, nullptr);
    note_launch();
    e = cudaGetLastError();
    alloc(&nrp, n + 1);
    if (e == cudaSuccess) e = launch_scan_lengths(n, row_len, nrp, scan_tmp, s);
    int64_t nn = 0;
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&nn, nrp + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) break;
    if (nn == cur_nnz) {  // no entry of this level
      drop(nrp);
      continue;
    }
    alloc(&nci, nn);
    alloc(&nlev, nn);
    if (e != cudaSuccess) break;
    k_fill_rows<true><<<(unsigned)grid, warps * 32, smem, s>>>(n, crp, cci, lev, ustart, p, words,
                                                              nullptr, nrp, nci, nlev);
    note_launch();
    // a launch that was refused has written no pattern for the next pass to read
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    drop(rp);
    drop(ci);
    drop(lev);
    rp = nrp;
    ci = nci;
    lev = nlev;
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
