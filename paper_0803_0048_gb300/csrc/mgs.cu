// mgs.cu -- a6: one Arnoldi step's modified Gram-Schmidt orthogonalisation in
// one launch: h_i = (w, v_i), w <- w - h_i v_i for i = 0 .. j, then h_{j+1} =
// ||w|| and v_{j+1} = w / h_{j+1}, with the fixed-shape inner product of
// krylov.cu (4096 partial sums, pairwise tree), so every bit is that of the
// one-launch-per-step form.
//
// 128 CTAs, one per SM, own 32 consecutive partials each, that is the
// elements p + 4096 r (a row of 32 for each r): they keep their part of w, and of
// the v_i as it passes, in shared memory for the whole step, so w is read
// once and each v_i once.  In a CTA the warps of three SM sub-partitions form
// the updates and products, a row at a time, while warp 0 adds the products in
// order (one chain per lane): a product's place holds a signalling NaN, which no
// product is, until it is there, and again once it is taken.  Against six busy
// warps a chain of additions still gets one in per 76 cycles, so that warp's own
// loads, votes and stores must not stand in its way: it takes Q products at a
// time and fetches the next Q, into registers of their own, and frees the places
// between the additions, whose latency hides both (before, four at a time ahead of
// their additions, a row took 118 cycles).  The tree runs over CTAs instead of
// through one CTA's memory: its strides 64 and 32 (in CTAs) inside a cluster of
// four, the partials pushed to the cluster's first CTA, its strides 16 .. 1
// over the 32 clusters' vectors, which travel through L2 and are summed by every
// cluster alike (four warps, eight vectors each), the last five levels as
// shuffles; the result is pushed to the cluster's CTAs.  Those values carry the
// step's tag in both 64-bit words, so they are their own flags and nothing is
// cleared in between.  (Clusters of eight would not all be resident: 15 fit.)
// What bounds it: per inner product the four FP64 operations an element on the
// 128 SMs' pipes, which is also the chain of n / 4096 additions (76 cycles each,
// 90 measured), and ~2.5 us of hand-offs and tree, instead of a launch, a counter
// and one CTA's tree.  Per inner product, launches included, one launch a step ->
// four products ahead of their additions -> this: n = 4,096 10.5 -> 2.9 -> 2.95 us,
// 65,536 11.7 -> 4.2 -> 3.8, 262,144 14.4 -> 7.2 -> 6.2, 729,000 20.5 -> 14.1 -> 11.6
// (a third of the warps or twice as many compute warps measured the same, and so
// did two or four rows at a time).
// All CTAs are resident (cooperative launch); every wait is bounded.
#include "internal.h"

namespace iluk {

constexpr int kMgsCluster = 4;
constexpr int kMgsClusters = kDotP / 32 / kMgsCluster;
constexpr int kMgsWarps = 8;
constexpr int kMgsThreads = kMgsWarps * 32;
constexpr int kMgsComputeWarps = kMgsWarps * 3 / 4;  // those of sub-partitions 1..3
constexpr unsigned long long kNoProduct = 0x7FF0DEADBEEFCAFEull;
static_assert(kMgsClusters == 32 && kMgsCluster == 4, "the tree below is written for 32 x 4");

struct MgsShared {
  uint4 slot[kMgsCluster][32];  // the cluster's partials (first CTA)
  uint4 part[4][32];            // the four warps' sums over the clusters (first CTA)
  uint4 h;                      // the inner product
};

// A double and its tag as two words, the tag in both (see the ring of sweeps.cu).
__device__ __forceinline__ void tag_words(double v, unsigned tag, unsigned long long &w0,
                                          unsigned long long &w1) {
  w0 = ((unsigned long long)tag << 32) | (unsigned)__double2loint(v);
  w1 = ((unsigned long long)tag << 32) | (unsigned)__double2hiint(v);
}

__device__ __forceinline__ bool tag_read(unsigned long long w0, unsigned long long w1,
                                         unsigned tag, double &v) {
  v = __hiloint2double((int)(unsigned)w1, (int)(unsigned)w0);
  return (unsigned)(w0 >> 32) == tag && (unsigned)(w1 >> 32) == tag;
}

__device__ __forceinline__ bool smem_try(const uint4 *p, unsigned tag, double &v) {
  unsigned long long w0, w1;
  asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];"
               : "=l"(w0), "=l"(w1)
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
  return tag_read(w0, w1, tag, v);
}

__device__ __forceinline__ void cluster_put(const uint4 *p, unsigned cta, double v, unsigned tag) {
  unsigned a;
  unsigned long long w0, w1;
  tag_words(v, tag, w0, w1);
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(a)
      : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(cta));
  asm volatile("st.relaxed.cluster.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(a), "l"(w0),
               "l"(w1)
               : "memory");
}

struct MgsWait {
  volatile int *fail;
  int64_t limit_ns;
  // try_ until it holds in every lane; false when the wait runs out or another has
  template <class F>
  __device__ __forceinline__ bool operator()(F try_) const {
    uint64_t t0 = 0;
    for (unsigned it = 0;; ++it) {
      if (__all_sync(FULL_MASK, try_())) return true;
      if ((it & 1023u) == 1023u) {
        if (t0 == 0) t0 = globaltimer_ns();
        const bool late = (int64_t)(globaltimer_ns() - t0) > limit_ns;
        if (__any_sync(FULL_MASK, late || *fail != 0)) {
          if (late) *fail = 1;
          return false;
        }
      }
    }
  }
};

template <int Q>
__global__ void __cluster_dims__(kMgsCluster, 1, 1) __launch_bounds__(kMgsThreads, 1)
k_mgs(int64_t n, int rows, const double *__restrict__ w, const double *__restrict__ V,
      int64_t ldv, int j, double *hc, double *vout, uint4 *xchg, unsigned tag0, int *fail,
      int64_t limit_ns) {
  extern __shared__ __align__(16) double sm[];  // w, v_even, v_odd, products: rows4 x 32 each
  __shared__ __align__(16) MgsShared sh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned rank, C;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  // the launch this kernel's tree is written for, or nothing
  if (C != kMgsCluster || gridDim.x != kMgsCluster * kMgsClusters) {
    if (threadIdx.x == 0) *fail = 1;
    return;
  }
  const size_t part = (size_t)rows * 32;
  const int cl = blockIdx.x / kMgsCluster;
  const int64_t p = (int64_t)(cl + kMgsClusters * (int)rank) * 32 + lane;
  double *sw = sm + lane, *sv = sw + part, *sp = sw + 3 * part;  // sv: even, then odd
  for (int t = threadIdx.x; t < (int)(sizeof(sh) / 4); t += blockDim.x)
    reinterpret_cast<unsigned *>(&sh)[t] = 0u;
  for (size_t t = threadIdx.x; t < part; t += blockDim.x)
    sm[3 * part + t] = __longlong_as_double((long long)kNoProduct);
  __syncthreads();
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");

  const MgsWait wait{fail, limit_ns};
  const int cw = (warp & 3) ? warp - (warp >> 2) - 1 : -1;  // compute warp, or -1
  const int ninner = j + 2;                                 // inner products of the step
  // The sums over the clusters' vectors q, q + 4, .., q + 28 (strides 16, 8, 4).
  auto cross = [&](int r, int q, double &x) -> bool {
    const uint4 *src = xchg + ((size_t)(r & 1) * kMgsClusters + q) * 32 + lane;
    const unsigned tag = tag0 + (unsigned)r;
    double a[8];
    const bool ok = wait([&] {
      bool all = true;
      unsigned long long w0[8], w1[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
                     : "=l"(w0[u]), "=l"(w1[u])
                     : "l"(src + u * 4 * 32)
                     : "memory");
#pragma unroll
      for (int u = 0; u < 8; ++u) all = tag_read(w0[u], w1[u], tag, a[u]) && all;
      return all;
    });
    if (!ok) return false;
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1)
#pragma unroll
      for (int u = 0; u < o; ++u) a[u] = __dadd_rn(a[u], a[u + o]);
    x = a[0];
    return true;
  };

  if (cw >= 0) {
    // this warp's rows: cw, cw + kMgsComputeWarps, ... (elements past the end
    // hold +0.0)
    auto fetch = [&](const double *src, double *dst, int r) {
      const int64_t i = p + (int64_t)r * kDotP;
      const unsigned a = (unsigned)__cvta_generic_to_shared(dst + (size_t)r * 32);
      if (i < n)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(a), "l"(src + i));
      else
        dst[(size_t)r * 32] = 0.0;
    };
    for (int r = cw; r < rows; r += kMgsComputeWarps) {
      fetch(w, sw, r);
      fetch(V, sv, r);
      if (j >= 1) fetch(V + ldv, sv + part, r);
    }
    bool ok = true;
    const bool sums = rank == 0 && warp <= 3;
    if (cw < rows || sums) {
      double h = 0.0;
      for (int s = 0; s < ninner; ++s) {
        if (s > 0) ok = wait([&] { return smem_try(&sh.h, tag0 + (unsigned)(s - 1), h); });
        if (!ok) break;
        asm volatile("cp.async.wait_all;" ::: "memory");
        double *vi = sv + (s & 1 ? 0 : part);                  // v_{s-1}
        const double *vn = s <= j ? sv + (s & 1 ? part : 0) : sw;  // v_s; at last w itself
        for (int r = cw; r < rows; r += kMgsComputeWarps) {
          const size_t o = (size_t)r * 32;
          double x = sw[o];
          if (s > 0) {
            x = __dsub_rn(x, __dmul_rn(h, vi[o]));
            sw[o] = x;
          }
          asm volatile("st.volatile.shared.f64 [%0], %1;" ::"r"(
                           (unsigned)__cvta_generic_to_shared(sp + o)),
                       "d"(__dmul_rn(x, vn[o])));
          // v_{s-1} is done with: v_{s+1} takes its place
          if (s > 0 && s + 1 <= j) fetch(V + (int64_t)(s + 1) * ldv, vi, r);
        }
        if (sums) {
          double x;
          ok = cross(s, warp, x);
          if (!ok) break;
          unsigned long long w0, w1;
          tag_words(x, tag0 + (unsigned)s, w0, w1);
          asm volatile("st.volatile.shared.v2.u64 [%0], {%1, %2};" ::"r"(
                           (unsigned)__cvta_generic_to_shared(&sh.part[warp][lane])),
                       "l"(w0), "l"(w1)
                       : "memory");
        }
      }
      if (ok) ok = wait([&] { return smem_try(&sh.h, tag0 + (unsigned)(ninner - 1), h); });
      if (ok && h != 0.0) {  // h = 0: a breakdown, v_{j+1} is not needed
        const DivPrep pd = div_prep(h);
        for (int r = cw; r < rows; r += kMgsComputeWarps) {
          const int64_t i = p + (int64_t)r * kDotP;
          if (i < n) vout[i] = div_fin(sw[(size_t)r * 32], pd);
        }
      }
    }
  } else if (warp == 0) {
    const int lane_rows = p < n ? (int)((n - p + kDotP - 1) / kDotP) : 0;
    const unsigned pa = (unsigned)__cvta_generic_to_shared(sp);
    double sum = 0.0, ya[Q], yb[Q];
    auto look = [&](double &y, int r) {
      asm volatile("ld.volatile.shared.f64 %0, [%1];" : "=d"(y) : "r"(pa + (unsigned)r * 256u));
    };
    auto release = [&](int r) {
      asm volatile("st.volatile.shared.u64 [%0], %1;" ::"r"(pa + (unsigned)r * 256u),
                   "l"(kNoProduct));
    };
    auto there = [&](const double (&y)[Q], int q) {
      bool all = true;
#pragma unroll
      for (int u = 0; u < Q; ++u)
        all = all && (u >= q || (unsigned long long)__double_as_longlong(y[u]) != kNoProduct);
      return all;
    };
    auto await = [&](double (&y)[Q], int r, int q) {  // the products of rows r .. r + q - 1
      return wait([&] {
#pragma unroll
        for (int u = 0; u < Q; ++u)
          if (u < q) look(y[u], r + u);
        return there(y, q);
      });
    };
    // adds the Q products y of rows r .. and fetches the q after them into z
    auto group = [&](const double (&y)[Q], double (&z)[Q], int r, int q) {
#pragma unroll
      for (int u = 0; u < Q; ++u) {
        asm volatile("add.rn.f64 %0, %0, %1;" : "+d"(sum) : "d"(y[u]));
        if (u < q) look(z[u], r + Q + u);
        release(r + u);
      }
      return __all_sync(FULL_MASK, there(z, q)) || await(z, r + Q, q);
    };
    // the last q products: a lane may have no element in the last row
    auto finish = [&](const double (&y)[Q], int r, int q) {
#pragma unroll
      for (int u = 0; u < Q; ++u)
        if (u < q) {
          if (r + u < lane_rows) sum = __dadd_rn(sum, y[u]);
          release(r + u);
        }
    };
    for (int s = 0; s < ninner; ++s) {
      const unsigned tag = tag0 + (unsigned)s;
      sum = 0.0;
      auto left = [&](int r) { return rows - r < Q ? rows - r : Q; };
      bool ok = await(ya, 0, left(0));
      int r = 0;
      for (; ok && r + 2 * Q < rows; r += 2 * Q) {
        ok = group(ya, yb, r, Q) &&
             group(yb, ya, r + Q, left(r + 2 * Q));
      }
      if (!ok) break;
      if (r + Q < rows) {
        if (!group(ya, yb, r, left(r + Q))) break;
        finish(yb, r + Q, left(r + Q));
      } else {
        finish(ya, r, left(r));
      }
      cluster_put(&sh.slot[rank][lane], 0u, sum, tag);
      if (rank == 0) {
        double a[kMgsCluster];
        ok = wait([&] {
          bool all = true;
#pragma unroll
          for (int t = 0; t < kMgsCluster; ++t) all = smem_try(&sh.slot[t][lane], tag, a[t]) && all;
          return all;
        });
        if (!ok) break;
        const double lo = __dadd_rn(a[0], a[2]), hi = __dadd_rn(a[1], a[3]);
        unsigned long long w0, w1;
        tag_words(__dadd_rn(lo, hi), tag, w0, w1);
        asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(
                         xchg + ((size_t)(s & 1) * kMgsClusters + cl) * 32 + lane),
                     "l"(w0), "l"(w1)
                     : "memory");
        double x0, x1 = 0.0, x2 = 0.0, x3 = 0.0;
        if (!cross(s, 0, x0)) break;
        ok = wait([&] {
          bool all = smem_try(&sh.part[1][lane], tag, x1);
          all = smem_try(&sh.part[2][lane], tag, x2) && all;
          return smem_try(&sh.part[3][lane], tag, x3) && all;
        });
        if (!ok) break;
        const double e = __dadd_rn(x0, x2), o = __dadd_rn(x1, x3);
        double x = __dadd_rn(e, o);
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
          const double y2 = __shfl_down_sync(FULL_MASK, x, d);
          if (lane < d) x = __dadd_rn(x, y2);
        }
        x = __shfl_sync(FULL_MASK, x, 0);
        if (s == ninner - 1) x = __dsqrt_rn(x);
        if (lane < kMgsCluster) cluster_put(&sh.h, (unsigned)lane, x, tag);
        if (cl == 0 && lane == 0) hc[s] = x;
      }
      // a CTA's next partials follow from its next products, which follow from h
    }
  }
  // every CTA arrives here: no shared memory is released while written to
  __syncwarp();
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// Products the adding warp takes at a time: larger groups hide more of its loads
// and votes, but it starts only when a whole one is there.  Per inner product
// with groups of 1, 4, 8: 1 row 2.95, 3.05, 3.12 us; 4 rows 3.17, 3.18, 3.23; 16 rows
// 4.07, 3.77, 3.97; 64 rows 7.73, 6.24, 6.23; 178 rows 16.4, 12.1, 11.6 us.
static int mgs_group(int rows) { return rows >= 64 ? 8 : rows >= 4 ? 4 : 1; }

// Shared memory for n elements, 0 when a CTA cannot hold its part.
static size_t mgs_smem(int64_t n, int *rows) {
  const int64_t r = (n + kDotP - 1) / kDotP;
  const size_t need = (size_t)r * 32 * 4 * sizeof(double);
  if (r < 1 || need + sizeof(MgsShared) + 1024 > (size_t)max_smem_optin()) return 0;
  *rows = (int)r;
  return need;
}

size_t mgs_scratch_bytes() { return (size_t)2 * kMgsClusters * 32 * sizeof(uint4); }

// One Arnoldi step j (see the top): hc[0 .. j + 1] and vout = V_{j+1}.  `ms` holds
// the launches' exchange buffer (zeroed before the first) and the next unused
// tag.  cudaErrorInvalidConfiguration when this form cannot run here: the
// caller then takes the steps one launch at a time.
cudaError_t launch_mgs(int64_t n, const double *w, const double *V, int64_t ldv, int j, double *hc,
                       double *vout, MgsScratch *ms, cudaStream_t s) {
  int rows = 0;
  const size_t smem = mgs_smem(n, &rows);
  if (smem == 0 || !ms->xchg) return cudaErrorInvalidConfiguration;
  ProfScope prof_scope(ILUK_PROF_DOT, s);
  const int group = mgs_group(rows);
  const auto kern = group == 8 ? k_mgs<8> : group == 4 ? k_mgs<4> : k_mgs<1>;
  cudaError_t e = allow_smem(kern, sizeof(MgsShared));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kMgsCluster * kMgsClusters));
  cfg.blockDim = dim3(kMgsThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const unsigned tag0 = ms->tag;
  ms->tag += (unsigned)(j + 2);
  e = cudaLaunchKernelEx(&cfg, kern, n, rows, w, V, ldv, j, hc, vout, (uint4 *)ms->xchg,
                         tag0, ms->fail, wait_limit());
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cudaErrorInvalidConfiguration;
  }
  note_launch();
  return cudaSuccess;
}

}  // namespace iluk
