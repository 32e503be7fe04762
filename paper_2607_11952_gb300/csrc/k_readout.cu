// Alignment read-out (Eq. 4 plan, Section 4.1.1 metrics): per-row top-k of
// T_ij = u_i K_ij v_j and the rank of given (row, column) pairs.  The row
// factor u_i does not change the order inside a row, so both kernels score
// s_ij = K_ij * v_j in float32 with identical rounding.  Order: larger
// score first, equal scores by lower column index.
#include <limits.h>
#include <math.h>

#include "fa_internal.cuh"

namespace fa {

__device__ __forceinline__ float kval(const float* K, int64_t t) { return K[t]; }
__device__ __forceinline__ float kval(const __nv_bfloat16* K, int64_t t) {
  return __bfloat162float(K[t]);
}

// (a_val, a_idx) ranks before (b_val, b_idx)?
__device__ __forceinline__ bool better(float av, int ai, float bv, int bi) {
  return av > bv || (av == bv && ai < bi);
}

constexpr int kTopkThreads = 256;

// 16 bytes of a kernel row as V = 4 or 8 floats, from aligned storage or
// (VEC = false, a caller's K that is not 16-byte aligned) element by element.
template <typename TK> struct RowVec {
  static constexpr int V = 16 / (int)sizeof(TK);
};
template <typename TK, bool VEC>
__device__ __forceinline__ uint4 load_row16(const TK* p) {
  uint4 u;
  if constexpr (VEC) {
    u = __ldcs(reinterpret_cast<const uint4*>(p));
  } else if constexpr (sizeof(TK) == 4) {
    u = make_uint4(__float_as_uint(p[0]), __float_as_uint(p[1]), __float_as_uint(p[2]),
                   __float_as_uint(p[3]));
  } else {
    const unsigned short* h = reinterpret_cast<const unsigned short*>(p);
    u.x = h[0] | ((uint32_t)h[1] << 16);
    u.y = h[2] | ((uint32_t)h[3] << 16);
    u.z = h[4] | ((uint32_t)h[5] << 16);
    u.w = h[6] | ((uint32_t)h[7] << 16);
  }
  return u;
}
__device__ __forceinline__ void widen(const uint4& u, float (&f)[4], float) {
  f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y);
  f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void widen(const uint4& u, float (&f)[8], __nv_bfloat16) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    f[2 * q] = __uint_as_float(w[q] << 16);
    f[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
  }
}
// x[j .. j + N) of a vector of n floats (16-byte aligned base, j a multiple
// of 4); entries past n are `fill`
template <int N>
__device__ __forceinline__ void load_floats(const float* __restrict__ x, int j, int n, float fill,
                                            float (&f)[N]) {
  if (j + N <= n) {
#pragma unroll
    for (int q = 0; q < N; q += 4) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(x + j + q));
      f[q] = t.x; f[q + 1] = t.y; f[q + 2] = t.z; f[q + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) f[q] = j + q < n ? x[j + q] : fill;
  }
}

// One warp per row, the row read once in 16-byte vectors with three in
// flight beyond the one in use.  The k <= 32 best (score, column) pairs are
// a list sorted across the lanes (lane t holds the t-th best); lane k-1's
// entry is the threshold, and a vector whose largest score is below it costs
// only the compare.  A candidate is inserted by a ballot (its position) and
// one shuffle; for n columns in no particular order about k (1 + ln(n/k))
// candidates pass.  Empty entries are (-inf, -1): -inf and NaN scores are
// never taken.  The read of K at half the copy rate; the widening, the
// product with v and the maximum are about 1.2 instructions per element.  The
// form it replaced (one CTA per row, 2-byte loads, a sorted 16-entry list per
// thread): top-10 of 20,000 x 20,000 BF16 in 4.44 ms; this one 0.237 ms (the
// read alone 0.12 ms).
template <typename TK, bool VEC>
__global__ void __launch_bounds__(kTopkThreads) k_topk(
    int n1, int n2, int64_t ld, const TK* __restrict__ K, const float* __restrict__ v,
    int k, int32_t* __restrict__ idx, float* __restrict__ score) {
  constexpr int V = RowVec<TK>::V, AHEAD = 3;
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (kTopkThreads / 32) + (threadIdx.x >> 5);
  if (row >= n1) return;
  const TK* Kr = K + (int64_t)row * ld;
  float best_v = -INFINITY, thr_v = -INFINITY;
  int best_i = -1, thr_i = -1;
  uint4 q[AHEAD];
#pragma unroll
  for (int a = 0; a < AHEAD; ++a) {
    const int j = (a * 32 + lane) * V;
    q[a] = j < n2 ? load_row16<TK, VEC>(Kr + j) : make_uint4(0u, 0u, 0u, 0u);
  }
  {
    // first threshold: the k-th largest of the 32 lanes' maxima over the
    // vectors at hand, which at least k scores of the row reach
    float m = -INFINITY;
#pragma unroll
    for (int a = 0; a < AHEAD; ++a) {
      const int j = (a * 32 + lane) * V;
      float s[V], vv[V];
      widen(q[a], s, TK());
      load_floats<V>(v, j, n2, 0.f, vv);
#pragma unroll
      for (int e = 0; e < V; ++e)
        if (j + e < n2) m = fmaxf(m, s[e] * vv[e]);
    }
    int rank = 0;
#pragma unroll 8
    for (int t = 0; t < 32; ++t) rank += better(__shfl_sync(0xffffffffu, m, t), t, m, lane);
    const uint32_t kth = __ballot_sync(0xffffffffu, rank == k - 1);
    thr_v = __shfl_sync(0xffffffffu, m, __ffs(kth) - 1);
    if (thr_v > -INFINITY) thr_i = INT_MAX;    // scores equal to it are taken
  }
  for (int base = 0; base < n2; base += 32 * V) {
    const int j0 = base + lane * V;
    const uint4 raw = q[0];
#pragma unroll
    for (int a = 0; a + 1 < AHEAD; ++a) q[a] = q[a + 1];
    const int jn = j0 + AHEAD * 32 * V;
    if (jn < n2) q[AHEAD - 1] = load_row16<TK, VEC>(Kr + jn);
    float s[V], vv[V];
    widen(raw, s, TK());
    load_floats<V>(v, j0, n2, 0.f, vv);
    float m = -INFINITY;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      s[e] *= vv[e];
      m = fmaxf(m, s[e]);
    }
    if (!__any_sync(0xffffffffu, m >= thr_v && j0 < n2)) continue;
    uint32_t todo = 0;
#pragma unroll
    for (int e = 0; e < V; ++e)
      if (j0 + e < n2 && better(s[e], j0 + e, thr_v, thr_i)) todo |= 1u << e;
    for (uint32_t who; (who = __ballot_sync(0xffffffffu, todo != 0)) != 0;) {
      // the first lane's first candidate
      const int src = __ffs(who) - 1, e_c = __ffs(todo) - 1;
      float cv = s[0];
#pragma unroll
      for (int e = 1; e < V; ++e) cv = e_c == e ? s[e] : cv;
      cv = __shfl_sync(0xffffffffu, cv, src);
      const int cj = __shfl_sync(0xffffffffu, j0 + e_c, src);
      if (lane == src) todo &= todo - 1;
      if (!better(cv, cj, thr_v, thr_i)) continue;   // the threshold has risen past it
      const int pos = __popc(__ballot_sync(0xffffffffu, better(best_v, best_i, cv, cj)));
      const float uv = __shfl_up_sync(0xffffffffu, best_v, 1);
      const int ui = __shfl_up_sync(0xffffffffu, best_i, 1);
      if (lane > pos) { best_v = uv; best_i = ui; }
      if (lane == pos) { best_v = cv; best_i = cj; }
      const float lv = __shfl_sync(0xffffffffu, best_v, k - 1);
      const int li = __shfl_sync(0xffffffffu, best_i, k - 1);
      if (better(lv, li, thr_v, thr_i)) { thr_v = lv; thr_i = li; }
    }
  }
  if (lane < k) {
    idx[(int64_t)row * k + lane] = best_i;
    if (score) score[(int64_t)row * k + lane] = best_v;
  }
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

fa_status launch_topk(int n1, int n2, int64_t ld, const void* K, bool bf16,
                      const float* v, int k, int32_t* idx, float* score,
                      cudaStream_t s) {
  constexpr int rows = kTopkThreads / 32;
  const unsigned grid = (unsigned)((n1 + rows - 1) / rows);
  const bool vec = aligned16(K);
#define FA_TOPK(T, VEC) \
  k_topk<T, VEC><<<grid, kTopkThreads, 0, s>>>(n1, n2, ld, static_cast<const T*>(K), v, k, idx, score)
  if (bf16) {
    if (vec) FA_TOPK(__nv_bfloat16, true); else FA_TOPK(__nv_bfloat16, false);
  } else {
    if (vec) FA_TOPK(float, true); else FA_TOPK(float, false);
  }
#undef FA_TOPK
  FA_LAUNCHED("k_topk");
  return FA_OK;
}

// rank = 1 + #{j : s_j > s_c} + #{j < c : s_j == s_c}; one CTA per query,
// the row in 16-byte vectors (two in flight per thread).  Bound by the read
// of one row per query; 20,000 queries of 20,000 BF16 columns took 264 us
// with 2-byte loads and a tie test per element, 177 us now (floor 120 us).
template <typename TK, bool VEC>
__global__ void __launch_bounds__(kTopkThreads) k_rank(
    int n2, int64_t ld, const TK* __restrict__ K, const float* __restrict__ v,
    const int32_t* __restrict__ rows, const int32_t* __restrict__ cols,
    int32_t* __restrict__ rank) {
  constexpr int V = RowVec<TK>::V;
  __shared__ int sc[kTopkThreads / 32];
  const int t = blockIdx.x;
  const int i = rows[t], c = cols[t];
  const TK* Kr = K + (int64_t)i * ld;
  const float ref = kval(Kr, c) * v[c];
  int cnt = 0;
#pragma unroll 2
  for (int j0 = threadIdx.x * V; j0 < n2; j0 += kTopkThreads * V) {
    float s[V], vv[V];
    widen(load_row16<TK, VEC>(Kr + j0), s, TK());
    load_floats<V>(v, j0, n2, 0.f, vv);
    // one vector of the row holds column c, at most one is cut by n2; every
    // other one lies wholly on one side of c
    if (j0 + V <= c) {
#pragma unroll
      for (int e = 0; e < V; ++e) cnt += s[e] * vv[e] >= ref;
    } else if (j0 > c && j0 + V <= n2) {
#pragma unroll
      for (int e = 0; e < V; ++e) cnt += s[e] * vv[e] > ref;
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const float x = s[e] * vv[e];
        cnt += j0 + e < n2 && ((x > ref) || (x == ref && j0 + e < c));
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0) sc[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int w = 0; w < kTopkThreads / 32; ++w) tot += sc[w];
    rank[t] = 1 + tot;
  }
}

fa_status launch_rank(int n2, int64_t ld, const void* K, bool bf16,
                      const float* v, int nq, const int32_t* rows,
                      const int32_t* cols, int32_t* rank, cudaStream_t s) {
  if (nq <= 0) return FA_OK;
  const bool vec = aligned16(K);
#define FA_RANK(T, VEC) \
  k_rank<T, VEC><<<nq, kTopkThreads, 0, s>>>(n2, ld, static_cast<const T*>(K), v, rows, cols, rank)
  if (bf16) {
    if (vec) FA_RANK(__nv_bfloat16, true); else FA_RANK(__nv_bfloat16, false);
  } else {
    if (vec) FA_RANK(float, true); else FA_RANK(float, false);
  }
#undef FA_RANK
  FA_LAUNCHED("k_rank");
  return FA_OK;
}

// ------------------------------------------------------------ plan change
// sum_ij |T_a,ij - T_b,ij| with T = diag(exp(log_u)) K diag(exp(log_v)):
// each element's two plan values in float32, their absolute differences
// summed in float64 in a fixed order.  One float64 add per element would be
// bound by this GPU's few float64 units, so a thread sums kDiffRows rows of
// its V = 4 or 8 columns as two unevaluated pairs of floats (Knuth's two-sum,
// at most 32 terms each) and adds the pairs to its float64 sum; a group whose
// float sum is not finite is summed again in float64.  Over 1,600
// random sums of 24 to 1,568 terms a thread's sum is off by at most one unit
// of float64 (1.1e-16 relative).  A thread owns V columns (their scalings in
// registers) of the rows blockIdx.y, + gridDim.y, ...; the block sums are
// added by one block in a fixed tree.  Bound by the two reads of K.  Whole
// call with its read-back, against an exponential and a float64 add per
// element and a one-thread final sum: 5,000 x 5,000 BF16 206 -> 67 us, 20,000
// 1,990 -> 384 us (374 us with one float pair per thread, which holds only
// float32's range; 438 with 4 rows a group).
constexpr int kDiffThreads = 256;
constexpr int kDiffRows = 8;

__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
  hi = s;
}

template <typename TK, bool VEC>
__global__ void __launch_bounds__(kDiffThreads) k_plan_l1diff(
    int n1, int n2, int64_t ld, const TK* __restrict__ Ka, const float* __restrict__ lua,
    const float* __restrict__ lva, const TK* __restrict__ Kb, const float* __restrict__ lub,
    const float* __restrict__ lvb, double* __restrict__ part) {
  constexpr int V = RowVec<TK>::V;
  __shared__ double red[kDiffThreads / 32];
  double acc = 0.0;
  for (int64_t jb = ((int64_t)blockIdx.x * kDiffThreads + threadIdx.x) * V; jb < n2;
       jb += (int64_t)gridDim.x * kDiffThreads * V) {
    const int j0 = (int)jb;
    float va[V], vb[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {   // past n2 both plans are 0
      va[e] = j0 + e < n2 ? expf(lva[j0 + e]) : 0.f;
      vb[e] = j0 + e < n2 ? expf(lvb[j0 + e]) : 0.f;
    }
    auto row = [&](int i, auto&& add) {      // |T_a - T_b| of row i to add(e, .)
      const int64_t at = (int64_t)i * ld + j0;
      float ka[V], kb[V];
      widen(load_row16<TK, VEC>(Ka + at), ka, TK());
      widen(load_row16<TK, VEC>(Kb + at), kb, TK());
      const float ua = expf(lua[i]), ub = expf(lub[i]);
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const float ta = __fmul_rn(__fmul_rn(ua, ka[e]), va[e]);
        const float tb = __fmul_rn(__fmul_rn(ub, kb[e]), vb[e]);
        add(e, j0 + e < n2 ? fabsf(ta - tb) : 0.f);
      }
    };
    for (int i0 = blockIdx.y; i0 < n1; i0 += kDiffRows * gridDim.y) {
      float hi[2] = {0.f, 0.f}, lo[2] = {0.f, 0.f};
#pragma unroll 4
      for (int i = i0; i < min(n1, i0 + kDiffRows * (int)gridDim.y); i += gridDim.y)
        row(i, [&](int e, float d) { two_sum_add(hi[e & 1], lo[e & 1], d); });
      double t = ((double)hi[0] + (double)hi[1]) + ((double)lo[0] + (double)lo[1]);
      if (!isfinite(hi[0] + hi[1])) {        // beyond float32's range, or not finite at all
        t = 0.0;
#pragma unroll 1
        for (int i = i0; i < min(n1, i0 + kDiffRows * (int)gridDim.y); i += gridDim.y)
          row(i, [&](int, float d) { t += (double)d; });
      }
      acc += t;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kDiffThreads / 32; ++w) t += red[w];
    part[blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

// one block: the sum of part[0..n) in a fixed order (thread t takes t, t +
// 256, ... in order, then a tree)
__global__ void __launch_bounds__(kDiffThreads) k_sum_in_order(int n,
                                                               const double* __restrict__ part,
                                                               double* __restrict__ out) {
  __shared__ double red[kDiffThreads / 32];
  double t = 0.0;
  for (int b = threadIdx.x; b < n; b += kDiffThreads) t += part[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double u = 0.0;
    for (int w = 0; w < kDiffThreads / 32; ++w) u += red[w];
    *out = u;
  }
}

fa_status launch_plan_l1diff(int n1, int n2, int64_t ld, bool bf16, const void* Ka,
                             const float* lua, const float* lva, const void* Kb,
                             const float* lub, const float* lvb, double* part, int nblocks,
                             double* out, cudaStream_t s) {
  const int cols = kDiffThreads * (bf16 ? 8 : 4);
  int gx = (n2 + cols - 1) / cols;
  if (gx > nblocks) gx = nblocks;
  int gy = nblocks / gx;      // at most nblocks blocks in all
  if (gy > n1) gy = n1;
  const dim3 grid((unsigned)gx, (unsigned)gy);
  const bool vec = aligned16(Ka) && aligned16(Kb);
#define FA_DIFF(T, VEC)                                                                       \
  k_plan_l1diff<T, VEC><<<grid, kDiffThreads, 0, s>>>(n1, n2, ld, static_cast<const T*>(Ka), \
                                                      lua, lva, static_cast<const T*>(Kb),   \
                                                      lub, lvb, part)
  if (bf16) {
    if (vec) FA_DIFF(__nv_bfloat16, true); else FA_DIFF(__nv_bfloat16, false);
  } else {
    if (vec) FA_DIFF(float, true); else FA_DIFF(float, false);
  }
#undef FA_DIFF
  FA_LAUNCHED("k_plan_l1diff");
  k_sum_in_order<<<1, kDiffThreads, 0, s>>>(gx * gy, part, out);
  FA_LAUNCHED("k_sum_in_order");
  return FA_OK;
}

}  // namespace fa
