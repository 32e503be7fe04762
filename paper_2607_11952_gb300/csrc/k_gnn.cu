// Learned warm start for the Sinkhorn solves (not in the paper): a 2-layer
// graph network on the column graph G2 predicts the correction
// y = log v* - log v1 between the converged column scaling of a solve and
// its cold first column update, from per-node features.
//
//   AF = Abar F,  A1 = AF W1 + b1,  H = relu(A1),  z2 = H w2,
//   a  = Abar z2 + c
//   L  = 1/n sum_j ((a_j - mean a) - (y_j - mean y))^2     (gauge invariant)
//
// W1 and w2 are used in BF16 (FP32 master copies are updated by Adam); all
// accumulation is FP32.  Reductions over nodes are deterministic (per-block
// partials summed in a fixed order).  Parameter vector layout:
// W1 [FA_GNN_FIN x 64 row-major] | b1 [64] | w2 [64] | c.
#include <math.h>

#include "fa_internal.cuh"

namespace fa {

constexpr int kFin = FA_GNN_FIN;
constexpr int kHid = FA_GNN_HIDDEN;
constexpr int kNP = FA_GNN_NPARAMS;
constexpr int kOffB1 = kFin * kHid;
constexpr int kOffW2 = kOffB1 + kHid;
constexpr int kOffC = kOffW2 + kHid;

// workspace (floats): AF n*kFin | A1 n*64 | z2 n | g n | partials nb*kNP | scal 8
struct GnnWs {
  float *AF, *A1, *z2, *g, *part, *scal;
  int nb;
};
constexpr int kGradThreads = 256;
static inline int grad_blocks(int n) {
  int nb = (n + 4 * (kGradThreads / 32) - 1) / (4 * (kGradThreads / 32));   // 4 nodes per warp
  return nb < 1 ? 1 : nb;
}
static GnnWs ws_layout(float* w, int n) {
  GnnWs s;
  s.AF = w;
  s.A1 = s.AF + (size_t)n * kFin;
  s.z2 = s.A1 + (size_t)n * kHid;
  s.g = s.z2 + n;
  s.part = s.g + n;
  s.nb = grad_blocks(n);
  s.scal = s.part + (size_t)s.nb * kNP;
  return s;
}
int64_t gnn_workspace_floats(int n) {
  return (int64_t)n * (kFin + kHid + 2) + (int64_t)grad_blocks(n) * kNP + 8;
}

// ------------------------------------------------------------ reductions
// The sums over nodes run in one block, and one SM adds only a few float64
// numbers per clock: the float64 forms of these kernels took 11 to 37 us at
// 4,000 to 5,000 nodes.  A thread's sum is therefore kept as an unevaluated
// pair of floats (Knuth's two-sum), products as the float product and its
// exact remainder; after kPairTerms terms the pair moves to a float64 sum, the
// pairs of a warp are added as pairs and the 32 warps' sums in float64.
// 240 vectors of 2,000 to 50,000 values and their squares: every result, in
// float32, is the correctly rounded one in either form; before that rounding
// the products' sums are off by up to 9e-15 relative, float64's by 4e-16.
// Fitted scale, 5,000 nodes 41 -> 29 us, 20,000 86 -> 35.
// What float32 cannot hold is summed again in float64 (sum64): a sum that is
// not finite, and products whose remainders may have underflowed.
constexpr int kPairTerms = 32;
struct PairSum {
  float hi = 0.f, lo = 0.f;
  double full = 0.0;                     // of the blocks of kPairTerms terms before
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
    hi = s;
  }
  // + (a + da) (b + db), da and db the small parts of a pair
  __device__ __forceinline__ void add_product(float a, float da, float b, float db) {
    const float p = __fmul_rn(a, b);
    add(p);
    lo += __fmaf_rn(a, b, -p) + (a * db + da * b);
  }
  __device__ __forceinline__ void flush() {
    full += (double)hi + (double)lo;
    hi = lo = 0.f;
  }
};
// term(i) for this thread's i < n, flush() after kPairTerms of them if more follow
template <typename T, typename F>
__device__ __forceinline__ void for_terms(int n, T term, F flush) {
  int i = threadIdx.x;
  while (true) {
    const int end = min(n, i + 1024 * kPairTerms);
    for (; i < end; i += 1024) term(i);
    if (i >= n) break;
    flush();
  }
}
// (a - m) as a pair, m = mh + ml
__device__ __forceinline__ void centre(float a, float mh, float ml, float& d, float& dd) {
  d = __fsub_rn(a, mh);
  const float t = __fsub_rn(d, a);
  dd = __fsub_rn(__fsub_rn(__fsub_rn(a, __fsub_rn(d, t)), __fadd_rn(mh, t)), ml);
}

// the warps' sums in float64, in every thread of a block of 1,024
__device__ __forceinline__ double add_warps(double mine, double* warp_sums) {
  __syncthreads();                       // warp_sums of the sum before are read
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = mine;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = warp_sums[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) warp_sums[0] = t;
  }
  __syncthreads();
  return warp_sums[0];
}
__device__ __forceinline__ double warp_sum64(double t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}
// sum_i f(i) over i < n in float64, in every thread (fixed order)
template <typename F>
__device__ double sum64(int n, double* warp_sums, F f) {
  double t = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) t += f(i);
  return add_warps(warp_sum64(t), warp_sums);
}
// Sum over a block of 1,024 threads with n terms in all, in every thread
// (fixed order: a tree inside the warps, then a tree over the warps' sums)
__device__ __forceinline__ double block_sum(PairSum x, int n, double* warp_sums) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(0xffffffffu, x.hi, o), l = __shfl_xor_sync(0xffffffffu, x.lo, o);
    // the same sum in both lanes: the remainder's terms do not depend on the order
    const float s = __fadd_rn(x.hi, h), b = __fsub_rn(s, x.hi);
    const float e = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, b)), __fsub_rn(h, b));
    x.lo = __fadd_rn(__fadd_rn(x.lo, l), e);
    x.hi = s;
  }
  double t = (double)x.hi + (double)x.lo;
  if (n > 1024 * kPairTerms) t += warp_sum64(x.full);
  return add_warps(t, warp_sums);
}
// a sum of n products is below this per term: their remainders, 2^-24 of
// terms of 2^-24 of the mean, are no longer normal floats
__device__ __forceinline__ bool products_too_small(double sum, int n) {
  return sum < (double)n * 0x1p-70;
}

// one block: out[0] = mean of x; when y (z) != null, out[1] (out[2]) = mean
// of y (z)
__global__ void __launch_bounds__(1024) k_means(int n, const float* __restrict__ x,
                                                const float* __restrict__ y,
                                                const float* __restrict__ z, float* out) {
  __shared__ double ws[32];
  PairSum ax, ay, az;
  for_terms(
      n,
      [&](int i) {
        ax.add(x[i]);
        if (y) ay.add(y[i]);
        if (z) az.add(z[i]);
      },
      [&] { ax.flush(); ay.flush(); az.flush(); });
  double tx = block_sum(ax, n, ws);
  double ty = y ? block_sum(ay, n, ws) : 0.0;
  double tz = z ? block_sum(az, n, ws) : 0.0;
  if (!isfinite(tx)) tx = sum64(n, ws, [=](int i) { return (double)x[i]; });
  if (!isfinite(ty)) ty = sum64(n, ws, [=](int i) { return (double)y[i]; });
  if (!isfinite(tz)) tz = sum64(n, ws, [=](int i) { return (double)z[i]; });
  if (threadIdx.x == 0) {
    out[0] = (float)(tx / n);
    if (y) out[1] = (float)(ty / n);
    if (z) out[2] = (float)(tz / n);
  }
}

// ------------------------------------------------------------ features
// F[j] = (log_v1_j - mean log_v1, corr_prev_j - mean corr_prev,
//         log(1 + deg_j), pot_prev_j - mean pot_prev, anchor_j, log(1 + t));
// the potentials are centred (they are defined up to a constant)
__global__ void k_gnn_features(int n, const int32_t* __restrict__ rp, const float* __restrict__ lv,
                               const float* __restrict__ corr, const float* __restrict__ pot,
                               const float* __restrict__ anc, float lt,
                               const float* __restrict__ mean, float* __restrict__ F) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  float* f = F + (size_t)j * kFin;
  f[0] = lv[j] - mean[0];
  f[1] = corr ? corr[j] - mean[1] : 0.f;
  f[2] = log1pf((float)(rp[j + 1] - rp[j]));
  f[3] = pot ? pot[j] - mean[2] : 0.f;
  f[4] = anc ? anc[j] : 0.f;
  f[5] = lt;
}

// ------------------------------------------------------------ forward
// AF[i] = sum_k Abar[i,k] F[k], A1 = AF W1 + b1, z2 = relu(A1) w2: one warp
// per node, the lanes over its edges, then over the hidden units (two per
// lane).  One thread per node walked a hub's 700 edges alone (26 us at 4,000
// nodes, and the hidden layer was a second launch); 4.6 us together now.
__global__ void __launch_bounds__(256) k_gnn_hidden(int n, const int32_t* __restrict__ rp,
                                                    const int32_t* __restrict__ ci,
                                                    const float* __restrict__ val,
                                                    const float* __restrict__ F,
                                                    const __nv_bfloat16* __restrict__ W1,
                                                    const float* __restrict__ theta,
                                                    const __nv_bfloat16* __restrict__ w2,
                                                    float* __restrict__ AF,
                                                    float* __restrict__ A1, float* __restrict__ z2) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  float fi[kFin];
#pragma unroll
  for (int f = 0; f < kFin; ++f) fi[f] = 0.f;
#pragma unroll 2
  for (int e = rp[i] + lane, e1 = rp[i + 1]; e < e1; e += 32) {
    const float w = val[e];
    const float* fk = F + (size_t)ci[e] * kFin;
#pragma unroll
    for (int f = 0; f < kFin; ++f) fi[f] += w * fk[f];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int f = 0; f < kFin; ++f) fi[f] += __shfl_xor_sync(0xffffffffu, fi[f], o);
#pragma unroll
  for (int f = 0; f < kFin; ++f)
    if (lane == f) AF[(size_t)i * kFin + f] = fi[f];
  float z = 0.f;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int h = lane + 32 * q;
    float a = theta[kOffB1 + h];
#pragma unroll
    for (int f = 0; f < kFin; ++f) a += fi[f] * __bfloat162float(W1[f * kHid + h]);
    A1[(size_t)i * kHid + h] = a;
    z += fmaxf(a, 0.f) * __bfloat162float(w2[h]);
  }
  for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  if (lane == 0) z2[i] = z;
}

// sum_k val[e] x[k] over node i's edges, in every lane of the warp
__device__ __forceinline__ float gather_sum(int e0, int e1, int lane, const int32_t* ci,
                                            const float* val, const float* x) {
  float s = 0.f;
#pragma unroll 2
  for (int e = e0 + lane; e < e1; e += 32) s += val[e] * x[ci[e]];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// out[i] = sum_k val[e] x[k] + theta[kOffC]  (warp per node)
__global__ void __launch_bounds__(256) k_gnn_out(int n, const int32_t* __restrict__ rp,
                                                 const int32_t* __restrict__ ci,
                                                 const float* __restrict__ val,
                                                 const float* __restrict__ x,
                                                 const float* __restrict__ theta,
                                                 float* __restrict__ out) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const float s = gather_sum(rp[i], rp[i + 1], lane, ci, val, x);
  if (lane == 0) out[i] = s + theta[kOffC];
}

// ------------------------------------------------------------ backward
// one block: residual r = (a - y) - mean(a - y), g = 2 r / n, loss = mean r^2,
// dL/dc = sum g
__global__ void __launch_bounds__(1024) k_gnn_resid(int n, const float* __restrict__ a,
                                                    const float* __restrict__ y,
                                                    float* __restrict__ g, float* loss,
                                                    float* __restrict__ grad) {
  __shared__ double ws[32];
  PairSum sa, sy;
  for_terms(
      n,
      [&](int i) {
        sa.add(a[i]);
        sy.add(y[i]);
      },
      [&] { sa.flush(); sy.flush(); });
  double ta = block_sum(sa, n, ws), ty = block_sum(sy, n, ws);
  if (!isfinite(ta)) ta = sum64(n, ws, [=](int i) { return (double)a[i]; });
  if (!isfinite(ty)) ty = sum64(n, ws, [=](int i) { return (double)y[i]; });
  const double m = (ta - ty) / n;
  const float mh = (float)m, ml = (float)(m - (double)mh);
  // a - y as a pair, then minus the mean
  auto resid = [=](int i) {
    const float d = __fsub_rn(a[i], y[i]), t = __fsub_rn(d, a[i]);
    const float dd = __fsub_rn(__fsub_rn(a[i], __fsub_rn(d, t)), __fadd_rn(y[i], t));
    float c, dc;
    centre(d, mh, ml, c, dc);
    return c + (dc + dd);
  };
  PairSum sl, sg;
  for_terms(
      n,
      [&](int i) {
        const float r = resid(i);
        const float gi = 2.f * r / (float)n;
        g[i] = gi;
        sl.add_product(r, 0.f, r, 0.f);
        sg.add(gi);
      },
      [&] { sl.flush(); sg.flush(); });
  double al = block_sum(sl, n, ws), ag = block_sum(sg, n, ws);
  if (!isfinite(al) || products_too_small(al, n))
    al = sum64(n, ws, [=](int i) { const double r = resid(i); return r * r; });
  if (!isfinite(ag)) ag = sum64(n, ws, [=](int i) { return (double)(2.f * resid(i) / (float)n); });
  if (threadIdx.x == 0) {
    if (loss) *loss = (float)(al / n);
    grad[kOffC] = (float)ag;
  }
}

// a = Abar z2 + c  =>  gz2 = dL/dz2 = Abar^T g (Abar^T[i,k] = 1/deg k), and
// the per-block partial gradients of W1, b1, w2 (warp per node, 4 nodes per
// warp: the node's edges over the lanes, then two hidden units per lane)
__global__ void __launch_bounds__(kGradThreads) k_gnn_grad_part(
    int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
    const float* __restrict__ val, const float* __restrict__ g, const float* __restrict__ AF,
    const float* __restrict__ A1, const __nv_bfloat16* __restrict__ w2,
    float* __restrict__ part) {
  __shared__ float red[kGradThreads / 32][kNP - 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float dW[kFin][2], db[2] = {0.f, 0.f}, dw[2] = {0.f, 0.f};
#pragma unroll
  for (int f = 0; f < kFin; ++f) dW[f][0] = dW[f][1] = 0.f;
  const float w2a = __bfloat162float(w2[lane]), w2b = __bfloat162float(w2[lane + 32]);
  const int base = (blockIdx.x * (kGradThreads / 32) + warp) * 4;
  for (int k = 0; k < 4; ++k) {
    const int i = base + k;
    if (i >= n) break;
    const float gi = gather_sum(rp[i], rp[i + 1], lane, ci, val, g);
    float af[kFin];
#pragma unroll
    for (int f = 0; f < kFin; ++f) af[f] = AF[(size_t)i * kFin + f];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float a = A1[(size_t)i * kHid + lane + 32 * q];
      const float h = fmaxf(a, 0.f);
      const float d = a > 0.f ? gi * (q == 0 ? w2a : w2b) : 0.f;
#pragma unroll
      for (int f = 0; f < kFin; ++f) dW[f][q] += af[f] * d;
      db[q] += d;
      dw[q] += gi * h;
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int h = lane + 32 * q;
#pragma unroll
    for (int f = 0; f < kFin; ++f) red[warp][f * kHid + h] = dW[f][q];
    red[warp][kOffB1 + h] = db[q];
    red[warp][kOffW2 + h] = dw[q];
  }
  __syncthreads();
  for (int p = threadIdx.x; p < kNP - 1; p += blockDim.x) {
    float s = 0.f;
    for (int w = 0; w < kGradThreads / 32; ++w) s += red[w][p];
    part[(size_t)blockIdx.x * kNP + p] = s;
  }
}

// grad[p] = sum over the blocks' partials: 32 parameters per block, the
// partials over 32 groups of lanes (b = group, + 32, ...), the groups added
// in order
__global__ void __launch_bounds__(1024) k_gnn_grad_reduce(int nb, const float* __restrict__ part,
                                                          float* __restrict__ grad) {
  __shared__ float red[32][33];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (p < kNP - 1) {
#pragma unroll 4
    for (int b = grp; b < nb; b += 32) s += part[(size_t)b * kNP + p];
  }
  red[grp][lane] = s;
  __syncthreads();
  if (grp == 0 && p < kNP - 1) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 32; ++k) t += red[k][lane];
    grad[p] = t;
  }
}

// ------------------------------------------------------------ optimiser
__global__ void k_gnn_adam(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ grad, float lr, float b1, float b2, float eps,
                           int step, __nv_bfloat16* __restrict__ W1,
                           __nv_bfloat16* __restrict__ w2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kNP) return;
  const float c1 = 1.f - powf(b1, (float)step);   // bias corrections
  const float c2 = 1.f - powf(b2, (float)step);
  const float g = grad[p];
  const float mp = b1 * m[p] + (1.f - b1) * g;
  const float vp = b2 * v[p] + (1.f - b2) * g * g;
  m[p] = mp;
  v[p] = vp;
  const float th = theta[p] - lr * (mp / c1) / (sqrtf(vp / c2) + eps);
  theta[p] = th;
  if (p < kOffB1) W1[p] = __float2bfloat16_rn(th);
  else if (p >= kOffW2 && p < kOffC) w2[p - kOffW2] = __float2bfloat16_rn(th);
}

__global__ void k_gnn_sync_bf16(const float* __restrict__ theta, __nv_bfloat16* __restrict__ W1,
                                __nv_bfloat16* __restrict__ w2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kOffB1) W1[p] = __float2bfloat16_rn(theta[p]);
  else if (p >= kOffW2 && p < kOffC) w2[p - kOffW2] = __float2bfloat16_rn(theta[p]);
}

__device__ __forceinline__ float clamp_pred(float p, float max_abs) {
  return isfinite(p) ? fminf(fmaxf(p, -max_abs), max_abs) : 0.f;
}

// warm start: out = log_v1 + scale * clamp(pred, -max_abs, max_abs); a
// non-finite prediction contributes 0 (the cold start for that column)
__global__ void k_gnn_warm(int n, const float* __restrict__ lv1, const float* __restrict__ pred,
                           float max_abs, const float* __restrict__ scale,
                           float* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = lv1[i] + (scale ? scale[0] : 1.f) * clamp_pred(pred[i], max_abs);
}

// one block: the centred least-squares scale of clamp(pred) against y,
// clipped to [0, 1] (two fixed-order passes: means, then moments)
__global__ void __launch_bounds__(1024) k_gnn_fit_scale(int n, const float* __restrict__ pred,
                                                        const float* __restrict__ y,
                                                        float max_abs, int shrink,
                                                        float* __restrict__ out) {
  __shared__ double ws[32];
  PairSum sp, sy;
  for_terms(
      n,
      [&](int i) {
        sp.add(clamp_pred(pred[i], max_abs));
        sy.add(y[i]);
      },
      [&] { sp.flush(); sy.flush(); });
  const double mp = block_sum(sp, n, ws) / n;
  double ty = block_sum(sy, n, ws);
  if (!isfinite(ty)) ty = sum64(n, ws, [=](int i) { return (double)y[i]; });
  const double my = ty / n;
  const float ph = (float)mp, pl = (float)(mp - (double)ph);
  const float yh = (float)my, yl = (float)(my - (double)yh);
  PairSum sxy, sxx, syy;
  float p_dev = 0.f, y_dev = 0.f;
  for_terms(
      n,
      [&](int i) {
        float p, dp, v, dv;
        centre(clamp_pred(pred[i], max_abs), ph, pl, p, dp);
        centre(y[i], yh, yl, v, dv);
        p_dev = fmaxf(p_dev, fabsf(p) + fabsf(dp));
        y_dev = fmaxf(y_dev, fabsf(v) + fabsf(dv));
        sxy.add_product(p, dp, v, dv);
        sxx.add_product(p, dp, p, dp);
        syy.add_product(v, dv, v, dv);
      },
      [&] { sxy.flush(); sxx.flush(); syy.flush(); });
  double txy = block_sum(sxy, n, ws), txx = block_sum(sxx, n, ws), tyy = block_sum(syy, n, ws);
  // constant vectors deviate by exactly 0: nothing has underflowed
  const bool p_varies = __syncthreads_or(p_dev != 0.f), y_varies = __syncthreads_or(y_dev != 0.f);
  if (!isfinite(txy + txx + tyy) || (p_varies && y_varies && (products_too_small(txx, n) ||
                                                               products_too_small(tyy, n)))) {
    double xy = 0.0, xx = 0.0, yy = 0.0;
    for (int i = threadIdx.x; i < n; i += 1024) {
      const double dp = (double)clamp_pred(pred[i], max_abs) - mp, dy = (double)y[i] - my;
      xy += dp * dy;
      xx += dp * dp;
      yy += dy * dy;
    }
    txy = add_warps(warp_sum64(xy), ws);
    txx = add_warps(warp_sum64(xx), ws);
    tyy = add_warps(warp_sum64(yy), ws);
  }
  if (threadIdx.x == 0) {
    double a = txx > 0.0 ? txy / txx : 0.0;
    a = a < 0.0 ? 0.0 : (a > 1.0 ? 1.0 : a);
    const double r2 = (txx > 0.0 && tyy > 0.0) ? (txy * txy) / (txx * tyy) : 0.0;
    if (shrink == 1) a *= r2;
    else if (shrink == 2) a *= sqrt(r2);
    out[0] = (float)a;
  }
}

__global__ void k_axpby(int n, float a, const float* __restrict__ x, float b,
                        const float* __restrict__ y, float* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = a * x[i] + (y ? b * y[i] : 0.f);
}

}  // namespace fa

// ------------------------------------------------------------ C ABI
struct fa_gnn {
  float* theta = nullptr;           // FP32 master parameters (kNP)
  float* m = nullptr;               // Adam first moment
  float* v = nullptr;               // Adam second moment
  __nv_bfloat16* W1 = nullptr;      // BF16 copy used by the forward pass
  __nv_bfloat16* w2 = nullptr;
  int64_t step = 0;
};

using namespace fa;

extern "C" {

fa_status fa_gnn_create(fa_gnn** out) {
  if (!out) { set_error("fa_gnn_create: out is NULL"); return FA_ERR_ARG; }
  *out = nullptr;
  fa_gnn* g = new fa_gnn();
  cudaError_t e;
  if ((e = cudaMalloc(&g->theta, kNP * 4)) != cudaSuccess || (e = cudaMalloc(&g->m, kNP * 4)) != cudaSuccess ||
      (e = cudaMalloc(&g->v, kNP * 4)) != cudaSuccess || (e = cudaMalloc(&g->W1, kOffB1 * 2)) != cudaSuccess ||
      (e = cudaMalloc(&g->w2, kHid * 2)) != cudaSuccess) {
    cudaGetLastError();
    set_error("fa_gnn_create: %s", cudaGetErrorString(e));
    fa_gnn_destroy(g);
    return FA_ERR_OOM;
  }
  if (cudaMemset(g->theta, 0, kNP * 4) != cudaSuccess || cudaMemset(g->m, 0, kNP * 4) != cudaSuccess ||
      cudaMemset(g->v, 0, kNP * 4) != cudaSuccess || cudaMemset(g->W1, 0, kOffB1 * 2) != cudaSuccess ||
      cudaMemset(g->w2, 0, kHid * 2) != cudaSuccess) {
    set_error("fa_gnn_create: memset failed");
    fa_gnn_destroy(g);
    return FA_ERR_CUDA;
  }
  *out = g;
  return FA_OK;
}

fa_status fa_gnn_destroy(fa_gnn* g) {
  if (!g) return FA_OK;
  if (g->theta) cudaFree(g->theta);
  if (g->m) cudaFree(g->m);
  if (g->v) cudaFree(g->v);
  if (g->W1) cudaFree(g->W1);
  if (g->w2) cudaFree(g->w2);
  delete g;
  return FA_OK;
}

fa_status fa_gnn_set_params(fa_gnn* g, const float* host_theta) {
  if (!g || !host_theta) { set_error("fa_gnn_set_params: NULL argument"); return FA_ERR_ARG; }
  FA_CUDA(cudaMemcpy(g->theta, host_theta, kNP * 4, cudaMemcpyHostToDevice));
  FA_CUDA(cudaMemset(g->m, 0, kNP * 4));
  FA_CUDA(cudaMemset(g->v, 0, kNP * 4));
  g->step = 0;
  k_gnn_sync_bf16<<<(kNP + 255) / 256, 256>>>(g->theta, g->W1, g->w2);
  FA_LAUNCHED("k_gnn_sync_bf16");
  FA_CUDA(cudaDeviceSynchronize());
  return FA_OK;
}

fa_status fa_gnn_get_params(const fa_gnn* g, float* host_theta) {
  if (!g || !host_theta) { set_error("fa_gnn_get_params: NULL argument"); return FA_ERR_ARG; }
  FA_CUDA(cudaMemcpy(host_theta, g->theta, kNP * 4, cudaMemcpyDeviceToHost));
  return FA_OK;
}

int64_t fa_gnn_workspace_floats(int32_t n) { return n < 1 ? -1 : gnn_workspace_floats(n); }

fa_status fa_gnn_features(const fa_graph* g2, const float* log_v1, const float* corr_prev,
                          const float* pot_prev, const float* anchor_mask, int32_t outer_index,
                          float* F, float* ws, fa_stream_t stream) {
  if (!g2 || !log_v1 || !F || !ws) { set_error("fa_gnn_features: NULL argument"); return FA_ERR_ARG; }
  if (outer_index < 0) { set_error("fa_gnn_features: outer_index < 0"); return FA_ERR_ARG; }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int n = g2->d.n;
  GnnWs w = ws_layout(ws, n);
  k_means<<<1, 1024, 0, s>>>(n, log_v1, corr_prev, pot_prev, w.scal);
  FA_LAUNCHED("k_means");
  k_gnn_features<<<(n + 255) / 256, 256, 0, s>>>(n, g2->d.row_ptr, log_v1, corr_prev, pot_prev,
                                                 anchor_mask, log1pf((float)outer_index), w.scal, F);
  FA_LAUNCHED("k_gnn_features");
  return FA_OK;
}

fa_status fa_gnn_forward(fa_gnn* g, const fa_graph* graph, const float* F, float* ws, float* a_out,
                         fa_stream_t stream) {
  if (!g || !graph || !F || !ws || !a_out) { set_error("fa_gnn_forward: NULL argument"); return FA_ERR_ARG; }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const DevGraph& d = graph->d;
  const int n = d.n;
  GnnWs w = ws_layout(ws, n);
  const unsigned blocks = (unsigned)(((int64_t)n * 32 + 255) / 256);   // a warp per node
  k_gnn_hidden<<<blocks, 256, 0, s>>>(n, d.row_ptr, d.col, d.val_row, F, g->W1, g->theta, g->w2,
                                      w.AF, w.A1, w.z2);
  FA_LAUNCHED("k_gnn_hidden");
  k_gnn_out<<<blocks, 256, 0, s>>>(n, d.row_ptr, d.col, d.val_row, w.z2, g->theta, a_out);
  FA_LAUNCHED("k_gnn_out");
  return FA_OK;
}

fa_status fa_gnn_backward(fa_gnn* g, const fa_graph* graph, const float* ws_in, const float* a_pred,
                          const float* target, float* grad, float* loss, fa_stream_t stream) {
  if (!g || !graph || !ws_in || !a_pred || !target || !grad) {
    set_error("fa_gnn_backward: NULL argument");
    return FA_ERR_ARG;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const DevGraph& d = graph->d;
  const int n = d.n;
  GnnWs w = ws_layout(const_cast<float*>(ws_in), n);
  k_gnn_resid<<<1, 1024, 0, s>>>(n, a_pred, target, w.g, loss, grad);
  FA_LAUNCHED("k_gnn_resid");
  k_gnn_grad_part<<<w.nb, kGradThreads, 0, s>>>(n, d.row_ptr, d.col, d.val_col, w.g, w.AF, w.A1,
                                                g->w2, w.part);
  FA_LAUNCHED("k_gnn_grad_part");
  k_gnn_grad_reduce<<<(kNP - 1 + 31) / 32, 1024, 0, s>>>(w.nb, w.part, grad);
  FA_LAUNCHED("k_gnn_grad_reduce");
  return FA_OK;
}

fa_status fa_gnn_adam_step(fa_gnn* g, const float* grad, float lr, float beta1, float beta2,
                           float eps, fa_stream_t stream) {
  if (!g || !grad) { set_error("fa_gnn_adam_step: NULL argument"); return FA_ERR_ARG; }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  g->step += 1;
  k_gnn_adam<<<(kNP + 255) / 256, 256, 0, s>>>(g->theta, g->m, g->v, grad, lr, beta1, beta2, eps,
                                               (int)g->step, g->W1, g->w2);
  FA_LAUNCHED("k_gnn_adam");
  return FA_OK;
}

fa_status fa_gnn_warm_start(int32_t n, const float* log_v1, const float* pred, float max_abs,
                            const float* scale, float* out, fa_stream_t stream) {
  if (n < 1 || !log_v1 || !pred || !out || !(max_abs > 0.f)) {
    set_error("fa_gnn_warm_start: bad argument");
    return FA_ERR_ARG;
  }
  k_gnn_warm<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, log_v1, pred, max_abs, scale, out);
  FA_LAUNCHED("k_gnn_warm");
  return FA_OK;
}

fa_status fa_gnn_fit_scale(int32_t n, const float* pred, const float* y, float max_abs,
                           int32_t shrink, float* scale, fa_stream_t stream) {
  if (n < 1 || !pred || !y || !scale || !(max_abs > 0.f)) {
    set_error("fa_gnn_fit_scale: bad argument");
    return FA_ERR_ARG;
  }
  k_gnn_fit_scale<<<1, 1024, 0, reinterpret_cast<cudaStream_t>(stream)>>>(n, pred, y, max_abs,
                                                                          shrink, scale);
  FA_LAUNCHED("k_gnn_fit_scale");
  return FA_OK;
}

fa_status fa_vec_axpby(int32_t n, float a, const float* x, float b, const float* y, float* out,
                       fa_stream_t stream) {
  if (n < 0 || (n > 0 && (!x || !out))) { set_error("fa_vec_axpby: bad argument"); return FA_ERR_ARG; }
  if (n == 0) return FA_OK;
  k_axpby<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(n, a, x, b, y, out);
  FA_LAUNCHED("k_axpby");
  return FA_OK;
}

}  // extern "C"
