// A whole Sinkhorn solve (Algorithm 1, Phase 3; Eq. 3) in one launch, for
// kernels K that fit in the SMs' shared memory together (up to about 2,600
// square in FP32, 3,600 in BF16).
//
// At these sizes an iteration is a few microseconds of latency, not of
// bandwidth: as two launches (sweep, column finalisation) it took 15 us at
// 1,000 x 1,000, 11 us of them in the kernels' own ramps and in the launches,
// and a tolerance test was a host round trip.  Here clusters of 8 CTAs keep
// their rows of K in shared memory for the whole solve and iterate together,
// without barriers beyond the block's own:
//
//   rows      u_i = mu_i / sum_j K_ij v_j, one warp per row
//   columns   the CTA's partial column sums sum_i K_ij u_i, each eighth of
//             the columns sent to its CTA of the cluster (st.async into
//             distributed shared memory, completing on the receiver's
//             mbarrier)
//   clusters  CTA q adds the 8 partials of its eighth and publishes every sum
//             in L2 together with the iteration's tag, 8 bytes at once; it
//             polls the other clusters' words of the eighth until they carry
//             the tag (no fence, no counter, one L2 round trip), adds them
//             in cluster order -- all clusters the same values -- and forms
//             the next v and the eighth's marginal error
//   v         goes to the cluster's 8 CTAs by st.async
//
// v is carried as nu / column sum, not through its logarithm: the rounding of
// a stored logarithm (5e-7 at |log v| = 10) and the biases of expf and logf
// moved u and v apart by 1e-5 in 50 iterations.  log v and log u are formed
// once, from the last iteration: log u for v = exp(log v) as it is returned.
// The tolerance is tested on the device: every CTA sees the same error and
// leaves in the same iteration.  The launch is cooperative (all CTAs
// resident).  Every wait is bounded; a CTA whose wait gave up sets ST_TIMEOUT
// and runs its remaining iterations without waiting.
// 1,000 x 1,000 FP32, 50 iterations: 764 -> 202 us (before: two launches per
// iteration with the split finalisation).  Counters and barriers in place of
// the tagged words and the sends: 382 us.
#include <math.h>

#include <algorithm>

#include "fa_internal.cuh"
#include "sweep_dev.cuh"

namespace fa {

namespace {

constexpr int kSQ = 8;            // CTAs per cluster
constexpr int kST = 512;          // threads per CTA
constexpr int kSW = kST / 32;
constexpr size_t kSmallSmem = 220 * 1024;

__host__ __device__ constexpr int small_max_rows(int n1, int C) {
  return (n1 + kSQ * C - 1) / (kSQ * C);
}
// K rows | v[2][ld] | red[8][ld / 8] | u, row sums [R]
static size_t small_smem(int R, int64_t ld, size_t b) {
  return (size_t)R * ld * b + 3 * (size_t)ld * 4 + 2 * (size_t)((R + 3) / 4 * 4) * 4;
}

constexpr int kMaxSmallC = 24;    // most clusters (polled words per column)

__device__ __forceinline__ void st_async_f32x4(uint32_t a, float4 v, uint32_t mbar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(a),
      "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
      "r"(__float_as_uint(v.w)), "r"(mbar)
      : "memory");
}
__device__ __forceinline__ void st_async_f64(uint32_t a, double v, uint32_t mbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
               "l"(__double_as_longlong(v)), "r"(mbar)
               : "memory");
}
// a column sum and the tag of its iteration, one 8-byte word
__device__ __forceinline__ void publish(uint2* p, float v, uint32_t tag) {
  asm volatile("st.relaxed.gpu.global.v2.b32 [%0], {%1, %2};" ::"l"(p), "r"(__float_as_uint(v)),
               "r"(tag)
               : "memory");
}
__device__ __forceinline__ uint2 peek(const uint2* p) {
  uint2 r;
  asm volatile("ld.relaxed.gpu.global.v2.b32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(p) : "memory");
  return r;
}

template <typename TK>
__global__ void __launch_bounds__(kST, 1) k_solve_small(
    const TK* __restrict__ K, int64_t ld, int n1, int n2, const float* log_v_in, float* log_u,
    float* log_v_out, float mu, float log_mu, float nu, int max_iter, double tol, int check_every,
    uint2* words, uint32_t tag0, double* err_out, int* iters_out, int* status) {
  constexpr int V = KT<TK>::V, V2 = V / 2;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t loaded, sums_bar, v_bar;
  __shared__ double errs[kSQ][kSW];
  __shared__ int s_dead;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q = (int)cluster_rank(), cl = blockIdx.x / kSQ, C = gridDim.x / kSQ;
  const int G = gridDim.x;
  const int r0 = (int)((int64_t)n1 * blockIdx.x / G);
  const int R = (int)((int64_t)n1 * (blockIdx.x + 1) / G) - r0;
  const int Rmax = small_max_rows(n1, C);
  const int S = (int)(ld / kSQ);                       // columns of an eighth
  const int NWS = (S + 31) / 32;                       // warps that own columns
  TK* Ks = reinterpret_cast<TK*>(smem);
  float* vbuf = reinterpret_cast<float*>(smem + (size_t)Rmax * ld * sizeof(TK));   // [2][ld]
  float* red = vbuf + 2 * ld;                          // [8][S]
  float* u_s = red + ld;
  float* rs_s = u_s + (Rmax + 3) / 4 * 4;

  if (tid == 0) {
    mbar_init(smem_u32(&loaded), 1);
    mbar_init(smem_u32(&sums_bar), 1);
    mbar_init(smem_u32(&v_bar), 1);
    fence_mbar_init();
    s_dead = 0;
    if (R > 0) {
      const uint32_t bytes = (uint32_t)(ld * sizeof(TK));
      mbar_expect_tx(smem_u32(&loaded), bytes * (uint32_t)R);
      for (int r = 0; r < R; ++r)
        bulk_g2s(smem_u32(Ks + (int64_t)r * ld), K + (int64_t)(r0 + r) * ld, bytes,
                 smem_u32(&loaded));
    }
  }
  for (int j = tid; j < ld; j += kST) vbuf[ld + j] = j < n2 ? expf(log_v_in[j]) : 0.f;
  // thread t of CTA q owns column q S + t in the finalisation
  const int jq = q * S + tid;
  const bool own = tid < S && jq < n2;
  const float lv_first = own ? log_v_in[jq] : 0.f;
  float v_own = own ? expf(lv_first) : 0.f;
  __syncthreads();
  if (R > 0 && !mbar_wait_bounded(smem_u32(&loaded), 0)) {
    atomicOr(status, ST_TIMEOUT);
    s_dead = 1;
  }
  cluster_arrive();      // every CTA's barriers exist before any remote store
  cluster_wait();

  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (s_dead == 0 && !mbar_wait_bounded(smem_u32(bar), parity)) {
      atomicOr(status, ST_TIMEOUT);
      s_dead = 1;
    }
  };
  // row sums and u of the CTA's rows
  auto row_pass = [&](const float* v) {
    for (int r = warp; r < R; r += kSW) {
      const uint32_t ka = smem_u32(Ks + (int64_t)r * ld), va = smem_u32(v);
      f2_t a[2] = {pk2(0.f, 0.f), pk2(0.f, 0.f)};
#pragma unroll 4
      for (int c = lane * V; c < (int)ld; c += 32 * V) {
        f2_t k[V2], x[V2];
        pairs(lds128a(ka + c * (uint32_t)sizeof(TK)), k, TK());
#pragma unroll
        for (int h = 0; h < V / 4; ++h) {
          const uint4 t = lds128a(va + (c + 4 * h) * 4);
          x[2 * h] = pk2u(t.x, t.y);
          x[2 * h + 1] = pk2u(t.z, t.w);
        }
#pragma unroll
        for (int h = 0; h < V2; ++h) a[h & 1] = ffma2(k[h], x[h], a[h & 1]);
      }
      const float2 p0 = upk2(a[0]), p1 = upk2(a[1]);
      float rs = (p0.x + p0.y) + (p1.x + p1.y);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
      if (lane == 0) {
        float ur = 0.f;
        if (rs > 0.f && isfinite(rs)) {
          ur = mu / rs;
          if (!isfinite(ur)) { ur = 0.f; atomicOr(status, ST_NUMERIC); }
        } else {
          atomicOr(status, ST_NUMERIC);
        }
        u_s[r] = ur;
        rs_s[r] = rs;
      }
    }
  };

  int it = 1;
  double err = -1.0;
  for (;; ++it) {
    const float* v = vbuf + (int64_t)(it & 1) * ld;
    const uint32_t par = (uint32_t)((it - 1) & 1);
    if (tid == 0) {
      mbar_expect_tx(smem_u32(&sums_bar), (uint32_t)(ld * 4));
      mbar_expect_tx(smem_u32(&v_bar), (uint32_t)(ld * 4 + kSQ * NWS * 8));
    }
    row_pass(v);
    __syncthreads();
    // ---- this CTA's partial column sums, each to the owner of its eighth
    for (int c = tid * V; c < (int)ld; c += kST * V) {
      f2_t a[V2];
#pragma unroll
      for (int h = 0; h < V2; ++h) a[h] = pk2(0.f, 0.f);
      const uint32_t ka = smem_u32(Ks + c);
#pragma unroll 4
      for (int r = 0; r < R; ++r) {
        const f2_t u2 = pk2(u_s[r], u_s[r]);
        f2_t k[V2];
        pairs(lds128a(ka + (uint32_t)(r * (int)ld * (int)sizeof(TK))), k, TK());
#pragma unroll
        for (int h = 0; h < V2; ++h) a[h] = ffma2(u2, k[h], a[h]);
      }
#pragma unroll
      for (int h = 0; h < V / 4; ++h) {
        const int cc = c + 4 * h, to = cc / S;         // an eighth is a multiple of 16 columns
        const float2 x = upk2(a[2 * h]), y = upk2(a[2 * h + 1]);
        st_async_f32x4(map_cluster(smem_u32(red + q * S + (cc - to * S)), (uint32_t)to),
                       make_float4(x.x, x.y, y.x, y.y), map_cluster(smem_u32(&sums_bar), (uint32_t)to));
      }
    }
    wait(&sums_bar, par);
    // ---- the column sums of the eighth: the cluster's, then all clusters'
    float cs = 0.f;
    if (tid < S) {
#pragma unroll
      for (int rank = 0; rank < kSQ; ++rank) cs += red[rank * S + tid];
      if (C > 1) {
        const uint32_t tag = tag0 + (uint32_t)it;
        uint2* w = words + (int64_t)(it & 1) * C * ld + jq;
        publish(w + (int64_t)cl * ld, cs, tag);
        uint2 x[kMaxSmallC];
        uint64_t t0 = 0;
        for (uint32_t spin = 0;; ++spin) {
          bool all = true;
#pragma unroll
          for (int k = 0; k < kMaxSmallC; ++k)
            if (k < C) {
              x[k] = peek(w + (int64_t)k * ld);
              all &= x[k].y == tag;
            }
          if (all || s_dead) break;
          if (spin == 0) t0 = global_ns();
          if ((spin & 63u) == 63u && global_ns() - t0 > kWaitNs) {
            atomicOr(status, ST_TIMEOUT);
            s_dead = 1;
            break;
          }
        }
        cs = 0.f;
#pragma unroll
        for (int k = 0; k < kMaxSmallC; ++k)
          if (k < C) cs += __uint_as_float(x[k].x);
      }
    }
    // ---- marginal error of the eighth and the next column scaling
    double e = 0.0;
    float v_next = 0.f;
    if (own) {
      e = fabs((double)v_own * (double)cs - (double)nu);
      if (cs > 0.f && isfinite(cs)) {
        v_next = nu / cs;
      } else {
        if (cl == 0) atomicOr(status, ST_NUMERIC);
        v_next = nu * 6.0760302e37f;   // e^87: keep finite; the status word reports it
      }
    }
    if (warp < NWS) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
      if (tid < S) {
        const uint32_t a = smem_u32(vbuf + (int64_t)((it + 1) & 1) * ld + jq);
#pragma unroll
        for (int rank = 0; rank < kSQ; ++rank)
          st_async_f32(map_cluster(a, (uint32_t)rank), v_next, map_cluster(smem_u32(&v_bar), (uint32_t)rank));
      }
      if (lane < kSQ)
        st_async_f64(map_cluster(smem_u32(&errs[q][warp]), (uint32_t)lane), e,
                     map_cluster(smem_u32(&v_bar), (uint32_t)lane));
    }
    wait(&v_bar, par);
    const bool check = tol >= 0.0 && it % check_every == 0;
    if (check || it == max_iter) {
      err = 0.0;
      for (int k = 0; k < kSQ; ++k)
        for (int w = 0; w < NWS; ++w) err += errs[k][w];
      if (it == max_iter || err <= tol) break;
      __syncthreads();     // errs is read out before the next iteration's arrive
    }
    v_own = v_next;
  }
  // ---- state (a_t, b_t) of the last iteration: log v, and log u for the v
  // that the returned logarithms stand for
  cluster_arrive();        // nothing is on its way to a CTA that leaves
  cluster_wait();
  if (it > 1) {
    float* v = vbuf + (int64_t)(it & 1) * ld;
    for (int j = tid; j < n2; j += kST) v[j] = expf(logf(v[j]));
    __syncthreads();
    row_pass(v);
    __syncthreads();
  }
  for (int r = tid; r < R; r += kST) log_u[r0 + r] = log_mu - logf(rs_s[r]);
  if (cl == 0 && own) log_v_out[jq] = it > 1 ? logf(v_own) : lv_first;
  if (blockIdx.x == 0 && tid == 0) {
    *err_out = err;
    *iters_out = it;
  }
}

void* small_fn(bool bf16) {
  return bf16 ? reinterpret_cast<void*>(&k_solve_small<__nv_bfloat16>)
              : reinterpret_cast<void*>(&k_solve_small<float>);
}

cudaLaunchConfig_t small_config(int C, size_t smem, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kSQ * C));
  cfg.blockDim = dim3(kST);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kSQ;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

}  // namespace

// Clusters of the one-launch solve, 0 where K does not fit: as many as are
// resident at once, but not more than leave each CTA a row.
int solve_small_clusters(int n1, int64_t ld, bool bf16) {
  const size_t b = bf16 ? 2 : 4;
  if (ld / kSQ > kST) return 0;
  const int most = (n1 + kSQ - 1) / kSQ;
  // a first bound without asking the device: 19 clusters of 8 on 152 SMs
  if (small_smem(small_max_rows(n1, std::min(most, 19)), ld, b) > kSmallSmem) return 0;
  void* fn = small_fn(bf16);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem) !=
      cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = small_config(1, kSmallSmem, attr, 0);
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const int C = std::min(std::min(most, n), kMaxSmallC);
  if (C < 1 || small_smem(small_max_rows(n1, C), ld, b) > kSmallSmem) return 0;
  return C;
}

fa_status launch_solve_small(int C, int n1, int n2, int64_t ld, const void* K, bool bf16,
                             const float* log_v_in, float* log_u, float* log_v_out, int max_iter,
                             double tol, int check_every, void* words, uint32_t tag0, double* err, int* iters, int* status, cudaStream_t s) {
  float mu = 1.0f / (float)n1, nu = 1.0f / (float)n2;
  float log_mu = logf(mu);
  const size_t smem = small_smem(small_max_rows(n1, C), ld, bf16 ? 2 : 4);
  void* fn = small_fn(bf16);
  FA_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem));
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = small_config(C, smem, attr, s);
  void* args[] = {(void*)&K, (void*)&ld, (void*)&n1, (void*)&n2, (void*)&log_v_in, (void*)&log_u,
                  (void*)&log_v_out, (void*)&mu, (void*)&log_mu, (void*)&nu, (void*)&max_iter, (void*)&tol, (void*)&check_every, (void*)&words, (void*)&tag0,
                  (void*)&err, (void*)&iters, (void*)&status};
  cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
  if (e != cudaSuccess) {
    set_error("k_solve_small launch (%d clusters, %zu bytes): %s", C, smem, cudaGetErrorString(e));
    cudaGetLastError();
    return FA_ERR_CUDA;
  }
  FA_LAUNCHED("k_solve_small");
  return FA_OK;
}

}  // namespace fa
