// A whole Sinkhorn solve (Algorithm 1, Phase 3; Eq. 3) in one launch, for
// kernels K that fit in the SMs' shared memory together (up to about 2,600
// square in FP32, 3,600 in BF16).
//
// At these sizes an iteration is a few microseconds of latency, not of
// bandwidth: as two launches (sweep, column finalisation) it took 15 us at
// 1,000 x 1,000, 11 us of them in the kernels' own ramps and in the launches,
// and a tolerance test was a host round trip.  Here each CTA, alone on its SM,
// keeps its rows of K in shared memory for the whole solve, and the CTAs
// exchange two kinds of words through L2 per iteration:
//
//   rows      u_i = mu_i / sum_j K_ij v_j, one warp per row
//   sums      the CTA's partial column sums sum_i K_ij u_i, published for
//             every column; CTA b owns a range of columns, polls all CTAs'
//             partial sums of them and adds them in CTA order
//   columns   the owner publishes the column sum; every CTA polls all of
//             them and forms the next v itself -- all CTAs the same values
//   errors    at a tolerance test the owners' parts of the marginal error
//             travel the same way
//
// A word is one 64-bit scalar, the value in its lower half and the
// iteration's tag in its upper half, written and read by relaxed accesses of
// GPU scope (two words in one vector store count as two scalar stores): a
// scalar access is single-copy atomic, so a word that carries the tag carries
// the value, and no fence or counter is needed.  Words are
// double-buffered by the iteration's parity: a CTA publishes iteration t + 2
// only after it has every column sum of t + 1, which the owners form after
// they have read all words of t.  Nothing but these words crosses a CTA.
//
// v is carried as nu / column sum, not through its logarithm: the rounding of
// a stored logarithm (5e-7 at |log v| = 10) and the biases of expf and logf
// moved u and v apart by 1e-5 in 50 iterations.  log v and log u are formed
// once, from the last iteration: log u for v = exp(log v) as it is returned.
// The tolerance is tested on the device: every CTA sees the same error and
// leaves in the same iteration.
//
// The launch is cooperative (all CTAs resident).  Every wait is bounded; a
// CTA whose wait gave up sets ST_TIMEOUT, publishes nothing more and leaves
// at the next block barrier, and its peers' waits run out in turn.  There are
// no asynchronous copies, remote shared-memory accesses or barriers across
// CTAs that could outlive a CTA.
//
// Measured (GB300), us per iteration: 300 x 300 FP32 3.9, 1,000 x 1,000 4.8,
// 2,000 x 1,500 5.9, 2,600 x 2,600 8.1, 3,000 x 3,000 BF16 8.1 (two launches
// per iteration: 12.1 at 2,000 x 1,500, 14.9 at 2,600, 17.6 at 3,000 BF16); a
// solve of 1,000 x 1,000 and 50 iterations 281 us.  Bound by two trips to L2
// per iteration: without its arithmetic 1,000 x 1,000 still took 4.4.  Clusters
// of CTAs that exchanged through distributed shared memory (one trip) took 4.0
// there, but a CTA that gave up left barriers undefined and stores on their
// way to it.  Tried: polling only the words that have not come (no gain); each
// lane storing its own columns instead of exchanging them for consecutive ones
// (8.3 -> 8.8 at 2,600, 7.9 -> 10.0 at 3,000 BF16).
#include <math.h>

#include <algorithm>

#include "fa_internal.cuh"
#include "sweep_dev.cuh"

namespace fa {

namespace {

constexpr int kST = 512;          // threads per CTA
constexpr int kSW = kST / 32;
constexpr size_t kSmallSmem = 220 * 1024;
constexpr int64_t kSmallMaxLd = 8 * kST;   // most columns: eight polled words per thread
constexpr int kPoll = 8;                   // words in flight per thread

__host__ __device__ constexpr int small_max_rows(int n1, int G) { return (n1 + G - 1) / G; }
// K rows | v[2][ld] | part[kST] | u, row sums [R]
static size_t small_smem(int R, int64_t ld, size_t b) {
  return (size_t)R * ld * b + 2 * (size_t)ld * 4 + kST * 4 + 2 * (size_t)((R + 3) / 4 * 4) * 4;
}

// a value and the tag of its iteration, one 64-bit word
__device__ __forceinline__ uint64_t word(uint32_t bits, uint32_t tag) {
  return (uint64_t)tag << 32 | bits;
}
__device__ __forceinline__ void publish(uint64_t* p, uint64_t w) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ uint64_t peek(const uint64_t* p) {
  uint64_t w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}

// What ends a wait: its limit, or another thread of the CTA that gave up.
struct Waits {
  volatile int* dead;
  int* status;
  uint64_t limit_ns;
};
// x[k] = the value of p[k stride], k < cnt, once all of them carry the tag
__device__ __forceinline__ void poll(const uint64_t* p, int64_t stride, int cnt, uint32_t tag,
                                     uint32_t (&x)[kPoll], const Waits& w) {
  uint64_t t0 = 0;
  for (uint32_t spin = 0; spin < (1u << 24); ++spin) {
    bool all = true;
#pragma unroll
    for (int k = 0; k < kPoll; ++k)
      if (k < cnt) {
        const uint64_t t = peek(p + k * stride);
        x[k] = (uint32_t)t;
        all &= (uint32_t)(t >> 32) == tag;
      }
    if (all) return;
    if (spin == 0) t0 = global_ns();
    if ((spin & 15u) == 15u && (*w.dead || global_ns() - t0 > w.limit_ns)) break;
  }
  atomicOr(w.status, ST_TIMEOUT);
  *w.dead = 1;
}

template <typename TK>
__global__ void __launch_bounds__(kST, 1) k_solve_small(
    const TK* __restrict__ K, int64_t ld, int n1, int n2, const float* log_v_in, float* log_u,
    float* log_v_out, float mu, float log_mu, float nu, int max_iter, double tol, int check_every,
    uint64_t* words, uint32_t tag0, double* err_out, int* iters_out, int* status,
    uint64_t limit_ns, int silent) {
  constexpr int V = KT<TK>::V, V2 = V / 2;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double errs[kSW], s_err;
  __shared__ int s_dead;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x, G = gridDim.x;
  const int r0 = (int)((int64_t)n1 * b / G);
  const int R = (int)((int64_t)n1 * (b + 1) / G) - r0;
  const int Rmax = small_max_rows(n1, G);
  TK* Ks = reinterpret_cast<TK*>(smem);
  float* vbuf = reinterpret_cast<float*>(smem + (size_t)Rmax * ld * sizeof(TK));   // [2][ld]
  float* part = vbuf + 2 * ld;
  float* u_s = part + kST;
  float* rs_s = u_s + (Rmax + 3) / 4 * 4;
  // words: partial sums [2][G][ld] | column sums [2][ld] | errors [2][2][G]
  uint64_t* col_words = words + 2 * (int64_t)G * ld;
  uint64_t* err_words = col_words + 2 * ld;
  // this CTA's columns [c0, c0 + nc), walked kST at a time: w columns side by
  // side, the partial sums of each over ng groups of threads
  const int S = (n2 + G - 1) / G, c0 = b * S, nc = max(0, min(S, n2 - c0));
  const int w = min(S, kST), ng = kST / w, grp = tid / w, cg = tid - grp * w;
  const int shift = w <= kST / 8 ? 3 : 0, c = tid >> shift, sub = tid & ((1 << shift) - 1);
  const int own_warps = (min(w << shift, kST) + 31) / 32;   // warps that hold column sums

  if (tid == 0) s_dead = 0;
  {
    const uint4* src = reinterpret_cast<const uint4*>(K + (int64_t)r0 * ld);
    uint4* dst = reinterpret_cast<uint4*>(Ks);
    const int n = (int)(R * ld / V);
#pragma unroll 8
    for (int i = tid; i < n; i += kST) dst[i] = __ldg(src + i);
  }
  for (int j = tid; j < ld; j += kST) {
    vbuf[j] = 0.f;
    vbuf[ld + j] = j < n2 ? expf(log_v_in[j]) : 0.f;
  }
  __syncthreads();
  const Waits waits{&s_dead, status, limit_ns};

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
    const int par = it & 1;
    float* v = vbuf + (int64_t)par * ld;
    float* v_next = vbuf + (int64_t)(par ^ 1) * ld;
    const uint32_t tag = tag0 + (uint32_t)it;
    const bool test = it == max_iter || (tol >= 0.0 && it % check_every == 0);
    row_pass(v);
    __syncthreads();
    // ---- this CTA's partial column sums
    uint64_t* sums = words + (int64_t)par * G * ld;
    for (int cw = warp * 32 * V; cw < n2; cw += kST * V) {   // a warp's 32 V columns
      f2_t a[V2];
#pragma unroll
      for (int h = 0; h < V2; ++h) a[h] = pk2(0.f, 0.f);
      const uint32_t ka = smem_u32(Ks + min(cw + lane * V, (int)ld - V));
#pragma unroll 4
      for (int r = 0; r < R; ++r) {
        const f2_t u2 = pk2(u_s[r], u_s[r]);
        f2_t k[V2];
        pairs(lds128a(ka + (uint32_t)(r * (int)ld * (int)sizeof(TK))), k, TK());
#pragma unroll
        for (int h = 0; h < V2; ++h) a[h] = ffma2(u2, k[h], a[h]);
      }
      if (b == silent) continue;       // failure-detection self-test
      // store h covers 64 consecutive columns, two per lane: pair lane % V2 of
      // the lane that holds them (padding columns have words too)
#pragma unroll
      for (int h = 0; h < V2; ++h) {
        f2_t got = 0;
#pragma unroll
        for (int q = 0; q < V2; ++q) {
          const f2_t t = __shfl_sync(0xffffffffu, a[q], (64 * h + 2 * lane) / V);
          if (lane % V2 == q) got = t;
        }
        const int col = cw + 64 * h + 2 * lane;
        const float2 f = upk2(got);
        if (col < (int)ld)
          asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(sums + (int64_t)b * ld + col),
                       "l"(word(__float_as_uint(f.x), tag)), "l"(word(__float_as_uint(f.y), tag))
                       : "memory");
      }
    }
    // ---- the sums of this CTA's columns over all CTAs
    double e = 0.0;
    for (int base = 0; base < nc; base += w) {
      float s = 0.f;
      if (grp < ng && base + cg < nc) {
        const uint64_t* p = sums + c0 + base + cg;
        for (int g = grp; g < G; g += kPoll * ng) {
          uint32_t x[kPoll];
          const int cnt = min(kPoll, (G - g + ng - 1) / ng);
          poll(p + (int64_t)g * ld, (int64_t)ng * ld, cnt, tag, x, waits);
#pragma unroll
          for (int k = 0; k < kPoll; ++k)
            if (k < cnt) s += __uint_as_float(x[k]);
        }
      }
      if (grp < ng) part[cg * ng + grp] = s;
      __syncthreads();
      // eight lanes per column (one where w > 64) add its ng partial sums
      float cs = 0.f;
      if (c < w)
        for (int k = sub; k < ng; k += 1 << shift) cs += part[c * ng + k];
      if (shift) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) cs += __shfl_xor_sync(0xffffffffu, cs, o);
      }
      if (sub == 0 && c < w && base + c < nc && s_dead == 0) {
        const int j = c0 + base + c;
        publish(col_words + par * ld + j, word(__float_as_uint(cs), tag));
        if (test) e += fabs((double)v[j] * (double)cs - (double)nu);
      }
      if (base + w < nc) __syncthreads();              // part is written again
    }
    if (test) {                        // this CTA's part of the error, as two words
      if (warp < own_warps) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if (lane == 0) errs[warp] = e;
      }
      __syncthreads();
      if (tid < 2 && s_dead == 0) {
        double t = 0.0;
        for (int k = 0; k < own_warps; ++k) t += errs[k];
        const uint64_t u = (uint64_t)__double_as_longlong(t);
        publish(err_words + (int64_t)(2 * par + tid) * G + b, word((uint32_t)(tid ? u >> 32 : u), tag));
      }
    }
    // ---- all column sums: the next column scaling
    {
      uint32_t x[kPoll];
      const int cnt = (n2 - tid + kST - 1) / kST;      // at most kPoll; <= 0 past the columns
      if (tid < n2) poll(col_words + par * ld + tid, kST, cnt, tag, x, waits);
#pragma unroll
      for (int k = 0; k < kPoll; ++k)
        if (tid + k * kST < n2) {
          const float cs = __uint_as_float(x[k]);
          float t = nu * 6.0760302e37f;      // e^87: keep finite; the status word reports it
          if (cs > 0.f && isfinite(cs)) t = nu / cs;
          else if (b == 0) atomicOr(status, ST_NUMERIC);
          v_next[tid + k * kST] = t;
        }
    }
    if (test && warp == 0) {           // all CTAs' parts of the error, in a fixed order
      double t = 0.0;
      for (int g = lane; g < G; g += 32) {
        uint32_t x[kPoll];
        poll(err_words + (int64_t)2 * par * G + g, G, 2, tag, x, waits);
        t += __longlong_as_double((long long)((uint64_t)x[1] << 32 | x[0]));
      }
      __syncwarp();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) s_err = t;
    }
    __syncthreads();
    if (s_dead != 0) return;           // the same in every thread: set before the barrier only
    if (test) {
      err = s_err;
      if (it == max_iter || err <= tol) break;
    }
  }
  // ---- state (a_t, b_t) of the last iteration: log v, and log u for the v
  // that the returned logarithms stand for
  float* v = vbuf + (int64_t)(it & 1) * ld;
  for (int j = tid; j < n2; j += kST) {
    const bool own = j >= c0 && j < c0 + nc;
    if (it > 1) {
      const float l = logf(v[j]);
      if (own) log_v_out[j] = l;
      v[j] = expf(l);
    } else if (own) {
      log_v_out[j] = log_v_in[j];
    }
  }
  __syncthreads();
  if (it > 1) {
    row_pass(v);
    __syncthreads();
  }
  for (int r = tid; r < R; r += kST) log_u[r0 + r] = log_mu - logf(rs_s[r]);
  if (b == 0 && tid == 0) {
    *err_out = err;
    *iters_out = it;
  }
}

void* small_fn(bool bf16) {
  return bf16 ? reinterpret_cast<void*>(&k_solve_small<__nv_bfloat16>)
              : reinterpret_cast<void*>(&k_solve_small<float>);
}

}  // namespace

// CTAs of the one-launch solve, 0 where K does not fit: one per pair of SMs
// where K fits these, else one per SM, but not more than leave each CTA a row.
// The two SMs of a pair share their way to L2, and an iteration is two trips
// there: 300 x 300 FP32 6.1 -> 3.9 us per iteration with half the CTAs, 1,000
// 6.2 -> 4.95, 2,000 x 1,500 7.3 -> 6.3 (three quarters of the CTAs: no gain).
int solve_small_ctas(int n1, int64_t ld, bool bf16) {
  if (ld > kSmallMaxLd) return 0;
  int dev = 0, sms = 0, coop = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const size_t b = bf16 ? 2 : 4;
  int G = std::min(n1, std::max(1, sms / 2));
  if (small_smem(small_max_rows(n1, G), ld, b) > kSmallSmem) G = std::min(n1, sms);
  if (!coop || G < 1 || small_smem(small_max_rows(n1, G), ld, b) > kSmallSmem) return 0;
  void* fn = small_fn(bf16);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kST, kSmallSmem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n >= 1 ? G : 0;
}

size_t solve_small_words(int G, int64_t ld) {
  return G > 0 ? (size_t)(2 * (int64_t)G * ld + 2 * ld + 4 * (int64_t)G) * 8 : 0;
}

fa_status launch_solve_small(int G, int n1, int n2, int64_t ld, const void* K, bool bf16,
                             const float* log_v_in, float* log_u, float* log_v_out, int max_iter,
                             double tol, int check_every, void* words, uint32_t tag0, double* err,
                             int* iters, int* status, cudaStream_t s, uint64_t limit_ns,
                             int silent) {
  float mu = 1.0f / (float)n1, nu = 1.0f / (float)n2;
  float log_mu = logf(mu);
  const size_t smem = small_smem(small_max_rows(n1, G), ld, bf16 ? 2 : 4);
  void* fn = small_fn(bf16);
  FA_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem));
  if (limit_ns == 0) limit_ns = kWaitNs;
  void* args[] = {(void*)&K, (void*)&ld, (void*)&n1, (void*)&n2, (void*)&log_v_in, (void*)&log_u,
                  (void*)&log_v_out, (void*)&mu, (void*)&log_mu, (void*)&nu, (void*)&max_iter,
                  (void*)&tol, (void*)&check_every, (void*)&words, (void*)&tag0, (void*)&err,
                  (void*)&iters, (void*)&status, (void*)&limit_ns, (void*)&silent};
  // self-test -2: more CTAs than any device holds, which the runtime refuses
  const int ask = silent == -2 ? 1 << 20 : G;
  cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)ask), dim3(kST), args, smem, s);
  if (e != cudaSuccess) {
    set_error("k_solve_small launch (%d CTAs, %zu bytes): %s", ask, smem, cudaGetErrorString(e));
    cudaGetLastError();
    // refused, not failed: the caller has another way
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources ||
                   e == cudaErrorNotSupported
               ? FA_ERR_UNSUPPORTED
               : FA_ERR_CUDA;
  }
  FA_LAUNCHED("k_solve_small");
  return FA_OK;
}

}  // namespace fa
