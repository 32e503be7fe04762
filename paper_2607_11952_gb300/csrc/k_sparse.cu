// Sparse x dense kernels of FastAlign (Section 3.3, "sparsity-aware"):
//   - RWR positional encoding, Algorithm 1 (SpMM with a tall-skinny dense R)
//   - SDDMM for the intra-network costs C1, C2, Algorithm 1
//   - the "SpMM on a wide dense matrix" pair  Z = P1 . D . P2^T
//     (Section 3.4; Algorithm 1 propagation, edge and neighbourhood costs), split into
//       left:  W  = P1 D   (row gathers of D, stored transposed as W^T)
//       right: Z  = W P2^T (row gathers of W^T), with a fused epilogue that
//              either stores Z (C_node propagation, Algorithm 1) or assembles
//              the cost (Algorithm 1 cost assembly, Eq. 2) and the log Gibbs kernel of the
//              proximal step.
// Storing the left product transposed turns both halves of the triple
// product into coalesced row gathers; the CTA order keeps one column panel
// of the gathered operand resident in L2 while every row tile uses it (the
// GPU form of the paper's column-blocked SpMM, Section 3.4).  The RWR, the
// left products and the propagation's right product are one kernel
// (k_spmm): a gather engine with a transposed or a row-major store.
#include <math.h>

#include "fa_internal.cuh"
#include "sweep_dev.cuh"

namespace fa {

// ------------------------------------------------------------ small helpers
__global__ void k_fill(float* p, int64_t n, float v) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (; i < n; i += stride) p[i] = v;
}

fa_status launch_fill(float* p, int64_t n, float v, cudaStream_t s) {
  if (n <= 0) return FA_OK;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  k_fill<<<(unsigned)blocks, 256, 0, s>>>(p, n, v);
  FA_LAUNCHED("k_fill");
  return FA_OK;
}

__global__ void k_exp_vec(int n, const float* __restrict__ x, float* __restrict__ y) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = expf(x[i]);
}

fa_status launch_exp_vec(int n, const float* x, float* y, cudaStream_t s) {
  if (n <= 0) return FA_OK;
  k_exp_vec<<<(n + 255) / 256, 256, 0, s>>>(n, x, y);
  FA_LAUNCHED("k_exp_vec");
  return FA_OK;
}

// ------------------------------------------------------------ edge records
// One CSR edge as the gather kernels read it: the neighbour (the gathered
// row), the output row and the weights of up to two value sets, already
// multiplied by the neighbour's scaling exp(log_scale[nb]).  Built once per
// product (16 bytes per stored entry) because every column panel of the
// product, hundreds of them, reads every edge again.
struct __align__(16) EdgeRec {
  int nb, row;
  float wa, wb;
};

__global__ void k_edge_records(int64_t nnz, const int32_t* __restrict__ ci,
                               const int32_t* __restrict__ ri, const float* __restrict__ va,
                               const float* __restrict__ vb, const float* __restrict__ log_scale,
                               EdgeRec* __restrict__ out) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nnz) return;
  const int k = ci[e];
  const float s = log_scale ? expf(log_scale[k]) : 1.f;
  out[e] = EdgeRec{k, ri[e], va[e] * s, vb ? vb[e] * s : 0.f};
}

fa_status launch_edge_records(const DevGraph& g, const float* va, const float* vb,
                              const float* log_scale, void* recs, cudaStream_t s) {
  if (g.nnz <= 0) return FA_OK;
  k_edge_records<<<(unsigned)((g.nnz + 255) / 256), 256, 0, s>>>(
      g.nnz, g.col, g.row, va, vb, log_scale, static_cast<EdgeRec*>(recs));
  FA_LAUNCHED("k_edge_records");
  return FA_OK;
}

__device__ __forceinline__ EdgeRec lds_edge(const EdgeRec* p) {
  const int4 v = *reinterpret_cast<const int4*>(p);
  return EdgeRec{v.x, v.y, __int_as_float(v.z), __int_as_float(v.w)};
}

// ------------------------------------------------------------ SpMM engine
// out = P D for NV value sets of the sparse P (n rows) and the dense D, one
// column panel of TJ = 32 V columns (V = 16 bytes of D per lane) and one
// tile of TI rows of P per CTA.  OUT_T stores the product transposed, Wt[j,
// i] (NV floats per element, TI consecutive i per column j); OUT_ROWS stores
// alpha times it row-major, plus beta where seeds[j] = i.
//
// The tile's edges are one contiguous CSR range, split evenly over the NW
// warps whatever the rows' degrees are: with one warp per row a hub row of
// 700 neighbours kept its CTA's other warps idle.  A warp walks its edges
// from the last to the first, the 512-byte gathers of kBatch of them in
// flight while the kBatch before are added.  A row ends when the next edge's
// row differs: its sum goes to the shared tile.  The last row of a warp may
// have begun in an earlier warp's range; its sum is parked in place of the
// warp's edge records and added in warp order, so every sum has a fixed
// order and there are no atomics.  A lane's columns lie 32 apart in the tile
// and its rows are RS = 1 (mod 32; 2 for tiles of 16 rows) apart: the
// stores, lanes over columns, and the transposed reads, lanes over rows, are
// free of bank conflicts.  blockIdx.x runs over row tiles first, so the panel
// of D (rows x 512 bytes) stays in L2 while every tile gathers from it;
// results are stored evict-first.
//
// What bounds it: the gathers of D's rows from L2, 512 bytes per edge and
// panel, with what the resident warps keep in flight (random 512-byte
// gathers alone, 128 KB in flight per SM: 20 TB/s).  Measured at 50,000 nodes
// of average degree 10, exponent 2.1 (GB300), before -> after this form: Pass
// A, BF16, two value sets, 25.1 -> 8.3 ms (50 GB of gathers, 25 GB of HBM);
// propagation, FP32, left 12.4 -> 7.7 ms, right 25.3 -> 7.7 ms (100 GB of
// gathers, 20 GB of HBM: 13 TB/s from L2); RWR step of 2,500 anchors 514 ->
// 421 us.  Pass A at 10,000 nodes in FP32: 599 -> 363 us.
// Tried on the same cases: batches of 4 (9.5 ms, 64 registers and fewer
// warps) and 8 (12.0 ms); single gathers replaced one by one, 4 to 8 deep
// (12 to 14 ms); gathers through a shared-memory ring by cp.async (10.3 ms,
// and 13.4 ms for the propagation: every element crosses shared memory
// twice); 16 warps (11.7 ms).  More resident warps beat deeper ones: the
// shapes below take 4 warps where the tile is small enough for 9 CTAs per SM.
enum { OUT_T = 0, OUT_ROWS = 1 };
constexpr int kBatch = 2;         // gathers per batch, two batches in turn

template <bool A16>
__device__ __forceinline__ uint4 ldg16(const char* p) {
  if constexpr (A16) {
    return __ldg(reinterpret_cast<const uint4*>(p));
  } else {                                       // 8-byte aligned operand
    const uint2 a = __ldg(reinterpret_cast<const uint2*>(p));
    const uint2 b = __ldg(reinterpret_cast<const uint2*>(p) + 1);
    return make_uint4(a.x, a.y, b.x, b.y);
  }
}

// A warp's edge records in 64 shared slots: the edge q steps before the
// range's end in slot q & 63, refilled 32 at a time as they are used up.
// Slots past the range hold its first edge, so that a gather running ahead
// of the range's end reads a valid row.
struct EdgeFeed {
  const int4* last;     // the record of the range's last edge
  int most;             // edges in the range - 1
  int4 later;           // this lane's record of the batch after next
  __device__ __forceinline__ EdgeFeed(const EdgeRec* recs, int ee, int cnt, EdgeRec* my, int lane)
      : last(reinterpret_cast<const int4*>(recs) + (ee - 1)), most(cnt - 1) {
    if (cnt > 0) {
      *reinterpret_cast<int4*>(my + lane) = at(lane);
      *reinterpret_cast<int4*>(my + 32 + lane) = at(32 + lane);
      later = at(64 + lane);
    }
  }
  __device__ __forceinline__ int4 at(int q) const { return __ldg(last - min(q, most)); }
  // edges before q are done; q a multiple of the chunk
  __device__ __forceinline__ void next(int q, EdgeRec* my, int lane) {
    if ((q & 31) == 0) {
      __syncwarp();
      *reinterpret_cast<int4*>(my + ((q + 32 + lane) & 63)) = later;
      later = at(q + 64 + lane);
      __syncwarp();
    }
  }
};

template <typename TD, int NV, int TI, int NW>
struct SpmmShape {
  static constexpr int V = 16 / (int)sizeof(TD);     // columns per lane
  static constexpr int TJ = 32 * V;                  // columns per panel
  static constexpr int F = TJ * NV;                  // floats per tile row
  static constexpr int RS = F + 32 / TI;             // tile row stride
  // per warp: 64 edge records, or a parked row
  static constexpr int kWarpBytes = F * 4 > 64 * 16 ? F * 4 : 64 * 16;
  static constexpr size_t smem = (size_t)NW * kWarpBytes + (size_t)TI * RS * sizeof(float);
};

template <typename TD, int NV, int TI, int NW, int MINB, int OUT, bool A16>
__global__ void __launch_bounds__(32 * NW, MINB) k_spmm(
    int n, int n_cols, int64_t ldd, int64_t ldo, const int32_t* __restrict__ rp,
    const EdgeRec* __restrict__ recs, const TD* __restrict__ D, float alpha, float beta,
    const int32_t* __restrict__ seeds, float* __restrict__ out) {
  using Sh = SpmmShape<TD, NV, TI, NW>;
  constexpr int V = Sh::V, TJ = Sh::TJ, F = Sh::F, RS = Sh::RS, V2 = V / 2;
  constexpr int B = kBatch;
  static_assert(32 % (2 * B) == 0, "records are staged 32 at a time");
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float* tile = reinterpret_cast<float*>(sm_raw + NW * Sh::kWarpBytes);  // [TI][RS]
  __shared__ int rps[TI + 1];
  __shared__ int head_row[NW];
  const int i0 = blockIdx.x * TI;
  const int j0 = blockIdx.y * TJ;
  const int warp = (int)threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* mine = sm_raw + warp * Sh::kWarpBytes;
  for (int t = threadIdx.x; t <= TI; t += 32 * NW) rps[t] = rp[min(i0 + t, n)];
  int cur = -1, cnt, eb;
  f2_t acc[NV][V2];
  auto clear = [&]() {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int k = 0; k < V2; ++k) acc[v][k] = pk2(0.f, 0.f);
  };
  auto store_row = [&](float* dst) {                  // column V lane + k at 32 k + lane
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int k = 0; k < V2; ++k) {
        const float2 a = upk2(acc[v][k]);
        dst[v * TJ + (2 * k) * 32 + lane] = a.x;
        dst[v * TJ + (2 * k + 1) * 32 + lane] = a.y;
      }
  };
  {
    const int E0 = rp[i0], len = rp[min(i0 + TI, n)] - E0;
    eb = E0 + (int)((int64_t)len * warp / NW);
    const int ee = E0 + (int)((int64_t)len * (warp + 1) / NW);
    cnt = ee - eb;
    // a lane past the operand's last column gathers the panel's first ones;
    // its results are never stored
    const int jl = j0 + lane * V < (int)ldd ? j0 + lane * V : j0;
    const char* dcol = reinterpret_cast<const char*>(D + jl);
    const uint32_t ldb = (uint32_t)(ldd * (int64_t)sizeof(TD));
    EdgeRec* my = reinterpret_cast<EdgeRec*>(mine);   // edge ee - 1 - q in slot q & 63
    EdgeFeed feed(recs, ee, cnt, my, lane);
    __syncwarp();
    uint4 da[B], db[B];
    auto gather = [&](uint4 (&d)[B], const EdgeRec* p) {
#pragma unroll
      for (int u = 0; u < B; ++u) d[u] = ldg16<A16>(dcol + (uint64_t)(uint32_t)p[u].nb * ldb);
    };
    auto add = [&](const uint4& d, const EdgeRec* p) {
      const EdgeRec er = lds_edge(p);
      if (er.row != cur) {
        if (cur >= 0) store_row(tile + (cur - i0) * RS);
        clear();
        cur = er.row;
      }
      f2_t x[V2];
      pairs(d, x, TD());
      const f2_t wa = pk2(er.wa, er.wa);
#pragma unroll
      for (int k = 0; k < V2; ++k) acc[0][k] = ffma2(wa, x[k], acc[0][k]);
      if constexpr (NV == 2) {
        const f2_t wb = pk2(er.wb, er.wb);
#pragma unroll
        for (int k = 0; k < V2; ++k) acc[NV - 1][k] = ffma2(wb, x[k], acc[NV - 1][k]);
      }
    };
    if (cnt > 0) {
      const EdgeRec* p = my;
      gather(da, p);
      int q = 0;
      for (; q + 2 * B <= cnt; q += 2 * B) {
        const EdgeRec* pn = my + ((q + 2 * B) & 63);
        gather(db, p + B);
#pragma unroll
        for (int u = 0; u < B; ++u) add(da[u], p + u);
        gather(da, pn);
#pragma unroll
        for (int u = 0; u < B; ++u) add(db[u], p + B + u);
        p = pn;
        feed.next(q + 2 * B, my, lane);
      }
      if (q < cnt) {                                  // the last 1 .. 2 B - 1 edges
        gather(db, p + B);
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (q + u < cnt) add(da[u], p + u);
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (q + B + u < cnt) add(db[u], p + B + u);
      }
    }
  }
  __syncthreads();                                    // rps; every warp is done with its records
  {
    const bool parked = cnt > 0 && rps[cur - i0] < eb;   // begun in an earlier warp's range
    if (cnt > 0)
      store_row(parked ? reinterpret_cast<float*>(mine) : tile + (cur - i0) * RS);
    if (lane == 0) head_row[warp] = parked ? cur - i0 : -1;
  }
  __syncthreads();
  // rows split between warps: the parked parts in warp order
  for (int f = threadIdx.x; f < F; f += 32 * NW) {
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      const int r = head_row[w];
      if (r >= 0) tile[r * RS + f] += reinterpret_cast<const float*>(sm_raw + w * Sh::kWarpBytes)[f];
    }
  }
  __syncthreads();
  if constexpr (OUT == OUT_T) {
    // 32 / TI columns per pass (side by side in the tile), lanes over rows
    constexpr int CP = 32 / TI;
    const int r = lane % TI, hi = lane / TI;
    const bool any = rps[r + 1] > rps[r];
    const float* trow = tile + r * RS;
    float* orow = out + (int64_t)(i0 + r) * NV;
#pragma unroll 4
    for (int p = warp * CP; p < TJ; p += NW * CP) {
      const int f = p + hi, j = j0 + V * (f & 31) + (f >> 5);
      if (j >= n_cols) continue;
      if constexpr (NV == 1) {
        __stcs(orow + (int64_t)j * ldo, any ? trow[f] : 0.f);
      } else {
        const float2 z = any ? make_float2(trow[f], trow[TJ + f]) : make_float2(0.f, 0.f);
        __stcs(reinterpret_cast<float2*>(orow + (int64_t)j * ldo * 2), z);
      }
    }
  } else {
    // warp per row, a lane's V columns (NV = 1, V = 4)
    static_assert(OUT == OUT_T || (NV == 1 && V == 4), "row-major store: one FP32 value set");
    const int j = j0 + 4 * lane;
    if (j < (int)ldo) {
      const int4 seed = __ldg(reinterpret_cast<const int4*>(seeds + j));
      for (int r = warp; r < TI && i0 + r < n; r += NW) {
        const int i = i0 + r;
        const float* t = tile + r * RS + lane;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rps[r + 1] > rps[r])
          o = make_float4(alpha * t[0], alpha * t[32], alpha * t[64], alpha * t[96]);
        if (seed.x == i) o.x += beta;
        if (seed.y == i) o.y += beta;
        if (seed.z == i) o.z += beta;
        if (seed.w == i) o.w += beta;
        *reinterpret_cast<float4*>(out + (int64_t)i * ldo + j) = o;
      }
    }
  }
}

template <typename TD, int NV, int TI, int NW, int MINB, int OUT, bool A16>
static fa_status run_spmm(const DevGraph& g, int n_cols, int64_t panel_cols, int64_t ldd,
                          int64_t ldo, const void* recs, const TD* D, float* out, cudaStream_t s,
                          float alpha = 1.f, float beta = 0.f, const int32_t* seeds = nullptr) {
  using Sh = SpmmShape<TD, NV, TI, NW>;
  auto* fn = &k_spmm<TD, NV, TI, NW, MINB, OUT, A16>;
  FA_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::smem));
  const dim3 grid((unsigned)((g.n + TI - 1) / TI), (unsigned)((panel_cols + Sh::TJ - 1) / Sh::TJ));
  fn<<<grid, 32 * NW, Sh::smem, s>>>(g.n, n_cols, ldd, ldo, g.row_ptr,
                                 static_cast<const EdgeRec*>(recs), D, alpha, beta, seeds,
                                     out);
  FA_LAUNCHED("k_spmm");
  return FA_OK;
}

// ------------------------------------------------------------ RWR (Algorithm 1)
// Rout[i,:] = (1-beta) sum_k Abar[i,k] Rin[k,:] + beta R^(0)[i,:], R^(0) the
// one-hot rows: column l is 1 at node seeds[l] (-1 in the padding columns).
// recs: Abar's records.
fa_status launch_rwr_step(const DevGraph& g, int64_t ldr, float beta, const void* recs,
                          const int32_t* seeds, const float* Rin, float* Rout, cudaStream_t s) {
  return run_spmm<float, 1, 32, 8, 5, OUT_ROWS, true>(g, (int)ldr, ldr, ldr, ldr, recs, Rin, Rout,
                                                      s, 1.0f - beta, beta, seeds);
}

// R^(0): 1 at R[nodes[l], l], 0 elsewhere (Algorithm 1)
__global__ void k_set_onehot(int L, int64_t ldr, const int32_t* __restrict__ nodes,
                             float* __restrict__ R) {
  int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l < L) R[(int64_t)nodes[l] * ldr + l] = 1.0f;
}

fa_status launch_onehot(int n, int L, int64_t ldr, const int32_t* nodes,
                        float* R, cudaStream_t s) {
  FA_TRY(launch_fill(R, (int64_t)n * ldr, 0.0f, s));
  if (L <= 0) return FA_OK;
  k_set_onehot<<<(L + 255) / 256, 256, 0, s>>>(L, ldr, nodes, R);
  FA_LAUNCHED("k_set_onehot");
  return FA_OK;
}

// ------------------------------------------------------------ SDDMM (Algorithm 1)
// out[e] = w[e] * <R[i,:], R[k,:]> for every stored entry e = (i, k); w is
// Abar (1/deg i) for C1 = (R1 R1^T) .* Abar1 or Abar^T (1/deg k) for
// C2 = (R2 R2^T) .* Abar2^T.  The dot product of (i, k) is that of (k, i), so
// only entries with k > i are formed and stored twice.  A warp takes
// kSddmmEdges consecutive entries (mostly of few rows, whose columns then
// come from L1) and walks the columns of four at a time, their eight loads in
// flight together: the work is spread by entry, where one warp per row left
// a hub row of 700 entries to 700 serial dot products.  Bound by the read of R's rows, about
// one per edge (R is larger than L2 at 50,000 nodes and 2,500 anchors): 4.2
// ms -> 0.44 ms per graph there, 177 -> 17 us at 10,000 nodes and 500 anchors.
constexpr int kSddmmEdges = 16;    // entries per warp, about half of them with k > i

__global__ void __launch_bounds__(256) k_sddmm(
    int64_t nnz, int64_t ldr, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
    const int32_t* __restrict__ ri, const float* __restrict__ w, const float* __restrict__ R,
    float* __restrict__ out) {
  constexpr int E = 4;              // entries whose columns are walked together
  const int64_t e = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * kSddmmEdges +
                    (threadIdx.x & 31);
  const int lane = threadIdx.x & 31;
  const bool in = lane < kSddmmEdges && e < nnz;
  const int i = in ? ri[e] : 0, k = in ? ci[e] : 0;
  uint32_t todo = __ballot_sync(0xffffffffu, k > i);
  const int nv = (int)(ldr / 4);
  float mine = 0.f;                 // lane t's own entry's dot product
  while (todo) {
    const float4* a_row[E];
    const float4* b_row[E];
    int src[E];
    float acc[E];
    int last = __ffs(todo) - 1;
#pragma unroll
    for (int t = 0; t < E; ++t) {   // a short group walks its last entry again
      if (todo) last = __ffs(todo) - 1;
      todo &= todo - 1;
      src[t] = last;
      a_row[t] = reinterpret_cast<const float4*>(R + (int64_t)__shfl_sync(0xffffffffu, i, last) * ldr);
      b_row[t] = reinterpret_cast<const float4*>(R + (int64_t)__shfl_sync(0xffffffffu, k, last) * ldr);
      acc[t] = 0.f;
    }
    for (int c = lane; c < nv; c += 32) {
      float4 a[E], b[E];
#pragma unroll
      for (int t = 0; t < E; ++t) {
        a[t] = __ldg(a_row[t] + c);
        b[t] = __ldg(b_row[t] + c);
      }
#pragma unroll
      for (int t = 0; t < E; ++t)
        acc[t] += a[t].x * b[t].x + a[t].y * b[t].y + a[t].z * b[t].z + a[t].w * b[t].w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int t = 0; t < E; ++t) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], o);
#pragma unroll
    for (int t = 0; t < E; ++t)
      if (lane == src[t]) mine = acc[t];
  }
  if (in && k > i) {
    out[e] = w[e] * mine;
    int lo = rp[k], hi = rp[k + 1];            // column i of row k: the mirrored entry
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (ci[mid] <= i) lo = mid; else hi = mid;
    }
    out[lo] = w[lo] * mine;
  }
}

// The dot products run over all ldr columns of R: the padding columns past
// the L anchors stay 0 through the RWR, so they add nothing.
fa_status launch_sddmm(const DevGraph& g, int64_t ldr, const float* R, bool weight_by_col,
                       float* out, cudaStream_t s) {
  if (g.nnz == 0) return FA_OK;
  const int64_t warps = (g.nnz + kSddmmEdges - 1) / kSddmmEdges;
  k_sddmm<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(
      g.nnz, ldr, g.row_ptr, g.col, g.row, weight_by_col ? g.val_col : g.val_row, R, out);
  FA_LAUNCHED("k_sddmm");
  return FA_OK;
}

// ------------------------------------------------------------ attributes
// Xh[i,:] = X[i,:] / |X[i,:]|_2 (or a plain copy), zero rows stay zero,
// padding columns [d, ldx) set to 0.  One warp per row.
__global__ void k_normalize_rows(int n, int d, const float* __restrict__ X,
                                 int64_t ldx, int normalize,
                                 float* __restrict__ Xh) {
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (warp >= n) return;
  const float* x = X + (int64_t)warp * d;
  float ss = 0.f;
  for (int c = lane; c < d; c += 32) ss += x[c] * x[c];
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  float scale = 1.0f;
  if (normalize) scale = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
  for (int c = lane; c < ldx; c += 32)
    Xh[(int64_t)warp * ldx + c] = c < d ? x[c] * scale : 0.f;
}

fa_status launch_normalize_rows(int n, int d, const float* X, int64_t ldx,
                                bool normalize, float* Xh, cudaStream_t s) {
  int64_t threads = (int64_t)n * 32;
  k_normalize_rows<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(
      n, d, X, ldx, normalize ? 1 : 0, Xh);
  FA_LAUNCHED("k_normalize_rows");
  return FA_OK;
}

// ------------------------------------------------------------ products P D, stored transposed
// Wt[j, i] = sum_k P[i,k] s_k D[k, j] for the two value sets of recs (Pass A:
// C1 and A1bar^T on the plan's kernel).
fa_status launch_spmm_pair_T(const DevGraph& g1, int n2, int64_t ldd, int64_t ldw,
                             const void* recs, const void* D, bool d_bf16, float* Wt,
                             cudaStream_t s) {
  if (d_bf16) {
    auto* Dp = static_cast<const __nv_bfloat16*>(D);
    if ((reinterpret_cast<uintptr_t>(D) & 15u) == 0)
      return run_spmm<__nv_bfloat16, 2, 16, 8, 4, OUT_T, true>(g1, n2, n2, ldd, ldw, recs, Dp,
                                                               Wt, s);
    return run_spmm<__nv_bfloat16, 2, 16, 8, 4, OUT_T, false>(g1, n2, n2, ldd, ldw, recs, Dp, Wt,
                                                              s);
  }
  return run_spmm<float, 2, 32, 8, 4, OUT_T, true>(g1, n2, n2, ldd, ldw, recs,
                                                   static_cast<const float*>(D), Wt, s);
}

// Wt[j, i] = sum_k P[i,k] D[k, j] for one value set and FP32 D: both halves
// of the C_node propagation A1bar C A2bar^T (Algorithm 1) -- (A1bar C)^T,
// then (A2bar (A1bar C)^T)^T.
fa_status launch_spmm_T(const DevGraph& g, int n_cols, int64_t ldd, int64_t ldw, const void* recs,
                        const float* D, float* Wt, cudaStream_t s) {
  return run_spmm<float, 1, 32, 4, 9, OUT_T, true>(g, n_cols, n_cols, ldd, ldw, recs, D, Wt,
                                                   s);
}

// ------------------------------------------------------------ right SpMM with cost
// Cost assembly + log Gibbs kernel (Phase 2 of Algorithm 1, Eq. 2, proximal step):
//   C   = C_node + lam_e Z_e - lam_n log max(Z_n, delta) + lam_a C_anc
//   x   = -C/eps + (lam_p/eps) (log u_i + log K_prev_ij + log v_j)
// stored as float32, plus the per-(row, 64-column tile) maximum of x, with
// Z[i, j] = sum_l P2[j, l] s_l W^T[l, i] for both value sets (recs: P2's
// records, W^T pairs interleaved).
template <bool VEC>
__device__ __forceinline__ float2 load_pair(const float* p) {
  if constexpr (VEC) return __ldcs(reinterpret_cast<const float2*>(p));
  return make_float2(p[0], p[1]);
}
__device__ __forceinline__ float2 load_kernel_pair(const float* p) {
  return __ldcs(reinterpret_cast<const float2*>(p));
}
__device__ __forceinline__ float2 load_kernel_pair(const __nv_bfloat16* p) {
  const uint32_t u = __ldcs(reinterpret_cast<const uint32_t*>(p));
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

// CTA tile: 64 columns j x 64 rows i.  The gathers are the engine's of
// k_spmm with the roles of rows and columns exchanged: the tile's columns'
// edges split evenly over the 8 warps, walked from the last to the first in
// two batches of gathers, a column split between warps parked and added in
// warp order (no atomics: two runs give identical bits).  A lane holds rows
// 2 lane and 2 lane + 1 as (e, n) pairs, so one paired FMA adds both value
// sets of a row with the record's weight pair.  The epilogue walks rows, a
// lane's columns 2 lane and 2 lane + 1, four rows at a time; their four
// maxima are reduced together (6 shuffles instead of 20).  The shared
// tile is column-major, columns 130 floats apart: 2-way conflicts both ways.
//
// What bounds it: 512-byte gathers of W^T from L2 (8 nnz2 n1 bytes) and the
// issue slots of the epilogue (two logarithms per element); HBM moves
// (16 + b) n1 n2 bytes.  Measured on GB300, 50,000 nodes of degree 10, BF16:
// 28.9 -> 18.7 ms (200 GB of gathers, 45 GB of HBM); 10,000 nodes FP32: 1.07
// -> 0.69 ms.  logf is 0.6 ms of it: the hardware's lg2 on a split argument
// took 18.1 ms, but it is off by up to 1.7e-7 absolutely where K is near 1
// and logf nearly exact.  Without its edges the kernel takes 0.3 ms at 10,000 nodes.
// 5 CTAs per SM with batches of 2 (48 registers): 20.8 ms; a scan of the
// row's anchors per element instead of the tile's flag: 19.8 ms.
constexpr int kRT = 64;    // rows per tile
constexpr int kCT = 64;    // columns per tile
constexpr int kZS = 2 * kRT + 2;   // floats between columns of the shared tile

template <typename TK, bool VEC>
__global__ void __launch_bounds__(256, 4) k_spmm_right_cost(
    int n1, int n2, int64_t ldw, int64_t ldo, const int32_t* __restrict__ rp,
    const EdgeRec* __restrict__ recs, const float* __restrict__ Wt, CostEpi ep) {
  constexpr int B = 4;                                // gathers per batch
  __shared__ __align__(16) float z[kCT * kZS];        // [column][row](e, n)
  __shared__ __align__(16) EdgeRec edges[8][64];      // records; then a parked column
  __shared__ int rps[kCT + 1], head_col[8], any_part[2];
  __shared__ uint32_t anc[kRT][2];                    // anchors of a row: bit per column
  __shared__ float lus[kRT];
  const int j0 = blockIdx.x * kCT, i0 = blockIdx.y * kRT;
  const int warp = (int)threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x <= kCT) rps[threadIdx.x] = rp[min(j0 + (int)threadIdx.x, n2)];
  if (threadIdx.x >= 128 && threadIdx.x < 128 + kRT) {
    // few tiles hold an anchor at all: one flag per tile, a bit per column
    const int r = threadIdx.x - 128, i = i0 + r;
    uint32_t m[2] = {0u, 0u};
    if (i < n1)
      for (int a = ep.anc_ptr[i], a1 = ep.anc_ptr[i + 1]; a < a1; ++a) {
        const int d = ep.anc_col[a] - j0;
        if (d >= 0 && d < kCT) m[d >> 5] |= 1u << (d & 31);
      }
    anc[r][0] = m[0];
    anc[r][1] = m[1];
    lus[r] = ep.log_u[min(i, n1 - 1)];
    const bool any = __any_sync(0xffffffffu, (m[0] | m[1]) != 0u);
    if ((threadIdx.x & 31) == 0) any_part[(threadIdx.x >> 5) & 1] = any;
  }
  int cur = -1, cnt, eb;
  float a0 = 0.f, b0 = 0.f, a1 = 0.f, b1 = 0.f;       // (e, n) of rows 2 lane, 2 lane + 1
  auto store_col = [&](float* dst) {
    *reinterpret_cast<float2*>(dst + 4 * lane) = make_float2(a0, b0);
    *reinterpret_cast<float2*>(dst + 4 * lane + 2) = make_float2(a1, b1);
  };
  {
    const int E0 = rp[min(j0, n2)], len = rp[min(j0 + kCT, n2)] - E0;
    eb = E0 + (int)((int64_t)len * warp / 8);
    const int ee = E0 + (int)((int64_t)len * (warp + 1) / 8);
    cnt = ee - eb;
    const char* wrow = reinterpret_cast<const char*>(Wt + (int64_t)(i0 + 2 * lane) * 2);
    const uint32_t ldb = (uint32_t)(ldw * 8);
    EdgeRec* my = edges[warp];                        // edge ee - 1 - q in slot q & 63
    EdgeFeed feed(recs, ee, cnt, my, lane);
    __syncwarp();
    uint4 da[B], db[B];
    auto gather = [&](uint4 (&d)[B], const EdgeRec* p) {
#pragma unroll
      for (int u = 0; u < B; ++u) d[u] = ldg16<true>(wrow + (uint64_t)(uint32_t)p[u].nb * ldb);
    };
    auto add = [&](const uint4& d, const EdgeRec* p) {
      const int4 er = *reinterpret_cast<const int4*>(p);
      if (er.y != cur) {
        if (cur >= 0) store_col(z + (cur - j0) * kZS);
        a0 = b0 = a1 = b1 = 0.f;
        cur = er.y;
      }
      const float wa = __int_as_float(er.z), wb = __int_as_float(er.w);
      a0 = fmaf(wa, __uint_as_float(d.x), a0);
      b0 = fmaf(wb, __uint_as_float(d.y), b0);
      a1 = fmaf(wa, __uint_as_float(d.z), a1);
      b1 = fmaf(wb, __uint_as_float(d.w), b1);
    };
    if (cnt > 0) {
      const EdgeRec* p = my;
      gather(da, p);
      int q = 0;
      for (; q + 2 * B <= cnt; q += 2 * B) {
        const EdgeRec* pn = my + ((q + 2 * B) & 63);
        gather(db, p + B);
#pragma unroll
        for (int u = 0; u < B; ++u) add(da[u], p + u);
        gather(da, pn);
#pragma unroll
        for (int u = 0; u < B; ++u) add(db[u], p + B + u);
        p = pn;
        feed.next(q + 2 * B, my, lane);
      }
      if (q < cnt) {
        gather(db, p + B);
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (q + u < cnt) add(da[u], p + u);
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (q + B + u < cnt) add(db[u], p + B + u);
      }
    }
  }
  __syncthreads();
  {
    const bool parked = cnt > 0 && rps[cur - j0] < eb;   // begun in an earlier warp's range
    if (cnt > 0)
      store_col(parked ? reinterpret_cast<float*>(edges[warp]) : z + (cur - j0) * kZS);
    if (lane == 0) head_col[warp] = parked ? cur - j0 : -1;
  }
  __syncthreads();
  if (threadIdx.x < 2 * kRT) {
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      const int c = head_col[w];
      if (c >= 0) z[c * kZS + threadIdx.x] += reinterpret_cast<const float*>(edges[w])[threadIdx.x];
    }
  }
  __syncthreads();

  // ---- epilogue: 8 rows per warp, four at a time
  const float inv_eps = 1.0f / ep.eps;
  const float prox = ep.lam_p * inv_eps;
  const float c_off = -logf(ep.eps_anc);          // C_anc off the anchors
  const float c_on = -logf(ep.eps_anc + 1.0f);    // C_anc on an anchor
  const TK* Kp = static_cast<const TK*>(ep.K_prev);
  const int c = 2 * lane, j = j0 + c;
  const bool in0 = j < n2, in1 = j + 1 < n2;
  const bool any0 = in0 && rps[c + 1] > rps[c], any1 = in1 && rps[c + 2] > rps[c + 1];
  const float lv0 = in0 ? ep.log_v[j] : 0.f, lv1 = in1 ? ep.log_v[j + 1] : 0.f;
  const float* z0 = z + c * kZS;
  const bool any_anchor = any_part[0] | any_part[1];
  // 32-bit offsets within the tile
  const int64_t tile0 = (int64_t)i0 * ldo + j;
  const float* Ct = ep.C_node + tile0;
  const TK* Kt = Kp + tile0;
  float* Xt = ep.X + tile0;
  const uint32_t ldo32 = (uint32_t)ldo;
  const int rlast = n1 - 1 - i0;                   // the last row, within the tile
#pragma unroll 1
  for (int r0 = warp * 8; r0 < warp * 8 + 8; r0 += 4) {
    float mx[4];
    float2 cn[4], kp[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {                  // rows past n1 read the last row again
      const uint32_t at = (uint32_t)min(r0 + t, rlast) * ldo32;
      cn[t] = load_pair<VEC>(Ct + at);
      kp[t] = prox != 0.f ? load_kernel_pair(Kt + at) : make_float2(1.f, 1.f);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int r = r0 + t;
      mx[t] = -INFINITY;
      if (r <= rlast) {                            // warp-uniform
        const float2 za = any0 ? *reinterpret_cast<const float2*>(z0 + 2 * r) : make_float2(0.f, 0.f);
        const float2 zb = any1 ? *reinterpret_cast<const float2*>(z0 + kZS + 2 * r) : make_float2(0.f, 0.f);
        const float lu = lus[r];
        float can0 = c_off, can1 = c_off;
        if (any_anchor) {
          const uint32_t m = anc[r][c >> 5] >> (c & 31);
          if (m & 1u) can0 = c_on;
          if (m & 2u) can1 = c_on;
        }
        const float n0 = fmaxf(za.y, ep.delta), n1v = fmaxf(zb.y, ep.delta);
        const float ln0 = logf(n0), ln1 = logf(n1v), lk0 = logf(kp[t].x), lk1 = logf(kp[t].y);
        const float C0 = cn[t].x + ep.lam_e * za.x - ep.lam_n * ln0 + ep.lam_a * can0;
        const float C1 = cn[t].y + ep.lam_e * zb.x - ep.lam_n * ln1 + ep.lam_a * can1;
        float x0 = -C0 * inv_eps, x1 = -C1 * inv_eps;
        if (prox != 0.f) {
          x0 += prox * (lu + lk0 + lv0);
          x1 += prox * (lu + lk1 + lv1);
        }
        if (!in0) x0 = -INFINITY;                  // padding columns
        if (!in1) x1 = -INFINITY;
        __stcs(reinterpret_cast<float2*>(Xt + (uint32_t)r * ldo32), make_float2(x0, x1));
        mx[t] = fmaxf(x0, x1);
      }
    }
    // four rows' maxima: lanes 0-7 end with row r0's, 8-15 r0 + 1's, ...
    {
      const bool hi = lane & 16;
      const float h0 = hi ? mx[2] : mx[0], h1 = hi ? mx[3] : mx[1];
      const float s0 = hi ? mx[0] : mx[2], s1 = hi ? mx[1] : mx[3];
      const float g0 = fmaxf(h0, __shfl_xor_sync(0xffffffffu, s0, 16));
      const float g1 = fmaxf(h1, __shfl_xor_sync(0xffffffffu, s1, 16));
      const bool lo = lane & 8;
      float m = fmaxf(lo ? g1 : g0, __shfl_xor_sync(0xffffffffu, lo ? g0 : g1, 8));
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      const int i = i0 + r0 + (lane >> 3);
      if ((lane & 7) == 0 && i < n1) ep.rowmax_part[(int64_t)blockIdx.x * n1 + i] = m;
    }
  }
}

fa_status launch_spmm_right_cost(const DevGraph& g2, int n1, int64_t ldw, int64_t ldo,
                                 const void* recs, const float* Wt, const CostEpi& ep,
                                 bool k_bf16, cudaStream_t s) {
  dim3 grid((unsigned)(ldo / kCT), (unsigned)((n1 + kRT - 1) / kRT));
  const EdgeRec* rec = static_cast<const EdgeRec*>(recs);
  const bool vec = (reinterpret_cast<uintptr_t>(ep.C_node) & 7u) == 0;
#define FA_PB(T, VEC) \
  k_spmm_right_cost<T, VEC><<<grid, 256, 0, s>>>(n1, g2.n, ldw, ldo, g2.row_ptr, rec, Wt, ep)
  if (k_bf16) {
    if (vec) FA_PB(__nv_bfloat16, true); else FA_PB(__nv_bfloat16, false);
  } else {
    if (vec) FA_PB(float, true); else FA_PB(float, false);
  }
#undef FA_PB
  FA_LAUNCHED("k_spmm_right_cost");
  return FA_OK;
}

// rowmax[i] = max over column tiles of the partial maxima.  An all -inf row
// (every entry underflowed) is reported and pinned to 0.
__global__ void k_rowmax_reduce(int n1, int ntiles, const float* __restrict__ part,
                                float* __restrict__ rowmax, int* status) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n1) return;
  float m = -INFINITY;
  for (int t = 0; t < ntiles; ++t) m = fmaxf(m, part[(int64_t)t * n1 + i]);
  if (!(m > -INFINITY) || isnan(m)) {
    atomicOr(status, ST_NUMERIC);
    m = 0.f;
  }
  rowmax[i] = m;
}

fa_status launch_rowmax_reduce(int n1, int ntiles, const float* part,
                               float* rowmax, int* status, cudaStream_t s) {
  k_rowmax_reduce<<<(n1 + 255) / 256, 256, 0, s>>>(n1, ntiles, part, rowmax, status);
  FA_LAUNCHED("k_rowmax_reduce");
  return FA_OK;
}

}  // namespace fa
