// ShortestPath graph embedding (Sec. 2.3, Eq. 8): for d target nodes,
//   X[i][t] = dist(v_i, target_t)  if that distance is <= l0,
//             l0 + 1               otherwise (or if no path exists),
// with l0 = sqrt(|E|) by default (distances are integers, so floor).
//
// All d breadth-first searches run together, level-synchronously: every node
// keeps two d-bit masks (targets that have reached it, and targets that
// reached it in the previous level).  Level L pulls, for each node, the OR of
// its neighbours' previous-level masks, keeps the bits it has not seen, and
// writes L for them.  One level is one pass over the adjacency (d/32 words
// per neighbour); nodes that every target has reached skip the pass.  The
// search ends at the first level that reaches no new (node, target) pair or at
// l0: a level whose predecessor reached none returns at once, and the host
// reads the levels' marks kSpBatch levels at a time (a read costs a level's time).
// The result is exact integer work, independent of scheduling.
#include <cmath>

#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

constexpr int kSpBatch = 4;  // levels between two looks of the host
constexpr int kSpMarks = 8;  // a ring of marks: level L found something; at least kSpBatch + 2
constexpr int kSpOwn = 32;   // longest row that one thread walks

__global__ void k_sp_init(int n, int words, uint32_t* __restrict__ frontier, uint32_t* __restrict__ seen,
                          uint32_t* __restrict__ marks) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  if (blockIdx.x == 0 && threadIdx.x < kSpMarks) marks[threadIdx.x] = threadIdx.x == 0 ? 1u : 0u;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < (int64_t)n * words; k += stride) {
    frontier[k] = 0u;
    seen[k] = 0u;
  }
}

// targets may repeat; each sets its own bit
__global__ void k_sp_seed(int d, int words, const int32_t* __restrict__ targets, uint32_t* __restrict__ frontier,
                          uint32_t* __restrict__ seen, float* __restrict__ X) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < d; t += gridDim.x * blockDim.x) {
    const int64_t v = targets[t];
    atomicOr(&frontier[v * words + (t >> 5)], 1u << (t & 31));
    atomicOr(&seen[v * words + (t >> 5)], 1u << (t & 31));
    X[v * d + t] = 0.f;
  }
}

template <int WORDS>
__device__ __forceinline__ void load_mask(const uint32_t* __restrict__ p, uint32_t (&m)[WORDS]) {
  if constexpr (WORDS % 4 == 0) {
#pragma unroll
    for (int w = 0; w < WORDS; w += 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(p + w);
      m[w] = q.x;
      m[w + 1] = q.y;
      m[w + 2] = q.z;
      m[w + 3] = q.w;
    }
  } else if constexpr (WORDS == 2) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    m[0] = q.x;
    m[1] = q.y;
  } else {
    m[0] = p[0];
  }
}

// X[v][t] = value for the bits t of node v's mask, node after node by the whole
// warp, so that a row is written 128 bytes at a time.  m: the lane's mask, none
// if the lane has no node.
template <int WORDS>
__device__ __forceinline__ void put_bits(const uint32_t (&m)[WORDS], int64_t v0, int d, float value,
                                         float* __restrict__ X) {
  const int lane = threadIdx.x & 31;
  uint32_t any = 0u;
#pragma unroll
  for (int w = 0; w < WORDS; ++w) any |= m[w];
  for (uint32_t todo = __ballot_sync(0xffffffffu, any != 0u); todo; todo &= todo - 1u) {
    const int src = __ffs((int)todo) - 1;
    float* const row = X + (v0 + src) * d + lane;
#pragma unroll
    for (int w = 0; w < WORDS; ++w)
      if ((__shfl_sync(0xffffffffu, m[w], src) >> lane) & 1u) row[32 * w] = value;
  }
}

// One level, a thread per node; rows longer than kSpOwn by the whole warp (one
// thread on a hub's row would be the level's time: R-MAT of 262,144 nodes, rows
// of up to 9,581 entries, 128 targets: 5.4 ms a call, 1.8 ms so; 128 instead of
// 32 entries is the same).  The rest is the stores of X and the gather of the
// neighbours' masks: 300,000 nodes of at most 23 neighbours, 128 targets, a
// level takes 26 us of 12 levels' average, 55 us with one store per new bit.
template <int WORDS>
__global__ void __launch_bounds__(256)
    k_sp_level(int n, int d, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
               const uint32_t* __restrict__ cur, uint32_t* __restrict__ next, uint32_t* __restrict__ seen,
               const uint32_t* __restrict__ full, int level, float* __restrict__ X, uint32_t* marks) {
  if (blockIdx.x == 0 && threadIdx.x == 0) marks[(level + 1) % kSpMarks] = 0u;
  if (__ldcg(marks + (level - 1) % kSpMarks) == 0u) return;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool found = false;
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); v0 < n; v0 += stride) {
    const int64_t v = v0 + lane;
    uint32_t s[WORDS], acc[WORDS];
    bool done = true;
#pragma unroll
    for (int w = 0; w < WORDS; ++w) s[w] = acc[w] = 0u;
    if (v < n) {
      load_mask<WORDS>(seen + v * WORDS, s);
#pragma unroll
      for (int w = 0; w < WORDS; ++w) done &= (s[w] == full[w]);
    }
    const int64_t a = done ? 0 : rp[v], b = done ? 0 : rp[v + 1];
    const bool hub = b - a > kSpOwn;
    if (!hub)
      for (int64_t e = a; e < b; ++e) {
        uint32_t q[WORDS];
        load_mask<WORDS>(cur + (int64_t)col[e] * WORDS, q);
#pragma unroll
        for (int w = 0; w < WORDS; ++w) acc[w] |= q[w];
      }
    for (uint32_t todo = __ballot_sync(0xffffffffu, hub); todo; todo &= todo - 1u) {
      const int src = __ffs((int)todo) - 1;
      const int64_t ha = __shfl_sync(0xffffffffu, a, src), hb = __shfl_sync(0xffffffffu, b, src);
      uint32_t sum[WORDS];
#pragma unroll
      for (int w = 0; w < WORDS; ++w) sum[w] = 0u;
#pragma unroll 4
      for (int64_t e = ha + lane; e < hb; e += 32) {
        uint32_t q[WORDS];
        load_mask<WORDS>(cur + (int64_t)col[e] * WORDS, q);
#pragma unroll
        for (int w = 0; w < WORDS; ++w) sum[w] |= q[w];
      }
#pragma unroll
      for (int w = 0; w < WORDS; ++w) {
        const uint32_t all = __reduce_or_sync(0xffffffffu, sum[w]);
        if (lane == src) acc[w] = all;
      }
    }
#pragma unroll
    for (int w = 0; w < WORDS; ++w) {
      acc[w] &= ~s[w];  // what is new (a node that is done gathered nothing)
      if (acc[w]) {
        found = true;
        seen[v * WORDS + w] = s[w] | acc[w];
      }
      if (v < n) next[v * WORDS + w] = acc[w];
    }
    put_bits<WORDS>(acc, v0, d, (float)level, X);
  }
  if (__any_sync(0xffffffffu, found) && lane == 0 && __ldcg(marks + level % kSpMarks) == 0u)
    atomicOr(marks + level % kSpMarks, 1u);
}

// The pairs that no level reached.
template <int WORDS>
__global__ void __launch_bounds__(256) k_sp_far(int n, int d, const uint32_t* __restrict__ seen,
                                                const uint32_t* __restrict__ full, float far, float* __restrict__ X) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); v0 < n; v0 += stride) {
    const int64_t v = v0 + (threadIdx.x & 31);
    uint32_t m[WORDS];
#pragma unroll
    for (int w = 0; w < WORDS; ++w) m[w] = 0u;
    if (v < n) {
      load_mask<WORDS>(seen + v * WORDS, m);
#pragma unroll
      for (int w = 0; w < WORDS; ++w) m[w] = full[w] & ~m[w];
    }
    put_bits<WORDS>(m, v0, d, far, X);
  }
}

template <int WORDS>
tsgne_status run_levels(int n, int d, const int64_t* rp, const int32_t* col, uint32_t* f0, uint32_t* f1,
                        uint32_t* seen, const uint32_t* full, int l0, float* X, uint32_t* marks, int grid,
                        cudaStream_t s) {
  uint32_t* cur = f0;
  uint32_t* nxt = f1;
  for (int L = 1, more = 1; more && L <= l0;) {
    int last = L;
    for (int k = 0; k < kSpBatch && L <= l0; ++k, last = L++) {
      k_sp_level<WORDS><<<grid, 256, 0, s>>>(n, d, rp, col, cur, nxt, seen, full, L, X, marks);
      TS_CUDA(cudaGetLastError());
      uint32_t* t = cur;
      cur = nxt;
      nxt = t;
    }
    if (L > l0) break;
    uint32_t h = 0;
    TS_CUDA(cudaMemcpyAsync(&h, marks + last % kSpMarks, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    TS_CUDA(cudaStreamSynchronize(s));
    more = h != 0u;
  }
  k_sp_far<WORDS><<<grid, 256, 0, s>>>(n, d, seen, full, (float)(l0 + 1), X);
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

}  // namespace

tsgne_status shortest_path_embedding(int n, const int64_t* rp, const int32_t* col, int64_t nnz,
                                     const int32_t* targets, int d, int l0, float* X, cudaStream_t s) {
  if (l0 <= 0) l0 = (int)std::floor(std::sqrt((double)(nnz / 2)));
  if (l0 < 0) l0 = 0;
  const int words = (d + 31) / 32;
  int W = 1;
  while (W < words) W <<= 1;
  if (W > 32) {
    last_msg() = "ShortestPath embedding supports at most 1024 targets";
    return TSGNE_ERR_INVALID_ARG;
  }
  int dev = 0, sms = 1;
  TS_CUDA(cudaGetDevice(&dev));
  TS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DevBuf<uint32_t> f0, f1, seen, full, marks;
  TS_TRY(f0.alloc((size_t)n * W));
  TS_TRY(f1.alloc((size_t)n * W));
  TS_TRY(seen.alloc((size_t)n * W));
  TS_TRY(full.alloc((size_t)W));
  TS_TRY(marks.alloc(kSpMarks));
  uint32_t hfull[32];
  for (int w = 0; w < W; ++w) {
    const int bits = d - 32 * w;
    hfull[w] = bits >= 32 ? 0xffffffffu : (bits <= 0 ? 0u : ((1u << bits) - 1u));
  }
  TS_CUDA(cudaMemcpyAsync(full.get(), hfull, sizeof(uint32_t) * W, cudaMemcpyHostToDevice, s));
  const int grid = sms * 8;
  k_sp_init<<<grid, 256, 0, s>>>(n, W, f0.get(), seen.get(), marks.get());
  k_sp_seed<<<(d + 255) / 256, 256, 0, s>>>(d, W, targets, f0.get(), seen.get(), X);
  TS_CUDA(cudaGetLastError());
  switch (W) {
    case 1: return run_levels<1>(n, d, rp, col, f0.get(), f1.get(), seen.get(), full.get(), l0, X, marks.get(), grid, s);
    case 2: return run_levels<2>(n, d, rp, col, f0.get(), f1.get(), seen.get(), full.get(), l0, X, marks.get(), grid, s);
    case 4: return run_levels<4>(n, d, rp, col, f0.get(), f1.get(), seen.get(), full.get(), l0, X, marks.get(), grid, s);
    case 8: return run_levels<8>(n, d, rp, col, f0.get(), f1.get(), seen.get(), full.get(), l0, X, marks.get(), grid, s);
    case 16: return run_levels<16>(n, d, rp, col, f0.get(), f1.get(), seen.get(), full.get(), l0, X, marks.get(), grid, s);
    default: return run_levels<32>(n, d, rp, col, f0.get(), f1.get(), seen.get(), full.get(), l0, X, marks.get(), grid, s);
  }
}

}  // namespace tsgne

extern "C" tsgne_status tsgne_shortest_path_embedding(int32_t n, const int64_t* row_ptr, const int32_t* col_idx,
                                                      const int32_t* targets, int32_t d, int32_t l0, float* X_out,
                                                      int32_t ptr_kind, void* cuda_stream) {
  using namespace tsgne;
  last_msg().clear();
  if (n < 1 || d < 1 || d > 1024 || !row_ptr || !targets || !X_out ||
      !(ptr_kind == TSGNE_PTR_HOST || ptr_kind == TSGNE_PTR_DEVICE)) {
    last_msg() = "need n >= 1, 1 <= d <= 1024, non-NULL row_ptr, targets and X_out, and a valid ptr_kind";
    return TSGNE_ERR_INVALID_ARG;
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  AllocScope as(s ? s : cudaStreamLegacy);
  const cudaMemcpyKind kin = ptr_kind == TSGNE_PTR_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  int64_t first = 0, m = 0;
  if (ptr_kind == TSGNE_PTR_HOST) {
    first = row_ptr[0];
    m = row_ptr[n];
    for (int t = 0; t < d; ++t)
      if (targets[t] < 0 || targets[t] >= n) return TSGNE_ERR_INVALID_ARG;
  } else {
    TS_CUDA(cudaMemcpy(&first, row_ptr, sizeof(int64_t), cudaMemcpyDeviceToHost));
    TS_CUDA(cudaMemcpy(&m, row_ptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost));
    int32_t* ht = new int32_t[d];
    cudaError_t e = cudaMemcpy(ht, targets, sizeof(int32_t) * d, cudaMemcpyDeviceToHost);
    bool bad = false;
    for (int t = 0; t < d && e == cudaSuccess; ++t) bad |= (ht[t] < 0 || ht[t] >= n);
    delete[] ht;
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy", __FILE__, __LINE__);
    if (bad) return TSGNE_ERR_INVALID_ARG;
  }
  if (first != 0 || m < 0) return TSGNE_ERR_BAD_CSR;
  if (m > 0 && !col_idx) return TSGNE_ERR_INVALID_ARG;
  DevBuf<int64_t> rp_in, rp, tslot;
  DevBuf<int32_t> col_in, col, tg;
  DevBuf<float> Xd;
  TS_TRY(rp_in.alloc((size_t)n + 1));
  TS_TRY(col_in.alloc((size_t)m));
  TS_TRY(tg.alloc((size_t)d));
  TS_CUDA(cudaMemcpyAsync(rp_in.get(), row_ptr, sizeof(int64_t) * ((size_t)n + 1), kin, s));
  if (m > 0) TS_CUDA(cudaMemcpyAsync(col_in.get(), col_idx, sizeof(int32_t) * (size_t)m, kin, s));
  TS_CUDA(cudaMemcpyAsync(tg.get(), targets, sizeof(int32_t) * d, kin, s));
  int64_t nnz = 0;
  TS_TRY(build_structure(n, rp_in.get(), col_in.get(), m, rp, col, tslot, &nnz, nullptr, s));
  float* Xo = X_out;
  if (ptr_kind == TSGNE_PTR_HOST) {
    TS_TRY(Xd.alloc((size_t)n * d));
    Xo = Xd.get();
  }
  TS_TRY(shortest_path_embedding(n, rp.get(), col.get(), nnz, tg.get(), d, l0, Xo, s));
  if (ptr_kind == TSGNE_PTR_HOST)
    TS_CUDA(cudaMemcpyAsync(X_out, Xo, sizeof(float) * (size_t)n * d, cudaMemcpyDeviceToHost, s));
  TS_CUDA(cudaStreamSynchronize(s));
  return TSGNE_OK;
}
