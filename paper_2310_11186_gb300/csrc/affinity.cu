// Affinities of t-SGNE on the neighbour structure.
//
// K1  conditional affinities (Eq. 2 with the denominator over N(i)):
//     p_{j|i} = exp(-beta_i (d_ij - m_i)) / S_i,  d_ij = ||x_i - x_j||^2,
//     m_i = min_j d_ij (the shift leaves p unchanged and keeps exp in range),
//     beta_i = 1 / (2 sigma_i^2) chosen by binary search so that the row
//     entropy H_i = ln S_i + beta_i E_p[d - m_i] equals ln(perplexity)
//     (Sec. 2.1: Perp = 2^H with H in bits).
//     Search: beta = 1, doubled / halved until the target is bracketed, then
//     midpoints; stop when |H - ln perp| <= tol or after max_iter entropy
//     evaluations; p is taken at the last evaluated beta.  A row with
//     |N(i)| <= perplexity cannot reach ln(perp) (its maximum entropy is
//     ln |N(i)|) and is set uniform.
//     Precision: distances, exp, entropy and p are FP64 and only p is rounded
//     to FP32.  FP32 throughout turns the rounding of d ~ 10^2 into ~1e-4
//     relative errors in p at small perplexities (large beta) and can flip
//     decisions near the stopping tolerance.
//     Cost: GB300 issues one FP64 instruction per warp and 16 cycles, however
//     few lanes are active, so FP64 work is packed and left out where it
//     decides nothing.  k_pair_dist sums each undirected pair once, one thread
//     per pair from a queue without gaps.  The search evaluates H in FP32
//     first and in FP64 only when that comes within tol + 2e-5 of the target.
//     The FP32 error near the target is below 1e-5: arguments x of exp are off
//     by 1.8e-7 |x|, so ln S by 1.8e-7 E[x] <= 1.8e-7 H, and E[x] by 1.8e-7
//     (E[x] + Var[x]), where Var[x] is at most 3.9 for 32 entries and 30 for
//     50,000; plus the sums' rounding (1e-8 per entry is allowed for).  Measured on rows of 6 to 50,000 entries: at most 3 % of
//     the margin.  Rows of up to 32 entries share a warp, 8 lanes each.
//     50,000 rows of 17 entries, d = 50, perplexity 5: 5.4 ms with one warp
//     per row and everything in FP64; distances now 0.14 ms (0.25 with
//     floats widened by conversion instructions), search 0.39 ms.
// K2  joint affinities (Eq. 3): p_ij = (p_{j|i} + p_{i|j}) / T with T the
//     FP64 total of all numerators, twice the sum of all p_{j|i} (T = 2n
//     without isolated nodes), so that sum P = 1; the total is a fixed-order
//     reduction.
#include <cmath>

#include "reduce.cuh"
#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

constexpr int kAffCta = 256;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_min_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Lists of the rows that need a search, by length (up to 32 entries, longer),
// in any order; saturated rows get their uniform p.  A CTA takes 256
// consecutive rows; their entries are consecutive too, so p is written
// coalesced, whatever the degrees.
constexpr int kGroupRow = 32;  // longest row of the packed search
__global__ void __launch_bounds__(kAffCta) k_row_kinds(int n, const int64_t* __restrict__ rp, float perp,
                                                       int32_t* __restrict__ list, int32_t* __restrict__ counts,
                                                       float* __restrict__ pcond) {
  __shared__ int64_t srp[kAffCta + 1];
  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * kAffCta;
  const int nr = (int)min((int64_t)kAffCta, (int64_t)n - r0);
  for (int t = tid; t <= nr; t += kAffCta) srp[t] = rp[r0 + t];
  __syncthreads();
  const int64_t k = tid < nr ? srp[tid + 1] - srp[tid] : 0;
  const bool search = k > 0 && !((float)k <= perp);
  const uint32_t below = (1u << (tid & 31)) - 1u;
#pragma unroll
  for (int c = 0; c < 2; ++c) {  // list[0..n): short rows, list[n..2n): long rows
    const uint32_t m = __ballot_sync(0xffffffffu, search && (k > kGroupRow) == (c == 1));
    if (m == 0u) continue;
    int base = 0;
    if ((tid & 31) == 0) base = atomicAdd(counts + c, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if ((m >> (tid & 31)) & 1u) list[(int64_t)c * n + base + __popc(m & below)] = (int32_t)(r0 + tid);
  }
  for (int64_t e = srp[0] + tid; e < srp[nr]; e += kAffCta) {
    int lo = 0, hi = nr - 1;  // the row of e: the last one that starts at or before it
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (srp[mid] <= e) lo = mid; else hi = mid - 1;
    }
    const int64_t d = srp[lo + 1] - srp[lo];
    if ((float)d <= perp) pcond[e] = 1.0f / (float)d;
  }
}

// d2 += (x - y)^2 in FP64.  kWalk: product and sum rounded apart, as the
// random-walk definition states them.
template <bool kWalk>
__device__ __forceinline__ double add_sq(double s, double x, double y) {
  const double t = __dsub_rn(x, y);
  return kWalk ? __dadd_rn(s, __dmul_rn(t, t)) : fma(t, t, s);
}

// (double)x by integer operations, for zeros and normal numbers: a conversion
// occupies the SM's FP64 pipe 16 cycles per warp like an FP64 sum does, the five
// instructions here 1 or 2, and a term of a distance needs two (1.0M pairs of
// 64 dimensions: 764 us with conversions, 488 us so).
__device__ __forceinline__ bool plain_float(float x) {
  const uint32_t m = __float_as_uint(x) & 0x7fffffffu;
  return m - 0x00800000u < 0x7f000000u || m == 0u;
}
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), m = b & 0x7fffffffu;
  const uint32_t hi = (m >> 3) + (m ? 0x38000000u : 0u);  // exponent bias 127 -> 1023
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}

// Squared distances, dimensions in index order, of every undirected pair that
// a row needs (kWalk: all; else those with an endpoint of more than perp
// entries), to both of its entries.  A CTA takes consecutive entries (the row
// of entry e is the column of its transpose), queues those it has to sum --
// the lower end sums a pair whose two rows both need it -- and works through
// the queue 256 at a time, one thread per pair.
constexpr int kPairEntries = 1024;  // entries per CTA
template <bool kWalk, int V>
__global__ void __launch_bounds__(kAffCta)
    k_pair_dist(int64_t nnz, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                const int64_t* __restrict__ tslot, const float* __restrict__ X, int d, float perp,
                const int32_t* __restrict__ counts, double* __restrict__ dist) {
  __shared__ int32_t qi[2 * kAffCta], qj[2 * kAffCta];
  __shared__ int64_t qe[2 * kAffCta];
  __shared__ int qn;
  if (!kWalk && counts[0] + counts[1] == 0) return;  // every row is saturated
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) qn = 0;
  __syncthreads();
  auto take = [&](int at) {  // one queued pair
    const int64_t i = qi[at], j = qj[at], e = qe[at];
    const float* __restrict__ x = X + i * d;
    const float* __restrict__ y = X + j * d;
    double s = 0.0;
    for (int c = 0; c < d; c += V) {
      alignas(16) float u[V], v[V];
      if constexpr (V == 4) {
        *reinterpret_cast<float4*>(u) = *reinterpret_cast<const float4*>(x + c);
        *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(y + c);
      } else if constexpr (V == 2) {
        *reinterpret_cast<float2*>(u) = *reinterpret_cast<const float2*>(x + c);
        *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(y + c);
      } else {
        u[0] = x[c];
        v[0] = y[c];
      }
      bool plain = true;
#pragma unroll
      for (int q = 0; q < V; ++q) plain = plain && plain_float(u[q]) && plain_float(v[q]);
      if (plain) {
#pragma unroll
        for (int q = 0; q < V; ++q) s = add_sq<kWalk>(s, widen(u[q]), widen(v[q]));
      } else {
#pragma unroll
        for (int q = 0; q < V; ++q) s = add_sq<kWalk>(s, (double)u[q], (double)v[q]);
      }
    }
    dist[e] = s;
    dist[tslot[e]] = s;
  };
  const int64_t e0 = (int64_t)blockIdx.x * kPairEntries;
  const int64_t e1 = e0 + kPairEntries < nnz ? e0 + kPairEntries : nnz;
  for (int64_t b = e0; b < e1; b += kAffCta) {
    const int64_t e = b + tid;
    bool need = false;
    int32_t i = 0, j = 0;
    if (e < e1) {
      j = col[e];
      i = col[tslot[e]];
      if (kWalk)
        need = i < j;
      else if (!((float)(rp[i + 1] - rp[i]) <= perp))
        need = i < j || (float)(rp[j + 1] - rp[j]) <= perp;
    }
    const uint32_t m = __ballot_sync(0xffffffffu, need);
    int base = 0;
    if (lane == 0 && m) base = atomicAdd(&qn, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (need) {
      const int at = base + __popc(m & ((1u << lane) - 1u));
      qi[at] = i;
      qj[at] = j;
      qe[at] = e;
    }
    __syncthreads();
    const int have = qn;  // below 512: fewer than 256 were left over
    if (have >= kAffCta) take(have - kAffCta + tid);
    __syncthreads();  // everyone has read qn and the queue's end
    if (have >= kAffCta) {
      if (tid == 0) qn = have - kAffCta;
      __syncthreads();
    }
  }
  if (tid < qn) take(tid);
}

// One step of the search for beta after an evaluation with H above (up) or
// below the target: halfway to the other bound, or doubled / halved while there
// is none.  One sum and one product, whichever it is (both branches' FP64
// instructions: 470 us for the search of 50,000 rows, 388 us so).
__device__ __forceinline__ void step_beta(bool up, double& beta, double& lo, double& hi) {
  const double other = up ? hi : lo;
  const bool open = (__double2hiint(other) & 0x7fffffff) == 0x7ff00000;  // infinite: never NaN
  if (up) lo = beta; else hi = beta;
  beta = (beta + (open ? 0.0 : other)) * (open && up ? 2.0 : 0.5);
}

// H may be taken from FP32 while it is this much further from the target than
// tol and finite: the sum of delta w passes FP32's range where delta is above
// about 1e37 (and beta too small to bring w down).
__device__ __forceinline__ float fp32_margin(int64_t k) { return 2e-5f + 1e-8f * (float)k; }
__device__ __forceinline__ bool fp32_decides(float far, float margin) {
  return fabsf(far) > margin && fabsf(far) < INFINITY;
}

// Rows of up to 32 entries: 8 lanes per row, 4 entries per lane in registers.
__global__ void __launch_bounds__(kAffCta)
    k_search_short(const int64_t* __restrict__ rp, const int32_t* __restrict__ list,
                   const int32_t* __restrict__ counts, double Hstar, double tol, int max_iter,
                   const double* __restrict__ dist, float* __restrict__ pcond) {
  constexpr int G = 8, U = kGroupRow / G;
  const int gl = threadIdx.x & (G - 1);
  const int count = counts[0];
  const int stride = (int)(gridDim.x * blockDim.x) / G;
  const int first = (int)(blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int wfirst = (int)(blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) / G;  // the warp's first group
  for (int base = 0; wfirst + base < count; base += stride) {
    const bool valid = first + base < count;
    const int64_t i = valid ? list[first + base] : 0;
    const int64_t a = valid ? rp[i] : 0;
    const int k = valid ? (int)(rp[i + 1] - a) : 0;
    double dl[U];
    float df[U];
    double m = INFINITY;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      dl[u] = gl + G * u < k ? dist[a + gl + G * u] : INFINITY;
      m = fmin(m, dl[u]);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
    int nu = 0;  // entries of the warp's longest lane
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool on = gl + G * u < k;
      dl[u] = on ? dl[u] - m : 0.0;
      df[u] = (float)dl[u];
      if (__any_sync(0xffffffffu, on)) nu = u + 1;
    }
    const float margin = (float)tol + fp32_margin(k), Hf = (float)Hstar;
    double beta = 1.0, lo = -INFINITY, hi = INFINITY, S = 1.0;
    // A row goes on in FP32 until it needs an FP64 evaluation, then waits for the
    // other rows of its warp: they need theirs at other steps, and an evaluation
    // takes as long for one row as for all four (50,000 rows of 17 entries,
    // perplexity 5: 687 us without waiting, 470 us so).
    double w[U];
#pragma unroll
    for (int u = 0; u < U; ++u) w[u] = 0.0;
    bool active = valid, waits = false;
    for (int it = 0; __any_sync(0xffffffffu, active);) {
      if (__any_sync(0xffffffffu, active && !waits)) {
        const float bf = (float)beta;
        float sf = 0.f, Ef = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (u < nu && gl + G * u < k) {
            const float wf = expf(-bf * df[u]);
            sf += wf;
            Ef += df[u] * wf;
          }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
          sf += __shfl_xor_sync(0xffffffffu, sf, o);
          Ef += __shfl_xor_sync(0xffffffffu, Ef, o);
        }
        const float far = logf(sf) + bf * Ef / sf - Hf;
        if (active && !waits) {
          if (it >= max_iter - 1 || !fp32_decides(far, margin)) {
            waits = true;
          } else {
            step_beta(far > 0.f, beta, lo, hi);
            ++it;
          }
        }
      } else {
        double s = 0.0, E = 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (u < nu && gl + G * u < k) {
            const double wu = exp(-beta * dl[u]);
            s += wu;
            E += dl[u] * wu;
            if (active) w[u] = wu;  // of the last evaluation: p's numerators
          }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
          s += __shfl_xor_sync(0xffffffffu, s, o);
          E += __shfl_xor_sync(0xffffffffu, E, o);
        }
        const double H = log(s) + beta * E / s;
        if (active) {
          S = s;
          if (fabs(H - Hstar) <= tol || it >= max_iter - 1) {
            active = false;
          } else {
            step_beta(H > Hstar, beta, lo, hi);
            ++it;
            waits = false;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u < nu && gl + G * u < k) pcond[a + gl + G * u] = (float)(w[u] / S);
  }
}

// Longer rows: one warp per row, its entries read from memory.
__global__ void __launch_bounds__(kAffCta)
    k_search_long(int n, const int64_t* __restrict__ rp, const int32_t* __restrict__ list,
                  const int32_t* __restrict__ counts, double Hstar, double tol, int max_iter,
                  const double* __restrict__ dist, float* __restrict__ pcond) {
  const int lane = threadIdx.x & 31;
  const int count = counts[1];
  const int warps = (int)(gridDim.x * blockDim.x) >> 5;
  for (int r = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < count; r += warps) {
    const int64_t i = list[(int64_t)n + r];
    const int64_t a = rp[i], b = rp[i + 1];
    double m = INFINITY;
    for (int64_t e = a + lane; e < b; e += 32) m = fmin(m, dist[e]);
    m = warp_min_d(m);
    const float margin = (float)tol + fp32_margin(b - a), Hf = (float)Hstar;
    double beta = 1.0, lo = -INFINITY, hi = INFINITY, S = 1.0;
    for (int it = 0; it < max_iter; ++it) {
      const bool last = it == max_iter - 1;
      const float bf = (float)beta;
      float sf = 0.f, Ef = 0.f;
      for (int64_t e = a + lane; e < b; e += 32) {
        const float delta = (float)(dist[e] - m);
        const float w = expf(-bf * delta);
        sf += w;
        Ef += delta * w;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        sf += __shfl_xor_sync(0xffffffffu, sf, o);
        Ef += __shfl_xor_sync(0xffffffffu, Ef, o);
      }
      const float far = logf(sf) + bf * Ef / sf - Hf;
      bool up = far > 0.f;
      if (last || !fp32_decides(far, margin)) {
        double s = 0.0, E = 0.0;
        for (int64_t e = a + lane; e < b; e += 32) {
          const double delta = dist[e] - m;
          const double w = exp(-beta * delta);
          s += w;
          E += delta * w;
        }
        S = warp_sum_d(s);
        E = warp_sum_d(E);
        const double H = log(S) + beta * E / S;
        if (fabs(H - Hstar) <= tol || last) break;
        up = H > Hstar;
      }
      step_beta(up, beta, lo, hi);
    }
    for (int64_t e = a + lane; e < b; e += 32) pcond[e] = (float)(exp(-beta * (dist[e] - m)) / S);
  }
}

// Total of the Eq. 3 numerators (FP64, fixed order) into sched->red[0]: every
// p_{j|i} is in two of them.
__global__ void __launch_bounds__(kAffCta) k_joint_total(int64_t nnz, const float* __restrict__ pcond,
                                                         double* __restrict__ parts, Sched* sched) {
  double acc = 0.0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) acc += (double)pcond[e];
  double bs = block_sum_d(acc);
  if (threadIdx.x == 0) parts[blockIdx.x] = bs;
  if (arrive_last(&sched->red_done)) {
    double T = 2.0 * sum_partials(parts, gridDim.x);
    if (threadIdx.x == 0) {
      sched->red[0] = T;
      if (!isfinite(T)) atomicOr(&sched->flags, kFlagNonfiniteP);
    }
  }
}

__global__ void __launch_bounds__(kAffCta) k_joint_scale(int64_t nnz, const float* __restrict__ pcond,
                                                         const int64_t* __restrict__ tslot, float* __restrict__ P,
                                                         Sched* sched) {
  const double inv = 1.0 / sched->red[0];  // one FP64 division per thread, not per entry
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 4
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) {
    const double v = ((double)pcond[e] + (double)pcond[tslot[e]]) * inv;
    const float p = (float)v;
    P[e] = p;
    if (!isfinite(p)) atomicOr(&sched->flags, kFlagNonfiniteP);
  }
}

template <bool kWalk>
tsgne_status launch_pair_dist(int64_t nnz, const int64_t* rp, const int32_t* col, const int64_t* tslot,
                              const float* X, int d, float perp, const int32_t* counts, double* dist,
                              cudaStream_t s) {
  if (nnz <= 0) return TSGNE_OK;
  const unsigned g = (unsigned)((nnz + kPairEntries - 1) / kPairEntries);
  const uintptr_t at = reinterpret_cast<uintptr_t>(X);
  if (d % 4 == 0 && (at & 15u) == 0)
    k_pair_dist<kWalk, 4><<<g, kAffCta, 0, s>>>(nnz, rp, col, tslot, X, d, perp, counts, dist);
  else if (d % 2 == 0 && (at & 7u) == 0)
    k_pair_dist<kWalk, 2><<<g, kAffCta, 0, s>>>(nnz, rp, col, tslot, X, d, perp, counts, dist);
  else
    k_pair_dist<kWalk, 1><<<g, kAffCta, 0, s>>>(nnz, rp, col, tslot, X, d, perp, counts, dist);
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

}  // namespace

tsgne_status walk_distances(int64_t nnz, const int64_t* rp, const int32_t* col, const int64_t* tslot, const float* X,
                            int d, double* dist, cudaStream_t s) {
  return launch_pair_dist<true>(nnz, rp, col, tslot, X, d, 0.f, nullptr, dist, s);
}

tsgne_status build_affinities(int n, const int64_t* rp, const int32_t* col, const int64_t* tslot, int64_t nnz,
                              const float* X, int d, float perplexity, float tol, int max_iter, float* P, Sched* sched,
                              cudaStream_t s) {
  int dev = 0, sms = 1;
  TS_CUDA(cudaGetDevice(&dev));
  TS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DevBuf<double> dist;
  DevBuf<float> pcond;
  DevBuf<int32_t> list, counts;
  TS_TRY(dist.alloc((size_t)nnz));
  TS_TRY(pcond.alloc((size_t)nnz));
  TS_TRY(list.alloc(2 * (size_t)n));
  TS_TRY(counts.alloc(2));
  const double Hstar = std::log((double)perplexity);
  TS_CUDA(cudaMemsetAsync(counts.get(), 0, 2 * sizeof(int32_t), s));
  k_row_kinds<<<(n + kAffCta - 1) / kAffCta, kAffCta, 0, s>>>(n, rp, perplexity, list.get(), counts.get(),
                                                              pcond.get());
  TS_CUDA(cudaGetLastError());
  TS_TRY(launch_pair_dist<false>(nnz, rp, col, tslot, X, d, perplexity, counts.get(), dist.get(), s));
  k_search_short<<<sms * 8, kAffCta, 0, s>>>(rp, list.get(), counts.get(), Hstar, tol, max_iter, dist.get(),
                                             pcond.get());
  k_search_long<<<sms * 8, kAffCta, 0, s>>>(n, rp, list.get(), counts.get(), Hstar, tol, max_iter, dist.get(),
                                            pcond.get());
  TS_CUDA(cudaGetLastError());
  TS_TRY(joint_affinities(nnz, pcond.get(), tslot, P, sched, s));
  return TSGNE_OK;
}

tsgne_status joint_affinities(int64_t nnz, const float* pcond, const int64_t* tslot, float* P, Sched* sched,
                              cudaStream_t s) {
  int dev = 0, sms = 1;
  TS_CUDA(cudaGetDevice(&dev));
  TS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int egrid = sms * 8;
  DevBuf<double> parts;
  TS_TRY(parts.alloc(egrid));
  k_joint_total<<<egrid, kAffCta, 0, s>>>(nnz, pcond, parts.get(), sched);
  k_joint_scale<<<egrid, kAffCta, 0, s>>>(nnz, pcond, tslot, P, sched);
  TS_CUDA(cudaGetLastError());
  TS_CUDA(cudaStreamSynchronize(s));  // temporaries are freed on return
  return TSGNE_OK;
}

}  // namespace tsgne
