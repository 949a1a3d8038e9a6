// Device code shared by the single-layout and the multi-layout symmetric
// repulsion kernels: the work of one tile pair (see repulsion_sym.cu for the
// decomposition and the ring schedule).
//
// Forces leave a unit as fixed-point integers: each FP32 partial (one
// point's sum over the other tile) is scaled by 2^s, rounded to the nearest
// int64 and added with an integer atomic into the point's accumulator
// acc[2 p + {0, 1}].  Integer addition is associative, so the total is the
// same bits whatever order the units finish in, and the accumulators take
// 16 bytes per point instead of one partial per tile.  fix_shift() picks s
// from n so that no sum can overflow (see tsgne_internal.cuh).
//
// Z: each lane's FP32 partial of a point covers one 64-point ring group
// (64 terms w in (0, 1]), is then added into a second FP32 partial over the
// unit's groups (at most 16 for 1,024-point tiles), and from there on the
// sums are exact integers (zsum.cuh).  The worst-case relative rounding of a
// unit's row sum is then about (63 + 15) 2^-24 = 4.6e-6, against 1,023 2^-24 =
// 6.1e-5 for one FP32 sum over the whole tile.  The integers also replace the
// FP64 sums that ended every unit and the last CTA's sum over all of them: on
// a 2,000-point layout these took 4.2 of 8 us (0.5 us the warp's double
// butterfly, 1.5 us the fence and the arrival counter, 2.2 us the last CTA).
#pragma once

#include "f32x2.cuh"
#include "storage.cuh"
#include "tsgne_internal.cuh"
#include "zsum.cuh"

namespace tsgne {

constexpr int kRI = 16;             // i-points per lane (default shape)
constexpr int kWarpsPerSm = 8;      // resident warps per SM the grid is sized for (16 i-points per lane)
constexpr int kGroup = 64;          // j-points per ring group (32 lanes x 2)
// Resident warps per SM the grid is sized for, by i-points per lane: 16
// i-points need about 200 registers a thread (8 warps), 8 about half.
__host__ __device__ constexpr int warps_per_sm(int RI) { return RI >= 16 ? 8 : 16; }

// Tile pairs of nt tiles, and the first one of diagonal a (products of two tile numbers pass 2^31 above 46,340 tiles).
__host__ __device__ __forceinline__ int tile_pairs(int nt) { return (int)((long long)nt * (nt + 1) / 2); }
__device__ __forceinline__ int row_start(int a, int nt) {
  return (int)((long long)a * nt - (long long)a * (a - 1) / 2);
}

// One j-point against the lane's 8 i-points; acc (x, y) is the running sum
// of w^2 (y_i - y_j) over i for this j.
template <int kH>
__device__ __forceinline__ void ring_pair(const float4 q, float& accx, float& accy, const u64 (&X2)[kH],
                                          const u64 (&Y2)[kH], u64 (&FX)[kH], u64 (&FY)[kH], u64 (&Z2)[kH],
                                          const u64 one2) {
  const u64 nx = pk(q.x, q.y);
  const u64 ny = pk(q.z, q.w);
  u64 PX = pk(accx, 0.f), PY = pk(accy, 0.f);
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    const u64 dx = add2(X2[h], nx);
    const u64 dy = add2(Y2[h], ny);
    u64 qq = fma2(dx, dx, one2);
    qq = fma2(dy, dy, qq);
    float q0, q1;
    upk(qq, q0, q1);
    const u64 w = pk(rcp_approx(q0), rcp_approx(q1));
    Z2[h] = add2(Z2[h], w);
    const u64 w2 = mul2(w, w);
    FX[h] = fma2(w2, dx, FX[h]);
    FY[h] = fma2(w2, dy, FY[h]);
    PX = fma2(w2, dx, PX);
    PY = fma2(w2, dy, PY);
  }
  float a0, a1;
  upk(PX, a0, a1);
  accx = a0 + a1;
  upk(PY, a0, a1);
  accy = a0 + a1;
}

// Adds v (one coordinate of a partial force) to a fixed-point accumulator.
__device__ __forceinline__ void red_int(unsigned long long* p, long long q) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"((unsigned long long)q) : "memory");
}
__device__ __forceinline__ void red_fix(unsigned long long* p, float v, float scale) {
  red_int(p, __float2ll_rn(v * scale));  // v * 2^s is exact: scale is a power of two
}

// One thread: the Z of a unit to its place: as a double (exact) in zunit, for
// a share of a sharded pass, or added to the words of zacc.
__device__ __forceinline__ void put_z(ZSum q, bool bad, double* zunit, u64* zacc, uint32_t* zbad) {
  if (zunit != nullptr) {
    *zunit = bad ? (double)NAN : z_double(q);
    return;
  }
  z_add(zacc, q);
  if (bad) atomicOr(zbad, 1u);
}

// The Z of a unit: the sum over a CTA of W warps of the threads' (valid in
// thread 0).  *bad: any thread's.  zs: 2 W words of shared memory, free again
// after a __syncthreads.
template <int W>
__device__ __forceinline__ ZSum cta_z(ZSum q, bool* bad, u64* zs) {
  const bool any = __any_sync(0xffffffffu, *bad);
  ZSum v = z_warp_sum(q);
  *bad = any;
  if (W == 1) return z_top53(v);
  if ((threadIdx.x & 31) == 0) {
    const int w = threadIdx.x >> 5;
    zs[2 * w] = any ? ~0ull : v.hi;
    zs[2 * w + 1] = v.lo;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    v = ZSum{};
    *bad = false;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      *bad |= zs[2 * w] == ~0ull;
      v.add(ZSum{zs[2 * w], zs[2 * w + 1]});
    }
  }
  return z_top53(v);
}

// The schedule of the iteration that follows a pass (one thread).
__device__ __forceinline__ void set_schedule(Sched* s, int advance, float ee, int ee_iters, float mom0, float mom1) {
  const int t = s->t;
  s->alpha = t < ee_iters ? ee : 1.0f;
  s->mu = t < ee_iters ? mom0 : mom1;
  if (advance) s->t = t + 1;
}

// The pairs of a unit: the lane's i-points against the G ring groups in sj,
// a != b with the j side in sacc, a == b as ordered pairs.  ZG: the lane's Z
// partials.  Ends, for a != b, with a __syncthreads.
template <int W, int kH>
__device__ __forceinline__ void unit_pairs(int G, bool off_diagonal, const float4* sj, float2* sacc,
                                           const u64 (&X2)[kH], const u64 (&Y2)[kH], u64 (&FX)[kH], u64 (&FY)[kH],
                                           u64 (&ZG)[kH]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u64 one2 = pk(1.f, 1.f);
  u64 Z2[kH];
#pragma unroll
  for (int h = 0; h < kH; ++h) Z2[h] = 0ull;
  if (off_diagonal) {
    for (int ph = 0; ph < G; ++ph) {
      const int g = (warp + ph) & (G - 1);
      const float4* gj = sj + g * kGroup;
      float2* ga = sacc + g * kGroup;
      float2 c0 = ga[2 * lane], c1 = ga[2 * lane + 1];
      float ax0 = c0.x, ay0 = c0.y, ax1 = c1.x, ay1 = c1.y;
      const int src = (lane + 1) & 31;
#pragma unroll 4
      for (int s = 0; s < 32; ++s) {
        const int jj = (lane + s) & 31;
        const float4 q0 = gj[2 * jj];
        const float4 q1 = gj[2 * jj + 1];
        ring_pair<kH>(q0, ax0, ay0, X2, Y2, FX, FY, Z2, one2);
        ring_pair<kH>(q1, ax1, ay1, X2, Y2, FX, FY, Z2, one2);
        ax0 = __shfl_sync(0xffffffffu, ax0, src);
        ay0 = __shfl_sync(0xffffffffu, ay0, src);
        ax1 = __shfl_sync(0xffffffffu, ax1, src);
        ay1 = __shfl_sync(0xffffffffu, ay1, src);
      }
      ga[2 * lane] = make_float2(ax0, ay0);
      ga[2 * lane + 1] = make_float2(ax1, ay1);
#pragma unroll
      for (int h = 0; h < kH; ++h) {  // the group's 64 terms into the unit's partial
        ZG[h] = add2(ZG[h], Z2[h]);
        Z2[h] = 0ull;
      }
      __syncthreads();
    }
    return;
  }
  // diagonal unit: ordered pairs within the tile, i side only, in groups
  // of 64 j-points for Z
  for (int j0 = 0; j0 < G * kGroup; j0 += kGroup) {
#pragma unroll 2
    for (int j = j0; j < j0 + kGroup; ++j) {
      const float4 q = sj[j];
      const u64 nx = pk(q.x, q.y);
      const u64 ny = pk(q.z, q.w);
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        const u64 dx = add2(X2[h], nx);
        const u64 dy = add2(Y2[h], ny);
        u64 qq = fma2(dx, dx, one2);
        qq = fma2(dy, dy, qq);
        float q0, q1;
        upk(qq, q0, q1);
        const u64 w = pk(rcp_approx(q0), rcp_approx(q1));
        Z2[h] = add2(Z2[h], w);
        const u64 w2 = mul2(w, w);
        FX[h] = fma2(w2, dx, FX[h]);
        FY[h] = fma2(w2, dy, FY[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < kH; ++h) {
      ZG[h] = add2(ZG[h], Z2[h]);
      Z2[h] = 0ull;
    }
  }
}

// TJ j-points from jb into shared memory, their accumulators cleared.
template <int W, class YT>
__device__ __forceinline__ void stage_j(const YT* __restrict__ Y, int jb, int TJ, float4* sj, float2* sacc) {
  for (int k = threadIdx.x; k < TJ; k += W * 32) {
    const float2 p = ld_y(Y, (size_t)jb + k);
    sj[k] = make_float4(-p.x, -p.x, -p.y, -p.y);
    sacc[k] = make_float2(0.f, 0.f);
  }
}

// Off-diagonal unit, j side: F_j = -sum_i w^2 (y_i - y_j) for the real j-points.
template <int W>
__device__ __forceinline__ void add_j(int jb, int TJ, int n, const float2* sacc, unsigned long long* acc,
                                      float fscale) {
  for (int k = threadIdx.x; k < TJ; k += W * 32)
    if (jb + k < n) {
      const float2 v = sacc[k];
      red_fix(acc + 2 * (size_t)(jb + k), -v.x, fscale);
      red_fix(acc + 2 * (size_t)(jb + k) + 1, -v.y, fscale);
    }
}

// The Z of N lane partials, those that count (the others are 0); *bad: a NaN
// among them.  The second half of the sum only where a lane of the warp needs
// it (15 iterations of 2,000 points: 254 us with it throughout, 245 us so; a
// BF16 gradient of 65,536 points: 783 and 768 us).
template <int N>
__device__ __forceinline__ ZSum lane_z(const float (&z)[N], bool* bad) {
  ZSum s;
  float zn = 0.f;  // NaN if any partial is
  bool small = false;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    s.hi += z_hi(z[k]);
    zn += z[k];
    small |= z[k] < kZWhole;
  }
  *bad = zn != zn;
  if (__any_sync(0xffffffffu, small && zn != 0.f)) {
#pragma unroll
    for (int k = 0; k < N; ++k) s.add(ZSum{0ull, z_lo(z[k])});
  }
  return s;
}

// The thread's Z from its lane partials (ordered pairs:
// twice the off-diagonal units', whose tile a holds no padding; the diagonal
// units' real points, w_ii = 1 included); *bad: a NaN among them.
template <int kH>
__device__ __forceinline__ ZSum unit_z(bool off_diagonal, int ibase, int n, const u64 (&ZG)[kH], bool* bad) {
  const float twice = off_diagonal ? 2.f : 1.f;
  float z[2 * kH];
#pragma unroll
  for (int h = 0; h < kH; ++h) {
    float z0, z1;
    upk(ZG[h], z0, z1);
    z[2 * h] = off_diagonal || ibase + (2 * h) * 32 < n ? twice * z0 : 0.f;
    z[2 * h + 1] = off_diagonal || ibase + (2 * h + 1) * 32 < n ? twice * z1 : 0.f;
  }
  return lane_z(z, bad);
}

// Loads of the lane's i-points of tile a: i = a T + warp 32 RI + r 32 + lane, r < RI.
template <int RI, class YT>
__device__ __forceinline__ void load_i(const YT* __restrict__ Y, int ibase, u64 (&X2)[RI / 2], u64 (&Y2)[RI / 2]) {
#pragma unroll
  for (int h = 0; h < RI / 2; ++h) {
    const float2 p0 = ld_y(Y, ibase + (2 * h) * 32);
    const float2 p1 = ld_y(Y, ibase + (2 * h + 1) * 32);
    X2[h] = pk(p0.x, p1.x);
    Y2[h] = pk(p0.y, p1.y);
  }
}

// i side of tile a's real points.
template <int RI>
__device__ __forceinline__ void add_i(int ibase, int n, const u64 (&FX)[RI / 2], const u64 (&FY)[RI / 2],
                                      unsigned long long* acc, float fscale) {
#pragma unroll
  for (int h = 0; h < RI / 2; ++h) {
    float fx0, fx1, fy0, fy1;
    upk(FX[h], fx0, fx1);
    upk(FY[h], fy0, fy1);
    const int p0 = ibase + (2 * h) * 32, p1 = ibase + (2 * h + 1) * 32;
    if (p0 < n) {
      red_fix(acc + 2 * (size_t)p0, fx0, fscale);
      red_fix(acc + 2 * (size_t)p0 + 1, fy0, fscale);
    }
    if (p1 < n) {
      red_fix(acc + 2 * (size_t)p1, fx1, fscale);
      red_fix(acc + 2 * (size_t)p1 + 1, fy1, fscale);
    }
  }
}

// sym_unit of a diagonal pair (a, a).  Out of line, as unit_tiles is: how the
// compiler schedules the ring loop, where a large pass spends its time,
// depends on what else is inlined beside it (300,000 points: 15.86 ms with
// both calls, 16.07 with this one alone, 16.2 with neither; 100,000: 1.80,
// 1.83, 1.92 ms).  A NaN comes back as hi = ~0.
template <int W, int RI, class YT>
static __device__ __noinline__ ZSum diag_unit(const YT* __restrict__ Y, int n, unsigned long long* __restrict__ acc,
                                             float fscale, int a, int sub, int G, float4* sj, float2* sacc) {
  constexpr int kH = RI / 2;
  const int TJ = G * kGroup;
  const int ibase = a * (W * 32 * RI) + (int)(threadIdx.x >> 5) * (32 * RI) + (int)(threadIdx.x & 31);
  u64 X2[kH], Y2[kH], FX[kH], FY[kH], ZG[kH];
  stage_j<W>(Y, a * (W * 32 * RI) + sub * TJ, TJ, sj, sacc);
  load_i<RI>(Y, ibase, X2, Y2);
#pragma unroll
  for (int h = 0; h < kH; ++h) FX[h] = FY[h] = ZG[h] = 0ull;
  __syncthreads();
  unit_pairs<W, kH>(G, false, sj, sacc, X2, Y2, FX, FY, ZG);
  bool bad;
  ZSum zt = unit_z<kH>(false, ibase, n, ZG, &bad);
  add_i<RI>(ibase, n, FX, FY, acc, fscale);
  if (bad) zt.hi = ~0ull;
  return zt;
}

// One unit of a layout: the points of tile a against the G ring groups of
// tile b that start at group sub * G (a <= b; G = groups, or T / 64, the whole
// tile, and sub = 0 for kWhole; see split_tiles).  Stages those j-points,
// evaluates the pairs and adds tile a's forces and (a < b) the j-points'
// forces into the fixed-point accumulators acc[2 p], acc[2 p + 1] of the real
// points (p < n).  Returns this thread's share of the unit's Z (unit_z).  Every
// thread of the CTA must call it; it ends with the shared tiles free for reuse
// only after a __syncthreads by the caller.  G is a power of two, at least W.
template <int W, int RI, class YT, bool kWhole>
__device__ __forceinline__ ZSum sym_unit(const YT* __restrict__ Y, int n, unsigned long long* __restrict__ acc,
                                        float fscale, int a, int b, int sub, int groups, float4* sj, float2* sacc,
                                        bool* bad) {
  constexpr int kH = RI / 2;  // FP32x2 pairs of i-points per lane
  constexpr int T = W * 32 * RI;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int G = kWhole ? T / kGroup : groups;  // a constant for whole tiles
  const int TJ = G * kGroup;
  if (a == b) {
    const ZSum z = diag_unit<W, RI, YT>(Y, n, acc, fscale, a, sub, G, sj, sacc);
    *bad = z.hi == ~0ull;
    return *bad ? ZSum{} : z;
  }
  const int jb = b * T + sub * TJ;  // first j-point
  stage_j<W>(Y, jb, TJ, sj, sacc);
  const int ibase = a * T + warp * (32 * RI) + lane;
  u64 X2[kH], Y2[kH], FX[kH], FY[kH], ZG[kH];
  load_i<RI>(Y, ibase, X2, Y2);
#pragma unroll
  for (int h = 0; h < kH; ++h) FX[h] = FY[h] = ZG[h] = 0ull;
  __syncthreads();
  unit_pairs<W, kH>(G, true, sj, sacc, X2, Y2, FX, FY, ZG);
  const ZSum zt = unit_z<kH>(true, ibase, n, ZG, bad);
  add_j<W>(jb, TJ, n, sacc, acc, fscale);
  add_i<RI>(ibase, n, FX, FY, acc, fscale);
  return zt;
}

// All S = T / (64 G) units of one tile pair by one CTA: the same FP32 partials,
// so the same bits, as S calls of sym_unit.  For a batch, whose members fill
// the GPU together: both tiles are loaded once, the i-points' integer sums
// stay in shared memory (si: T long2, each thread its own points) and reach
// the accumulators once instead of S times.  Returns the sum of the units' Z
// in thread 0 (a NaN as hi = ~0).  zs: 2 W words of shared memory.
template <int W, int RI, class YT>
static __device__ __noinline__ ZSum sym_units(const YT* __restrict__ Y, int n, unsigned long long* __restrict__ acc,
                                             float fscale, int a, int b, int G, float4* sj, float2* sacc,
                                             longlong2* si, u64* zs) {
  constexpr int kH = RI / 2;
  constexpr int T = W * 32 * RI;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ibase = a * T + warp * (32 * RI) + lane;
  longlong2* const mine = si + warp * (32 * RI) + lane;
  u64 X2[kH], Y2[kH];
  stage_j<W>(Y, b * T, T, sj, sacc);
  load_i<RI>(Y, ibase, X2, Y2);
  __syncthreads();
  ZSum zt;
  bool bad = false;
  for (int j0 = 0; j0 < T; j0 += G * kGroup) {
    u64 FX[kH], FY[kH], ZG[kH];
#pragma unroll
    for (int h = 0; h < kH; ++h) FX[h] = FY[h] = ZG[h] = 0ull;
    unit_pairs<W, kH>(G, a != b, sj + j0, sacc + j0, X2, Y2, FX, FY, ZG);
    bool nan;
    zt.add(cta_z<W>(unit_z<kH>(a != b, ibase, n, ZG, &nan), &nan, zs));
    bad |= nan;
    if (W > 1) __syncthreads();
#pragma unroll
    for (int h = 0; h < kH; ++h) {
      float fx[2], fy[2];
      upk(FX[h], fx[0], fx[1]);
      upk(FY[h], fy[0], fy[1]);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        longlong2 v = j0 == 0 ? make_longlong2(0, 0) : mine[(2 * h + k) * 32];
        v.x += __float2ll_rn(fx[k] * fscale);
        v.y += __float2ll_rn(fy[k] * fscale);
        mine[(2 * h + k) * 32] = v;
      }
    }
  }
  if (a != b) add_j<W>(b * T, T, n, sacc, acc, fscale);
#pragma unroll
  for (int r = 0; r < RI; ++r)
    if (ibase + r * 32 < n) {
      const longlong2 v = mine[r * 32];
      red_int(acc + 2 * (size_t)(ibase + r * 32), v.x);
      red_int(acc + 2 * (size_t)(ibase + r * 32) + 1, v.y);
    }
  if (bad) zt.hi = ~0ull;
  return zt;
}

// The small pass (layouts of at most kSmallPoints points).  Such a pass has
// too few pairs to fill the GPU: what counts is the length of the chain of
// dependent instructions, not the work.  Every ordered pair is evaluated, so
// no accumulator travels round a ring (a step of the ring waits 190 cycles
// for its shuffle; the whole 64-point group takes 3 us) and nothing is added
// on the j side.  A unit is one CTA of 4 warps: 256 i-points, two per lane,
// against a chunk of j-points in shared memory.  Twice the arithmetic of the
// symmetric pass, on units a quarter of its smallest: 2,000 points make 256
// CTAs.  The chunk is the FP32 partial of a point's force and depends on n
// alone, so a member of a batch gets the bits of a layout on its own.
constexpr int kSmallWarps = 4;
constexpr int kSmallBlock = 64 * kSmallWarps;  // i-points per unit
constexpr int kSmallMaxChunk = 128;
__host__ __device__ inline int small_chunk(int n) { return n <= 3072 ? 64 : 128; }
__host__ __device__ inline int small_chunks(int n) { return (n + small_chunk(n) - 1) / small_chunk(n); }
__host__ __device__ inline int small_units(int n) { return ((n + kSmallBlock - 1) / kSmallBlock) * small_chunks(n); }

template <class YT>
__device__ __forceinline__ ZSum small_unit(const YT* __restrict__ Y, int n, unsigned long long* __restrict__ acc,
                                          float fscale, int ib, int c, float4* sj, bool* bad) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u64 one2 = pk(1.f, 1.f);
  const int TJ = small_chunk(n);
  const int i0 = ib * kSmallBlock + warp * 64 + lane, i1 = i0 + 32;
  const float2 p0 = ld_y(Y, i0), p1 = ld_y(Y, i1);  // padded: the sentinel above n
  for (int k = tid; k < TJ; k += 32 * kSmallWarps) {
    const float2 p = ld_y(Y, c * TJ + k);
    sj[k] = make_float4(-p.x, -p.x, -p.y, -p.y);
  }
  const u64 X2 = pk(p0.x, p1.x), Y2 = pk(p0.y, p1.y);
  u64 FX = 0ull, FY = 0ull, ZG = 0ull;
  __syncthreads();
  for (int j0 = 0; j0 < TJ; j0 += kGroup) {
    u64 Z2 = 0ull;
#pragma unroll 16
    for (int j = j0; j < j0 + kGroup; ++j) {
      const float4 q = sj[j];
      const u64 dx = add2(X2, pk(q.x, q.y));
      const u64 dy = add2(Y2, pk(q.z, q.w));
      u64 qq = fma2(dx, dx, one2);
      qq = fma2(dy, dy, qq);
      float q0, q1;
      upk(qq, q0, q1);
      const u64 w = pk(rcp_approx(q0), rcp_approx(q1));
      Z2 = add2(Z2, w);
      const u64 w2 = mul2(w, w);
      FX = fma2(w2, dx, FX);
      FY = fma2(w2, dy, FY);
    }
    ZG = add2(ZG, Z2);
  }
  float z0, z1, fx0, fx1, fy0, fy1;
  upk(ZG, z0, z1);
  upk(FX, fx0, fx1);
  upk(FY, fy0, fy1);
  if (i0 < n) {
    red_fix(acc + 2 * (size_t)i0, fx0, fscale);
    red_fix(acc + 2 * (size_t)i0 + 1, fy0, fscale);
  }
  if (i1 < n) {
    red_fix(acc + 2 * (size_t)i1, fx1, fscale);
    red_fix(acc + 2 * (size_t)i1 + 1, fy1, fscale);
  }
  const float z[2] = {i0 < n ? z0 : 0.f, i1 < n ? z1 : 0.f};
  return lane_z(z, bad);
}

// Units per tile pair: j sub-tiles, a power of two.  Passes on tiles of 8
// i-points per lane (see kMidPoints) cut their tile pairs until the units make 2.2 waves of
// the grid, down to one ring group per warp: 10,000 points take 30.8 us with
// four sub-tiles and 40.1 us whole, 20,000 points 95.8 us with two and 98.5 us
// whole; at 30,000 (whole tiles: 2.8 waves) cutting gains nothing.  Tiles of 16
// i-points are not cut.  The cut depends on the layout's size and the shape
// alone: a member of a batch is cut as the layout on its own.
inline int split_tiles(long pairs, long slots, int RI) {
  int s = 1;
  while (RI == 8 && s < RI / 2 && 5 * pairs * s < 11 * slots) s *= 2;
  return s;
}

// (a, b) of tile pair u of a layout with nt tiles, numbered diagonal by diagonal:
// diagonal d = b - a holds the nt - d units (0, d), (1, d + 1), ..., so it
// starts at sum_{d' < d} (nt - d') = row_start(d, nt).  Units taken one after
// the other by the persistent grid then touch different tiles: the integer
// atomics of concurrently finishing units go to different points instead of
// all to the shared tile a of one row of the triangle.
static __device__ __noinline__ int2 unit_tiles(int u, int nt) {
  int d = 0, hi = nt - 1;  // largest d with row_start(d) <= u
  while (d < hi) {
    const int mid = (d + hi + 1) >> 1;
    if (row_start(mid, nt) <= u) d = mid; else hi = mid - 1;
  }
  const int a = u - row_start(d, nt);
  return make_int2(a, a + d);
}

}  // namespace tsgne
