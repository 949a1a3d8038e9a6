// Symmetric exact repulsion (Sec. 2.1, Eq. 4): each unordered pair {i, j} is
// evaluated once and its force is applied to both points,
//   w = (1 + ||y_i - y_j||^2)^-1,  F^r_i += w^2 (y_i - y_j),  F^r_j -= w^2 (y_i - y_j),
//   Z += 2 w  (Z sums ordered pairs k != l).
// Per unordered pair this is 10 FP32 lane-ops and one MUFU reciprocal, i.e.
// 5 lane-ops and half a reciprocal per ordered pair (the ordered kernel in
// repulsion.cu spends 8 and 1).  Forces go to per-point fixed-point
// accumulators with integer atomics (sym_unit.cuh), so the pass needs 16
// bytes per point whatever the number of tiles, and its result does not
// depend on the order in which units finish.
//
// Decomposition.  Points are padded to n_pad = nt * T (T = 32 W points for each
// of a lane's 8 or 16 i-points) with the sentinel point.  A unit of work is a
// tile pair (a, b), a <= b, or one of the j sub-tiles that split_tiles cuts it
// into; a persistent grid (warps_per_sm: 8 warps per SM with 16 i-points; 2-warp
// CTAs once there are enough tile pairs, else 1-warp CTAs) takes one unit per
// CTA and then the rest from a global queue.  Sixteen i-points per lane and few
// warps beat eight i-points and 24 warps per SM on GB300 where there are tile
// pairs enough: the longer independent chains per lane hide the reciprocal
// latency better than more warps do.  Unit (a, b), a < b, adds the forces of
// tile a's points and of its j-points into their accumulators; a diagonal unit
// evaluates its ordered pairs with the i-side only.  Z: each unit adds its exact
// value to the words of the slot of this pass; the rows that use the forces turn
// them into 1 / Z, so the pass ends with its units.  Layouts of at most
// kSmallPoints points take k_repulsion_small instead.
//
// Inside a unit (a < b), with 16 i-points per lane (8: half of each).  Each of
// the W warps holds 512 points of tile a in registers (as eight FP32x2 pairs).  Tile b sits in shared
// memory as {-x, -x, -y, -y} plus an FP32 force accumulator per point, cut
// into 8W groups of 64 points.  In phase p warp w works on group (w + p) mod
// 8W, so no two warps touch the same accumulators at once and no atomics are
// needed.  Within a warp, lane l starts with the accumulators of the group's
// points 2l and 2l+1; each of 32 steps evaluates the lane's 16 i-points
// against those 2 j-points, then passes the j accumulators one lane down the
// ring (shuffle); after 32 steps every j has met all 512 i of the warp and
// its accumulators are back home.  Only sentinel points lie in the last tile,
// and a < b means tile a never holds any, so sentinel-sentinel pairs (w = 1)
// occur only in the diagonal unit, where they are masked out of Z.
#include "f32x2.cuh"
#include "sym_unit.cuh"
#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

// The part of a whole pass that is not the units': the other slot's sums and
// queue are cleared for the next pass and the schedule is set.  Nobody else
// reads or writes these during the pass, so one thread of it does.
__device__ __forceinline__ void open_pass(Sched* s, int slot, int advance, float ee, int ee_iters, float mom0,
                                          float mom1) {
  const int o = slot ^ 1;
  for (u64& w : s->zacc[o]) w = 0ull;
  s->zbad[o] = 0u;
  s->work_next[o] = 0u;
  set_schedule(s, advance, ee, ee_iters, mom0, mom1);
}

// Units [u0, u1) of the tile pairs' units (all of them on one GPU; one
// rank's share when the pass is sharded, zunit != NULL: the caller sums the
// unit partials over the ranks and launches k_finalize_z).
template <int W, int RI, class YT, bool kWhole>
__global__ void __launch_bounds__(W * 32, warps_per_sm(RI) / W)
    k_repulsion_sym(const YT* __restrict__ Y, int n, int nt, int split, unsigned long long* __restrict__ acc,
                    float fscale, double* __restrict__ zunit, Sched* sched, int slot, int u0, int u1, int advance,
                    float ee, int ee_iters, float mom0, float mom1) {
  constexpr int T = W * 32 * RI;
  constexpr int G = T / kGroup;
  extern __shared__ float4 smem[];
  const int TJ = kWhole ? T : T / split;
  float4* sj = smem;                                    // TJ x {-x, -x, -y, -y}
  float2* sacc = reinterpret_cast<float2*>(smem + TJ);  // TJ x force accumulator
  __shared__ int s_unit, s_a, s_b;
  __shared__ u64 s_z[2 * W];
  const int tid = threadIdx.x;
  const int pairs = tile_pairs(nt);
  if (blockIdx.x == 0 && tid == 0 && zunit == nullptr) open_pass(sched, slot, advance, ee, ee_iters, mom0, mom1);

  for (bool first = true;; first = false) {
    if (tid == 0) {
      // the first unit of a CTA needs no queue: one round trip to L2 less
      const int u = u0 + (first ? (int)blockIdx.x : (int)(gridDim.x + atomicAdd(&sched->work_next[slot], 1u)));
      const int2 ab = u < u1 ? unit_tiles(u % pairs, nt) : make_int2(0, 0);
      s_unit = u;
      s_a = ab.x;
      s_b = ab.y;
    }
    __syncthreads();
    const int u = s_unit, a = s_a, b = s_b, sub = u / pairs;
    if (u >= u1) break;
    if (!(TS_IN(a, 0, nt, &sched->flags) && TS_IN(b, a, nt, &sched->flags))) {  // debug build only
      if (tid == 0 && zunit != nullptr) zunit[u] = 0.0;
      __syncthreads();
      continue;
    }
    bool bad;
    const ZSum zt = sym_unit<W, RI, YT, kWhole>(Y, n, acc, fscale, a, b, sub, G / split, sj, sacc, &bad);
    const ZSum zb = cta_z<W>(zt, &bad, s_z);
    if (tid == 0) put_z(zb, bad, zunit ? zunit + u : nullptr, sched->zacc[slot], &sched->zbad[slot]);
    __syncthreads();  // shared tiles are rewritten by the next unit
  }
}

// The small pass: one unit per CTA, units [u0, u0 + gridDim.x).
template <class YT>
__global__ void __launch_bounds__(32 * kSmallWarps)
    k_repulsion_small(const YT* __restrict__ Y, int n, unsigned long long* __restrict__ acc, float fscale,
                      double* __restrict__ zunit, Sched* sched, int slot, int u0, int advance, float ee,
                      int ee_iters, float mom0, float mom1) {
  __shared__ float4 sj[kSmallMaxChunk];
  __shared__ u64 s_z[2 * kSmallWarps];
  const int u = u0 + (int)blockIdx.x, nc = small_chunks(n);
  if (blockIdx.x == 0 && threadIdx.x == 0 && zunit == nullptr)
    open_pass(sched, slot, advance, ee, ee_iters, mom0, mom1);
  bool bad;
  const ZSum zt = small_unit<YT>(Y, n, acc, fscale, u / nc, u % nc, sj, &bad);
  const ZSum zb = cta_z<kSmallWarps>(zt, &bad, s_z);
  if (threadIdx.x == 0) put_z(zb, bad, zunit ? zunit + u : nullptr, sched->zacc[slot], &sched->zbad[slot]);
}

// Z of a sharded pass: the unit partials' integers summed into sched->zacc,
// as the units of a whole pass add them.
__global__ void __launch_bounds__(1024)
    k_finalize_z(const double* __restrict__ zunit, int units, Sched* sched, int slot, int advance, float ee,
                 int ee_iters, float mom0, float mom1) {
  __shared__ u64 sum[kZWords];
  __shared__ uint32_t nan;
  if (threadIdx.x < kZWords) sum[threadIdx.x] = 0ull;
  if (threadIdx.x == 0) nan = 0u;
  __syncthreads();
  u64 words[kZWords] = {};
  bool bad = false;
  for (int k = threadIdx.x; k < units; k += blockDim.x) {
    const double z = zunit[k];
    bad |= z != z;
    const ZSum v = z_fix(z);
#pragma unroll
    for (int w = 0; w < kZWords; ++w) words[w] += z_word(v, w);
  }
#pragma unroll
  for (int w = 0; w < kZWords; ++w) atomicAdd(&sum[w], words[w]);
  if (bad) atomicOr(&nan, 1u);
  __syncthreads();
  if (threadIdx.x == 0) {
    open_pass(sched, slot, advance, ee, ee_iters, mom0, mom1);
    for (int w = 0; w < kZWords; ++w) sched->zacc[slot][w] = sum[w];
    sched->zbad[slot] = nan;
  }
}

template <int W, int RI>
size_t smem_bytes() {
  constexpr int T = W * 32 * RI;
  return (size_t)T * (sizeof(float4) + sizeof(float2));
}

template <int W, int RI>
tsgne_status prepare() {
  const int most = (int)smem_bytes<W, RI>();
  constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  TS_CUDA(cudaFuncSetAttribute(k_repulsion_sym<W, RI, float2, true>, attr, most));
  TS_CUDA(cudaFuncSetAttribute(k_repulsion_sym<W, RI, bf162, true>, attr, most));
  TS_CUDA(cudaFuncSetAttribute(k_repulsion_sym<W, RI, float2, false>, attr, most));
  TS_CUDA(cudaFuncSetAttribute(k_repulsion_sym<W, RI, bf162, false>, attr, most));
  return TSGNE_OK;
}

struct PassArgs {
  const RepShape* sh;
  int n;
  const void* Y;
  int y_bf16;
  unsigned long long* acc;
  double* zunit;  // NULL: a whole pass
  Sched* sched;
  int slot, u0, u1, advance;
  float ee;
  int ee_iters;
  float mom0, mom1;
};

template <int W, int RI, class YT>
void launch(const PassArgs& p, int grid, cudaStream_t s) {
  auto kernel = p.sh->split == 1 ? k_repulsion_sym<W, RI, YT, true> : k_repulsion_sym<W, RI, YT, false>;
  kernel<<<grid, W * 32, p.sh->smem, s>>>(static_cast<const YT*>(p.Y), p.n, p.sh->chunks, p.sh->split, p.acc,
                                          fix_scale(p.n), p.zunit, p.sched, p.slot, p.u0, p.u1, p.advance, p.ee,
                                          p.ee_iters, p.mom0, p.mom1);
}

template <class YT>
tsgne_status dispatch_t(const PassArgs& p, cudaStream_t s) {
  const RepShape& sh = *p.sh;
  const int units = p.u1 - p.u0;
  const int grid = units < sh.grid ? units : sh.grid;
  if (sh.small)
    k_repulsion_small<YT><<<units, 32 * kSmallWarps, 0, s>>>(static_cast<const YT*>(p.Y), p.n, p.acc,
                                                             fix_scale(p.n), p.zunit, p.sched, p.slot, p.u0,
                                                             p.advance, p.ee, p.ee_iters, p.mom0, p.mom1);
  else if (sh.warps == 2 && sh.R == 16)
    launch<2, 16, YT>(p, grid, s);
  else if (sh.warps == 1 && sh.R == 16)
    launch<1, 16, YT>(p, grid, s);
  else if (sh.warps == 2 && sh.R == 8)
    launch<2, 8, YT>(p, grid, s);
  else if (sh.warps == 1 && sh.R == 8)
    launch<1, 8, YT>(p, grid, s);
  else {
    last_msg() = "no compiled repulsion shape with these warps / i-points per lane";
    return TSGNE_ERR_INVALID_ARG;
  }
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

tsgne_status dispatch(const PassArgs& p, cudaStream_t s) {
  return p.y_bf16 ? dispatch_t<bf162>(p, s) : dispatch_t<float2>(p, s);
}

}  // namespace

RepShape repulsion_shape_sym_fixed(int n, int sm_count, int W, int RI) {
  RepShape sh;
  if (n <= kSmallPoints) {
    sh.small = true;
    sh.warps = kSmallWarps;
    sh.block = 32 * kSmallWarps;
    sh.R = 2;
    sh.jtile = small_chunk(n);
    sh.chunks = small_chunks(n);
    sh.n_iblk = (n + kSmallBlock - 1) / kSmallBlock;
    sh.n_jtiles = sh.chunks;
    sh.n_pad = sh.n_iblk * kSmallBlock;
    sh.units = small_units(n);
    sh.grid = sh.units;
    return sh;
  }
  if (n <= kMidPoints) {
    W = 1;
    RI = 8;
  }
  const int T = 32 * RI * W;
  const int nt = (n + T - 1) / T;
  const int pairs = tile_pairs(nt);
  const int slots = sm_count * (warps_per_sm(RI) / W);
  sh.warps = W;
  sh.block = 32 * W;
  sh.R = RI;
  sh.split = split_tiles(pairs, slots, RI);
  sh.jtile = T / sh.split;
  sh.chunks = nt;
  sh.n_pad = nt * T;
  sh.n_iblk = nt;
  sh.n_jtiles = nt * sh.split;
  sh.units = pairs * sh.split;
  sh.grid = sh.units < slots ? sh.units : slots;
  sh.smem = (size_t)sh.jtile * (sizeof(float4) + sizeof(float2));
  return sh;
}

// The default shape: 16 i-points per lane (above kMidPoints), with 2-warp
// CTAs once their tile pairs make 7 waves (one and two warps: 1,206 and 1,249
// us at 80,000 points, 1,876 and 1,803 at 100,000).
RepShape repulsion_shape_sym(int n, int sm_count) {
  const long nt = ((long)n + 64 * kRI - 1) / (64 * kRI);
  const bool two = nt * (nt + 1) / 2 >= 7L * sm_count * (kWarpsPerSm / 2);
  return repulsion_shape_sym_fixed(n, sm_count, two ? 2 : 1, kRI);
}

tsgne_status repulsion_sym_prepare(const RepShape& sh) {
  if (sh.small) return TSGNE_OK;
  if (sh.warps == 2 && sh.R == 16) return prepare<2, 16>();
  if (sh.warps == 1 && sh.R == 16) return prepare<1, 16>();
  if (sh.warps == 2 && sh.R == 8) return prepare<2, 8>();
  if (sh.warps == 1 && sh.R == 8) return prepare<1, 8>();
  last_msg() = "no compiled repulsion shape with these warps / i-points per lane";
  return TSGNE_ERR_INVALID_ARG;
}

tsgne_status launch_repulsion_sym(const RepShape& sh, int n, const void* Y, int y_bf16, unsigned long long* acc,
                                  Sched* sched, int slot, int advance, float ee, int ee_iters, float mom0,
                                  float mom1, cudaStream_t s) {
  return dispatch(PassArgs{&sh, n, Y, y_bf16, acc, nullptr, sched, slot, 0, sh.units, advance, ee, ee_iters, mom0,
                           mom1},
                  s);
}

tsgne_status launch_repulsion_sym_units(const RepShape& sh, int n, const void* Y, int y_bf16,
                                        unsigned long long* acc, double* zpart, Sched* sched, int slot, int u0,
                                        int u1, cudaStream_t s) {
  if (u1 <= u0) return TSGNE_OK;
  return dispatch(PassArgs{&sh, n, Y, y_bf16, acc, zpart, sched, slot, u0, u1, 0, 1.f, 0, 0.f, 0.f}, s);
}

tsgne_status launch_finalize_z(const RepShape& sh, const double* zpart, Sched* sched, int slot, int advance, float ee,
                               int ee_iters, float mom0, float mom1, cudaStream_t s) {
  k_finalize_z<<<1, 1024, 0, s>>>(zpart, sh.units, sched, slot, advance, ee, ee_iters, mom0, mom1);
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

}  // namespace tsgne
