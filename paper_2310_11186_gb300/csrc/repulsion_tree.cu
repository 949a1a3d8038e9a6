// Tree-code approximation of the repulsive sums and of Z (an extension: the
// paper sums Eq. 4 exactly, at O(|V|^2) cost, Sec. 2.1 "Time complexity").
//
// Definition (the oracle restates the same steps in plain C):
//  1. bounding square of the layout (FP32): lo = (min x, min y), side = the
//     longer extent (floored at 1e-30); scale = 2^32 / side in FP64;
//  2. cell of a point per axis = trunc((v - lo) * scale) in FP64, clamped
//     to [0, 2^32 - 1]; key = 64-bit Morton interleave (x in the even bits).
//     32 bits per axis keep the bulk resolved when a few outliers stretch
//     the square to thousands of times its size;
//  3. points sorted by (key, index); sorted position k has the 96-bit
//     augmented key (key, k);
//  4. the binary radix tree of the augmented keys (a node over positions
//     [f, l] splits at the highest bit in which keys f and l differ);
//  5. node summaries in FP32: coordinate sums (left + right), box, centre =
//     sums / count, r2 = (longer box side)^2;
//  6. groups: the maximal subtrees of at most 32 points (nodes of <= 32
//     points whose parent has more), in sorted order -- compact Morton
//     cells, so no group box straddles a jump of the curve;
//  7. per group, a depth-first walk from the root, left child first: a leaf
//     is an exact interaction; a node whose r2 < theta^2 d2 (d = distance
//     from its centre to the group box) is one interaction of weight count
//     at its centre; an opened node of at most kTreeBucket points is
//     summed exactly over its points; other nodes are opened.
// Every decision (keys, tree shape, acceptance) is taken with IEEE FP32 /
// FP64 operations written as _rn intrinsics, so no FMA contraction changes
// it and the CPU reference takes the same decisions.
//
// GPU mapping.  Keys: one thread per point, which also counts the digits of
// all eight sort passes.  Sort: LSD radix sort, 8 stable passes of 8 bits,
// one launch each: a CTA ranks a tile of 2048 keys (ballots within warps,
// offsets across warps) and takes the tile's global offsets from the
// tiles before it by a decoupled look-back (a bounded wait).  The last pass
// also gathers the layout into sorted order.  Tree, summaries and group
// starts: bottom up in shared memory, tile by tile, one thread per leaf climbing
// (each node's parent follows from two neighbouring key prefixes) until it is the
// first of two children to arrive; the marks of the group starts are then listed.
// Walk: a persistent grid takes groups from a queue, one warp per group,
// lane = point; per round the lanes decide up to 32 stack entries at once and
// then all apply the round's accepted nodes and exact points, so the dependent
// node loads along the tree are issued 32 at a time.  Z: FP32 partial sums of a
// round, added without loss into a pair of FP32 sums per lane, the pairs over
// the warp's lanes, and every group's total as an exact integer (zsum.cuh) --
// the same bits in whatever order groups finish.
#include <cmath>

#include "f32x2.cuh"
#include "reduce.cuh"
#include "tsgne_internal.cuh"
#include "zsum.cuh"

namespace tsgne {

namespace {

constexpr int kRadixPasses = 8;  // 8-bit digits of the 64-bit keys
constexpr int kRadixBins = 256;
constexpr int kSortTile = 2048;  // keys per tile (per CTA)
constexpr int kWalkWarps = 8;

__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ---------------------------------------------------------- 1. bounding box

// Min / max over a 256-thread CTA (exact in any order); valid in thread 0.
__device__ __forceinline__ float4 block_box(float lx, float ly, float hx, float hy, float4* ws) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  lx = warp_min(lx);
  ly = warp_min(ly);
  hx = warp_max(hx);
  hy = warp_max(hy);
  if (lane == 0) ws[w] = make_float4(lx, ly, hx, hy);
  __syncthreads();
  float4 b = ws[0];
  if (threadIdx.x == 0)
    for (int k = 1; k < 8; ++k) {
      b.x = fminf(b.x, ws[k].x);
      b.y = fminf(b.y, ws[k].y);
      b.z = fmaxf(b.z, ws[k].z);
      b.w = fmaxf(b.w, ws[k].w);
    }
  __syncthreads();
  return b;
}

// Also clears the sort's digit counts, tile counters and tile status words
// (zero[0..nzero)), the group starts, the number of groups and the stall mark
// for the build that follows.
__global__ void __launch_bounds__(256) k_tree_box(const float2* __restrict__ Y, int n, float4* __restrict__ part,
                                                  TreeState* st, uint32_t* __restrict__ zero, int64_t nzero,
                                                  uint32_t* __restrict__ starts) {
  __shared__ float4 ws[8];
  for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < nzero; k += (int64_t)gridDim.x * 256) zero[k] = 0u;
  for (int k = blockIdx.x * 256 + threadIdx.x; k <= n / 32; k += gridDim.x * 256) starts[k] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->sort_stall = 0u;
    st->groups = 0u;
    st->climb_global = 0u;
  }
  float lx = INFINITY, ly = INFINITY, hx = -INFINITY, hy = -INFINITY;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
    const float2 p = Y[i];
    lx = fminf(lx, p.x);
    ly = fminf(ly, p.y);
    hx = fmaxf(hx, p.x);
    hy = fmaxf(hy, p.y);
  }
  float4 b = block_box(lx, ly, hx, hy, ws);
  if (threadIdx.x == 0) part[blockIdx.x] = b;
  if (arrive_last(&st->box_done)) {
    lx = ly = INFINITY;
    hx = hy = -INFINITY;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) {
      const float4 q = __ldcg(part + k);
      lx = fminf(lx, q.x);
      ly = fminf(ly, q.y);
      hx = fmaxf(hx, q.z);
      hy = fmaxf(hy, q.w);
    }
    b = block_box(lx, ly, hx, hy, ws);
    if (threadIdx.x == 0) {
      const float side = fmaxf(fmaxf(__fsub_rn(b.z, b.x), __fsub_rn(b.w, b.y)), 1e-30f);
      st->lo_x = b.x;
      st->lo_y = b.y;
      st->scale = __ddiv_rn(4294967296.0, (double)side);
    }
  }
}

// ---------------------------------------------------------------- 2. keys

__device__ __forceinline__ uint64_t spread32(uint32_t v) {
  uint64_t x = v;
  x = (x | (x << 16)) & 0x0000ffff0000ffffull;
  x = (x | (x << 8)) & 0x00ff00ff00ff00ffull;
  x = (x | (x << 4)) & 0x0f0f0f0f0f0f0f0full;
  x = (x | (x << 2)) & 0x3333333333333333ull;
  x = (x | (x << 1)) & 0x5555555555555555ull;
  return x;
}

__device__ __forceinline__ uint32_t cell32(float v, double lo, double scale) {
  const double c = __dmul_rn(__dsub_rn((double)v, lo), scale);
  if (!(c >= 0.0)) return 0u;
  if (c >= 4294967295.0) return 0xffffffffu;
  return (uint32_t)c;
}

// Keys and the identity permutation, plus the counts of every 8-bit digit
// of every key for all eight passes at once (ghist[pass][digit], zeroed by
// k_tree_box): one read of the layout serves the whole sort.  One large CTA
// per SM: the counts of a CTA are 2,048 global additions, and the FP64 pipe
// (14 instructions per point and warp, 16 cycles each) needs warps to overlap
// with (300,000 points: 13.7 us with 8 warps per SM, 11.2 us with 32).
constexpr int kKeyThreads = 1024;
__global__ void __launch_bounds__(kKeyThreads) k_tree_keys(const float2* __restrict__ Y, int n,
                                                   const TreeState* __restrict__ st, uint64_t* __restrict__ keys,
                                                   int32_t* __restrict__ vals, uint32_t* __restrict__ ghist) {
  __shared__ uint32_t h[kRadixPasses * kRadixBins];
  for (int k = threadIdx.x; k < kRadixPasses * kRadixBins; k += kKeyThreads) h[k] = 0u;
  __syncthreads();
  const double lx = st->lo_x, ly = st->lo_y, sc = st->scale;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float2 p = Y[i];
    const uint64_t key = spread32(cell32(p.x, lx, sc)) | (spread32(cell32(p.y, ly, sc)) << 1);
    keys[i] = key;
    vals[i] = i;
#pragma unroll
    for (int q = 0; q < kRadixPasses; ++q) atomicAdd(&h[q * kRadixBins + (int)((key >> (8 * q)) & 255u)], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < kRadixPasses * kRadixBins; k += kKeyThreads)
    if (h[k]) atomicAdd(ghist + k, h[k]);
}

// ---------------------------------------------------------------- 3. sort

// One stable pass of the LSD radix sort, digit (key >> 8 pass) & 255, as a
// single launch (one-sweep: the digit counts of all passes come from
// k_tree_keys; the offsets of a tile come from its predecessors through a
// decoupled look-back, Merrill & Garland's single-pass prefix scan, instead
// of a separate count / scan / scatter per pass).
//
// A CTA takes tiles in launch order from a counter (ctl[pass]), so it only
// ever waits on tiles that running CTAs own.  Tile t covers keys
// [t T, t T + T), T = kSortTile; warp w holds K = T / (32 kWarps) rounds of 32
// keys, w 32 K + 32 r + lane, r < K, so (w, r, lane) order is input order.
//  1. ranks within the warp: per round of 32 keys eight ballots, one per bit of
//     the digit, group equal digits (__match_any_sync takes longer for 32
//     digits that mostly differ: an iteration of 2,097,152 points 1466 us, 1439
//     with ballots); rank = running count of the digit in the warp + the number
//     of lower lanes with the same digit;
//  2. per digit d (thread d): the warps' exclusive offsets and the tile's
//     count c_d, published at once as status[pass][t][d] = (AGG, c_d)
//     (tile 0: (INCL, c_d));
//  3. look-back, thread d: walk tiles t-1, t-2, ... (8 status words loaded
//     at once) adding AGG counts until an INCL one (the inclusive count of
//     digit d over all tiles before);
//     then publish (INCL, excl + c_d).  A wait for a tile that has published
//     nothing yet spins at most `budget` clock cycles; past that the pass
//     records sort_stall and publishes what it has, so no wait chains on it,
//     every later kernel of the build sees the stall and does nothing, and
//     the walk reports kFlagWaitTimeout;
//  4. keys staged in shared memory in (digit, input) order, then written
//     out: element i of the staged tile, digit d, goes to
//     digit_start[d] + excl_d + (i - local_start[d]), so consecutive threads
//     write consecutive addresses inside a digit's run.
// With Y != NULL (last pass) the layout is gathered into sorted order.
// status words: bits 31..30 flag (0 empty, 1 AGG, 2 INCL), 29..0 count
// (n < 2^30).
constexpr uint32_t kStAgg = 1u << 30, kStIncl = 2u << 30, kStCount = (1u << 30) - 1u;
constexpr int kLookWindow = 8;  // predecessor tiles a look-back step reads at once

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u32(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Exclusive scans over the threads of a CTA of two values at once
// (thread x gets the sums over threads < x).
__device__ __forceinline__ void block_excl_scan2(uint32_t a, uint32_t b, uint32_t& ea, uint32_t& eb,
                                                 uint2* wsum) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t ia = a, ib = b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t ua = __shfl_up_sync(0xffffffffu, ia, o), ub = __shfl_up_sync(0xffffffffu, ib, o);
    if (lane >= o) {
      ia += ua;
      ib += ub;
    }
  }
  if (lane == 31) wsum[w] = make_uint2(ia, ib);
  __syncthreads();
  uint32_t oa = 0u, ob = 0u;
  for (int v = 0; v < w; ++v) {
    oa += wsum[v].x;
    ob += wsum[v].y;
  }
  ea = oa + ia - a;
  eb = ob + ib - b;
}

template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
    k_radix_onesweep(const uint64_t* __restrict__ kin, const int32_t* __restrict__ vin, int n, int pass,
                     const uint32_t* __restrict__ ghist, uint32_t* ctl, uint32_t* status, int ntiles,
                     long long budget, TreeState* st, uint64_t* __restrict__ kout, int32_t* __restrict__ vout,
                     const float2* __restrict__ Y, float2* __restrict__ ys) {
  constexpr int kThreads = 32 * kWarps, kItems = kSortTile / kThreads;  // keys per lane
  static_assert(kThreads >= kRadixBins, "the look-back maps one thread to one digit");
  __shared__ uint32_t hw[kWarps][kRadixBins];
  __shared__ uint64_t skey[kSortTile];
  __shared__ int32_t sval[kSortTile];
  __shared__ uint32_t lstart[kRadixBins], gbase[kRadixBins];
  __shared__ uint2 wsum[kWarps];
  __shared__ int tile_s;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  if (tid == 0) tile_s = (int)atomicAdd(ctl + pass, 1u);
  for (int k = tid; k < kWarps * kRadixBins; k += kThreads) (&hw[0][0])[k] = 0u;
  // up to here beside the end of the pass before (its CTAs release this launch
  // after their own wait, so everything older is complete)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
  if (__ldcg(&st->sort_stall)) return;  // an earlier pass gave up: nothing of this build is valid
  const int t = tile_s;
  if (t >= ntiles) return;  // uniform: more CTAs than tiles never happens, kept as a guard
  const int64_t t0 = (int64_t)t * kSortTile;
  const int tn = (int)min((int64_t)kSortTile, (int64_t)n - t0);
  const int shift = 8 * pass;
  const uint32_t lt = (1u << lane) - 1u;
  const int wb = w * (32 * kItems) + lane;
  uint64_t key[kItems];
  int32_t val[kItems];
  uint32_t rk[kItems];
#pragma unroll
  for (int r = 0; r < kItems; ++r) {  // all loads of the tile in flight at once
    const int i = wb + 32 * r;
    key[r] = i < tn ? kin[t0 + i] : 0ull;
    val[r] = i < tn ? vin[t0 + i] : 0;
  }
  // 1. ranks within the warp
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const bool valid = wb + 32 * r < tn;
    const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
    uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool one = (d >> q) & 1u;
      const uint32_t ones = __ballot_sync(0xffffffffu, one);
      peers &= one ? ones : ~ones;
    }
    const uint32_t before = valid ? hw[w][d] : 0u;
    rk[r] = before + (uint32_t)__popc(peers & lt);
    __syncwarp();
    if (valid && (peers & lt) == 0u) hw[w][d] = before + (uint32_t)__popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // 2. per digit: offsets of the warps, count of the tile, published
  const int d = tid;
  const bool digit = kThreads == kRadixBins || d < kRadixBins;
  uint32_t cnt = 0u;
  if (digit) {
#pragma unroll
    for (int v = 0; v < kWarps; ++v) {
      const uint32_t x = hw[v][d];
      hw[v][d] = cnt;
      cnt += x;
    }
  }
  uint32_t* const sbase = status + (size_t)pass * ntiles * kRadixBins;
  if (digit) st_relaxed_u32(sbase + (size_t)t * kRadixBins + d, (t == 0 ? kStIncl : kStAgg) | cnt);
  uint32_t dstart, lst;
  block_excl_scan2(digit ? __ldg(ghist + pass * kRadixBins + d) : 0u, cnt, dstart, lst, wsum);
  // 3. look-back
  uint32_t excl = 0u;
  if (t > 0 && digit) {
    const long long c0 = clock64();
    bool stalled = false, done = false;
    // windows of kLookWindow predecessors, loaded at once, read nearest first
    for (int k = t - 1; !done && !stalled; k -= kLookWindow) {
      uint32_t sw[kLookWindow];
#pragma unroll
      for (int u = 0; u < kLookWindow; ++u)
        sw[u] = k - u >= 0 ? ld_relaxed_u32(sbase + (size_t)(k - u) * kRadixBins + d) : kStIncl;
#pragma unroll
      for (int u = 0; u < kLookWindow; ++u) {
        uint32_t v = sw[u];
        while ((v >> 30) == 0u) {  // tile k - u (>= 0: tiles < 0 read as INCL 0) has published nothing yet
          if (clock64() - c0 > budget) {
            stalled = true;
            break;
          }
          v = ld_relaxed_u32(sbase + (size_t)(k - u) * kRadixBins + d);
        }
        if (stalled) break;
        excl += v & kStCount;
        if ((v & kStIncl) != 0u) {  // tile 0 always publishes INCL
          done = true;
          break;
        }
      }
    }
    if (stalled) atomicExch(&st->sort_stall, 1u);
    st_relaxed_u32(sbase + (size_t)t * kRadixBins + d, kStIncl | ((excl + cnt) & kStCount));
  }
  if (digit) {
    gbase[d] = dstart + excl;
    lstart[d] = lst;
  }
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;");  // the next pass may set up beside the writes
  // 4. stage in (digit, input) order, then write out
#pragma unroll
  for (int r = 0; r < kItems; ++r)
    if (wb + 32 * r < tn) {
      const uint32_t dg = (uint32_t)(key[r] >> shift) & 255u;
      const uint32_t lp = lstart[dg] + hw[w][dg] + rk[r];
      skey[lp] = key[r];
      sval[lp] = val[r];
    }
  __syncthreads();
  for (int i = tid; i < tn; i += kThreads) {
    const uint64_t kk = skey[i];
    const uint32_t dg = (uint32_t)(kk >> shift) & 255u;
    const uint32_t pos = gbase[dg] + ((uint32_t)i - lstart[dg]);
    if (pos < (uint32_t)n) {  // always true unless a wait ran out
      const int32_t v = sval[i];
      kout[pos] = kk;
      vout[pos] = v;
      if (ys != nullptr && (uint32_t)v < (uint32_t)n) ys[pos] = Y[v];
    }
  }
}

// ---------------------------------------------------------------- 4. tree

// Tree, summaries and group starts bottom up (agglomerative construction of the
// binary radix tree, Apetrei 2014): the thread of leaf k holds a node with
// range [L, R] and climbs.  The parent of [L, R] is the node split between R
// and R + 1 if the augmented keys R, R + 1 share a longer prefix than keys
// L - 1, L (a range end counts as -1), else the node split between L - 1 and L;
// this gives exactly the tree of the definition (the one whose node over
// [f, l] splits at the highest differing bit).  Internal node ids are their
// split positions (node g has children over [f, g] and [g + 1, l]); leaves are
// ~position.  A child reaching its parent exchanges (the end of the parent's
// range it knows, its own id) with the parent's slot: the first arrival
// leaves, the second learns the sibling, computes the parent (left + right:
// FP32 addition is commutative, so it does not matter which child's thread
// that is) and climbs on.  A completed node of more than kGroupMax points marks
// the first positions of its children that hold at most kGroupMax (the groups:
// maximal subtrees of at most kGroupMax points).
//
// A climb is a chain of exchanges, 32 deep for 300,000 spread points.  Through
// L2 an exchange with its fence and the load of the sibling's summary take
// 2 us, so nearly all of them are made in shared memory, over tiles of
// at most 1,024 consecutive nodes:
//   1. the leaves: a tile builds every node whose range lies inside it and
//      hands on the rest of its forest, about 11 subtrees;
//   2. while there are more than kUpTiles tiles: the subtrees of kUpTiles tiles
//      each, likewise;
//   3. what is left, by one CTA.
// The finished nodes are written afterwards, thread j the one split before
// starting node j: side by side, and all divisions at once (written in the climb,
// each exchange waits for the stores: 66 us for 300,000 points instead of 52).
// Whether a node's parent lies inside the tile is known beforehand: it does not
// exactly if the prefix it splits at is also shared with the key beyond the
// tile's end, i.e. if no shorter prefix lies between (a running minimum over
// the tile).  If a tile of steps 2 or 3 would hold more than 1,024 subtrees
// (points nested around the tiles' ends; one tile can leave 193), step 3
// climbs from all subtrees of step 1 through global memory instead.
// 300,000 points: 69 us with every exchange in L2, 17 + 14 + 11 us now; 2,097,152
// points: 237 us, 85 + 15 + 14 us now.
constexpr int kGroupMax = 32;
constexpr unsigned long long kSlotEmpty = ~0ull;

// Common-prefix length of the augmented keys (ka, a) and (kb, b).
__device__ __forceinline__ int aug_prefix(uint64_t ka, uint64_t kb, int a, int b) {
  return ka != kb ? __clzll((long long)(ka ^ kb)) : 64 + __clz((uint32_t)a ^ (uint32_t)b);
}

__device__ __forceinline__ void mark_start(uint32_t* starts, int k) { atomicOr(starts + (k >> 5), 1u << (k & 31)); }

// Where finished nodes go.
struct TreeOut {
  float4* nodeA;
  int4* nodeB;
  uint32_t* starts;
  TreeState* st;
};

// The node split after position p with range [pL, pR], children left and right.
__device__ __forceinline__ void put_node(const TreeOut& o, int p, int pL, int pR, int left, int right, float4 box,
                                         float2 sum) {
  const int count = pR - pL + 1;
  const float cnt = (float)count;
  const float r = fmaxf(__fsub_rn(box.z, box.x), __fsub_rn(box.w, box.y));
  o.nodeA[p] = make_float4(__fdiv_rn(sum.x, cnt), __fdiv_rn(sum.y, cnt), __fmul_rn(r, r), cnt);
  o.nodeB[p] = make_int4(left, right, pL, pR);
  if (count > kGroupMax) {
    if (p - pL + 1 <= kGroupMax) mark_start(o.starts, pL);  // left child [pL, p]
    if (pR - p <= kGroupMax) mark_start(o.starts, p + 1);   // right child [p + 1, pR]
  }
}
__device__ __forceinline__ void put_root(const TreeOut& o, int id, int count) {
  o.st->root = id;
  if (count <= kGroupMax) mark_start(o.starts, 0);
}
__device__ __forceinline__ float4 box_union(float4 a, float4 b) {
  return make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
}

// Subtrees handed on by tiles: tile t's are entries t kItemCap ... in
// position order, counts[t] of them.
constexpr int kTileLeaves = 1024;  // nodes a tile starts from, one per thread
constexpr int kItemCap = 256;      // a tile leaves at most 2 * 96 + 1 subtrees: one per prefix length and side
constexpr int kUpTiles = 48;       // tiles whose subtrees one CTA of step 2 joins (about 520)
struct Items {
  int4* at;  // first, last position, id
  float4* box;
  float2* sum;
  int32_t* counts;
};

// Shared memory of a tile.  Boundary j lies between nodes j - 1 and j.
struct ClimbTile {
  uint32_t slot[kTileLeaves];            // exchange at boundary j: far end << 16 | ref
  float4 box[kTileLeaves];               // of the node built at boundary j
  float4 ibox[kTileLeaves];              // of starting node j
  float2 sum[kTileLeaves], isum[kTileLeaves];
  ushort2 child[kTileLeaves];            // refs of the children of the node built at boundary j
  short2 ends[kTileLeaves];              // starting nodes it reaches from and to (y < 0: none built)
  int32_t first[kTileLeaves], last[kTileLeaves], id[kTileLeaves];  // of starting node j
  int8_t d[kTileLeaves + 1];   // common prefix across boundary j (-1: no key beyond)
  int8_t dl[kTileLeaves + 1];  // least of d[0..j]
  int8_t dr[kTileLeaves + 1];  // least of d[j..c]
  uint32_t on[kTileLeaves];    // subtree from starting node j that is handed on: to << 16 | ref
  uint32_t more[kTileLeaves];  // climbs that go on: from << 22 | to << 12 | ref (11 bits, kBuilt as bit 10)
  int32_t wl[32], wr[32];
  uint32_t nmore;
};

// Exclusive scan of v over the CTA's 1,024 threads; *total its sum.
__device__ __forceinline__ int climb_scan(ClimbTile& t, int v, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) t.wl[w] = inc;
  __syncthreads();
  if (w == 0) {
    int u = t.wl[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int p = __shfl_up_sync(0xffffffffu, u, o);
      if (lane >= o) u += p;
    }
    t.wl[lane] = u;
  }
  __syncthreads();
  const int before = (w > 0 ? t.wl[w - 1] : 0) + inc - v;
  *total = t.wl[31];
  __syncthreads();
  return before;
}

// Running minima of d over the boundaries 0..c (c <= 1,024; boundary 0 apart).
__device__ __forceinline__ void climb_minima(ClimbTile& t, int c) {
  const int x = threadIdx.x, lane = x & 31, w = x >> 5;
  // prefix: thread x covers boundary x; suffix: boundary x + 1
  int a = x <= c ? t.d[x] : 127, b = x + 1 <= c ? t.d[x + 1] : 127;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, a, o), v = __shfl_down_sync(0xffffffffu, b, o);
    if (lane >= o) a = min(a, u);
    if (lane + o < 32) b = min(b, v);
  }
  if (lane == 31) t.wl[w] = a;
  if (lane == 0) t.wr[w] = b;
  __syncthreads();
  if (w == 0) {
    int u = t.wl[lane], v = t.wr[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int p = __shfl_up_sync(0xffffffffu, u, o), q = __shfl_down_sync(0xffffffffu, v, o);
      if (lane >= o) u = min(u, p);
      if (lane + o < 32) v = min(v, q);
    }
    t.wl[lane] = u;
    t.wr[lane] = v;
  }
  __syncthreads();
  if (w > 0) a = min(a, t.wl[w - 1]);
  if (w < 31) b = min(b, t.wr[w + 1]);
  if (x <= c) t.dl[x] = (int8_t)a;
  if (x + 1 <= c) t.dr[x + 1] = (int8_t)b;
  __syncthreads();
}

// Order of a thread's shared memory accesses around an exchange.  (No store to
// global memory is in flight in the climb: the fence would wait for it.)
__device__ __forceinline__ void fence_cta() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

constexpr uint32_t kBuilt = 0x8000u;
__device__ __forceinline__ int ref_id(const ClimbTile& t, uint32_t ref) {
  return ref & kBuilt ? t.last[(ref & ~kBuilt) - 1] : t.id[ref];
}

// At most `steps` exchanges of the climb from the node over starting nodes
// [a, b]; false once it has ended.
__device__ __forceinline__ bool climb_steps(ClimbTile& t, bool top, const TreeOut& o, int steps, int& a, int& b,
                                            uint32_t& ref) {
  float4 bc = ref & kBuilt ? t.box[ref & ~kBuilt] : t.ibox[ref];
  float2 sc = ref & kBuilt ? t.sum[ref & ~kBuilt] : t.isum[ref];
  for (int k = 0; k < steps; ++k) {
    const int dl = t.d[a], dr = t.d[b + 1];
    if (dl < 0 && dr < 0) {
      put_root(o, ref_id(t, ref), t.last[b] - t.first[a] + 1);
      return false;
    }
    const bool toward_right = dr > dl;  // this node is the left child
    if (!top && (toward_right ? dr == t.dr[b + 1] : dl == t.dl[a])) {
      t.on[a] = ((uint32_t)b << 16) | ref;
      return false;
    }
    const int j = toward_right ? b + 1 : a;  // the parent's boundary
    fence_cta();                             // the summary before the exchange
    const uint32_t old = atomicExch(&t.slot[j], ((uint32_t)(toward_right ? a : b) << 16) | ref);
    if (old == 0xffffffffu) return false;
    fence_cta();
    const uint32_t sref = old & 0xffffu;
    const float4 bs = sref & kBuilt ? t.box[sref & ~kBuilt] : t.ibox[sref];
    const float2 ss = sref & kBuilt ? t.sum[sref & ~kBuilt] : t.isum[sref];
    if (toward_right) b = (int)(old >> 16); else a = (int)(old >> 16);
    sc = make_float2(__fadd_rn(sc.x, ss.x), __fadd_rn(sc.y, ss.y));
    bc = box_union(bc, bs);
    t.box[j] = bc;
    t.sum[j] = sc;
    t.child[j] = toward_right ? make_ushort2(ref, sref) : make_ushort2(sref, ref);
    t.ends[j] = make_short2((short)a, (short)b);
    ref = kBuilt | (uint32_t)j;
  }
  return true;
}

// Climbs from the tile's c starting nodes, one per thread, whose first, last,
// id, ibox, isum and boundary prefixes are in shared memory.  ref: a node within
// the tile, starting node j (j) or the one built at boundary j (kBuilt | j).
// Subtrees whose parent reaches beyond the tile go to out (tile index tile);
// out.counts == NULL: the top, where none does.  An exchange ends one climb of
// two, so after kFirstSteps of them 1 in 15 is left: those go on side by side
// in full warps (all in their own warps: 32 warps issue each step to the end,
// 21 us for the leaves of 300,000 points instead of 17).
constexpr int kFirstSteps = 3;
__device__ void climb_tile(ClimbTile& t, int c, const TreeOut& o, Items out, int tile, float4* gbox, float2* gsum) {
  const int x = threadIdx.x;
  const bool top = out.counts == nullptr;
  t.slot[x] = 0xffffffffu;
  t.on[x] = 0xffffffffu;
  t.ends[x] = make_short2(0, -1);
  if (x == 0) t.nmore = 0u;
  climb_minima(t, c);
  int a = x, b = x;
  uint32_t ref = (uint32_t)x;
  if (x < c && climb_steps(t, top, o, kFirstSteps, a, b, ref))
    t.more[atomicAdd(&t.nmore, 1u)] =
        ((uint32_t)a << 22) | ((uint32_t)b << 12) | (ref & kBuilt ? 0x400u : 0u) | (ref & 0x3ffu);
  __syncthreads();
  if (x < (int)t.nmore) {
    const uint32_t m = t.more[x];
    a = (int)(m >> 22);
    b = (int)((m >> 12) & 0x3ffu);
    ref = (m & 0x3ffu) | (m & 0x400u ? kBuilt : 0u);
    climb_steps(t, top, o, kTileLeaves, a, b, ref);  // ends: each step takes in a starting node at least
  }
  __syncthreads();
  if (x < c && t.ends[x].y >= 0)
    put_node(o, t.last[x - 1], t.first[t.ends[x].x], t.last[t.ends[x].y], ref_id(t, t.child[x].x),
             ref_id(t, t.child[x].y), t.box[x], t.sum[x]);
  if (top) return;
  const uint32_t on = t.on[x];
  const bool hand_on = on != 0xffffffffu;
  int total;
  const int rank = climb_scan(t, hand_on ? 1 : 0, &total);
  if (hand_on) {
    ref = on & 0xffffu;
    const int id = ref_id(t, ref);
    const float4 bc = ref & kBuilt ? t.box[ref & ~kBuilt] : t.ibox[ref];
    const float2 sc = ref & kBuilt ? t.sum[ref & ~kBuilt] : t.isum[ref];
    if (rank < kItemCap) {
      const size_t at = (size_t)tile * kItemCap + rank;
      out.at[at] = make_int4(t.first[x], t.last[on >> 16], id, 0);
      out.box[at] = bc;
      out.sum[at] = sc;
    }
    if (id >= 0) {  // where the climb through global memory looks for it
      gbox[id] = bc;
      gsum[id] = sc;
    }
  }
  if (x == 0) out.counts[tile] = total;
}

// Prefix across the boundary after position r (-1 at the last key).
__device__ __forceinline__ int8_t prefix_after(const uint64_t* __restrict__ keys, int r, int n) {
  return r < n - 1 ? (int8_t)aug_prefix(keys[r], keys[r + 1], r, r + 1) : (int8_t)-1;
}

// Step 1: the leaves.
__global__ void __launch_bounds__(kTileLeaves)
    k_climb_leaves(int n, const uint64_t* __restrict__ keys, const float2* __restrict__ ys, TreeOut o, Items out,
                   float4* gbox, float2* gsum) {
  extern __shared__ __align__(16) unsigned char climb_smem[];
  ClimbTile& t = *reinterpret_cast<ClimbTile*>(climb_smem);
  if (__ldcg(&o.st->sort_stall)) return;
  const int x = threadIdx.x, t0 = (int)blockIdx.x * kTileLeaves;
  const int c = min(kTileLeaves, n - t0), k = t0 + x;
  if (x < c) {
    const float2 q = ys[k];
    t.ibox[x] = make_float4(q.x, q.y, q.x, q.y);
    t.isum[x] = q;
    t.first[x] = t.last[x] = k;
    t.id[x] = ~k;
    t.d[x + 1] = prefix_after(keys, k, n);
    if (x == 0) t.d[0] = t0 > 0 ? prefix_after(keys, t0 - 1, n) : (int8_t)-1;
  }
  __syncthreads();
  climb_tile(t, c, o, out, (int)blockIdx.x, gbox, gsum);
}

// Loads the subtrees of tiles [t0, t1) of `in` (t1 - t0 <= 1,024) into a tile;
// returns how many there are, nothing loaded above 1,024.
__device__ int load_items(ClimbTile& t, const Items& in, int t0, int t1, int n, const uint64_t* __restrict__ keys) {
  const int x = threadIdx.x;
  const int mine = t0 + x < t1 ? in.counts[t0 + x] : 0;
  int total;
  const int before = climb_scan(t, mine, &total);
  if (total > kTileLeaves) return total;
  int32_t* src = reinterpret_cast<int32_t*>(t.more);  // free until the climb
  for (int q = 0; q < mine; ++q) src[before + q] = (t0 + x) * kItemCap + q;
  __syncthreads();
  if (x < total) {
    const int4 it = in.at[src[x]];
    t.first[x] = it.x;
    t.last[x] = it.y;
    t.id[x] = it.z;
    t.ibox[x] = in.box[src[x]];
    t.isum[x] = in.sum[src[x]];
    t.d[x + 1] = prefix_after(keys, it.y, n);
    if (x == 0) t.d[0] = it.x > 0 ? prefix_after(keys, it.x - 1, n) : (int8_t)-1;
  }
  __syncthreads();
  return total;
}

// Step 2: the subtrees of kUpTiles tiles of the launch before.
__global__ void __launch_bounds__(kTileLeaves)
    k_climb_items(int n, const uint64_t* __restrict__ keys, Items in, int ntiles, TreeOut o, Items out, float4* gbox,
                  float2* gsum) {
  extern __shared__ __align__(16) unsigned char climb_smem[];
  ClimbTile& t = *reinterpret_cast<ClimbTile*>(climb_smem);
  if (__ldcg(&o.st->sort_stall)) return;
  const int t0 = (int)blockIdx.x * kUpTiles, t1 = min(ntiles, t0 + kUpTiles);
  // another CTA of this launch may be setting it: one thread looks for all
  const bool gave_up = __syncthreads_or(threadIdx.x == 0 && __ldcg(&o.st->climb_global) != 0u);
  const int c = gave_up ? 0 : load_items(t, in, t0, t1, n, keys);
  if (gave_up || c > kTileLeaves) {
    if (threadIdx.x == 0) {
      if (!gave_up) o.st->climb_global = 1u;
      out.counts[blockIdx.x] = 0;
    }
    return;
  }
  climb_tile(t, c, o, out, (int)blockIdx.x, gbox, gsum);
}

// Exchange at a node in global memory: acquire-release, so the summary a
// child's thread stored before its exchange is visible to the sibling's thread
// after its own.
__device__ __forceinline__ unsigned long long atom_exch_acq_rel(unsigned long long* p, unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.acq_rel.gpu.global.exch.b64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
  return old;
}

// The climb of subtree (L, R, id) through global memory to the root.
__device__ void climb_global(int n, const uint64_t* __restrict__ keys, const float2* __restrict__ ys,
                             unsigned long long* slot, float4* box, float2* sum, const TreeOut& o, int4 it, float4 bc,
                             float2 sc) {
  int L = it.x, R = it.y, id = it.z;
  for (;;) {
    const int dl = L > 0 ? prefix_after(keys, L - 1, n) : -1;
    const int dr = prefix_after(keys, R, n);
    if (dl < 0 && dr < 0) {
      put_root(o, id, R - L + 1);
      return;
    }
    const bool toward_right = dr > dl;
    const int p = toward_right ? R : L - 1;
    const unsigned long long old =
        atom_exch_acq_rel(slot + p, ((unsigned long long)(uint32_t)(toward_right ? L : R) << 32) | (uint32_t)id);
    if (old == kSlotEmpty) return;
    slot[p] = kSlotEmpty;  // both arrivals are in: ready for the next pass
    const int sid = (int)(uint32_t)old;
    float4 bs;
    float2 ss;
    if (sid < 0) {
      ss = ys[~sid];
      bs = make_float4(ss.x, ss.y, ss.x, ss.y);
    } else {
      bs = __ldcg(box + sid);
      ss = __ldcg(sum + sid);
    }
    if (toward_right) R = (int)(old >> 32); else L = (int)(old >> 32);
    sc = make_float2(__fadd_rn(sc.x, ss.x), __fadd_rn(sc.y, ss.y));
    bc = box_union(bc, bs);
    box[p] = bc;
    sum[p] = sc;
    put_node(o, p, L, R, toward_right ? id : sid, toward_right ? sid : id, bc, sc);
    id = p;
  }
}

// Step 3: the subtrees of all tiles of `in` by one CTA; or, if they are too
// many or a tile of step 2 gave up, those of step 1 (leaf) by all CTAs.
__global__ void __launch_bounds__(kTileLeaves)
    k_climb_top(int n, const uint64_t* __restrict__ keys, const float2* __restrict__ ys, Items in, int ntiles,
                Items leaf, int leaf_tiles, unsigned long long* slot, float4* gbox, float2* gsum, TreeOut o) {
  extern __shared__ __align__(16) unsigned char climb_smem[];
  ClimbTile& t = *reinterpret_cast<ClimbTile*>(climb_smem);
  if (__ldcg(&o.st->sort_stall)) return;
  int c = kTileLeaves + 1;
  if (ntiles <= kTileLeaves && !__ldcg(&o.st->climb_global)) c = load_items(t, in, 0, ntiles, n, keys);
  if (c <= kTileLeaves) {
    if (blockIdx.x == 0 && c > 0) climb_tile(t, c, o, Items{}, 0, gbox, gsum);
    return;
  }
  const int64_t entries = (int64_t)leaf_tiles * kItemCap, stride = (int64_t)gridDim.x * kTileLeaves;
  for (int64_t e = (int64_t)blockIdx.x * kTileLeaves + threadIdx.x; e < entries; e += stride)
    if ((int)(e % kItemCap) < leaf.counts[e / kItemCap])
      climb_global(n, keys, ys, slot, gbox, gsum, o, leaf.at[e], leaf.box[e], leaf.sum[e]);
}

// --------------------------------------------------------------- 6. groups

// The groups (first position, end) from the marks, one thread per 32
// positions; a CTA's groups are listed in order at a place of its own, CTAs in
// any order (nothing depends on it).  A group holds at most 32 points, so it
// ends at the next mark of its word or of the next one, or at n.
__global__ void __launch_bounds__(256) k_tree_groups(int n, TreeState* st, const uint32_t* __restrict__ starts,
                                                     int2* __restrict__ groups) {
  __shared__ uint2 wsum[8];
  __shared__ uint32_t base;
  if (__ldcg(&st->sort_stall)) return;
  const int words = (n + 31) / 32;
  const int w = blockIdx.x * 256 + threadIdx.x;
  const uint32_t m = w < words ? starts[w] : 0u;
  const uint32_t next = w + 1 < words ? starts[w + 1] : 0u;
  uint32_t at, unused;
  const uint32_t cnt = (uint32_t)__popc(m);
  block_excl_scan2(cnt, 0u, at, unused, wsum);
  if (threadIdx.x == 255) base = atomicAdd(&st->groups, at + cnt);
  __syncthreads();
  const int after = next ? 32 * (w + 1) + __ffs((int)next) - 1 : n;
  uint32_t left = m;
  for (uint32_t k = 0; k < cnt; ++k) {
    const int b = __ffs((int)left) - 1;
    left &= left - 1u;
    groups[base + at + k] = make_int2(32 * w + b, left ? 32 * w + __ffs((int)left) - 1 : after);
  }
}

// ---------------------------------------------------------------- 7. walk

// Walk of one group, 32 stack entries per round: each lane takes one entry
// (the top of the stack), loads its node record and decides: accept (r2 <
// theta^2 d2: one interaction of weight count at the centre), sum exactly
// (at most kTreeBucket points) or open (push both children).  Ballots
// compact the three outcomes into shared-memory lists in lane order; then
// every lane applies all accepted nodes and all exact points of the round
// to its own point.  A leaf (sorted position j) is the record (y_j, r2 = 0,
// count 1): accepting it is the exact interaction with its point, and it is
// never accepted by its own group (distance 0 to the box), which takes the
// exact path with the self term removed.  The set of interactions is the
// definition's; only the order of the sums differs from a depth-first walk.
// A round's interactions form one list: an accepted node is one item
// (centre, count), an exact entry is one item per point (point, 1).  The
// deciding lanes write their items at offsets from ballots over the item
// counts, as negated x, negated y and weight arrays, so two items are read as
// three FP32x2 words and go through the packed arithmetic unchanged.  A
// lane's own point, when an exact entry holds it, is summed like any other
// item: its force term is exactly zero (dx = dy = 0) and its Z term, 1 / (1 +
// 0) as computed, is subtracted once at the end (the entries mark which lanes
// they cover) instead of masking every item.  An accepted node may also hold
// the group's own points (coincident points: a centre one rounding away from
// them, a box of size zero); it is then one monopole term as the definition
// says, with nothing subtracted.
// Stack bound: a round that starts at <= kWalkStack - 200 entries pops up to
// 32 and pushes up to 64, ending at <= kWalkStack - 168; above kWalkStack -
// 200 rounds pop one entry (a depth-first walk, which adds at most one entry
// per tree level, and the tree has at most 94 levels: 64 key bits and 30
// index bits), so the stack stays below kWalkStack - 74.
constexpr int kWalkStack = 512;
static_assert(kTreeBucket <= 7, "a lane's items of a round are counted in three bits");
constexpr int kWalkList = 32 * kTreeBucket + 4;  // items of one round at most, plus padding (even)

// Two interactions at once: items (-x, -y, c) packed in pairs against p; FX,
// FY, Z hold two partial sums each.
__device__ __forceinline__ void interact2(u64 PX, u64 PY, u64 NX, u64 NY, u64 C, u64& FX, u64& FY, u64& Z) {
  const u64 dx = add2(PX, NX);
  const u64 dy = add2(PY, NY);
  u64 q = fma2(dx, dx, pk(1.0f, 1.0f));
  q = fma2(dy, dy, q);
  float q0, q1;
  upk(q, q0, q1);
  const u64 w = pk(rcp_approx(q0), rcp_approx(q1));
  const u64 cw = mul2(C, w);
  Z = add2(Z, cw);
  const u64 cw2 = mul2(cw, w);
  FX = fma2(cw2, dx, FX);
  FY = fma2(cw2, dy, FY);
}

// Sums without loss: two FP32 sums (s, e) whose exact sum is that of the terms
// up to about 2^-47 of it (Knuth's two-sum; e collects its errors).  Packed
// FP32x2 for the two halves a lane accumulates, scalar across lanes.  FP64
// would be as exact, but a double conversion or addition occupies the SM's FP64
// pipe for 16 cycles: with four a round it was 59 % busy and the walk waited
// for it (a walk over 300,000 spread
// points: 157 us, 139 us with these sums and the item counts from ballots).
__device__ __forceinline__ void two_sum2(u64& S, u64& E, u64 z) {
  const u64 m1 = pk(-1.f, -1.f);
  const u64 s = add2(S, z);
  const u64 b = fma2(S, m1, s);          // s - S
  const u64 a = fma2(b, m1, s);          // s - b
  const u64 e = add2(fma2(a, m1, S), fma2(b, m1, z));
  S = s;
  E = add2(E, e);
}
__device__ __forceinline__ void two_sum(float& s, float& e, float t, float te) {
  const float r = __fadd_rn(s, t);
  const float b = __fsub_rn(r, s);
  const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(r, b)), __fsub_rn(t, b));
  s = r;
  e = __fadd_rn(__fadd_rn(e, te), d);
}

__global__ void __launch_bounds__(32 * kWalkWarps, 4)
    k_tree_walk(int n, const float2* __restrict__ ys, const int32_t* __restrict__ perm,
                const float4* __restrict__ nodeA, const int4* __restrict__ nodeB, const int2* __restrict__ groups,
                float theta2, float2* __restrict__ frep, Sched* sched, TreeState* st, int advance, float ee,
                int ee_iters, float mom0, float mom1) {
  __shared__ int stk[kWalkWarps][kWalkStack];
  __shared__ __align__(8) float lnx[kWalkWarps][kWalkList];
  __shared__ __align__(8) float lny[kWalkWarps][kWalkList];
  __shared__ __align__(8) float lc[kWalkWarps][kWalkList];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  // A sort wait that ran out leaves no valid tree: the pass only zeroes the
  // forces and reports the timeout.
  const bool stalled = __ldcg(&st->sort_stall) != 0u;
  const int ngroups = stalled ? 0 : (int)__ldcg(&st->groups);
  const int root = __ldcg(&st->root);  // internal node id, or ~0 for a single point
  if (stalled)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
      frep[i] = make_float2(0.f, 0.f);
  for (;;) {
    int g = 0;
    if (lane == 0) g = (int)atomicAdd(&st->next_group, 1u);
    g = __shfl_sync(0xffffffffu, g, 0);
    if (g >= ngroups) break;
    const int2 gr = groups[g];
    const int k0 = gr.x, k1 = gr.y;
    const int k = k0 + lane;
    const bool act = k < k1;
    const float2 p = ys[act ? k : k0];
    const float gx0 = warp_min(p.x), gy0 = warp_min(p.y), gx1 = warp_max(p.x), gy1 = warp_max(p.y);
    const u64 PX = pk(p.x, p.x), PY = pk(p.y, p.y);
    u64 FX = 0ull, FY = 0ull;
    u64 ZS = 0ull, ZE = 0ull;
    bool overflow = false;
    uint32_t seen = 0u;  // lanes whose own point an exact entry held
    if (lane == 0) stk[w][0] = root;
    int sp = 1;
    while (sp > 0) {
      __syncwarp();
      const int take = sp > kWalkStack - 200 ? 1 : (sp < 32 ? sp : 32);
      const bool has = lane < take;
      const int v = has ? stk[w][sp - take + lane] : 0;
      sp -= take;
      int kind = 0;  // 1 accept, 2 exact, 3 open
      float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
      int4 B = make_int4(0, 0, 0, 0);
      const bool vok = !has || (v < 0 ? TS_IN(~v, 0, n, &sched->flags) : TS_IN(v, 0, n - 1, &sched->flags));
      if (has && vok) {
        if (v < 0) {
          const float2 q = ys[~v];
          A = make_float4(q.x, q.y, 0.f, 1.f);
          B = make_int4(-1, -1, ~v, ~v);
        } else {
          A = nodeA[v];
          B = nodeB[v];
        }
        const float dx = fmaxf(fmaxf(__fsub_rn(gx0, A.x), __fsub_rn(A.x, gx1)), 0.0f);
        const float dy = fmaxf(fmaxf(__fsub_rn(gy0, A.y), __fsub_rn(A.y, gy1)), 0.0f);
        const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
        kind = A.z < __fmul_rn(theta2, d2) ? 1 : (B.w - B.z + 1 <= kTreeBucket ? 2 : 3);
      }
      const uint32_t mo = __ballot_sync(0xffffffffu, kind == 3);
      // list offsets: the items per lane, summed over the lanes below bit by
      // bit; from ballots, so that the compiler knows the number of items to
      // be the same in every lane (uniform loop and addresses below: 5 %)
      const int cnt = kind == 1 ? 1 : (kind == 2 ? B.w - B.z + 1 : 0);
      int off = 0, ni = 0;
#pragma unroll
      for (int bit = 0; bit < 3; ++bit) {
        const uint32_t m = __ballot_sync(0xffffffffu, (cnt >> bit) & 1);
        off += __popc(m & lt) << bit;
        ni += __popc(m) << bit;
      }
      if (kind == 1 && TS_IN(off, 0, kWalkList, &sched->flags)) {
        lnx[w][off] = -A.x;
        lny[w][off] = -A.y;
        lc[w][off] = A.w;
      }
      uint32_t cover = 0u;
      if (kind == 2) {
#pragma unroll
        for (int u = 0; u < kTreeBucket; ++u)
          if (u < cnt && TS_IN(B.z + u, 0, n, &sched->flags) && TS_IN(off + u, 0, kWalkList, &sched->flags)) {
            const float2 q = ys[B.z + u];
            lnx[w][off + u] = -q.x;
            lny[w][off + u] = -q.y;
            lc[w][off + u] = 1.0f;
          }
        const int lo = max(B.z, k0) - k0, hi = min(B.w, k1 - 1) - k0;  // lanes whose points it holds
        if (lo <= hi) cover = ((1u << (hi - lo + 1)) - 1u) << lo;  // hi - lo < kTreeBucket
      }
      seen |= __reduce_or_sync(0xffffffffu, cover);
      if (lane == 0 && (ni & 1) && TS_IN(ni, 0, kWalkList, &sched->flags)) {  // pad to a whole pair with a zero-weight item
        lnx[w][ni] = 0.f;
        lny[w][ni] = 0.f;
        lc[w][ni] = 0.f;
      }
      __syncwarp();  // every lane has read its entry before the pushes reuse the slots
      const int npush = 2 * __popc(mo);
      if (sp + npush <= kWalkStack) {
        if (kind == 3 && TS_IN(sp + 2 * __popc(mo & lt) + 1, 0, kWalkStack, &sched->flags)) {
          const int slot = sp + 2 * __popc(mo & lt);
          stk[w][slot] = B.y;  // right below, left on top
          stk[w][slot + 1] = B.x;
        }
        sp += npush;
      } else {
        overflow = true;  // excluded by the bound above; recorded, never written past
      }
      __syncwarp();
      u64 Z = 0ull;
      for (int t = 0; t < ni && TS_IN(t + 1, 0, kWalkList, &sched->flags); t += 2)
        interact2(PX, PY, *reinterpret_cast<const u64*>(&lnx[w][t]), *reinterpret_cast<const u64*>(&lny[w][t]),
                  *reinterpret_cast<const u64*>(&lc[w][t]), FX, FY, Z);
      two_sum2(ZS, ZE, Z);
    }
    float zs, ze, z1, e1;
    upk(ZS, zs, z1);
    upk(ZE, ze, e1);
    two_sum(zs, ze, z1, e1);
    if ((seen >> lane) & 1u) two_sum(zs, ze, -rcp_approx(1.0f), 0.f);  // the lane's own term out
    if (!act) zs = ze = 0.f;                                          // idle lanes add nothing
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      two_sum(zs, ze, __shfl_xor_sync(0xffffffffu, zs, o), __shfl_xor_sync(0xffffffffu, ze, o));
    if (lane == 0) {
      const double z = (double)zs + (double)ze;
      z_add(st->zsum, z_fix(z));
      if (z != z) atomicOr(&st->zbad, 1u);
      if (overflow) atomicOr(&sched->flags, kFlagTreeOverflow);
    }
    if (act) {
      float fx0, fx1, fy0, fy1;
      upk(FX, fx0, fx1);
      upk(FY, fy0, fy1);
      if (TS_IN(perm[k], 0, n, &sched->flags)) frep[perm[k]] = make_float2(fx0 + fx1, fy0 + fy1);
    }
  }
  if (arrive_last(&st->walk_done)) {
    if (threadIdx.x == 0) {
      unsigned long long words[kZWords];
      for (int k = 0; k < kZWords; ++k) {
        words[k] = __ldcg(&st->zsum[k]);
        st->zsum[k] = 0ull;
      }
      const double total = z_value(words, __ldcg(&st->zbad), 0);
      st->zbad = 0u;
      st->next_group = 0u;
      if (stalled)
        atomicOr(&sched->flags, kFlagWaitTimeout);
      else {
        sched->Z = total;
        sched->inv_z = (float)(1.0 / total);
      }
      const int t = sched->t;
      sched->alpha = t < ee_iters ? ee : 1.0f;
      sched->mu = t < ee_iters ? mom0 : mom1;
      if (advance) sched->t = t + 1;
    }
  }
}

int grid_for(int64_t items, int per_block, int cap) {
  int64_t g = (items + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

}  // namespace

tsgne_status TreeBufs::alloc(int n_points, int sm_count, cudaStream_t s) {
  n = n_points;
  if (n >= (1 << 30)) {
    last_msg() = "the tree code takes fewer than 2^30 points";
    return TSGNE_ERR_INVALID_ARG;
  }
  ntiles = (n + kSortTile - 1) / kSortTile;
  box_blocks = grid_for(n, 256, 2 * sm_count);
  keys_blocks = grid_for(n, kKeyThreads, sm_count);
  int per_sm = 0;
  TS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tree_walk, 32 * kWalkWarps, 0));
  walk_blocks = sm_count * (per_sm > 0 ? per_sm : 1);
  const size_t nn = (size_t)(n > 1 ? n - 1 : 1);
  TS_TRY(keys[0].alloc((size_t)n));
  TS_TRY(keys[1].alloc((size_t)n));
  TS_TRY(vals[0].alloc((size_t)n));
  TS_TRY(vals[1].alloc((size_t)n));
  TS_TRY(ys.alloc((size_t)n));
  TS_TRY(sortmem.alloc(sort_words()));
  TS_TRY(starts.alloc((size_t)n / 32 + 1));
  TS_TRY(groups.alloc((size_t)n));
  TS_TRY(nodeA.alloc(nn));
  TS_TRY(nodeB.alloc(nn));
  TS_TRY(box.alloc(nn));
  TS_TRY(sum.alloc(nn));
  TS_TRY(slot.alloc(nn));
  size_t tiles = ((size_t)n + kTileLeaves - 1) / kTileLeaves;
  for (int k = 0; k < 3; ++k, tiles = (tiles + kUpTiles - 1) / kUpTiles) {
    TS_TRY(item_at[k].alloc(tiles * kItemCap));
    TS_TRY(item_box[k].alloc(tiles * kItemCap));
    TS_TRY(item_sum[k].alloc(tiles * kItemCap));
    TS_TRY(item_count[k].alloc(tiles));
  }
  this->sm_count = sm_count;
  TS_CUDA(cudaFuncSetAttribute(k_climb_leaves, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClimbTile)));
  TS_CUDA(cudaFuncSetAttribute(k_climb_items, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClimbTile)));
  TS_CUDA(cudaFuncSetAttribute(k_climb_top, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClimbTile)));
  TS_TRY(boxpart.alloc((size_t)box_blocks));
  TS_TRY(state.alloc(1));
  TS_CUDA(cudaMemsetAsync(slot.get(), 0xff, sizeof(unsigned long long) * nn, s));  // every slot empty
  TS_CUDA(cudaMemsetAsync(state.get(), 0, sizeof(TreeState), s));
  return TSGNE_OK;
}

tsgne_status launch_tree_build(TreeBufs& tb, const float2* Y, cudaStream_t s) {
  const int n = tb.n;
  TreeState* st = tb.state.get();
  uint32_t* ghist = tb.sortmem.get();
  uint32_t* ctl = ghist + kRadixPasses * kRadixBins;
  uint32_t* status = ctl + kRadixPasses;
  k_tree_box<<<tb.box_blocks, 256, 0, s>>>(Y, n, tb.boxpart.get(), st, tb.sortmem.get(), (int64_t)tb.sort_words(),
                                           tb.starts.get());
  k_tree_keys<<<tb.keys_blocks, kKeyThreads, 0, s>>>(Y, n, st, tb.keys[0].get(), tb.vals[0].get(), ghist);
  TS_CUDA(cudaGetLastError());
  // 16 warps of 4 keys a lane while every SM has at most one tile: a tile is a
  // serial chain, shorter with fewer keys a lane (an iteration at 300,000 points,
  // 147 tiles: 291 us with 8 warps, 281 with 16).  With more tiles the SMs are
  // full and half the counts in shared memory are cheaper (2,097,152 points: 1439
  // us with 8 warps, 1476 with 16).
  // A pass may set up beside the end of the one before.  Its CTAs are then
  // placed among those still running, unevenly, which costs more than the
  // set-up where the tiles fill the SMs almost exactly once or twice
  // (us per iteration without / with it: 98 tiles 228 / 226, 147 tiles 280 /
  // 291, 293 tiles 480 / 494, 489 tiles 740.6 / 739.3; launched one by one
  // the eight passes gain 10 to 23 us outside that range).
  const int sms = tb.sm_count;
  const bool one_wave = tb.ntiles <= sms, beside = 3 * tb.ntiles <= 2 * sms || tb.ntiles >= 3 * sms;
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)tb.ntiles);
  cfg.blockDim = dim3(one_wave ? 512u : 256u);
  cfg.stream = s;
  cfg.attrs = &early;
  cfg.numAttrs = 0;  // the first pass waits for the keys as usual
  for (int pass = 0; pass < kRadixPasses; ++pass) {
    const int in = pass & 1, out = in ^ 1;
    const bool last = pass == kRadixPasses - 1;
    TS_CUDA(cudaLaunchKernelEx(&cfg, one_wave ? k_radix_onesweep<16> : k_radix_onesweep<8>,
                               (const uint64_t*)tb.keys[in].get(), (const int32_t*)tb.vals[in].get(), n, pass,
                               (const uint32_t*)ghist, ctl, status, tb.ntiles, (long long)tb.spin_budget, st,
                               tb.keys[out].get(), tb.vals[out].get(), last ? Y : (const float2*)nullptr,
                               last ? tb.ys.get() : (float2*)nullptr));
    if (beside) cfg.numAttrs = 1;
  }
  // an even number of passes: sorted keys / permutation are back in slot 0
  static_assert(kRadixPasses % 2 == 0, "sorted keys end in slot 0");
  const TreeOut o{tb.nodeA.get(), tb.nodeB.get(), tb.starts.get(), st};
  const size_t smem = sizeof(ClimbTile);
  const int leaf_tiles = (n + kTileLeaves - 1) / kTileLeaves;
  auto items = [&](int k) {
    return Items{tb.item_at[k].get(), tb.item_box[k].get(), tb.item_sum[k].get(), tb.item_count[k].get()};
  };
  k_climb_leaves<<<leaf_tiles, kTileLeaves, smem, s>>>(n, tb.keys[0].get(), tb.ys.get(), o, items(0), tb.box.get(),
                                                       tb.sum.get());
  int tiles = leaf_tiles, at = 0;
  while (tiles > kUpTiles) {
    const int up = (tiles + kUpTiles - 1) / kUpTiles, to = at == 1 ? 2 : 1;
    k_climb_items<<<up, kTileLeaves, smem, s>>>(n, tb.keys[0].get(), items(at), tiles, o, items(to), tb.box.get(),
                                                tb.sum.get());
    tiles = up;
    at = to;
  }
  if (tiles > 1)
    k_climb_top<<<tb.sm_count, kTileLeaves, smem, s>>>(n, tb.keys[0].get(), tb.ys.get(), items(at), tiles,
                                                          items(0), leaf_tiles, tb.slot.get(), tb.box.get(),
                                                          tb.sum.get(), o);
  TS_CUDA(cudaGetLastError());
  k_tree_groups<<<grid_for((n + 31) / 32, 256, 1 << 30), 256, 0, s>>>(n, st, tb.starts.get(), tb.groups.get());
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

tsgne_status launch_tree_walk(TreeBufs& tb, float theta, float2* frep, Sched* sched, int advance, float ee,
                              int ee_iters, float mom0, float mom1, cudaStream_t s) {
  const float theta2 = theta * theta;
  k_tree_walk<<<tb.walk_blocks, 32 * kWalkWarps, 0, s>>>(tb.n, tb.ys.get(), tb.vals[0].get(), tb.nodeA.get(),
                                                         tb.nodeB.get(), tb.groups.get(), theta2, frep, sched,
                                                         tb.state.get(), advance, ee, ee_iters, mom0, mom1);
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

}  // namespace tsgne
