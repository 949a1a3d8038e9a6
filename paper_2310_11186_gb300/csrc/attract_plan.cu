// Attraction + update (S3 + S5 fused) on a schedule fixed when P is
// installed.  The terms and the order in which each row adds them are those
// of k_attract (iterate.cu) -- the definition the gradient export, the batch
// engine and the oracle parity tests share -- so the results are the same
// bits; what changes is how the work is laid out over threads.
//
// The order of a row's sum, by degree d:
//   d <= 32:   8 slot chains, slot s adding entries s, s + 8, ... in order
//              (at most 4), then the 8 slots in xor-butterfly order;
//   d > 32:    chunks of 1024 entries; within a chunk 32 lane chains, lane l
//              adding entries l, l + 32, ... in order, then the 32 lanes in
//              xor-butterfly order; the chunk sums in chunk order.
// A row of 33 to 128 entries is one chunk whose lane chains hold at most 4
// entries.  One warp per such row leaves most lanes with one or two entries
// and pays the warp's fixed costs per row; R-MAT 2^21 has 122,000 of them.
// So rows up to 128 entries are cut into their chains ("pairs" of row and
// slot: 8 per row up to 32 entries, 32 per row above), one thread per chain,
// and rows above 128 entries keep one warp per chunk.
//
// The schedule (built on the device from row_ptr, once per P):
//   short CTAs  rows [256 c, 256 c + 256): the chains of their rows of at most
//               32 entries; then one thread per row adds its 8 slots and
//               updates the row (rows above 32 entries are left to the others;
//               rows without entries get F^a = 0);
//   medium CTAs up to 64 rows of 33..128 entries (listed): their 32 chains
//               each; then one warp per row adds the 32 chains with the same
//               shuffle butterfly the chunk warps use, and one thread per row
//               updates it;
//   big CTAs    one warp per 1024-entry chunk of the rows above 128 entries,
//               as k_attract's fused hub branch.
// Within a CTA the chains are sorted by length (longest first), so the chains
// still running at level k are a prefix [0, cnt[k]) of the list and entry k
// of chain q sits at ent + off[k] + q in copies of col and P made in that
// order: every level's loads are coalesced, and each thread issues the loads
// of all entries of its chain before the first gather returns.  A CTA starts
// by prefetching into L2 the streams it reads (chain codes, col and P in chain
// order, its rows' optimiser state; a hub chunk's col and P).
#include "row_update.cuh"
#include "storage.cuh"
#include "tsgne_internal.cuh"

namespace tsgne {

namespace {

constexpr int kPlanThreads = 256;
constexpr int kShortRowsPerCta = 256;  // at most (short_rows)
constexpr int kMedRowsPerCta = 64;
constexpr int kSlotsShort = 8;
constexpr int kSlotsMed = 32;
static_assert(kShortRowsPerCta * kSlotsShort == kMedRowsPerCta * kSlotsMed, "one shared partial array");
constexpr int kPartials = kShortRowsPerCta * kSlotsShort;  // 2048

// L2 prefetch of the 128-byte lines of [lo, hi), spread over nt threads; every
// address touched lies inside the range.  A hint: the CTA's streams (chain
// codes, col and P in chain order, the rows' optimiser state; a hub chunk's
// col and P) are on their way from DRAM while its first gathers run.
template <class T>
__device__ __forceinline__ void prefetch_range(const T* lo, const T* hi, int t, int nt) {
  const uintptr_t a = (uintptr_t)lo, b = (uintptr_t)hi;
  for (uintptr_t q = (a & ~(uintptr_t)127) + (uintptr_t)t * 128; q < b; q += (uintptr_t)nt * 128)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(q < a ? a : q));
}

// One entry's term of F^a, as attract_entries adds it.
template <class PT, class YT>
__device__ __forceinline__ void add_term(float2 yi, float2 yj, float p, float& ax, float& ay) {
  const float dx = yi.x - yj.x, dy = yi.y - yj.y;
  const float w = 1.0f / fmaf(dy, dy, fmaf(dx, dx, 1.0f));
  const float pw = p * w;
  ax = fmaf(pw, dx, ax);
  ay = fmaf(pw, dy, ay);
}

template <class PT, class YT>
__global__ void __launch_bounds__(kPlanThreads, 6)
    k_attract_plan(AttractArgs a, PlanView pv, int big_blocks) {
  __shared__ float2 spart[kPartials];
  __shared__ float2 sfa[kMedRowsPerCta];
  __shared__ float s_invz;
  const RowForce rf{a.frep, a.facc, a.unscale};
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PT* __restrict__ P = static_cast<const PT*>(a.P);
  const YT* __restrict__ Y = static_cast<const YT*>(a.Yr);
  bf162* Ynext16 = static_cast<bf162*>(a.Ynext16);
  uint32_t* dbg = &a.sched->flags;  // index checks of the debug build
  (void)dbg;

  if ((int)blockIdx.x < big_blocks) {  // one warp per chunk of a row above 128 entries
    const HeavyRows& hv = a.hv;
    const int stride = big_blocks * (kPlanThreads / 32);
    for (int k = blockIdx.x * (kPlanThreads / 32) + warp; k < pv.n_big; k += stride) {
      const int c = pv.big[k];
      if (!TS_IN(c, 0, hv.chunks, dbg)) continue;
      const int64_t i = hv.chunk_row[c];
      if (!TS_IN(i, 0, a.n, dbg)) continue;
      prefetch_range(a.col + hv.chunk_begin[c], a.col + hv.chunk_end[c], lane, 32);
      prefetch_range(P + hv.chunk_begin[c], P + hv.chunk_end[c], lane, 32);
      float ax = 0.f, ay = 0.f;
      attract_entries<32, PT, YT>(hv.chunk_begin[c], hv.chunk_end[c], a.col, P, Y, i, lane, ld_y(Y, i), ax, ay,
                                  a.n, dbg);
      ax = group_sum<32>(ax);
      ay = group_sum<32>(ay);
      if (lane == 0) {
        hv.fa[c] = make_float2(ax, ay);
        const int h = hv.chunk_heavy[c];
        const int c0 = hv.chunk_off[h], c1 = hv.chunk_off[h + 1];
        if (atom_add_acq_rel_u32(&hv.arrivals[h], 1u) == (unsigned)(c1 - c0 - 1)) {  // last chunk of the row
          hv.arrivals[h] = 0u;
          float sx = 0.f, sy = 0.f;
          for (int q = c0; q < c1; ++q) {
            const float2 f = __ldcg(hv.fa + q);
            sx += f.x;
            sy += f.y;
          }
          finish_row<false>(i, make_float2(sx, sy), rf, pass_inv_z(a.sched, a.zslot, a.n), a.sched, 0.f, nullptr,
                            a.Ym, a.Ynext, Ynext16, a.upd, a.gains, a.eta, a.min_gain);
        }
      }
    }
    return;
  }

  const int cb = (int)blockIdx.x - big_blocks;
  const bool med = cb < pv.n_med;
  const PlanCta m = med ? pv.med[cb] : pv.shorts[cb - pv.n_med];
  const int shift = med ? 5 : 3;
  const int64_t row0 = med ? 0 : (int64_t)(cb - pv.n_med) * pv.short_rows;
  {
    const int64_t tot = (int64_t)m.cnt[0] + m.cnt[1] + m.cnt[2] + m.cnt[3];
    prefetch_range(pv.code + m.pair, pv.code + m.pair + m.cnt[0], tid, kPlanThreads);
    prefetch_range(pv.colS + m.ent, pv.colS + m.ent + tot, tid, kPlanThreads);
    const PT* PS = static_cast<const PT*>(pv.PS);
    prefetch_range(PS + m.ent, PS + m.ent + tot, tid, kPlanThreads);
  }
  if (!med) {
    const int64_t r1 = row0 + m.nrows;
    prefetch_range(a.rp + row0, a.rp + r1 + 1, tid, kPlanThreads);
    if (a.facc) prefetch_range(a.facc + 2 * row0, a.facc + 2 * r1, tid, kPlanThreads);
    else prefetch_range(a.frep + row0, a.frep + r1, tid, kPlanThreads);
    prefetch_range(a.upd + row0, a.upd + r1, tid, kPlanThreads);
    prefetch_range(a.gains + row0, a.gains + r1, tid, kPlanThreads);
    prefetch_range(a.Ym + row0, a.Ym + r1, tid, kPlanThreads);
  }
  if (tid == 0) s_invz = pass_inv_z(a.sched, a.zslot, a.n);
  for (int k = tid; k < m.nrows << shift; k += kPlanThreads) spart[k] = make_float2(0.f, 0.f);
  __syncthreads();

  // the chains: thread per chain, every entry's loads issued up front
  const int64_t off1 = m.cnt[0], off2 = off1 + m.cnt[1], off3 = off2 + m.cnt[2];
  for (int q = tid; q < m.cnt[0]; q += kPlanThreads) {
    if (!TS_IN(m.pair + q, 0, pv.n_codes, dbg)) continue;
    const int code = pv.code[m.pair + q];
    const int r = code >> shift, s = code & ((1 << shift) - 1);
    if (!TS_IN(r, 0, m.nrows, dbg) || (med && !TS_IN(m.rows + r, 0, pv.n_med_rows, dbg))) continue;
    const int64_t i = med ? (int64_t)pv.med_rows[m.rows + r] : row0 + r;
    if (!TS_IN(i, 0, a.n, dbg)) continue;
    const int depth = 1 + (q < m.cnt[1]) + (q < m.cnt[2]) + (q < m.cnt[3]);
    const int64_t e[4] = {m.ent + q, m.ent + off1 + q, m.ent + off2 + q, m.ent + off3 + q};
    int32_t j[4];
    float p[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool ld = k < depth && TS_IN(e[k], 0, pv.entries, dbg);
      j[k] = ld ? pv.colS[e[k]] : (int32_t)i;
      p[k] = ld ? ld_p(static_cast<const PT*>(pv.PS), e[k]) : 0.f;
      if (!TS_IN(j[k], 0, a.n, dbg)) j[k] = (int32_t)i;
    }
    const float2 yi = ld_y(Y, i);
    float2 yj[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) yj[k] = ld_y(Y, j[k]);
    float ax = 0.f, ay = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < depth) add_term<PT, YT>(yi, yj[k], p[k], ax, ay);
    spart[(r << shift) + s] = make_float2(ax, ay);
  }
  __syncthreads();

  if (!med) {  // one thread per row of at most 32 entries: slots in butterfly order, then the update
    if (tid >= m.nrows) return;
    const int64_t i = row0 + tid;
    if (a.rp[i + 1] - a.rp[i] > kHeavyDeg) return;  // a medium or big CTA updates it
    const float2* sp = spart + tid * kSlotsShort;
    float2 a0 = sp[0], a1 = sp[1], t = sp[4];
    a0 = make_float2(a0.x + t.x, a0.y + t.y);  // o = 4
    t = sp[5];
    a1 = make_float2(a1.x + t.x, a1.y + t.y);
    float2 a2 = sp[2];
    t = sp[6];
    a2 = make_float2(a2.x + t.x, a2.y + t.y);
    float2 a3 = sp[3];
    t = sp[7];
    a3 = make_float2(a3.x + t.x, a3.y + t.y);
    a0 = make_float2(a0.x + a2.x, a0.y + a2.y);  // o = 2
    a1 = make_float2(a1.x + a3.x, a1.y + a3.y);
    const float2 fa = make_float2(a0.x + a1.x, a0.y + a1.y);  // o = 1
    finish_row<false>(i, fa, rf, s_invz, a.sched, 0.f, nullptr, a.Ym, a.Ynext, Ynext16, a.upd, a.gains, a.eta,
                      a.min_gain);
    return;
  }
  // medium rows: the 32 chains of a row with the chunk warps' shuffle
  // butterfly, then (one chunk) its sum starting from 0 as the chunk-sum loop
  for (int r = warp; r < m.nrows; r += kPlanThreads / 32) {
    const float2 v = spart[r * kSlotsMed + lane];
    const float ax = group_sum<32>(v.x), ay = group_sum<32>(v.y);
    if (lane == 0) sfa[r] = make_float2(0.f + ax, 0.f + ay);
  }
  __syncthreads();
  if (tid < m.nrows && TS_IN(m.rows + tid, 0, pv.n_med_rows, dbg))
    finish_row<false>(pv.med_rows[m.rows + tid], sfa[tid], rf, s_invz, a.sched, 0.f, nullptr, a.Ym, a.Ynext, Ynext16,
                      a.upd, a.gains, a.eta, a.min_gain);
}

// ------------------------------------------------ building the schedule
//
// Four small launches over blocks of 256 consecutive rows (a block is a short
// CTA of the schedule), one host wait for the sizes of the lists:
//   k_row_totals   what each block's rows add to every list
//   k_row_scan     exclusive scan of those totals over the blocks (CTA f: list f)
//   k_row_lists    the hub rows with their chunks, the medium rows, the chunks
//                  of the rows above 128 entries, each in row order
//   k_plan_chains  a CTA's chains sorted longest first (by counting: a row's
//                  chains have at most two lengths, so four counters packed in
//                  one 64-bit scan give every chain its place), then col and P
//                  copied level by level, coalesced.
// Bound by the reads of row_ptr, col and P and the writes of their copies
// (16 B per entry).  A whole P build of 300,000 rows and 2.0M entries (device
// arrays) took 16.5 ms with the lists built by host loops over a copy of
// row_ptr, and 2.72 ms with these kernels instead (0.47 ms since allocations
// come from kept blocks and a canonical structure is copied).
enum RowList { kCodes = 0, kEntries, kHeavyRows, kChunks, kMedRows, kMedEntries, kBigChunks, kRowLists };

struct RowAdds {
  uint32_t v[kRowLists];
};

// What one row of d entries adds to each list.
__device__ __forceinline__ RowAdds row_adds(int64_t d) {
  RowAdds a{};
  if (d <= kHeavyDeg) {
    a.v[kCodes] = (uint32_t)(d < kSlotsShort ? d : kSlotsShort);
    a.v[kEntries] = (uint32_t)d;
    return a;
  }
  a.v[kHeavyRows] = 1u;
  a.v[kChunks] = (uint32_t)((d + kHeavyChunk - 1) / kHeavyChunk);
  if (d <= kMedDeg) {
    a.v[kMedRows] = 1u;
    a.v[kMedEntries] = (uint32_t)d;
  } else {
    a.v[kBigChunks] = a.v[kChunks];
  }
  return a;
}

// tot[list][block] = sum of the block's rows.
__global__ void __launch_bounds__(kPlanThreads)
    k_row_totals(int n, const int64_t* __restrict__ rp, int per, int nb, int64_t* __restrict__ tot) {
  __shared__ uint32_t sum[kRowLists];
  if (threadIdx.x < kRowLists) sum[threadIdx.x] = 0u;
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * per + threadIdx.x;
  const RowAdds a = row_adds((int)threadIdx.x < per && i < n ? rp[i + 1] - rp[i] : 0);
#pragma unroll
  for (int f = 0; f < kRowLists; ++f) {
    const uint32_t w = __reduce_add_sync(0xffffffffu, a.v[f]);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(&sum[f], w);
  }
  __syncthreads();
  if (threadIdx.x < kRowLists) tot[(int64_t)threadIdx.x * nb + blockIdx.x] = sum[threadIdx.x];
}

// Exclusive scan over the threads of a CTA (at most 1,024); *total: the sum.
template <class T>
__device__ __forceinline__ T cta_excl_scan(T v, T* total) {
  __shared__ T ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  T base = 0, all = 0;
  for (int k = 0; k < nw; ++k) {
    if (k < w) base += ws[k];
    all += ws[k];
  }
  *total = all;
  __syncthreads();
  return base + x - v;
}

// CTA f: tot[f][0..nb) to its exclusive scan, the total to sums[f].
__global__ void __launch_bounds__(1024) k_row_scan(int nb, int64_t* __restrict__ tot, int64_t* __restrict__ sums) {
  int64_t* t = tot + (int64_t)blockIdx.x * nb;
  int64_t carry = 0;
  for (int c0 = 0; c0 < nb; c0 += 1024) {
    const int c = c0 + threadIdx.x;
    int64_t all;
    const int64_t ex = cta_excl_scan<int64_t>(c < nb ? t[c] : 0, &all);
    if (c < nb) t[c] = carry + ex;
    carry += all;
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = carry;
}

// The lists of rows and chunks (see HeavyStore and AttractPlan).  med_ent
// (NULL: no plan wanted): first entry, in the copies, of each medium CTA.
__global__ void __launch_bounds__(kPlanThreads)
    k_row_lists(int n, const int64_t* __restrict__ rp, int per, int nb, const int64_t* __restrict__ tot,
                int32_t* __restrict__ rows, int32_t* __restrict__ chunk_off, int32_t* __restrict__ chunk_row,
                int32_t* __restrict__ chunk_heavy, int64_t* __restrict__ chunk_begin, int64_t* __restrict__ chunk_end,
                int32_t* __restrict__ med_rows, int64_t* __restrict__ med_ent, int32_t* __restrict__ big) {
  const int64_t i = (int64_t)blockIdx.x * per + threadIdx.x;
  const bool mine = (int)threadIdx.x < per && i < n;
  const int64_t a = mine ? rp[i] : 0, b = mine ? rp[i + 1] : 0;
  const RowAdds ra = row_adds(b - a);
  if (!__syncthreads_or((int)ra.v[kHeavyRows])) return;
  uint32_t ex[kRowLists], all;
#pragma unroll
  for (int f = kHeavyRows; f < kRowLists; ++f) ex[f] = cta_excl_scan<uint32_t>(ra.v[f], &all);
  if (!ra.v[kHeavyRows]) return;
  auto at = [&](int f) { return tot[(int64_t)f * nb + blockIdx.x] + ex[f]; };
  const int64_t h = at(kHeavyRows), c0 = at(kChunks);
  rows[h] = (int32_t)i;
  chunk_off[h + 1] = (int32_t)(c0 + ra.v[kChunks]);
  const int64_t bg = at(kBigChunks);
  for (uint32_t k = 0; k < ra.v[kChunks]; ++k) {
    const int64_t x = a + (int64_t)k * kHeavyChunk;
    chunk_row[c0 + k] = (int32_t)i;
    chunk_heavy[c0 + k] = (int32_t)h;
    chunk_begin[c0 + k] = x;
    chunk_end[c0 + k] = x + kHeavyChunk < b ? x + kHeavyChunk : b;
    if (med_ent != nullptr && ra.v[kBigChunks]) big[bg + k] = (int32_t)(c0 + k);
  }
  if (med_ent != nullptr && ra.v[kMedRows]) {
    const int64_t m = at(kMedRows);
    med_rows[m] = (int32_t)i;
    if (m % kMedRowsPerCta == 0) med_ent[m / kMedRowsPerCta] = at(kMedEntries);
  }
}

// Chain codes, copies of col and P in chain order and the PlanCta of one CTA:
// medium CTA blockIdx.x < n_med, else short CTA blockIdx.x - n_med.  Chain
// (row r, slot s) of a row of d = S q + m entries (S slots) holds q + 1
// entries if s < m, else q; the chains lie longest first, within a length by
// row and slot.
template <class PT>
__global__ void __launch_bounds__(kPlanThreads)
    k_plan_chains(int n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col, const PT* __restrict__ P,
                  int n_med, int64_t n_med_rows, int64_t med_entries, const int32_t* __restrict__ med_rows,
                  const int64_t* __restrict__ med_ent, int per, int nb, const int64_t* __restrict__ tot,
                  PlanCta* __restrict__ cta, uint16_t* __restrict__ code, int32_t* __restrict__ colS,
                  PT* __restrict__ PS) {
  __shared__ int64_t sfirst[kPartials];  // first entry of each chain, in chain order
  __shared__ int64_t sa[kShortRowsPerCta];
  __shared__ int sq[kShortRowsPerCta], sm[kShortRowsPerCta];
  __shared__ unsigned long long sex[kShortRowsPerCta];
  const int tid = threadIdx.x;
  const bool med = (int)blockIdx.x < n_med;
  const int c = med ? (int)blockIdx.x : (int)blockIdx.x - n_med;
  const int shift = med ? 5 : 3, slots = 1 << shift;
  int64_t r0 = 0;
  int nrows;
  int64_t i = -1;
  if (med) {
    r0 = (int64_t)c * kMedRowsPerCta;
    nrows = (int)min((int64_t)kMedRowsPerCta, n_med_rows - r0);
    if (tid < nrows) i = med_rows[r0 + tid];
  } else {
    r0 = (int64_t)c * per;
    nrows = (int)min((int64_t)per, (int64_t)n - r0);
    if (tid < nrows) i = r0 + tid;
  }
  int64_t a = 0, d = 0;
  if (i >= 0) {
    a = rp[i];
    d = rp[i + 1] - a;
    if (!med && d > kHeavyDeg) d = 0;  // a medium or big CTA's row
  }
  const int q = (int)(d >> shift), m = (int)d & (slots - 1);
  // chains of length L = 1..4 in bits 16 (L - 1); at most 2,048 of a length
  unsigned long long cnt = 0ull;
  if (m > 0) cnt += (unsigned long long)m << (16 * q);
  if (q > 0) cnt += (unsigned long long)(slots - m) << (16 * (q - 1));
  unsigned long long all;
  sex[tid] = cta_excl_scan<unsigned long long>(cnt, &all);
  sa[tid] = a;
  sq[tid] = q;
  sm[tid] = m;
  __syncthreads();
  int num[4], start[4];
  {
    int at = 0;
#pragma unroll
    for (int L = 3; L >= 0; --L) {
      num[L] = (int)(all >> (16 * L)) & 0xffff;
      start[L] = at;
      at += num[L];
    }
  }
  const int64_t pair0 = med ? r0 * kSlotsMed : n_med_rows * kSlotsMed + tot[(int64_t)kCodes * nb + c];
  const int64_t ent0 = med ? med_ent[c] : med_entries + tot[(int64_t)kEntries * nb + c];
  for (int k = tid; k < nrows << shift; k += kPlanThreads) {
    const int r = k >> shift, s = k & (slots - 1);
    const bool lng = s < sm[r];
    const int len = sq[r] + (lng ? 1 : 0);
    if (len == 0) continue;
    int st = start[0];
#pragma unroll
    for (int L = 1; L < 4; ++L)
      if (len == L + 1) st = start[L];
    const int at = st + ((int)(sex[r] >> (16 * (len - 1))) & 0xffff) + (lng ? s : s - sm[r]);
    code[pair0 + at] = (uint16_t)((r << shift) | s);
    sfirst[at] = sa[r] + s;
  }
  __syncthreads();
  int64_t ent = ent0;
  int more = num[0] + num[1] + num[2] + num[3];  // chains of more than k entries: a prefix of the list
  PlanCta pc{};
  pc.ent = ent0;
  pc.pair = (int32_t)pair0;
  pc.rows = med ? (int32_t)r0 : 0;
  pc.nrows = nrows;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    pc.cnt[k] = more;
    for (int x = tid; x < more; x += kPlanThreads) {
      const int64_t e = sfirst[x] + (int64_t)slots * k;
      colS[ent + x] = col[e];
      PS[ent + x] = P[e];
    }
    ent += more;
    more -= num[k];
  }
  if (tid == 0) cta[blockIdx.x] = pc;
}

// Rows of a short CTA: the fewest (a power of two, at least 32) that still
// make one wave of the 6 CTAs an SM holds.  A CTA is a chain of dependent
// loads, so few rows per CTA shorten small passes (2,000 points: 10.5 us with
// 128 rows, 8.7 us with 32; 30,000: 13.3 us with 256, 11.1 us with 64) and a
// second wave costs more than that (130,000: 20.8 us with 128, 18.8 us with 256).
int short_rows(int n, int sms) {
  int r = 32;
  while (r < kShortRowsPerCta && (n + r - 1) / r > 6 * sms) r *= 2;
  return r;
}

// The hub rows of a structure and, if plan is not NULL, the schedule.
tsgne_status build_row_schedule(int n, const int64_t* rp, const int32_t* col, const float* P, const bf16* P16,
                                HeavyStore& hs, AttractPlan* plan, cudaStream_t s) {
  int dev = 0, sms = 1;
  TS_CUDA(cudaGetDevice(&dev));
  TS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int per = plan ? short_rows(n, sms) : kShortRowsPerCta;
  const int nb = (n + per - 1) / per;
  DevBuf<int64_t> tot, med_ent;
  TS_TRY(tot.alloc((size_t)nb * kRowLists + kRowLists));
  int64_t* const sums = tot.get() + (size_t)nb * kRowLists;
  k_row_totals<<<nb, kPlanThreads, 0, s>>>(n, rp, per, nb, tot.get());
  k_row_scan<<<kRowLists, 1024, 0, s>>>(nb, tot.get(), sums);
  TS_CUDA(cudaGetLastError());
  int64_t h[kRowLists];
  TS_CUDA(cudaMemcpyAsync(h, sums, sizeof(h), cudaMemcpyDeviceToHost, s));
  TS_CUDA(cudaStreamSynchronize(s));
  auto at_least_1 = [](int64_t v) { return (size_t)(v > 0 ? v : 1); };
  hs.count = (int)h[kHeavyRows];
  hs.chunks = (int)h[kChunks];
  TS_TRY(hs.rows.alloc(at_least_1(h[kHeavyRows])));
  TS_TRY(hs.chunk_off.alloc((size_t)h[kHeavyRows] + 1));
  TS_TRY(hs.chunk_row.alloc(at_least_1(h[kChunks])));
  TS_TRY(hs.chunk_begin.alloc(at_least_1(h[kChunks])));
  TS_TRY(hs.chunk_end.alloc(at_least_1(h[kChunks])));
  TS_TRY(hs.fa.alloc(at_least_1(h[kChunks])));
  TS_TRY(hs.chunk_heavy.alloc(at_least_1(h[kChunks])));
  TS_TRY(hs.arrivals.alloc(at_least_1(h[kHeavyRows])));
  TS_CUDA(cudaMemsetAsync(hs.arrivals.get(), 0, sizeof(uint32_t) * at_least_1(h[kHeavyRows]), s));
  TS_CUDA(cudaMemsetAsync(hs.chunk_off.get(), 0, sizeof(int32_t), s));
  if (plan) {
    *plan = AttractPlan();
    plan->n_med = (int)((h[kMedRows] + kMedRowsPerCta - 1) / kMedRowsPerCta);
    plan->n_short = nb;
    plan->short_rows = per;
    plan->n_big = (int)h[kBigChunks];
    plan->n_med_rows = h[kMedRows];
    plan->n_codes = h[kMedRows] * kSlotsMed + h[kCodes];
    plan->entries = h[kMedEntries] + h[kEntries];
    TS_TRY(plan->cta.alloc((size_t)(plan->n_med + plan->n_short)));
    TS_TRY(plan->code.alloc((size_t)plan->n_codes));
    TS_TRY(plan->med_rows.alloc((size_t)plan->n_med_rows));
    TS_TRY(plan->big.alloc((size_t)plan->n_big));
    TS_TRY(plan->colS.alloc((size_t)plan->entries));
    TS_TRY(med_ent.alloc((size_t)plan->n_med));
    if (P16) TS_TRY(plan->PS16.alloc((size_t)plan->entries));
    else TS_TRY(plan->PS.alloc((size_t)plan->entries));
  }
  if (h[kHeavyRows] > 0)
    k_row_lists<<<nb, kPlanThreads, 0, s>>>(n, rp, per, nb, tot.get(), hs.rows.get(), hs.chunk_off.get(),
                                            hs.chunk_row.get(), hs.chunk_heavy.get(), hs.chunk_begin.get(),
                                            hs.chunk_end.get(), plan ? plan->med_rows.get() : nullptr,
                                            plan ? med_ent.get() : nullptr, plan ? plan->big.get() : nullptr);
  if (plan) {
    const int grid = plan->n_med + plan->n_short;
    if (P16)
      k_plan_chains<bf16><<<grid, kPlanThreads, 0, s>>>(
          n, rp, col, P16, plan->n_med, plan->n_med_rows, h[kMedEntries], plan->med_rows.get(), med_ent.get(), per,
          nb, tot.get(), plan->cta.get(), plan->code.get(), plan->colS.get(), plan->PS16.get());
    else
      k_plan_chains<float><<<grid, kPlanThreads, 0, s>>>(
          n, rp, col, P, plan->n_med, plan->n_med_rows, h[kMedEntries], plan->med_rows.get(), med_ent.get(), per,
          nb, tot.get(), plan->cta.get(), plan->code.get(), plan->colS.get(), plan->PS.get());
  }
  TS_CUDA(cudaGetLastError());
  TS_CUDA(cudaStreamSynchronize(s));  // tot and med_ent are freed on return
  if (plan) plan->ready = true;
  return TSGNE_OK;
}

}  // namespace

tsgne_status find_heavy_rows(int n, const int64_t* rp, HeavyStore& hs, cudaStream_t s) {
  return build_row_schedule(n, rp, nullptr, nullptr, nullptr, hs, nullptr, s);
}

tsgne_status build_attract_plan(int n, const int64_t* rp, const int32_t* col, const float* P, const bf16* P16,
                                HeavyStore& hs, AttractPlan& plan, cudaStream_t s) {
  return build_row_schedule(n, rp, col, P, P16, hs, &plan, s);
}

PlanView AttractPlan::view() const {
  PlanView v;
  v.med = cta.get();
  v.shorts = cta.get() + n_med;
  v.code = code.get();
  v.colS = colS.get();
  v.PS = PS16.get() ? (const void*)PS16.get() : (const void*)PS.get();
  v.med_rows = med_rows.get();
  v.big = big.get();
  v.n_med = n_med;
  v.n_short = n_short;
  v.n_big = n_big;
  v.short_rows = short_rows;
  v.entries = entries;
  v.n_codes = n_codes;
  v.n_med_rows = n_med_rows;
  return v;
}

tsgne_status launch_attract_plan(const AttractArgs& a, const PlanView& pv, cudaStream_t s) {
  int big_blocks = (pv.n_big + kPlanThreads / 32 - 1) / (kPlanThreads / 32);
  if (big_blocks > 4096) big_blocks = 4096;
  const int grid = big_blocks + pv.n_med + pv.n_short;
  if (grid <= 0) return TSGNE_OK;
  if (a.p_bf16 && a.y_bf16)
    k_attract_plan<bf16, bf162><<<grid, kPlanThreads, 0, s>>>(a, pv, big_blocks);
  else if (!a.p_bf16 && !a.y_bf16)
    k_attract_plan<float, float2><<<grid, kPlanThreads, 0, s>>>(a, pv, big_blocks);
  else {
    last_msg() = "P and Y must share a storage precision";
    return TSGNE_ERR_INVALID_ARG;
  }
  TS_CUDA(cudaGetLastError());
  return TSGNE_OK;
}

}  // namespace tsgne
