// spk_items.cuh -- entries of a thread-block item in registers.
//
// A thread-block item (a CTA-class column, or one row window of a heavy
// column) holds the entries of k input segments.  Flattened, they are
// positions [0, total): segment after segment.  A block of B threads owns a
// chunk of at most 16 B positions at a time; each warp takes an equal run of
// it, `ns` times 32 positions, slot t holding positions 32 t to 32 t + 31 of
// the run (coalesced inside each segment).  An item of at most 16 B entries
// reads every row from memory once, into registers, whatever
// number of passes follow.  Longer items go chunk by chunk and read the rows
// once per pass.
//
// Finding a position's segment is what the walk costs.  Searching per entry
// (five shuffles, or a division for equal lengths) in each of three passes
// took most of the 13 warp instructions an entry used to cost.  Here
// each non-empty segment sets one bit at its first position in a shared
// start-bit map, and every 32-position block stores the segment holding its
// first position: a position's segment is one broadcast load and one popcount.
#pragma once

#include "spk_common.cuh"

namespace spk {

constexpr int ITEM_SLOTS = 16;
constexpr int ITEM_GROUP = 2;  // slots per unrolled group (of four: up to three empty ones; R-MAT 25.7 -> 24.8 ms)

// Shared memory of the entry map of a block of B threads.
template <int B>
struct ItemMap {
  static constexpr int NW = B / 32;
  static constexpr int CAP = B * ITEM_SLOTS;   // positions per chunk
  static constexpr int KT = 512;               // inputs per segment table
  static constexpr int KPT = (KT + B - 1) / B; // inputs per thread
  static_assert(NW % 4 == 0 && KT % FP32_PHASE_INPUTS == 0, "segment table");
  ulonglong2 seg[KT];            // non-empty segments: row and value addresses minus their first position
  int first[KT + 1];             // first position of every non-empty segment, then the total
  int ne;                        // non-empty segments
  uint2 blk[CAP / 32];           // per 32 positions: start bits (kept zero between chunks), first segment
  alignas(16) int red[2][2 * NW];  // scan totals, two buffers used in turn
  int phase[KT / FP32_PHASE_INPUTS + 1];  // first position of every 128th input
};

// Block-wide exclusive scan with one barrier.  Two scans in a row must use
// different buffers.
template <int B>
__device__ __forceinline__ int item_scan(int x, int* red, int* total) {
  constexpr int NW = B / 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int inc = warp_incl_scan(x, lane);
  if (lane == 31) red[wid] = inc;
  __syncthreads();
  int before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < NW; w += 4) {
    const int4 v = *reinterpret_cast<const int4*>(red + w);
    before += (w < wid ? v.x : 0) + (w + 1 < wid ? v.y : 0) + (w + 2 < wid ? v.z : 0) + (w + 3 < wid ? v.w : 0);
    sum += v.x + v.y + v.z + v.w;
  }
  *total = sum;
  return before + inc - x;
}

// Bounds of a thread's inputs (KPT thread, ...) of a segment table, as loaded:
// nothing is computed from them before the table is built, so bounds loaded an
// item ahead are not waited for.
template <int B>
struct ItemBounds {
  int beg[ItemMap<B>::KPT], end[ItemMap<B>::KPT];
};

// Bounds of inputs [k_lo, k_lo + nk), nk <= KT: seg(i, &beg, &end) gives input
// i's part of the item.
template <int B, typename SegF>
__device__ __forceinline__ ItemBounds<B> item_bounds(int k_lo, int nk, SegF& seg) {
  constexpr int KPT = ItemMap<B>::KPT;
  ItemBounds<B> F;
#pragma unroll
  for (int h = 0; h < KPT; ++h) {
    F.beg[h] = 0;
    F.end[h] = 0;
    const int i = KPT * (int)threadIdx.x + h;
    if (i < nk) seg(k_lo + i, &F.beg[h], &F.end[h]);
  }
  return F;
}

// Start bits and first segments of the chunk at c0 that segment o, positions
// [p0, p1) less c0, calls for.
template <int B>
__device__ __forceinline__ void item_mark(ItemMap<B>& M, int o, int p0, int p1) {
  if (p0 >= 0 && p0 < ItemMap<B>::CAP) atomicOr(&M.blk[p0 >> 5].x, 1u << (p0 & 31));
  const int b1 = min(p1 - 1, ItemMap<B>::CAP - 1) >> 5;
  if (p1 > 0)
    for (int b = p0 <= 0 ? 0 : (p0 + 31) >> 5; b <= b1; ++b) M.blk[b].y = (uint32_t)o;
}

// Segment table of inputs [k_lo, k_lo + nk) and (MAP) the map of its first
// chunk; returns its positions' number.  VS: bytes of a value (0: rows only).
// Contains one barrier; the caller's next barrier publishes the table.
template <int VS, bool PREF, bool MAP, int B>
__device__ __forceinline__ int item_table(ItemMap<B>& M, const Inputs& in, int off, int k_lo, int nk,
                                          const ItemBounds<B>& F, int* red) {
  constexpr int KPT = ItemMap<B>::KPT, NW = ItemMap<B>::NW;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int len[KPT], ne = 0, lsum = 0;
#pragma unroll
  for (int h = 0; h < KPT; ++h) {
    len[h] = F.end[h] - F.beg[h];
    // Split windows of rows out of order: the end, the next window's start, may lie before the start.
    if constexpr (VS > 0) len[h] = max(0, len[h]);
    ne += len[h] > 0;
    lsum += len[h];
  }
  const bool holds = 32 * KPT * wid < nk;  // (warp-uniform) this warp holds inputs
  int li = 0, oi = 0;
  if (holds) {
    li = warp_incl_scan(lsum, lane);
    oi = warp_incl_scan(ne, lane);
    if (lane == 31) {
      red[wid] = li;
      red[NW + wid] = oi;
    }
  }
  __syncthreads();
  int P = 0, total = 0;
  for (int w = 0; 32 * KPT * w < nk; ++w) {  // the warps that hold inputs
    P = w == wid ? total : P;
    total += red[w];
  }
  if (!holds) return total;
  int o = oi - ne;
  for (int w = 0; w < wid; ++w) o += red[NW + w];
  P += li - lsum;
#pragma unroll
  for (int h = 0; h < KPT; ++h) {
    const int i = KPT * (int)threadIdx.x + h;
    if (VS && i % FP32_PHASE_INPUTS == 0) M.phase[i / FP32_PHASE_INPUTS] = P;
    if (len[h] > 0) {
      const int64_t d = (int64_t)F.beg[h] - P;
      ulonglong2 s;
      s.x = reinterpret_cast<unsigned long long>(in.ri[off + k_lo + i]) + (unsigned long long)(d * 4);
      s.y = 0ull;
      if constexpr (VS > 0) {
        const unsigned long long v = reinterpret_cast<unsigned long long>(in.val[off + k_lo + i]);
        s.y = v + (unsigned long long)(d * VS);
        if constexpr (PREF)
          l2_prefetch(reinterpret_cast<const void*>(v + (unsigned long long)F.beg[h] * VS), (size_t)len[h] * VS);
      }
      M.seg[o] = s;
      M.first[o] = P;
      if constexpr (MAP) item_mark(M, o, P, P + len[h]);
      ++o;
      P += len[h];
    }
    if (i == nk - 1) {
      M.ne = o;
      M.first[o] = total;
    }
  }
  return total;
}

// The map of the chunk at c0 of a published table; the caller's next barrier
// publishes it.
template <int B>
__device__ __forceinline__ void item_map(ItemMap<B>& M, int c0) {
  const int ne = M.ne;
  for (int o = threadIdx.x; o < ne; o += B) item_mark(M, o, M.first[o] - c0, M.first[o + 1] - c0);
}

template <int B>
__device__ __forceinline__ void item_unmap(ItemMap<B>& M) {
  if (threadIdx.x < ItemMap<B>::CAP / 32) M.blk[threadIdx.x].x = 0u;
}

// A thread's slots of one chunk: slot t (t < ns) is position run + 32 t + lane.
// A lane past the end of its warp's run repeats the run's last position, and a
// slot past ns its last slot: what is done with rows may be done twice (a bit
// set again), what must not be (a value added) asks live().
template <int B>
struct ItemSlots {
  int ns;    // slots of this warp (warp-uniform)
  int run;   // the warp's first position in the chunk
  int end;   // and its last one, plus one
  __device__ __forceinline__ void init(int c0, int total) {
    const int n = min(total - c0, ItemMap<B>::CAP);
    const int full = (n + B - 1) / B;
    run = ((int)threadIdx.x & ~31) * full;
    end = min(n, run + 32 * full);
    ns = end > run ? (end - run + 31) >> 5 : 0;
  }
  __device__ __forceinline__ bool live(int t) const { return run + 32 * t + ((int)threadIdx.x & 31) < end; }
  // The position slot t stands for.
  __device__ __forceinline__ int pos(int t) const {
    return min(run + 32 * min(t, ns - 1) + ((int)threadIdx.x & 31), end - 1);
  }
};

// Segment of slot t's position.  (Lanes past the last position of the run's
// last block see no later start bit, so they get the last segment.)
template <int B>
__device__ __forceinline__ int item_seg(const ItemMap<B>& M, const ItemSlots<B>& S, int t) {
  const uint2 b = M.blk[(S.run >> 5) + min(t, S.ns - 1)];
  return (int)b.y + __popc(b.x & (0xfffffffeu & (0xffffffffu >> (31 - (threadIdx.x & 31)))));
}

// Positions [p0, p1) of a published table without chunks or barriers: each warp
// walks an equal run of them, segment by segment, 32 U at a time.
// f(rows, vals, n): the lane's entries are at rows[32 t] (and vals[32 t]) for
// t < U with 32 t < n.
template <int B, typename V, int U, typename F>
__device__ __forceinline__ void item_walk(const ItemMap<B>& M, int64_t p0, int64_t p1, F&& f) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t run = (p1 - p0 + ItemMap<B>::NW - 1) / ItemMap<B>::NW;
  int64_t p = p0 + wid * run;
  const int64_t pe = min(p1, p + run);
  int o = 0, oe = M.ne;  // the last segment that starts at or before p
  while (oe - o > 1) {
    const int mid = (o + oe) >> 1;
    if (M.first[mid] <= p) o = mid;
    else oe = mid;
  }
  for (; p < pe; ++o) {
    const ulonglong2 seg = M.seg[o];
    const int64_t end = min(pe, (int64_t)M.first[o + 1]);
    const int32_t* rows = reinterpret_cast<const int32_t*>(seg.x) + p + lane;
    const V* vals = reinterpret_cast<const V*>(seg.y) + p + lane;
    for (int n = (int)(end - p); n > 0; n -= 32 * U) {  // (warp-uniform)
      f(rows, vals, n - lane);
      rows += 32 * U;
      vals += 32 * U;
    }
    p = end;
  }
}

// Issues the loads of the chunk's rows.  Slots are handled in groups; groups
// past ns are skipped here and by every pass.
template <int B>
__device__ __forceinline__ void item_rows(const ItemMap<B>& M, const ItemSlots<B>& S, int c0,
                                          uint32_t (&r)[ITEM_SLOTS]) {
#pragma unroll
  for (int t0 = 0; t0 < ITEM_SLOTS; t0 += ITEM_GROUP) {
    if (t0 >= S.ns) break;  // (warp-uniform)
#pragma unroll
    for (int t = t0; t < t0 + ITEM_GROUP; ++t)
      r[t] = (uint32_t)__ldg(reinterpret_cast<const int32_t*>(M.seg[item_seg(M, S, t)].x) + (c0 + S.pos(t)));
  }
}

}  // namespace spk
