// spk_numeric.cu -- a4/a5 of the hot path for thread-block work items: the
// CTA-class columns and the row windows of heavy columns.  Accumulate the
// values and write each item's output rows sorted.
//
// Alg. 5 (HashAdd) keeps an insert-or-add table keyed by row and sorts it at
// the end; Sec. II-D allows a dense accumulator in place of the hash.  Here the
// table is indexed by the exact output rank of the row, taken from a bitmap of
// the item's rows (the symbolic pass's structure, rebuilt in shared memory):
//
//   pass A   every entry sets bit (r - lo) of a 64-bit-word row bitmap; the
//            first bit set in a word also sets the word's bit in a summary
//            bitmap (one bit per word)
//   rank     the non-empty words (found through the summary) get the
//            exclusive popcount prefix of the words before them, and are
//            listed in row order
//   pass B   every entry adds its value at acc[rank(r)], rank(r) =
//            prefix(word) + popcount(word & bits below r)
//   write    the listed words are expanded to rows in rank order (one thread
//            per word) and rows and acc[rank] are written out coalesced,
//            already in row order; the touched words are cleared for the next
//            item.
//
// The bitmap covers a slab of 2^slab_log2 rows (at most 2^20): an item whose
// rows span more is processed slab by slab.
//
// k_num_items (below) is this accumulator with the entries' rows in registers,
// as a flat bitmap or a compact word table; k_num_bitmap, which walks the
// entries once per pass, runs only for block_accumulator = 1 on slabs of more
// than 2^17 rows (from 2^20 on the bitmap fills the SM).
#include <mutex>
#include <type_traits>

#include "spk_common.cuh"
#include "spk_items.cuh"
#include "spk_launch.h"

namespace spk {

constexpr int NUM_SLAB_LOG2_MAX = 20;  // 2^20 rows: 128 KB of bitmap

__device__ __forceinline__ unsigned long long warp_incl_scan_u64(unsigned long long x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(SPK_FULL, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Block-wide exclusive scan of one 64-bit value per thread; `tmp` holds
// BLOCK/32 + 1 entries.  Contains __syncthreads().
template <int BLOCK>
__device__ __forceinline__ unsigned long long block_excl_scan_u64(unsigned long long x, unsigned long long* tmp,
                                                                  unsigned long long* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned long long inc = warp_incl_scan_u64(x, lane);
  if (lane == 31) tmp[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const unsigned long long v = lane < BLOCK / 32 ? tmp[lane] : 0ull;
    const unsigned long long vi = warp_incl_scan_u64(v, lane);
    if (lane < BLOCK / 32) tmp[lane] = vi - v;
    if (lane == 31) tmp[BLOCK / 32] = vi;
  }
  __syncthreads();
  const unsigned long long r = tmp[wid] + inc - x;
  *total = tmp[BLOCK / 32];
  __syncthreads();
  return r;
}

// Shared-memory layout of the bitmap kernel.
struct BitmapSmem {
  unsigned long long* bm;  // W64 words: row bitmap of the slab (kept zero between slabs)
  uint16_t* wpre;          // W64: exclusive popcount prefix of each non-empty word
  uint32_t* summ;          // NSW = max(1, W64/32): one bit per bitmap word (kept zero between slabs)
  uint16_t* nel;           // umax: the non-empty words in row order
  int32_t* rows;           // umax: output rows of the slab in rank order
  unsigned char* acc;      // umax values
  unsigned long long* red; // BLOCK/32 + 1 scan slots
  int W64, NSW, umax;
};

// Bitmap words per thread for `nwords` words: a power of two <= 32, so a
// thread's run of words sits inside one summary word.
template <int BLOCK>
__device__ __forceinline__ int words_per_thread(int nwords) {
  int per = 1;
  while (per * BLOCK < nwords && per < 32) per <<= 1;
  return per;
}

// The summary bits of words [w0, w0 + per) (per a power of two <= 32, w0 a multiple of per).
__device__ __forceinline__ uint32_t own_word_mask(const uint32_t* summ, int w0, int per, int nwords) {
  if (w0 >= nwords) return 0u;
  const uint32_t all = summ[w0 >> 5] >> (w0 & 31);
  return per == 32 ? all : (all & ((1u << per) - 1u));
}

// Item filter of a launch over one problem kind (a check: the records it is
// given are grouped by kind, so it keeps them all): 0 float, 1 double, 2
// float with k <= FP32_ACC_TERMS, 3 float with FP32_ACC_TERMS < k <=
// FP32_PHASED_MAX_K, 4 float with larger k; -1 (a batch of one kind) keeps
// every item.
__device__ __forceinline__ bool item_selected(int sel, const Inst* I) {
  if (sel == 1) return I->dtype == 1;
  if (I->dtype != 0) return false;
  if (sel == 2) return I->k <= FP32_ACC_TERMS;
  if (sel == 3) return I->k > FP32_ACC_TERMS && I->k <= FP32_PHASED_MAX_K;
  if (sel == 4) return I->k > FP32_PHASED_MAX_K;
  return true;
}

// Pass B of an item's slab: every entry's value added at its rank.  Without
// phases the sums stay in acc for the caller's write (returns false).
// PHASED (float sums of problems with k > FP32_ACC_TERMS): a slab whose
// s_ent entries on slab_u rows can give a row more than FP32_ACC_TERMS
// terms runs its inputs in phases of FP32_PHASE_INPUTS; after each phase the
// slab's first `lim` partial sums are added into B's values (the first phase
// stores them) and acc is zeroed (returns true: the values are written).
template <typename V, typename A, bool PHASED, int BLOCK, int U, typename SegF, typename FAdd>
__device__ __forceinline__ bool add_values(const Inputs& in, int k, int off, SegF& seg, FAdd& add, SegCache& sc,
                                           A* acc, V* oval, int slab_u, int lim, int s_ent) {
  auto none = [](uint32_t, int32_t, V) {};
  if constexpr (PHASED)
    if (s_ent - slab_u >= FP32_ACC_TERMS) {
      for (int p0 = 0; p0 < k; p0 += FP32_PHASE_INPUTS) {
        SegCache fresh{0, 0, false};  // a phase's chunks differ from pass A's
        block_for_each_entry<true, V, BLOCK, U>(in, p0, min(k, p0 + FP32_PHASE_INPUTS), off, seg, add, none, fresh);
        __syncthreads();
        for (int q = threadIdx.x; q < slab_u; q += BLOCK) {
          if (q < lim) oval[q] = p0 == 0 ? (V)acc[q] : oval[q] + (V)acc[q];
          acc[q] = A(0);
        }
        __syncthreads();
      }
      return true;
    }
  block_for_each_entry<true, V, BLOCK, U>(in, 0, k, off, seg, add, none, sc);
  return false;
}

// One item (a CTA-class column or a heavy column's row window [r_lo, r_hi),
// Alg. 8: B(r1:r2, j) <- HashAdd(A_1(r1:r2, j), ..., A_k(r1:r2, j))).
template <typename V, typename A, bool PHASED, int BLOCK, int U>
__device__ __forceinline__ void bitmap_item(const Inputs& in, const Window& W, const Inst* I, const int32_t* offs,
                                            int32_t* __restrict__ out_row, V* __restrict__ out_val,
                                            const BitmapSmem& sm, int slab_log2, Counters* ctr_w) {
  const int k = I->k, off = I->ptr_off, j = W.col - I->colbase;
  A* acc = reinterpret_cast<A*>(sm.acc);
  const int64_t S = (int64_t)1 << slab_log2;
  const int64_t span = (int64_t)W.r_hi - W.r_lo;
  const int nsl = span <= 0 ? 0 : (int)((span + S - 1) >> slab_log2);
  int u_done = 0;
  bool bad = false;
  for (int t = 0; t < nsl; ++t) {
    const int lo = W.r_lo + (int)(t * S);
    const int hi = (int)min((int64_t)W.r_hi, (int64_t)lo + S);
    const uint32_t width = (uint32_t)(hi - lo);
    // The item's entries of input i that fall in [lo, hi).
    auto seg = [&](int i, int* beg, int* len) {
      int b, e;
      if (W.search < 0) {
        const int32_t* cp = in.cp[off + i];
        b = __ldg(cp + j);
        e = __ldg(cp + j + 1);
      } else {
        const int32_t* o = offs + ((int64_t)W.search * in.kmax + i) * 2;
        b = o[0];
        e = max(b, o[1]);  // (rows out of order: the next window may start further down)
      }
      if (nsl > 1 && in.sorted) {  // unordered inputs: the whole segment, rows outside the slab skipped
        const int32_t* ri = in.ri[off + i];
        b = lower_bound_i32(ri, b, e, lo);
        e = lower_bound_i32(ri, b, e, hi);
      }
      *beg = b;
      *len = e - b;
    };
    // Pass A: row bits (rows outside the slab are ignored: they cannot occur
    // for valid inputs, and shared-memory accesses stay in bounds).
    int n_ent = 0;  // PHASED: entries this thread met in the slab
    auto setbit = [&](int32_t r, V) -> uint32_t {
      const uint32_t rr = (uint32_t)(r - lo);
      if constexpr (PHASED) n_ent += rr < width;
      return (rr < width && set_row_bit(sm.bm, rr)) ? 1u : 0u;
    };
    auto mark_word = [&](uint32_t fresh, int32_t r, V) {
      if (fresh) {
        const uint32_t w = (uint32_t)(r - lo) >> 6;
        atomicOr(&sm.summ[w >> 5], 1u << (w & 31));
      }
    };
    SegCache sc{0, 0, false};
    block_for_each_entry<false, V, BLOCK, U, decltype(seg), decltype(setbit), decltype(mark_word), true>(
        in, k, off, seg, setbit, mark_word, sc);
    __syncthreads();
    int s_ent = 0;
    if constexpr (PHASED) block_excl_scan<BLOCK>(n_ent, reinterpret_cast<int*>(sm.red), &s_ent);
    // Rank prefix: thread t owns bitmap words [t*per, t*per + per); their
    // non-empty ones are the set bits of `mine` (kept for the clear below).
    const int nwords = (int)((width + 63) >> 6);
    const int per = words_per_thread<BLOCK>(nwords);
    if (per * BLOCK < nwords) {  // the host sizes blocks so this cannot happen; never skip words silently
      if (threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
      bad = true;
    }
    const int w0 = threadIdx.x * per;
    const uint32_t mine = own_word_mask(sm.summ, w0, per, nwords);
    unsigned long long loc = (unsigned long long)__popc(mine) << 32;  // (non-empty words << 32) | rows
    for (uint32_t bits = mine; bits; bits &= bits - 1) loc += (unsigned long long)__popcll(sm.bm[w0 + __ffs(bits) - 1]);
    unsigned long long tot;
    const unsigned long long ex = block_excl_scan_u64<BLOCK>(loc, sm.red, &tot);
    const int slab_u = (int)(tot & 0xffffffffull);
    const int slab_ne = (int)(tot >> 32);
    const bool fits = u_done + slab_u <= sm.umax && !bad;
    if (fits) {
      int rank = (int)(ex & 0xffffffffull), pos = (int)(ex >> 32);
      for (uint32_t bits = mine; bits; bits &= bits - 1) {
        const int w = w0 + __ffs(bits) - 1;
        sm.wpre[w] = (uint16_t)rank;
        sm.nel[pos++] = (uint16_t)w;
        rank += __popcll(sm.bm[w]);
      }
      for (int q = threadIdx.x; q < slab_u; q += BLOCK) acc[q] = A(0);
    } else {
      bad = true;
    }
    __syncthreads();
    if (fits) {
      // Pass B: values at their rank.
      auto add = [&](int32_t r, V v) -> uint32_t {
        const uint32_t rr = (uint32_t)(r - lo);
        if (rr < width) {
          const uint32_t w = rr >> 6;
          const unsigned long long bits = sm.bm[w];
          const uint32_t below = rr & 63;
          const int q = (int)sm.wpre[w] + __popcll(below ? (bits << (64 - below)) : 0ull);
          if (bits && q < slab_u) atomicAdd(&acc[q], (A)v);
        }
        return 0u;
      };
      // Ranks past the symbolic count are never written (B holds W.u rows
      // here); they can only arise if the inputs changed between the passes.
      const bool written = add_values<V, A, PHASED, BLOCK, U>(in, k, off, seg, add, sc, acc, out_val + u_done, slab_u,
                                                              min(slab_u, W.u - u_done), s_ent);
      // Rows in rank order: one thread per non-empty word.
      for (int p = threadIdx.x; p < slab_ne; p += BLOCK) {
        const int w = sm.nel[p];
        int q = sm.wpre[w];
        const int rbase = lo + (w << 6);
        for (unsigned long long bits = sm.bm[w]; bits; bits &= bits - 1) sm.rows[q++] = rbase + __ffsll(bits) - 1;
      }
      __syncthreads();
      // Coalesced write of the slab's rows and values.
      const int lim = min(slab_u, W.u - u_done);
      int32_t* orow = out_row + u_done;
      V* oval = out_val + u_done;
      for (int q = threadIdx.x; q < lim; q += BLOCK) {
        orow[q] = sm.rows[q];
        if (!written) oval[q] = (V)acc[q];
      }
      u_done += slab_u;
    }
    // Clear this thread's words; then the summary.
    for (uint32_t bits = mine; bits; bits &= bits - 1) sm.bm[w0 + __ffs(bits) - 1] = 0ull;
    __syncthreads();
    for (int x = threadIdx.x; x < ((nwords + 31) >> 5); x += BLOCK) sm.summ[x] = 0u;
    __syncthreads();
  }
  if (threadIdx.x == 0 && (bad || u_done != W.u)) atomicOr(&ctr_w->err, ERR_INTERNAL);
}

// ---------------------------------------------------------------------------
// Items in registers (spk_items.cuh): the same exact-rank accumulator, with a
// layout picked per item slab:
//
//   flat     (at most 2^17 rows) one bit per row
//     pass A   every entry sets its row's bit
//     rank     popcount prefix over all words: wpre[w]
//     pass B   acc[wpre[w] + popcount(bits of w below r)] += value
//   compact  (up to 2^20 rows, at most umax of them present) a summary bit
//            per 32-row word, and a table of the non-empty words in row order
//     pass A1  every entry sets its word's summary bit
//     rank 1   popcount prefix over the summary: word w gets the compact index
//              c(w) = spre[w / 32] + popcount(summary bits below w)
//     pass A2  every entry sets its row's bit in cw[c(w)]
//     rank 2   popcount prefix over cw: wpre[c]
//     pass B   acc[wpre[c] + popcount(cw[c] & bits below r)] += value
//   write    values copied out in rank order; then the words expanded to rows
//            in the accumulator's slots (free once the values are out) and
//            copied out, so both are written coalesced
//
// The rows are read once, into registers, for items of one chunk; the value
// segments start toward L2 while the rows are ranked.
// What bounds it: issue slots and shared-memory wavefronts at once (60% and 55%
// busy on 2^15 columns of 2048 entries, 128 distinct rows; the rest is barriers).
// Measured against three walks over the entries with a segment search each:
// 131072 such columns (float) 3.23 -> 2.14 ms, R-MAT scale 20 k = 64 12.7 ->
// 10.6 ms, 65537 unordered ragged columns 1.20 -> 0.60 ms.
// ---------------------------------------------------------------------------
constexpr int FLAT_LOG2 = 17;  // rows of a flat slab: 16 KB of bits
constexpr int FLAT_ROWS = 1 << FLAT_LOG2;

// A flat bitmap word's place: four pad words after every 16, so that threads
// owning 16 consecutive words each start their 16-byte loads on their own banks.
__host__ __device__ constexpr int pad_word(int w) { return w + ((w >> 4) << 2); }

// Shared-memory layout.  WIDE: slabs above FLAT_ROWS occur (both forms may run).
template <bool WIDE, int B>
struct ItemLayout {
  int wflat;      // words of the flat bitmap
  int zero;       // words kept zero between slabs: flat bits, or summary + compact words
  int pre;        // bytes of prefixes: flat wpre, or spre + compact wpre
  size_t acc;     // bytes of the accumulator (at least 4 per rank: it holds the rows at the end)
  __host__ __device__ ItemLayout(int slab_log2, int umax, int asize) {
    const int fl = slab_log2 < FLAT_LOG2 ? slab_log2 : FLAT_LOG2;
    wflat = 1 << (fl - 5);
    if (wflat < 4 * B) wflat = 4 * B;
    zero = pad_word(wflat);
    pre = 2 * wflat;
    if (WIDE) {
      if (zero < 1024 + umax) zero = 1024 + umax;
      if (pre < 2 * (1024 + umax)) pre = 2 * (1024 + umax);
    }
    zero = (zero + 3) & ~3;
    pre = (pre + 15) & ~15;
    acc = ((size_t)umax * asize + 15) & ~(size_t)15;
  }
  __host__ __device__ size_t bytes() const { return acc + (size_t)zero * 4 + pre + sizeof(ItemMap<B>) + 2 * sizeof(Window); }
};

template <int B>
struct ItemSmem {
  unsigned char* acc;
  uint32_t* zero;  // flat bits / summary, then cw
  uint16_t* pre;   // flat wpre / spre, then compact wpre
  ItemMap<B>* map;
  Window* win;     // this item's record and the next one's, by turns
  int umax;
};

// Threads per block: 256 for CTA-class columns (at most 4096 entries: one chunk,
// four blocks per SM), 384 for the windows of heavy columns (window_max distinct
// rows, mostly under 6144 entries; 512 threads measured 808 against 750 us on 96
// columns of 480,000 entries, since more warps run with part of their slots).
constexpr int CTA_ITEM_BLOCK = 256, HEAVY_ITEM_BLOCK = 384;
// Rows in registers, chunk by chunk (one chunk in CTA-class columns); the same,
// but items of several chunks and long segments walked in runs; all walked.
enum : int { ITEM_CHUNK, ITEM_BOTH, ITEM_WALK };
// Entries per segment from which an item of more than a chunk is walked in runs.
constexpr int ITEM_LONG = 128;

// Input i's part of the item of window W in column j.
__device__ __forceinline__ void window_seg(const Inputs& in, const Window& W, const int32_t* offs, int off, int j, int i,
                                           int* beg, int* end) {
  if (W.search < 0) {
    const int32_t* cp = in.cp[off + i];
    *beg = __ldg(cp + j);
    *end = __ldg(cp + j + 1);
  } else {
    const int32_t* o = offs + ((int64_t)W.search * in.kmax + i) * 2;
    *beg = o[0];
    *end = o[1];
  }
}

// One item, the record at sm.win[turn].  F holds the bounds of its first segment
// table (read while the previous item ran) and leaves with those of the next
// item, whose record (null: none) goes to sm.win[turn ^ 1].
template <typename V, typename A, bool PHASED, bool WIDE, int B, int MODE>
__device__ __forceinline__ void reg_item(const Inputs& in, const Window* next, int turn, ItemBounds<B>& F,
                                         const int32_t* offs, int32_t* __restrict__ out_row, V* __restrict__ out_val,
                                         const ItemSmem<B>& sm, int slab_log2, int flat_rows, Counters* ctr_w) {
  constexpr int KT = ItemMap<B>::KT, CAP = ItemMap<B>::CAP;
  constexpr bool WALK = MODE != ITEM_CHUNK, REGS = MODE != ITEM_WALK;
  const int tid = threadIdx.x;
  const Window& W = sm.win[turn];
  const Inst* I = in.inst + inst_of(in, W.col);
  const int k = I->k, off = I->ptr_off, j = W.col - I->colbase;
  int next_word = 0;
  if (next && tid < (int)(sizeof(Window) / 4)) next_word = reinterpret_cast<const int32_t*>(next)[tid];
  auto next_bounds = [&]() {
    const Window& Wn = sm.win[turn ^ 1];
    const Inst* In = in.inst + inst_of(in, Wn.col);
    const int jn = Wn.col - In->colbase, offn = In->ptr_off;
    auto segn = [&](int i, int* beg, int* end) { window_seg(in, Wn, offs, offn, jn, i, beg, end); };
    return item_bounds<B>(0, min(In->k, KT), segn);
  };
  A* acc = reinterpret_cast<A*>(sm.acc);
  ItemMap<B>& M = *sm.map;
  uint32_t* bits = sm.zero;      // flat
  uint16_t* wpre = sm.pre;
  uint32_t* summ = sm.zero;      // compact
  uint32_t* cw = sm.zero + 1024;
  uint16_t* spre = sm.pre;
  uint16_t* cpre = sm.pre + 1024;
  const int64_t S = (int64_t)1 << slab_log2;
  const int64_t span = (int64_t)W.r_hi - W.r_lo;
  const int nsl = span <= 0 ? 0 : (int)((span + S - 1) >> slab_log2);
  // Several slabs: of a CTA-class column, one chunk, every slab takes all entries
  // and skips the rows outside it.  A binary search's dozen dependent loads take
  // longer than reading the rows again (25000 columns of 1200 entries in 16 inputs,
  // 2^21 rows, float: 2369 -> 1950 us).  (Larger items would search, but the windows
  // of a heavy column end with its slabs.)
  constexpr bool KEEP = B == CTA_ITEM_BLOCK && MODE == ITEM_CHUNK;
  int u_done = 0;
  bool bad = false;
  for (int t = 0; t < nsl; ++t) {
    const int lo = W.r_lo + (int)(t * S);
    const int hi = (int)min((int64_t)W.r_hi, (int64_t)lo + S);
    const uint32_t width = (uint32_t)(hi - lo);
    const bool flat = !WIDE || width <= (uint32_t)flat_rows;
    // The item's entries of input i.
    auto seg = [&](int i, int* beg, int* end) {
      int b, e;
      window_seg(in, W, offs, off, j, i, &b, &e);
      if (!KEEP && nsl > 1 && in.sorted) {
        const int32_t* ri = in.ri[off + i];
        b = lower_bound_i32(ri, b, e, lo);
        e = lower_bound_i32(ri, b, e, hi);
      }
      *beg = b;
      *end = e;
    };
    uint32_t r[REGS ? ITEM_SLOTS : 1];  // rows less lo
    ItemSlots<B> L;
    int total = 0;  // positions of the current segment table
    L.ns = 0;
    const int nib = (k + KT - 1) / KT;
    bool single = false;  // the whole item sits in r[]
    int s_ent = 0;
    auto table = [&](int ib, bool first, int* red) {
      const int k_lo = ib * KT, nk = min(KT, k - k_lo);
      if (!(first && ib == 0 && (KEEP ? t == 0 || nib == 1 : nsl == 1))) F = item_bounds<B>(k_lo, nk, seg);
      if (!first) {
        total = item_table<sizeof(V), false, false>(M, in, off, k_lo, nk, F, red);
        return;
      }
      total = item_table<sizeof(V), true, REGS>(M, in, off, k_lo, nk, F, red);
      if (t == 0 && ib == 0 && next && tid < (int)(sizeof(Window) / 4))  // (every thread is past the previous item)
        reinterpret_cast<int32_t*>(&sm.win[turn ^ 1])[tid] = next_word;
      s_ent += total;
      single = REGS && nib == 1 && total <= CAP;
    };
    const uint32_t wmax = width - 1u;
    // Loaded rows to rows less lo; those outside the slab become 0xffffffff.
    auto relative = [&]() {
      if constexpr (REGS) {
#pragma unroll
        for (int q0 = 0; q0 < ITEM_SLOTS; q0 += ITEM_GROUP) {
          if (q0 >= L.ns) break;  // (warp-uniform)
#pragma unroll
          for (int q = q0; q < q0 + ITEM_GROUP; ++q) {
            r[q] -= (uint32_t)lo;
            r[q] = r[q] <= wmax ? r[q] : 0xffffffffu;
          }
        }
      }
    };
    // Compact index of a row's word.
    auto compact = [&](uint32_t c) {
      const uint32_t wd = c >> 5;
      return (int)spre[wd >> 5] + __popc(summ[wd >> 5] & ((1u << (wd & 31)) - 1u));
    };
    // Long segments: barrier-free runs instead of chunks.  (The table is published.)
    auto long_segments = [&]() { return !REGS || (WALK && total > CAP && total >= ITEM_LONG * M.ne); };
    // Runs mark(row less lo) over the rows.  A single-chunk item is loaded by the
    // first call only; others reload their rows (and rebuild the map) each time.
    auto rows_pass = [&](bool first, auto&& mark) {
      auto slots = [&]() {
        if constexpr (REGS) {
#pragma unroll
          for (int q0 = 0; q0 < ITEM_SLOTS; q0 += ITEM_GROUP) {
            if (q0 >= L.ns) break;  // (warp-uniform)
#pragma unroll
            for (int q = q0; q < q0 + ITEM_GROUP; ++q) mark(r[q]);
          }
        }
      };
      if (!first && single) {
        slots();
        return;
      }
      for (int ib = 0; ib < nib; ++ib) {
        if (first || nib > 1) {
          if (nib > 1) __syncthreads();
          table(ib, first, M.red[0]);
          if (!first) __syncthreads();
        }
        if (WALK && (!REGS || total > CAP)) {
          if (first) __syncthreads();
          if (long_segments()) {
            item_walk<B, V, 8>(M, 0, total, [&](const int32_t* rows, const V*, int n) {
              uint32_t x[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                x[u] = 0xffffffffu;
                if (32 * u < n) x[u] = (uint32_t)__ldg(rows + 32 * u) - (uint32_t)lo;
              }
#pragma unroll
              for (int u = 0; u < 8; ++u) mark(x[u]);
            });
            if (REGS && first) {
              __syncthreads();
              item_unmap(M);
            }
            continue;
          }
        }
        if constexpr (REGS) {
          for (int c0 = 0; total > 0; c0 += CAP) {
            if (!first || c0 > 0) item_map(M, c0);
            __syncthreads();
            L.init(c0, total);
            item_rows(M, L, c0, r);
            relative();
            slots();
            if (single) break;
            __syncthreads();
            item_unmap(M);
            __syncthreads();
            if (total - c0 <= CAP) break;
          }
        }
      }
    };
    int slab_u = 0, ne = 0;
    bool fits;
    const int nwords = (int)((width + 31) >> 5);
    // Ownership of words for the rank scans: `per` consecutive words a thread.
    const int per = nwords <= 4 * B ? 4 : (nwords <= 8 * B ? 8 : 16);
    // The passes have no branches: addresses come from the row clamped into
    // the slab, and only the atomic itself is predicated.
    rows_pass(true, [&](uint32_t x) {
      const uint32_t c = min(x, wmax);
      uint32_t* w = flat ? &bits[pad_word((int)(c >> 5))] : &summ[c >> 10];
      const uint32_t bit = 1u << (flat ? c & 31 : (c >> 5) & 31);
      if (x <= wmax) atomicOr(w, bit);
    });
    __syncthreads();
    if (t == nsl - 1 && nib == 1 && next) F = next_bounds();  // used when the next item starts
    if (flat) {
      const uint4* own = reinterpret_cast<const uint4*>(bits + pad_word(tid * per));
      int loc = 0;
      if (tid * per < nwords)
        for (int x = 0; x < per / 4; ++x) {
          const uint4 w = own[x];
          loc += __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
        }
      int run = item_scan<B>(loc, M.red[1], &slab_u);
      fits = u_done + slab_u <= sm.umax && !bad;
      if (tid * per < nwords)
        for (int x = 0; x < per / 4; ++x) {
          const uint4 w = own[x];
          const int a1 = run + __popc(w.x), a2 = a1 + __popc(w.y), a3 = a2 + __popc(w.z);
          uint2 p;
          p.x = (uint32_t)run | ((uint32_t)a1 << 16);
          p.y = (uint32_t)a2 | ((uint32_t)a3 << 16);
          *reinterpret_cast<uint2*>(wpre + tid * per + 4 * x) = p;
          run = a3 + __popc(w.w);
        }
    } else {
      // Rank 1: thread t < 256 owns summary words [4t, 4t + 4) (1024 in all).
      const bool sum4 = tid < 256;
      uint4 w = make_uint4(0u, 0u, 0u, 0u);
      if (sum4) w = *reinterpret_cast<const uint4*>(summ + 4 * tid);
      const int n0 = __popc(w.x), n1 = __popc(w.y), n2 = __popc(w.z);
      const int run1 = item_scan<B>(n0 + n1 + n2 + __popc(w.w), M.red[1], &ne);
      uint2 p;
      p.x = (uint32_t)run1 | ((uint32_t)(run1 + n0) << 16);
      p.y = (uint32_t)(run1 + n0 + n1) | ((uint32_t)(run1 + n0 + n1 + n2) << 16);
      if (sum4) *reinterpret_cast<uint2*>(spre + 4 * tid) = p;
      __syncthreads();
      fits = ne <= sm.umax && !bad;
      if (fits) {
        rows_pass(false, [&](uint32_t x) {
          const uint32_t c = min(x, wmax);
          const int cc = compact(c);
          if (x <= wmax && cc < ne) atomicOr(&cw[cc], 1u << (c & 31));
        });
        __syncthreads();
        const int pc = ne <= 4 * B ? 4 : (ne <= 8 * B ? 8 : 16);
        int loc = 0;
        for (int c = tid * pc; c < min(ne, tid * pc + pc); ++c) loc += __popc(cw[c]);
        int run = item_scan<B>(loc, M.red[0], &slab_u);
        fits = u_done + slab_u <= sm.umax;
        if (fits)
          for (int c = tid * pc; c < min(ne, tid * pc + pc); ++c) {
            cpre[c] = (uint16_t)run;
            run += __popc(cw[c]);
          }
      }
    }
    if (fits)
      for (int q = tid; q < slab_u; q += B) acc[q] = A(0);
    else
      bad = true;
    __syncthreads();
    // Ranks past the symbolic count are never written (B holds W.u rows
    // here); they can only arise if the inputs changed between the passes.
    const int lim = min(slab_u, W.u - u_done);
    int32_t* orow = out_row + u_done;
    V* oval = out_val + u_done;
    const bool phased = PHASED && s_ent - slab_u >= FP32_ACC_TERMS;
    const bool by_entry = single && !phased;  // rows are written from r[]
    if (fits && slab_u > 0) {
      // Pass B.
      for (int ib = 0; ib < nib; ++ib) {
        const int nk = min(KT, k - ib * KT);
        if (nib > 1) {
          __syncthreads();
          table(ib, false, M.red[1]);
          __syncthreads();
        }
        const int nph = phased ? (nk + FP32_PHASE_INPUTS - 1) / FP32_PHASE_INPUTS : 1;
        for (int ph = 0; ph < nph; ++ph) {
          const int e_lo = phased ? M.phase[ph] : 0;
          const int e_hi = phased && ph + 1 < nph ? M.phase[ph + 1] : total;
          // Rank of row x less lo (none for rows outside the slab).
          auto rank_of = [&](uint32_t x) {
            const uint32_t c = min(x, wmax);
            uint32_t wbits;
            int base;
            if (flat) {
              wbits = bits[pad_word((int)(c >> 5))];
              base = wpre[c >> 5];
            } else {
              const int cc = min(ne - 1, compact(c));
              wbits = cw[cc];
              base = cpre[cc];
            }
            const uint32_t rank = (uint32_t)(base + __popc(wbits & ((1u << (c & 31)) - 1u)));
            return x > wmax ? 0xffffffffu : rank;
          };
          const bool walk = !single && long_segments();
          if (WALK && walk && e_lo < e_hi)
            item_walk<B, V, 4>(M, e_lo, e_hi, [&](const int32_t* rows, const V* vals, int n) {
              uint32_t x[4];
              V v[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                x[u] = 0xffffffffu;
                v[u] = V(0);
                if (32 * u < n) {
                  x[u] = (uint32_t)__ldg(rows + 32 * u) - (uint32_t)lo;
                  v[u] = __ldg(vals + 32 * u);
                }
              }
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const uint32_t rank = rank_of(x[u]);
                if (rank < (uint32_t)slab_u) atomicAdd(&acc[rank], (A)v[u]);
              }
            });
          for (int c0 = 0; REGS && !walk && e_lo < e_hi; c0 += CAP) {
            if (c0 + (CAP - 1) >= e_lo) {
              if (!single) {
                item_map(M, c0);
                __syncthreads();
                L.init(c0, total);
                if constexpr (REGS) item_rows(M, L, c0, r);
                relative();
              }
              if constexpr (REGS) {
#pragma unroll
                for (int q0 = 0; q0 < ITEM_SLOTS; q0 += ITEM_GROUP) {
                  if (q0 >= L.ns) break;  // (warp-uniform)
                  uint32_t rank[ITEM_GROUP];
                  V v[ITEM_GROUP];
#pragma unroll
                  for (int x = 0; x < ITEM_GROUP; ++x)
                    v[x] = __ldg(reinterpret_cast<const V*>(M.seg[item_seg(M, L, q0 + x)].y) + (c0 + L.pos(q0 + x)));
#pragma unroll
                  for (int x = 0; x < ITEM_GROUP; ++x) {
                    const int q = q0 + x;
                    rank[x] = rank_of(r[q]);
                    // Row and rank together (20 + 12 bits) for the rows' write below.
                    if (by_entry) r[q] = r[q] <= wmax ? r[q] | (rank[x] << 20) : 0xffffffffu;
                    bool ok = L.live(q);
                    if (PHASED && phased) {
                      const int e = c0 + L.run + 32 * q + (tid & 31);
                      ok = ok && e >= e_lo && e < e_hi;
                    }
                    if (!ok) rank[x] = 0xffffffffu;
                  }
#pragma unroll
                  for (int x = 0; x < ITEM_GROUP; ++x)
                    if (rank[x] < (uint32_t)slab_u) atomicAdd(&acc[rank[x]], (A)v[x]);
                }
              }
              if (!single) {
                __syncthreads();
                item_unmap(M);
                __syncthreads();
              }
            }
            if (single || e_hi - c0 <= CAP) break;
          }
          if (phased) {
            // The phase's sums join B's values (the first phase stores them).
            __syncthreads();
            for (int q = tid; q < slab_u; q += B) {
              if (q < lim) oval[q] = ib + ph == 0 ? (V)acc[q] : oval[q] + (V)acc[q];
              acc[q] = A(0);
            }
            __syncthreads();
          }
        }
      }
      __syncthreads();
      if (!phased)
        for (int q = tid; q < lim; q += B) oval[q] = (V)acc[q];
      // The non-empty words in row order, in the segment table's place (free now).
      uint16_t* nel = reinterpret_cast<uint16_t*>(M.seg);
      if (!flat && !by_entry && tid < 256) {
        const uint4 w4 = *reinterpret_cast<const uint4*>(summ + 4 * tid);
        int c = spre[4 * tid];
#pragma unroll
        for (int x = 0; x < 4; ++x)
          for (uint32_t wb = x == 0 ? w4.x : x == 1 ? w4.y : x == 2 ? w4.z : w4.w; wb; wb &= wb - 1)
            nel[c++] = (uint16_t)((4 * tid + x) * 32 + __ffs(wb) - 1);
      }
      __syncthreads();
      int32_t* rows = reinterpret_cast<int32_t*>(acc);  // slab_u <= umax slots of at least 4 bytes
      if (REGS && by_entry) {
        // Every entry writes its row at its rank (equal rows write the same).
        // All ones marks a slot without a row; its rank, 4095, is below slab_u
        // only for a whole column of 4096 rows, where every entry has one.
        if constexpr (REGS) {
#pragma unroll
          for (int q0 = 0; q0 < ITEM_SLOTS; q0 += ITEM_GROUP) {
            if (q0 >= L.ns) break;  // (warp-uniform)
#pragma unroll
            for (int q = q0; q < q0 + ITEM_GROUP; ++q)
              if ((r[q] >> 20) < (uint32_t)slab_u) rows[r[q] >> 20] = lo + (int)(r[q] & 0xfffffu);
          }
        }
      } else if (flat) {
        for (int w = tid; w < nwords; w += B) {
          int q = wpre[w];
          for (uint32_t wb = bits[pad_word(w)]; wb; wb &= wb - 1) rows[q++] = lo + (w << 5) + __ffs(wb) - 1;
        }
      } else {
        for (int c = tid; c < ne; c += B) {
          int q = cpre[c];
          const int rbase = lo + ((int)nel[c] << 5);
          for (uint32_t wb = cw[c]; wb; wb &= wb - 1) rows[q++] = rbase + __ffs(wb) - 1;
        }
      }
      item_unmap(M);
      __syncthreads();
      for (int q = tid; q < lim; q += B) orow[q] = rows[q];
      u_done += slab_u;
    } else {
      item_unmap(M);
    }
    // Zero words again, each thread its own (every reader is past the last barrier).
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    if (flat) {
      uint4* mine = reinterpret_cast<uint4*>(bits + pad_word(tid * per));
      if (tid * per < nwords)
        for (int x = 0; x < per / 4; ++x) mine[x] = z;
    } else {
      if (tid < 256) *reinterpret_cast<uint4*>(summ + 4 * tid) = z;
      for (int c = tid; c < min(ne, sm.umax); c += B) cw[c] = 0u;
    }
    // (The next slab's or item's table has two barriers before anything here is reused.)
  }
  if (next && k > KT) F = next_bounds();  // (tables of more inputs go through F)
  if (tid == 0 && (bad || u_done != W.u)) atomicOr(&ctr_w->err, ERR_INTERNAL);
}

// DT: 0 = float values, 1 = double values; ACC: 0 sums in the value type, 1
// float sums in phases, 2 float values summed in double.

template <int DT, int ACC, bool WIDE, int B, int MODE>
__global__ void __launch_bounds__(B, B == CTA_ITEM_BLOCK ? 4 : 2)
    k_num_items(Inputs in, const Window* __restrict__ win, int nwin, const int32_t* __restrict__ offs,
                const int64_t* __restrict__ col_ptr, Outs o, int slab_log2, int umax, int flat_rows, int only_dtype,
                Counters* ctr_w) {
  using V = typename std::conditional<DT == 1, double, float>::type;
  using A = typename std::conditional<DT == 1 || ACC == 2, double, float>::type;  // accumulator
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const ItemLayout<WIDE, B> L(slab_log2, umax, (int)sizeof(A));
  ItemSmem<B> sm;
  sm.umax = umax;
  sm.acc = sm_raw;
  sm.zero = reinterpret_cast<uint32_t*>(sm.acc + L.acc);
  sm.pre = reinterpret_cast<uint16_t*>(sm.zero + L.zero);
  sm.map = reinterpret_cast<ItemMap<B>*>(reinterpret_cast<unsigned char*>(sm.pre) + L.pre);
  sm.win = reinterpret_cast<Window*>(sm.map + 1);
  for (int x = threadIdx.x; x < L.zero; x += B) sm.zero[x] = 0u;
  item_unmap(*sm.map);
  // While an item runs, the next one's record and segment bounds are on their
  // way.  (The item filter only checks: every record belongs to this launch.)
  const int step = gridDim.x;
  int wi = blockIdx.x;
  if (wi >= nwin) return;
  if (threadIdx.x < sizeof(Window) / 4)
    reinterpret_cast<int32_t*>(sm.win)[threadIdx.x] = reinterpret_cast<const int32_t*>(win + wi)[threadIdx.x];
  __syncthreads();
  auto bounds = [&](const Window& W) {
    const Inst* I = in.inst + inst_of(in, W.col);
    const int j = W.col - I->colbase, off = I->ptr_off;
    auto seg = [&](int i, int* beg, int* end) { window_seg(in, W, offs, off, j, i, beg, end); };
    return item_bounds<B>(0, min(I->k, ItemMap<B>::KT), seg);
  };
  ItemBounds<B> F = bounds(sm.win[0]);
  for (int turn = 0;; turn ^= 1) {
    const Window& W = sm.win[turn];
    const int q = inst_of(in, W.col);
    const Inst* I = in.inst + q;
    if (only_dtype >= 0 && !item_selected(only_dtype, I)) {  // (cannot happen)
      if (threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
      return;
    }
    const bool more = wi + step < nwin;
    if (W.r_hi <= W.r_lo) {
      // An empty window: the column's last cut fell into the slab's last word.
      // It writes nothing, but the items after it are still this block's.
      if (threadIdx.x == 0 && W.u != 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
      if (!more) break;
      wi += step;
      __syncthreads();  // every thread is past the item before, whose record is replaced
      if (threadIdx.x < sizeof(Window) / 4)
        reinterpret_cast<int32_t*>(sm.win + (turn ^ 1))[threadIdx.x] =
            reinterpret_cast<const int32_t*>(win + wi)[threadIdx.x];
      __syncthreads();
      F = bounds(sm.win[turn ^ 1]);
      continue;
    }
    const int64_t out = col_ptr[W.col] - (in.col_inst ? col_ptr[I->colbase] : 0) + W.out_off;
    reg_item<V, A, ACC == 1, WIDE, B, MODE>(in, more ? win + wi + step : nullptr, turn, F, offs, out_row_of(o, q) + out,
                                      static_cast<V*>(out_val_of(o, q)) + out, sm, slab_log2, flat_rows, ctr_w);
    if (!more) break;
    wi += step;
  }
}

// DT: 0 = float values, 1 = double values; ACC: 0 sums in the value type, 1
// float sums in phases, 2 float values summed in double.  A batch of several
// problem kinds runs the kernel once per kind over that kind's records
// (only_dtype: the item filter above).
template <int DT, int ACC, int BLOCK, int U>
__global__ void __launch_bounds__(BLOCK) k_num_bitmap(Inputs in, const Window* __restrict__ win, int nwin,
                                                      const int32_t* __restrict__ offs,
                                                      const int64_t* __restrict__ col_ptr, Outs o, int slab_log2,
                                                      int umax, int only_dtype, Counters* ctr_w) {
  using V = typename std::conditional<DT == 1, double, float>::type;
  using A = typename std::conditional<DT == 1 || ACC == 2, double, float>::type;  // accumulator
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ unsigned long long red[BLOCK / 32 + 1];
  BitmapSmem sm;
  sm.W64 = 1 << (slab_log2 - 6);
  sm.NSW = (sm.W64 + 31) >> 5;
  sm.umax = umax;
  sm.bm = reinterpret_cast<unsigned long long*>(sm_raw);
  sm.acc = reinterpret_cast<unsigned char*>(sm.bm + sm.W64);
  sm.wpre = reinterpret_cast<uint16_t*>(sm.acc + (size_t)umax * sizeof(A));
  sm.summ = reinterpret_cast<uint32_t*>(sm.wpre + ((sm.W64 + 1) & ~1));
  sm.rows = reinterpret_cast<int32_t*>(sm.summ + sm.NSW);
  sm.nel = reinterpret_cast<uint16_t*>(sm.rows + umax);
  sm.red = red;
  for (int x = threadIdx.x; x < sm.W64; x += BLOCK) sm.bm[x] = 0ull;
  for (int x = threadIdx.x; x < sm.NSW; x += BLOCK) sm.summ[x] = 0u;
  __syncthreads();
  // The next item's window record is fetched while the current item runs.
  Window Wn{};
  if (blockIdx.x < nwin) Wn = win[blockIdx.x];
  for (int wi = blockIdx.x; wi < nwin; wi += gridDim.x) {
    const Window W = Wn;
    if (wi + (int)gridDim.x < nwin) Wn = win[wi + gridDim.x];
    const int q = inst_of(in, W.col);
    const Inst* I = in.inst + q;
    if (only_dtype >= 0 && !item_selected(only_dtype, I)) continue;
    const int64_t out = col_ptr[W.col] - (in.col_inst ? col_ptr[I->colbase] : 0) + W.out_off;
    bitmap_item<V, A, ACC == 1, BLOCK, U>(in, W, I, offs, out_row_of(o, q) + out, static_cast<V*>(out_val_of(o, q)) + out, sm,
                             slab_log2, ctr_w);
  }
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
// Lets a kernel's launches on the current device ask for all the dynamic shared
// memory that a block can have there.  The limit belongs to the kernel and the
// device, not to a launch: it is set once, to a number that depends on nothing
// else, so host threads launching the same kernel with other sizes never lower
// it under one another.
cudaError_t allow_smem(const void* fn) {
  struct Entry {
    int dev;
    const void* fn;
  };
  static std::mutex mu;
  static Entry done[512];
  static int ndone = 0;
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < ndone; ++i)
    if (done[i].fn == fn && done[i].dev == dev) return cudaSuccess;
  cudaFuncAttributes fa;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, fn);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  if (e == cudaSuccess && ndone < 512) done[ndone++] = Entry{dev, fn};
  return e;
}

// Resident blocks per SM of a kernel at a block size and dynamic shared
// memory size (registers, shared memory and threads all counted), or 0 on
// error; its launches may then ask for that size.  Cached per device: the
// query is not free.
int resident_blocks(const void* fn, int block, size_t smem) {
  struct Entry {
    int dev;
    const void* fn;
    int block;
    size_t smem;
    int blocks;
  };
  static std::mutex mu;
  static Entry cache[256];
  static int ncache = 0;
  int dev = 0, b = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();  // not sticky: leave no stale error for the next check
    return 0;
  }
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < ncache; ++i)
    if (cache[i].fn == fn && cache[i].block == block && cache[i].smem == smem && cache[i].dev == dev)
      return cache[i].blocks;
  if (allow_smem(fn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, block, smem) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  if (b > 0 && ncache < 256) cache[ncache++] = Entry{dev, fn, block, smem, b};
  return b;
}

// Shared bytes of the flat-bitmap kernel for a slab of 2^slab_log2 rows, umax ranks.
static size_t bitmap_smem_bytes(int slab_log2, int umax, size_t vsize) {
  const size_t w64 = (size_t)1 << (slab_log2 - 6);
  const size_t nsw = (w64 + 31) / 32;
  return w64 * 8 + (size_t)umax * vsize + ((w64 + 1) & ~(size_t)1) * 2 + nsw * 4 + (size_t)umax * 4 +
         (size_t)umax * 2 + 16;
}

template <typename K>
static cudaError_t launch_items(K kern, int block, int blocks_per_sm, const Inputs& in, const Window* win, int n_win,
                                const int32_t* offs, const int64_t* col_ptr, const Outs& out, int slab_log2, int umax,
                                size_t smem, int only_dtype, Counters* ctr_w, const DeviceInfo& dev, cudaStream_t st) {
  if (blocks_per_sm < 1) return cudaErrorInvalidConfiguration;
  int grid = dev.sms * blocks_per_sm;
  if (grid > n_win) grid = n_win;
  if (grid < 1) return cudaSuccess;
  kern<<<grid, block, smem, st>>>(in, win, n_win, offs, col_ptr, out, slab_log2, umax, only_dtype, ctr_w);
  return cudaGetLastError();
}

template <int DT, int ACC, bool WIDE, int B, int MODE>
static cudaError_t launch_reg_items(const Inputs& in, const Window* win, int n_win, const int32_t* offs,
                                    const int64_t* col_ptr, const Outs& out, int slab_log2, int umax, int flat_rows,
                                    int only_dtype, Counters* ctr_w, const DeviceInfo& dev, cudaStream_t st) {
  auto kern = k_num_items<DT, ACC, WIDE, B, MODE>;
  const size_t smem = ItemLayout<WIDE, B>(slab_log2, umax, (DT == 1 || ACC == 2) ? 8 : 4).bytes();
  const int bps = resident_blocks((const void*)kern, B, smem);
  if (bps < 1) return cudaErrorInvalidConfiguration;
  int grid = dev.sms * bps;
  if (grid > n_win) grid = n_win;
  if (grid < 1) return cudaSuccess;
  kern<<<grid, B, smem, st>>>(in, win, n_win, offs, col_ptr, out, slab_log2, umax, flat_rows, only_dtype, ctr_w);
  return cudaGetLastError();
}

// accumulator: 0 = automatic (slabs of at most FLAT_ROWS rows flat, larger
// ones compact), 1 = flat bitmap, 2 = compact word table.  A flat bitmap of
// more than FLAT_ROWS rows fills the SM: one 1024-thread block.
template <int DT, int ACC>
static cudaError_t launch_num_cta_t(const Inputs& in, const Window* win, int n_win, bool heavy, const int32_t* offs,
                                    const int64_t* col_ptr, const Outs& out, int umax, int accumulator,
                                    int64_t heavy_mean, int only_dtype, Counters* ctr_w, const DeviceInfo& dev,
                                    cudaStream_t st) {
  constexpr size_t VS = (DT == 1 || ACC == 2) ? 8 : 4;  // accumulator bytes
  int slab_log2 = 10;
  while (slab_log2 < NUM_SLAB_LOG2_MAX && ((int64_t)1 << slab_log2) < (int64_t)in.mmax) ++slab_log2;
  if (accumulator == 1 && slab_log2 > FLAT_LOG2) {
    const size_t sf = bitmap_smem_bytes(slab_log2, umax, VS);
    const bool small = sf <= (size_t)dev.smem_per_sm / 2 - 2048;  // room for several blocks
    auto kern = small ? k_num_bitmap<DT, ACC, 256, 8> : k_num_bitmap<DT, ACC, 1024, 4>;
    const int block = small ? 256 : 1024;
    const int bf = sf <= (size_t)dev.smem_optin ? resident_blocks((const void*)kern, block, sf) : 0;
    return launch_items(kern, block, bf, in, win, n_win, offs, col_ptr, out, slab_log2, umax, sf, only_dtype, ctr_w,
                        dev, st);
  }
  const bool wide = accumulator == 2 || slab_log2 > FLAT_LOG2;
  const int flat_rows = accumulator == 2 ? 0 : FLAT_ROWS;
  // Heavy windows of flat slabs: blocks of 256 threads, or 384 while there are few
  // windows (750 columns of 40000 entries in 16 inputs, 2^15 rows, float: 458 us with
  // 384, 374 with 256; 122 windows of R-MAT scale 14: the call 222 and 232 us).
  // Compact ones: 384 (tall columns 719 against 903 us with 256), chunk by chunk (12
  // inputs of 1.7 M rows, 201 columns of 200,000 entries, double: the walk's code
  // spills, 710 -> 760 us, and windows hold little more than a chunk); but in unordered
  // inputs, whose windows read whole columns, 256 and walked from the start when the
  // columns are long and their segments too (2500 columns of 12000 entries in 16
  // inputs, 2^20 rows, float 1084 -> 981 us; of 6000 entries 1021 -> 1105 us).
  auto launch = wide ? launch_reg_items<DT, ACC, true, CTA_ITEM_BLOCK, ITEM_CHUNK>
                     : launch_reg_items<DT, ACC, false, CTA_ITEM_BLOCK, ITEM_CHUNK>;
  if (heavy && wide)
    launch = !in.sorted && heavy_mean >= 8192 && heavy_mean >= 100 * (int64_t)in.kmax
                 ? launch_reg_items<DT, ACC, true, CTA_ITEM_BLOCK, ITEM_WALK>
                 : launch_reg_items<DT, ACC, true, HEAVY_ITEM_BLOCK, ITEM_CHUNK>;
  else if (heavy)
    launch = n_win <= 4 * dev.sms ? launch_reg_items<DT, ACC, false, HEAVY_ITEM_BLOCK, ITEM_BOTH>
                                  : launch_reg_items<DT, ACC, false, CTA_ITEM_BLOCK, ITEM_BOTH>;
  return launch(in, win, n_win, offs, col_ptr, out, slab_log2, umax, flat_rows, only_dtype, ctr_w, dev, st);
}

// Batches of several problem kinds: after the symbolic phase the
// thread-block items' records are copied, grouped by class (CTA, then heavy)
// and kind (count, then place with warp-aggregated appends; order inside a
// group is arbitrary), so that each numeric launch reads only its own items.
// The numbers of records are read from the counters (at most `cap` in all).
__device__ __forceinline__ int record_group(const Inputs& in, const Window* win, int cap, int n_cta, int x,
                                            Window* W) {
  *W = x < n_cta ? win[x] : win[cap - 1 - (x - n_cta)];
  return item_kind(in.inst + inst_of(in, W->col)) + (x < n_cta ? 0 : 4);
}

__global__ void k_kind_count(Inputs in, const Window* __restrict__ win, int cap, Counters* ctr_w) {
  const int n_cta = min(ctr_w->n_windows, cap), nwin = min(n_cta + ctr_w->n_hwin, cap);
  const int stride = gridDim.x * blockDim.x;
  for (int w0 = blockIdx.x * blockDim.x; w0 < nwin; w0 += stride) {  // (block-uniform)
    const int x = w0 + (int)threadIdx.x;
    Window W;
    const int grp = x < nwin ? record_group(in, win, cap, n_cta, x, &W) : -1;
    for (int q = 0; q < 8; ++q) {
      const unsigned m = __ballot_sync(SPK_FULL, grp == q);
      if (m && (threadIdx.x & 31) == 0) atomicAdd(&ctr_w->kind_n[q], __popc(m));
    }
  }
}

__global__ void k_kind_place(Inputs in, const Window* __restrict__ win, int cap, Window* __restrict__ wsort,
                             Counters* ctr_w) {
  __shared__ int base[8];
  if (threadIdx.x == 0) {
    int b = 0;
    for (int q = 0; q < 8; ++q) {
      base[q] = b;
      b += ctr_w->kind_n[q];
    }
  }
  __syncthreads();
  const int n_cta = min(ctr_w->n_windows, cap), nwin = min(n_cta + ctr_w->n_hwin, cap);
  const int lane = threadIdx.x & 31;
  const int stride = gridDim.x * blockDim.x;
  for (int w0 = blockIdx.x * blockDim.x; w0 < nwin; w0 += stride) {  // (block-uniform)
    const int x = w0 + (int)threadIdx.x;
    Window W{};
    const int grp = x < nwin ? record_group(in, win, cap, n_cta, x, &W) : -1;
    for (int q = 0; q < 8; ++q) {
      const unsigned m = __ballot_sync(SPK_FULL, grp == q);
      if (!m) continue;
      const int leader = __ffs(m) - 1;
      int pos = 0;
      if (lane == leader) pos = atomicAdd(&ctr_w->kind_fill[q], __popc(m));
      pos = __shfl_sync(SPK_FULL, pos, leader);
      if (grp == q) wsort[base[q] + pos + __popc(m & ((1u << lane) - 1u))] = W;
    }
  }
}

int num_cta_kinds(int dt, int f32_kinds) { return (dt != 1 ? (f32_kinds & 7) : 0) | (dt != 0 ? 8 : 0); }

cudaError_t launch_kind_sort(const Inputs& in, const Window* win, int cap, Window* wsort, Counters* ctr_w,
                             const DeviceInfo& dev, cudaStream_t st) {
  if (cap <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(&ctr_w->kind_n[0], 0, 16 * sizeof(int32_t), st);  // kind_n, kind_fill
  if (e != cudaSuccess) return e;
  int blocks = (cap + 255) / 256;
  if (blocks > dev.sms * 8) blocks = dev.sms * 8;
  k_kind_count<<<blocks, 256, 0, st>>>(in, win, cap, ctr_w);
  k_kind_place<<<blocks, 256, 0, st>>>(in, win, cap, wsort, ctr_w);
  return cudaGetLastError();
}

cudaError_t launch_num_cta(const Inputs& in, int dt, int f32_kinds, const Window* win, int64_t win_cap, int n_cta,
                           int n_heavy, const Window* wsort, const int32_t* kind_n, const int32_t* offs,
                           const int64_t* col_ptr, const Outs& out, int window_max, int accumulator,
                           int64_t heavy_mean, Counters* ctr_w, const DeviceInfo& dev, cudaStream_t st,
                           int* launches) {
  *launches = 0;
  if (n_cta + n_heavy <= 0) return cudaSuccess;
  // Float problems: k <= FP32_ACC_TERMS sum in float, up to
  // FP32_PHASED_MAX_K in float by phases, beyond in double; each kind that
  // the batch holds gets its own launches, over its own groups of the records
  // (the item filter of kind q, sel[q], only checks that).
  const int kinds = num_cta_kinds(dt, f32_kinds);
  const bool alone = __builtin_popcount(kinds) == 1;
  constexpr int sel[4] = {2, 3, 4, 1};
  int base = 0;
  cudaError_t e = cudaSuccess;
  for (int g = 0; g < 8 && e == cudaSuccess; ++g) {
    const int q = g & 3;
    const bool heavy = g >= 4;
    if (!((kinds >> q) & 1)) continue;
    // A batch of one kind: its records where the symbolic phase left them
    // (CTA-class from the array's start, heavy at its end).
    const Window* w = alone ? (heavy ? win + (win_cap - n_heavy) : win) : wsort + base;
    const int n = alone ? (heavy ? n_heavy : n_cta) : kind_n[g];
    base += alone ? 0 : n;
    if (n <= 0) continue;
    ++*launches;
    const int f = alone ? -1 : sel[q];
    auto launch = q == 0 ? launch_num_cta_t<0, 0> : q == 1 ? launch_num_cta_t<0, 1>
                  : q == 2 ? launch_num_cta_t<0, 2> : launch_num_cta_t<1, 0>;
    e = launch(in, w, n, heavy, offs, col_ptr, out, window_max, accumulator, heavy_mean, f, ctr_w, dev, st);
  }
  return e;
}

}  // namespace spk
