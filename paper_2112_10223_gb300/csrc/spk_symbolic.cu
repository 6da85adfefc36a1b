// spk_symbolic.cu -- a2 of the hot path: nnz(B(:,j)) per column.
//
// Warp class (s_j <= warp_max): see spk_warp.cu.
// CTA class (s_j <= cta_max): one thread block per column, counting the bits its
//   rows are first to set (at most 2^20 rows), or an open-addressing table with
//   a multiplicative hash.  Emits one numeric work item per column.
// Heavy class: one thread block per column with a shared-memory bitmap of a
//   slab of up to 2^20 rows (the dense-accumulator form of the symbolic step,
//   which Sec. II-D allows in place of the hash).  Popcounts give nnz(B(:,j))
//   and cut the column into row windows of fewer than window_max distinct rows
//   each (Alg. 7/8's sliding windows, sized to shared memory and balanced by
//   count rather than by equal row ranges).  An optional compact form
//   (k_sym_heavy_compact) does the same from a summary bit per 32-row word
//   and a bounded table of non-empty words.
#include "spk_common.cuh"
#include "spk_items.cuh"
#include "spk_launch.h"

namespace spk {

template <int BLOCK, int U>
__global__ void __launch_bounds__(BLOCK) k_sym_cta(Inputs in, const int32_t* __restrict__ list,
                                                   const int32_t* __restrict__ s_arr, const Counters* __restrict__ ctr,
                                                   int32_t* __restrict__ u_out, Window* __restrict__ win,
                                                   int64_t win_cap, int tmax, Counters* ctr_w) {
  extern __shared__ int32_t keys[];
  __shared__ int red[BLOCK / 32 + 1];
  constexpr int NW = BLOCK / 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ncols = ctr->n_cta;
  for (int c = blockIdx.x; c < ncols; c += gridDim.x) {
    const int g = list[c];
    const Inst* I = in.inst + inst_of(in, g);
    const int k = I->k, off = I->ptr_off, j = g - I->colbase;
    const int s = s_arr[g];
    const int q = max(6, ceil_log2(2 * s));
    const int T = 1 << q;
    if (T > tmax) {
      if (threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
      continue;
    }
    for (int p = threadIdx.x; p < T; p += BLOCK) keys[p] = -1;
    __syncthreads();
    int newc = 0;
    const int nch = (k + 31) >> 5;
    const int groups = min(nch, NW);
    const int per = NW / groups;
    const int gid = wid / per, lw = wid - gid * per;
    for (int cb = gid * 32; gid < groups && cb < k; cb += groups * 32) {
      const int i = cb + lane;
      int beg = 0, len = 0;
      if (i < k) {
        const int32_t* cp = in.cp[off + i];
        beg = __ldg(cp + j);
        len = __ldg(cp + j + 1) - beg;
      }
      SegWalk w;
      w.init(beg, len, lane);
      for (int e0 = lw * 32 * U; e0 < w.total; e0 += per * 32 * U) {
        int32_t r[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
          r[t] = -1;
          if (e0 + t * 32 >= w.total) continue;  // (warp-uniform) slot wholly past the chunk's end
          const int e = e0 + t * 32 + lane;
          const int seg = w.find(e);
          const int idx = w.index_in_input(e, seg);
          if (e < w.total) r[t] = __ldg(in.ri[off + cb + seg] + idx);
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
          if (r[t] < 0) continue;
          uint32_t h = hash_scrambled(r[t], q);
          for (int probes = 0; probes < T; ++probes) {  // T > s_j keys: an empty slot is always found
            const int old = atomicCAS(&keys[h], -1, r[t]);
            if (old == -1) {
              ++newc;
              break;
            }
            if (old == r[t]) break;
            h = (h + 1) & (T - 1);
          }
        }
      }
    }
    int total;
    block_excl_scan<BLOCK>(newc, red, &total);
    if (threadIdx.x == 0) {
      u_out[g] = total;
      const int wi = atomicAdd(&ctr_w->n_windows, 1);
      if (wi < win_cap - ctr->n_hwin) {
        Window w;
        w.col = g;
        w.r_lo = 0;
        w.r_hi = I->m;
        w.u = total;
        w.out_off = 0;
        w.search = -1;
        win[wi] = w;
      } else {
        atomicOr(&ctr_w->err, ERR_WINDOW_CAP);
      }
    }
    __syncthreads();
  }
}

// CTA-class columns of at most 2^20 rows: the entries' rows in registers
// (spk_items.cuh), counted as the bits they are first to set.
//   !WIDE (at most 2^SYM_FLAT_LOG2 rows) one bit per row; a column of one
//         chunk clears the words it set, entry by entry.
//   WIDE  a summary bit per 32-row word first; then the row bits in a table of
//         the non-empty words, indexed by the summary's popcount prefix.
// Against the open-addressing table of k_sym_cta (a probe loop per entry, a
// five-shuffle segment search): 131072 columns of 2048 entries 1.64 -> 0.80 ms,
// R-MAT scale 20 1.11 -> 0.72 ms.  The table stays for more than 2^20 rows.
// Threads per block of the flat form: what an item costs beyond its entries
// (table, map, barriers: some 220 instructions a warp) is paid by fewer warps.
// (256 threads: 65537 unordered columns 855 against 833 us, a batch of 20 1069
// against 1042; 131072 columns of 2048 entries the same.)  Bitmaps of more than
// 2^17 rows leave shared memory for five blocks: those have 256 threads (R-MAT
// scale 18: 310 against 402 us).
constexpr int SYM_BLOCK = 128;
constexpr int SYM_FLAT_LOG2 = 18;  // 32 KB of bits

template <bool WIDE, int B>
__global__ void __launch_bounds__(B, 1280 / B) k_sym_items(Inputs in, const int32_t* __restrict__ list,
                                                             const Counters* __restrict__ ctr,
                                                             int32_t* __restrict__ u_out, Window* __restrict__ win,
                                                             int64_t win_cap, int words, const int32_t* __restrict__ s_arr,
                                                             DupList dup, Counters* ctr_w) {
  static_assert(!WIDE || B == 256, "four summary words a thread");
  using Map = ItemMap<B>;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  Map& M = *reinterpret_cast<Map*>(sm_raw);
  uint32_t* bits = reinterpret_cast<uint32_t*>(sm_raw + sizeof(Map));  // !WIDE: `words` words, kept zero
  uint32_t* summ = bits;                                                    // WIDE: 1024 words, kept zero
  uint32_t* cw = bits + 1024;                                               //   CTA_MAX_LIMIT words, kept zero
  uint16_t* spre = reinterpret_cast<uint16_t*>(cw + CTA_MAX_LIMIT);         //   1024 prefixes
  const int tid = threadIdx.x;
  __shared__ DupTally tally;
  if (tid == 0) tally.clear();
  for (int x = tid; x < (WIDE ? 1024 + CTA_MAX_LIMIT : words); x += B) bits[x] = 0u;
  item_unmap(M);
  __syncthreads();
  const int ncols = ctr->n_cta;
  // A column's bounds of its first segment table, read while the column before it runs.
  auto bounds = [&](int g, const Inst* I, int k_lo) {
    const int j = g - I->colbase, off = I->ptr_off;
    auto seg = [&](int i, int* beg, int* end) {
      const int32_t* cp = in.cp[off + i];
      *beg = __ldg(cp + j);
      *end = __ldg(cp + j + 1);
    };
    return item_bounds<B>(k_lo, min(Map::KT, I->k - k_lo), seg);
  };
  int c = blockIdx.x;
  if (c >= ncols) return;
  int gn = list[c];
  const Inst* In = in.inst + inst_of(in, gn);
  ItemBounds<B> Fn = bounds(gn, In, 0);
  for (; c < ncols; c += gridDim.x) {
    const int g = gn;
    const Inst* I = In;
    ItemBounds<B> F = Fn;
    const int k = I->k, off = I->ptr_off;
    const uint32_t m = (uint32_t)I->m;
    if (c + (int)gridDim.x < ncols) gn = list[c + gridDim.x];
    const int nib = (k + Map::KT - 1) / Map::KT;
    bool single = false;
    uint32_t r[ITEM_SLOTS];
    int total = 0;
    ItemSlots<B> L;
    auto rows_pass = [&](bool first, auto&& op) {
      if (!first && single) {
        op();
        return;
      }
      for (int ib = 0; ib < nib; ++ib) {
        const bool built = first || nib > 1;
        if (built) {
          if (nib > 1) __syncthreads();
          if (!first || ib > 0) F = bounds(g, I, ib * Map::KT);
          total = item_table<0, false, true>(M, in, off, ib * Map::KT, min(Map::KT, k - ib * Map::KT), F, M.red[0]);
          single = nib == 1 && total <= Map::CAP;
        }
        for (int c0 = 0; total > 0; c0 += Map::CAP) {
          if (!built || c0 > 0) item_map(M, c0);
          __syncthreads();
          L.init(c0, total);
          item_rows(M, L, c0, r);
          op();
          if (single) break;
          __syncthreads();
          item_unmap(M);
          __syncthreads();
          if (total - c0 <= Map::CAP) break;
        }
      }
    };
    const uint32_t mmax = m - 1u;
    // Applies f(row clamped into [0, m), row inside [0, m)) to the rows: no
    // branches, only the shared-memory writes themselves are predicated.
    auto each_row = [&](auto&& f) {
#pragma unroll
      for (int q0 = 0; q0 < ITEM_SLOTS; q0 += ITEM_GROUP) {
        if (q0 >= L.ns) break;  // (warp-uniform)
#pragma unroll
        for (int q = q0; q < q0 + ITEM_GROUP; ++q) f(min(r[q], mmax), r[q] <= mmax);
      }
    };
    // The block's total of a per-thread count, read by thread 0 alone.
    auto add_up = [&](int x) {
      const int w = __reduce_add_sync(SPK_FULL, x);
      if ((tid & 31) == 0) M.red[1][tid >> 5] = w;
      __syncthreads();
      int sum = 0;
      if (tid == 0)
        for (int v = 0; v < Map::NW; ++v) sum += M.red[1][v];
      return sum;
    };
    int fresh = 0, ne = 0, u;
    int s = 0, kind = 0;  // thread 0's, loaded while the rows are counted
    if (!WIDE) {
      rows_pass(true, [&]() {
        each_row([&](uint32_t x, bool in_m) {
          const uint32_t bit = 1u << (x & 31);
          uint32_t old = 0xffffffffu;
          if (in_m) old = atomicOr(&bits[x >> 5], bit);
          fresh += !(old & bit);
        });
      });
      if (c + (int)gridDim.x < ncols) {
        In = in.inst + inst_of(in, gn);
        Fn = bounds(gn, In, 0);
      }
      if (tid == 0 && dup.cols) {
        s = s_arr[g];
        kind = item_kind(I);
      }
      u = add_up(fresh);
      if (single) {
        each_row([&](uint32_t x, bool) { bits[x >> 5] = 0u; });
      } else {
        for (int x = tid; x < (int)((m + 31) >> 5); x += B) bits[x] = 0u;
      }
    } else {
      rows_pass(true, [&]() {
        each_row([&](uint32_t x, bool in_m) {
          if (in_m) atomicOr(&summ[x >> 10], 1u << ((x >> 5) & 31));
        });
      });
      if (c + (int)gridDim.x < ncols) {
        In = in.inst + inst_of(in, gn);
        Fn = bounds(gn, In, 0);
      }
      __syncthreads();
      const uint4 w = *reinterpret_cast<const uint4*>(summ + 4 * tid);
      const int n0 = __popc(w.x), n1 = __popc(w.y), n2 = __popc(w.z);
      const int run = item_scan<B>(n0 + n1 + n2 + __popc(w.w), M.red[1], &ne);
      uint2 p;
      p.x = (uint32_t)run | ((uint32_t)(run + n0) << 16);
      p.y = (uint32_t)(run + n0 + n1) | ((uint32_t)(run + n0 + n1 + n2) << 16);
      *reinterpret_cast<uint2*>(spre + 4 * tid) = p;
      __syncthreads();
      ne = min(ne, CTA_MAX_LIMIT);
      rows_pass(false, [&]() {
        each_row([&](uint32_t x, bool in_m) {
          const uint32_t wd = x >> 5;
          const int cc = (int)spre[wd >> 5] + __popc(summ[wd >> 5] & ((1u << (wd & 31)) - 1u));
          const uint32_t bit = 1u << (x & 31);
          uint32_t old = 0xffffffffu;
          if (in_m && cc < ne) old = atomicOr(&cw[cc], bit);
          fresh += !(old & bit);
        });
      });
      if (tid == 0 && dup.cols) {
        s = s_arr[g];
        kind = item_kind(I);
      }
      u = add_up(fresh);  // (a barrier lies between the two uses of red[1])
      *reinterpret_cast<uint4*>(summ + 4 * tid) = make_uint4(0u, 0u, 0u, 0u);
      for (int x = tid; x < ne; x += B) cw[x] = 0u;
    }
    item_unmap(M);
    if (tid == 0 && dup.cols && dup_column(s, u)) {
      u_out[g] = u;
      dup_append(dup, tally, g, s, kind, ctr_w);
    } else if (tid == 0) {
      u_out[g] = u;
      const int wi = atomicAdd(&ctr_w->n_windows, 1);
      if (wi < win_cap - ctr->n_hwin) {
        Window w;
        w.col = g;
        w.r_lo = 0;
        w.r_hi = I->m;
        w.u = u;
        w.out_off = 0;
        w.search = -1;
        win[wi] = w;
      } else {
        atomicOr(&ctr_w->err, ERR_WINDOW_CAP);
      }
    }
  }
  if (tid == 0) tally.flush(ctr_w);
}

constexpr int HEAVY_BLOCK = 1024;
constexpr int MAX_SLAB_WINDOWS = 1100;  // 2^20 rows / (1024 - 64) + 2
constexpr int FILTER_WINDOWS = 3;       // see the window records below
constexpr int FILTER_SEG = 64;

// Heavy columns: one thread block per column (from a work counter, columns
// with s_j > BIG_S first).  Rows of one slab of 2^20 rows
// at a time go into a 64-bit-word bitmap plus a summary bitmap (one bit per
// non-empty word), both kept zero between slabs, so the work per slab grows
// with the rows present, not with the slab.  The popcount prefix over the
// non-empty words gives nnz(B(:,j)) and cuts the column into windows of at
// most win_target + 63 distinct rows (boundaries on 64-row words).  The rows
// come through the entry map of spk_items.cuh, the next column's bounds while
// this one is counted (15669 columns of 9000 entries, m = 20011: 0.81 -> 0.33 ms;
// with the 128 KB bitmap of 2^20 rows one block holds the SM and the prefix and
// its barriers decide: R-MAT scale 20 5.06 -> 4.94 ms).
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, BLOCK >= 1024 ? 1 : 4) k_sym_heavy(Inputs in, const int32_t* __restrict__ list,
                                                     const int32_t* __restrict__ s_arr,
                                                     const Counters* __restrict__ ctr, int32_t* __restrict__ u_out,
                                                     Window* __restrict__ win, int32_t* __restrict__ search_list,
                                                     int64_t win_cap, int win_target, int slab_log2,
                                                     DupList dup, Counters* ctr_w) {
  using Map = ItemMap<BLOCK>;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ int red[BLOCK / 32 + 1];
  __shared__ int bnd[MAX_SLAB_WINDOWS + 1];
  __shared__ int cval[MAX_SLAB_WINDOWS + 1];
  __shared__ int s_col_u, s_wbase, s_sbase;
  const int W64 = 1 << (slab_log2 - 6);
  const int NSW = (W64 + 31) >> 5;
  Map& M = *reinterpret_cast<Map*>(sm_raw);
  unsigned long long* bm = reinterpret_cast<unsigned long long*>(sm_raw + sizeof(Map));
  uint32_t* summ = reinterpret_cast<uint32_t*>(bm + W64);
  for (int x = threadIdx.x; x < W64; x += BLOCK) bm[x] = 0ull;
  for (int x = threadIdx.x; x < NSW; x += BLOCK) summ[x] = 0u;
  item_unmap(M);
  __shared__ DupTally tally;
  if (threadIdx.x == 0) tally.clear();
  __syncthreads();
  const int n_big = ctr->n_big;
  const int ncols = n_big + ctr->n_heavy;
  const int slab_rows = 1 << slab_log2;
  // Columns are handed out by a work counter, the largest list first; the
  // next column's ticket is taken while the current one runs.
  __shared__ int s_tk[2];
  if (threadIdx.x == 0) s_tk[0] = atomicAdd(&ctr_w->heavy_next, 1);
  __syncthreads();
  // A column's bounds of its first segment table; those of a one-slab column
  // are read while the column before it runs.
  auto column = [&](int c) { return c < n_big ? list[in.ncols + c] : list[c - n_big]; };
  auto bounds = [&](int g, const Inst* I, int k_lo) {
    const int j = g - I->colbase, off = I->ptr_off;
    auto seg = [&](int i, int* beg, int* end) {
      const int32_t* cp = in.cp[off + i];
      *beg = __ldg(cp + j);
      *end = __ldg(cp + j + 1);
    };
    return item_bounds<BLOCK>(k_lo, min(Map::KT, I->k - k_lo), seg);
  };
  ItemBounds<BLOCK> F;
  if (s_tk[0] < ncols) {
    const int g = column(s_tk[0]);
    F = bounds(g, in.inst + inst_of(in, g), 0);
  }
  for (int it = 0;; ++it) {
    const int c = s_tk[it & 1];
    if (c >= ncols) break;
    if (threadIdx.x == 0) s_tk[(it + 1) & 1] = atomicAdd(&ctr_w->heavy_next, 1);
    const int g = column(c);
    const Inst* I = in.inst + inst_of(in, g);
    const int k = I->k, off = I->ptr_off, m = I->m;
    const int nslabs = (int)(((int64_t)m + slab_rows - 1) / slab_rows);
    if (threadIdx.x == 0) s_col_u = 0;
    for (int slab = 0; slab < nslabs; ++slab) {
      const int lo = slab * slab_rows;
      const int hi = (int)min((int64_t)m, (int64_t)lo + slab_rows);
      const uint32_t width = (uint32_t)(hi - lo);
      const int nib = (k + Map::KT - 1) / Map::KT;
      for (int ib = 0; ib < nib; ++ib) {
        const int k_lo = ib * Map::KT;
        if (ib > 0 || nslabs > 1) {
          F = bounds(g, I, k_lo);
          if (nslabs > 1 && in.sorted) {  // unordered inputs: the whole column, rows outside the slab skipped
#pragma unroll
            for (int h = 0; h < Map::KPT; ++h)
              if (F.beg[h] < F.end[h]) {
                const int32_t* ri = in.ri[off + k_lo + Map::KPT * (int)threadIdx.x + h];
                F.beg[h] = lower_bound_i32(ri, F.beg[h], F.end[h], lo);
                F.end[h] = lower_bound_i32(ri, F.beg[h], F.end[h], hi);
              }
          }
          __syncthreads();
        }
        // Row bit, and the summary mark of the word whose half it is first in.
        auto set_row = [&](uint32_t row) {
          const uint32_t rr = row - (uint32_t)lo;
          const uint32_t cl = min(rr, width - 1u);
          uint32_t old = 1u;
          if (rr < width) old = atomicOr(reinterpret_cast<uint32_t*>(bm) + (cl >> 5), 1u << (cl & 31));
          if (old == 0u) atomicOr(&summ[cl >> 11], 1u << ((cl >> 6) & 31));
        };
        const int total = item_table<0, false, true>(M, in, off, k_lo, min(Map::KT, k - k_lo), F, M.red[0]);
        __syncthreads();
        if (total <= Map::CAP || total < 256 * M.ne) {  // chunk by chunk, all of a chunk's loads in flight
          for (int c0 = 0; total > 0; c0 += Map::CAP) {
            if (c0 > 0) {
              item_map(M, c0);
              __syncthreads();
            }
            ItemSlots<BLOCK> L;
            uint32_t r[ITEM_SLOTS];
            L.init(c0, total);
            item_rows(M, L, c0, r);
#pragma unroll
            for (int q0 = 0; q0 < ITEM_SLOTS; q0 += ITEM_GROUP) {
              if (q0 >= L.ns) break;  // (warp-uniform)
#pragma unroll
              for (int q = q0; q < q0 + ITEM_GROUP; ++q) set_row(r[q]);
            }
            if (total - c0 <= Map::CAP) break;
            __syncthreads();
            item_unmap(M);
            __syncthreads();
          }
        } else {
          // Long segments: each warp walks an equal run of the positions, segment
          // by segment, without barriers (96 columns of 480,000 entries: 263 us
          // in chunks, 232 us so; columns of 250 segments of 34: 0.33 and 1.08 ms).
          const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
          const int run = (int)(((int64_t)total + Map::NW - 1) / Map::NW);
          const int64_t p1 = min((int64_t)total, (int64_t)(wid + 1) * run);
          int64_t p = (int64_t)wid * run;
          int o = 0, oe = M.ne;  // the last segment that starts at or before p
          while (oe - o > 1) {
            const int mid = (o + oe) >> 1;
            if (M.first[mid] <= p) o = mid;
            else oe = mid;
          }
          for (; p < p1; ++o) {
            const int32_t* rows = reinterpret_cast<const int32_t*>(M.seg[o].x);
            const int64_t end = min(p1, (int64_t)M.first[o + 1]);
            for (; p < end; p += 256) {
              uint32_t r[8];
#pragma unroll
              for (int t = 0; t < 8; ++t) r[t] = (uint32_t)__ldg(rows + min(p + 32 * t + lane, end - 1));
#pragma unroll
              for (int t = 0; t < 8; ++t)
                if (p + 32 * t < end) set_row(r[t]);  // (warp-uniform)
            }
            p = end;
          }
        }
        __syncthreads();
        item_unmap(M);
      }
      __syncthreads();
      if (slab == nslabs - 1 && s_tk[(it + 1) & 1] < ncols) {  // the next column's bounds, used when it starts
        const int gn = column(s_tk[(it + 1) & 1]);
        F = bounds(gn, in.inst + inst_of(in, gn), 0);
      }
      // Popcount prefix over the non-empty words: thread t owns bitmap words
      // [t*per, t*per + per) (a power of two <= 32, inside one summary word);
      // `mine` holds which of them are non-empty.
      const int nwords = (int)((width + 63) >> 6);
      int per = 1;
      while (per * BLOCK < nwords && per < 32) per <<= 1;
      if (per * BLOCK < nwords && threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);  // host sizing prevents it
      const int w0 = threadIdx.x * per;
      uint32_t mine = 0u;
      if (w0 < nwords) {
        mine = summ[w0 >> 5] >> (w0 & 31);
        if (per < 32) mine &= (1u << per) - 1u;
      }
      int loc = 0;
      for (uint32_t bits = mine; bits; bits &= bits - 1) loc += __popcll(bm[w0 + __ffs(bits) - 1]);
      int slab_u;
      const int ex = block_excl_scan<BLOCK>(loc, red, &slab_u);
      const int P = slab_u == 0 ? 0 : (slab_u + win_target - 1) / win_target;
      const bool whole = (nslabs == 1 && P == 1);
      // Windows read per-input offsets found by binary search when the inputs
      // are sorted, except in a column of one slab cut into at most
      // FILTER_WINDOWS windows whose input segments are short (s_j <=
      // FILTER_SEG * k): there every window reads the whole column and keeps
      // its rows, since a few extra passes over short segments cost less
      // than k binary searches per window.  Unordered inputs always do so.
      const bool searched = !whole && in.sorted &&
                            (nslabs > 1 || P > FILTER_WINDOWS || (int64_t)s_arr[g] > (int64_t)FILTER_SEG * k);
      if (whole && dup.cols && dup_column(s_arr[g], slab_u)) {
        if (threadIdx.x == 0) dup_append(dup, tally, g, s_arr[g], item_kind(I), ctr_w);
      } else if (P > MAX_SLAB_WINDOWS) {  // win_target is validated on the host; guard anyway
        if (threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
      } else if (P > 0) {
        if (threadIdx.x == 0) {
          bnd[0] = 0;
          cval[0] = 0;
          bnd[P] = nwords;
          cval[P] = slab_u;
          s_wbase = atomicAdd(&ctr_w->n_hwin, P);
          s_sbase = searched ? atomicAdd(&ctr_w->n_search, P) : -1;
        }
        // Window p starts after the word in which the running count first
        // reaches p * win_target.
        if (P > 1) {
          int run = ex;
          for (uint32_t bits = mine; bits; bits &= bits - 1) {
            const int wd = w0 + __ffs(bits) - 1;
            const int before = run;
            run += __popcll(bm[wd]);
            const int pb = before / win_target, pa = run / win_target;
            if (pa > pb && pa >= 1 && pa <= P - 1) {
              bnd[pa] = wd + 1;
              cval[pa] = run;
            }
          }
        }
        __syncthreads();
        const int col_u = s_col_u;
        for (int p = threadIdx.x; p < P; p += BLOCK) {
          const int wi = (int)win_cap - 1 - (s_wbase + p);  // from the array's end
          if (wi >= 0 && (!searched || s_sbase + p < win_cap)) {
            Window w;
            w.col = g;
            w.r_lo = whole ? 0 : lo + 64 * bnd[p];
            w.r_hi = whole ? m : (int)min((int64_t)hi, (int64_t)lo + 64 * (int64_t)bnd[p + 1]);
            w.u = cval[p + 1] - cval[p];
            w.out_off = col_u + cval[p];
            w.search = searched ? s_sbase + p : -1;
            win[wi] = w;
            if (searched) search_list[s_sbase + p] = wi;
          } else {
            atomicOr(&ctr_w->err, ERR_WINDOW_CAP);
          }
        }
      }
      // Clear this thread's words, then the summary, for the next slab or column.
      for (uint32_t bits = mine; bits; bits &= bits - 1) bm[w0 + __ffs(bits) - 1] = 0ull;
      __syncthreads();
      for (int x = threadIdx.x; x < ((nwords + 31) >> 5); x += BLOCK) summ[x] = 0u;
      if (threadIdx.x == 0) s_col_u += slab_u;
      __syncthreads();
    }
    if (threadIdx.x == 0) u_out[g] = s_col_u;
    __syncthreads();
  }
  if (threadIdx.x == 0) tally.flush(ctr_w);
}

// Heavy columns, compact form: the same count and window cuts from a summary
// bit per 32-row word and a table of at most `cap` non-empty words, instead of
// a bitmap over the whole slab (128 KB at 2^20 rows), so that several columns
// are in flight per SM.  Per slab:
//
//   pass A1  every entry sets its word's summary bit
//   rank 1   popcount prefix over the summary words; the slab is cut into
//            sub-ranges of whole summary words holding at most `cap`
//            non-empty words each (one sub-range unless the column is huge)
//   per sub-range:
//     pass A2  every entry of the sub-range sets its row bit in the table
//              (sorted inputs: the sub-range's slice found by binary search)
//     rank 2   popcount prefix over the table: distinct rows, and the window
//              cuts where the running count reaches multiples of win_target
//              (on 32-row words: a window holds at most win_target + 31 rows)
template <int BLOCK, int U>
__global__ void __launch_bounds__(BLOCK) k_sym_heavy_compact(Inputs in, const int32_t* __restrict__ list,
                                                             const int32_t* __restrict__ s_arr,
                                                             const Counters* __restrict__ ctr,
                                                             int32_t* __restrict__ u_out, Window* __restrict__ win,
                                                             int32_t* __restrict__ search_list, int64_t win_cap,
                                                             int win_target, int slab_log2, int cap,
                                                             Counters* ctr_w) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ int red[BLOCK / 32 + 1];
  __shared__ int bnd[MAX_SLAB_WINDOWS + 1];
  __shared__ int cval[MAX_SLAB_WINDOWS + 1];
  __shared__ int s_col_u, s_wbase, s_sbase;
  const int NSW = 1 << (slab_log2 - 10);
  uint32_t* summ = reinterpret_cast<uint32_t*>(sm_raw);     // NSW: one bit per 32-row word (kept zero)
  uint32_t* cw = summ + NSW;                                // cap: row bits of non-empty words (kept zero)
  int32_t* spre = reinterpret_cast<int32_t*>(cw + cap);     // NSW: exclusive prefix of non-empty words
  int32_t* srs = spre + NSW;                                // NSW: first summary word of each sub-range
  for (int x = threadIdx.x; x < NSW; x += BLOCK) summ[x] = 0u;
  for (int x = threadIdx.x; x < cap; x += BLOCK) cw[x] = 0u;
  __syncthreads();
  const int n_big = ctr->n_big;
  const int ncols = n_big + ctr->n_heavy;
  const int slab_rows = 1 << slab_log2;
  const int capw = cap - 32;  // a sub-range starts below capw words: it ends below cap
  // Columns are handed out by a work counter, the largest list first; the
  // next column's ticket is taken while the current one runs.
  __shared__ int s_tk[2];
  if (threadIdx.x == 0) s_tk[0] = atomicAdd(&ctr_w->heavy_next, 1);
  __syncthreads();
  for (int it = 0;; ++it) {
    const int c = s_tk[it & 1];
    if (c >= ncols) break;
    if (threadIdx.x == 0) s_tk[(it + 1) & 1] = atomicAdd(&ctr_w->heavy_next, 1);
    const int g = c < n_big ? list[in.ncols + c] : list[c - n_big];
    const Inst* I = in.inst + inst_of(in, g);
    const int k = I->k, off = I->ptr_off, m = I->m, j = g - I->colbase;
    const int nslabs = (int)(((int64_t)m + slab_rows - 1) / slab_rows);
    if (threadIdx.x == 0) s_col_u = 0;
    for (int slab = 0; slab < nslabs; ++slab) {
      const int lo = slab * slab_rows;
      const int hi = (int)min((int64_t)m, (int64_t)lo + slab_rows);
      const uint32_t width = (uint32_t)(hi - lo);
      // The column's entries of input i in rows [a, b) of this slab.
      auto seg_rows = [&](int i, int a, int b, int* beg, int* len) {
        const int32_t* cp = in.cp[off + i];
        int x = __ldg(cp + j), y = __ldg(cp + j + 1);
        if (in.sorted && (a > 0 || b < m)) {  // unordered inputs: all entries, rows outside skipped
          const int32_t* ri = in.ri[off + i];
          x = lower_bound_i32(ri, x, y, a);
          y = lower_bound_i32(ri, x, y, b);
        }
        *beg = x;
        *len = y - x;
      };
      auto seg_slab = [&](int i, int* beg, int* len) { seg_rows(i, nslabs > 1 ? lo : 0, nslabs > 1 ? hi : m, beg, len); };
      auto none = [](uint32_t, int32_t, float) {};
      auto mark = [&](int32_t r, float) -> uint32_t {
        const uint32_t rr = (uint32_t)(r - lo);
        if (rr < width) {
          const uint32_t w = rr >> 5, bit = 1u << (w & 31);
          if (!(summ[w >> 5] & bit)) atomicOr(&summ[w >> 5], bit);
        }
        return 0u;
      };
      SegCache sc{0, 0, false};
      block_for_each_entry<false, float, BLOCK, U>(in, k, off, seg_slab, mark, none, sc);
      __syncthreads();
      // Rank 1: thread t owns summary words [x0, x1).
      const int nwords = (int)((width + 31) >> 5);
      const int nsw = (nwords + 31) >> 5;
      const int ps = (nsw + BLOCK - 1) / BLOCK;
      const int x0 = min(nsw, (int)threadIdx.x * ps), x1 = min(nsw, x0 + ps);
      int loc = 0;
      for (int x = x0; x < x1; ++x) loc += __popc(summ[x]);
      int ne;
      int run = block_excl_scan<BLOCK>(loc, red, &ne);
      {
        int prev_sub = x0 > 0 ? (run - __popc(summ[x0 - 1])) / capw : -1;  // sub-range of word x0 - 1
        for (int x = x0; x < x1; ++x) {
          const int sub = run / capw;
          if (sub != prev_sub) srs[sub] = x;  // the prefix grows by <= 32 <= capw per word: no sub-range skipped
          prev_sub = sub;
          spre[x] = run;
          run += __popc(summ[x]);
        }
      }
      __syncthreads();
      const int R = spre[nsw - 1] / capw + 1;
      int slab_run = 0;
      for (int sub = 0; sub < R; ++sub) {
        const int xa = srs[sub], xb = sub + 1 < R ? srs[sub + 1] : nsw;
        const int cbase = spre[xa];
        const int nsub = (xb < nsw ? spre[xb] : ne) - cbase;
        if (nsub > cap) {  // cannot happen (see capw); never index past the table
          if (threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
          continue;
        }
        // Pass A2: row bits of the sub-range's non-empty words.
        auto setbit = [&](int32_t r, float) -> uint32_t {
          const uint32_t rr = (uint32_t)(r - lo);
          if (rr < width) {
            const uint32_t w = rr >> 5;
            const int x = (int)(w >> 5);
            if (x >= xa && x < xb) {
              const int cc = spre[x] + __popc(summ[x] & ((1u << (w & 31)) - 1u)) - cbase;
              const uint32_t bit = 1u << (rr & 31);
              if (cc < nsub && !(cw[cc] & bit)) atomicOr(&cw[cc], bit);  // cc < nsub: pass A1 set w's bit
            }
          }
          return 0u;
        };
        if (R == 1) {
          block_for_each_entry<false, float, BLOCK, U>(in, k, off, seg_slab, setbit, none, sc);
        } else {
          const int ra = lo + xa * 1024, rb = (int)min((int64_t)hi, (int64_t)lo + (int64_t)xb * 1024);
          auto seg_sub = [&](int i, int* beg, int* len) { seg_rows(i, ra, rb, beg, len); };
          SegCache sc2{0, 0, false};
          block_for_each_entry<false, float, BLOCK, U>(in, k, off, seg_sub, setbit, none, sc2);
        }
        __syncthreads();
        // Rank 2, by summary word: thread t owns summary words [y0, y1) of the sub-range.
        const int nx = xb - xa;
        const int ps2 = (nx + BLOCK - 1) / BLOCK;
        const int y0 = xa + min(nx, (int)threadIdx.x * ps2), y1 = xa + min(nx, (int)threadIdx.x * ps2 + ps2);
        int l2 = 0;
        for (int x = y0; x < y1; ++x) {
          int cc = spre[x] - cbase;
          for (int t = __popc(summ[x]); t > 0; --t) l2 += __popc(cw[cc++]);
        }
        int sub_u;
        int run2 = slab_run + block_excl_scan<BLOCK>(l2, red, &sub_u);
        // Window p starts after the word in which the running count first reaches p * win_target.
        for (int x = y0; x < y1; ++x) {
          int cc = spre[x] - cbase;
          for (uint32_t bits = summ[x]; bits; bits &= bits - 1) {
            const int wd = x * 32 + __ffs(bits) - 1;
            const int before = run2;
            run2 += __popc(cw[cc++]);
            const int pb = before / win_target, pa = run2 / win_target;
            if (pa > pb && pa >= 1 && pa <= MAX_SLAB_WINDOWS - 1) {
              bnd[pa] = wd + 1;
              cval[pa] = run2;
            }
          }
        }
        __syncthreads();
        for (int cc = threadIdx.x; cc < nsub; cc += BLOCK) cw[cc] = 0u;
        slab_run += sub_u;
        __syncthreads();
      }
      const int slab_u = slab_run;
      const int P = slab_u == 0 ? 0 : (slab_u + win_target - 1) / win_target;
      const bool whole = (nslabs == 1 && P == 1);
      // As in the bitmap form: split windows of sorted inputs are searched
      // unless the column has one slab, at most FILTER_WINDOWS windows and
      // short segments.
      const bool searched = !whole && in.sorted &&
                            (nslabs > 1 || P > FILTER_WINDOWS || (int64_t)s_arr[g] > (int64_t)FILTER_SEG * k);
      if (P > MAX_SLAB_WINDOWS) {
        if (threadIdx.x == 0) atomicOr(&ctr_w->err, ERR_INTERNAL);
      } else if (P > 0) {
        if (threadIdx.x == 0) {
          bnd[0] = 0;
          cval[0] = 0;
          bnd[P] = nwords;
          cval[P] = slab_u;
          s_wbase = atomicAdd(&ctr_w->n_hwin, P);
          s_sbase = searched ? atomicAdd(&ctr_w->n_search, P) : -1;
        }
        __syncthreads();
        const int col_u = s_col_u;
        for (int p = threadIdx.x; p < P; p += BLOCK) {
          const int wi = (int)win_cap - 1 - (s_wbase + p);  // from the array's end
          if (wi >= 0 && (!searched || s_sbase + p < win_cap)) {
            Window w;
            w.col = g;
            w.r_lo = whole ? 0 : lo + 32 * bnd[p];
            w.r_hi = whole ? m : (int)min((int64_t)hi, (int64_t)lo + 32 * (int64_t)bnd[p + 1]);
            w.u = cval[p + 1] - cval[p];
            w.out_off = col_u + cval[p];
            w.search = searched ? s_sbase + p : -1;
            win[wi] = w;
            if (searched) search_list[s_sbase + p] = wi;
          } else {
            atomicOr(&ctr_w->err, ERR_WINDOW_CAP);
          }
        }
      }
      for (int x = x0; x < x1; ++x) summ[x] = 0u;
      __syncthreads();
      if (threadIdx.x == 0) s_col_u += slab_u;
      __syncthreads();
    }
    if (threadIdx.x == 0) u_out[g] = s_col_u;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
static int blocks_per_sm(const DeviceInfo& dev, size_t smem_per_block, int threads_per_block) {
  const size_t reserve = 1024;  // per-block system shared memory
  int b = (int)(dev.smem_per_sm / (smem_per_block + reserve));
  int bt = 2048 / threads_per_block;
  if (b > bt) b = bt;
  if (b > 32) b = 32;
  return b < 1 ? 1 : b;
}

static int pow2_at_least(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

cudaError_t launch_sym_cta(const Inputs& in, const int32_t* list, const int32_t* s, const Counters* ctr, int32_t* u,
                           Window* win, int64_t win_cap, Counters* ctr_w, int cta_max, const DupList& dup,
                           const DeviceInfo& dev, cudaStream_t st) {
  if (in.mmax <= (1 << SLAB_BITS)) {
    const bool wide = in.mmax > (1 << SYM_FLAT_LOG2);
    const int words = pow2_at_least((in.mmax + 31) / 32);  // (few sizes: their occupancy is looked up once)
    auto go = [&](auto kern, int block, size_t smem) {
      const int bps = resident_blocks((const void*)kern, block, smem);
      if (bps < 1) return cudaErrorInvalidConfiguration;
      kern<<<dev.sms * bps, block, smem, st>>>(in, list, ctr, u, win, win_cap, words, s, dup, ctr_w);
      return cudaGetLastError();
    };
    if (wide) return go(k_sym_items<true, 256>, 256, sizeof(ItemMap<256>) + (1024 + CTA_MAX_LIMIT) * 4 + 1024 * 2);
    if (words > (1 << 12)) return go(k_sym_items<false, 256>, 256, sizeof(ItemMap<256>) + (size_t)words * 4);
    return go(k_sym_items<false, SYM_BLOCK>, SYM_BLOCK, sizeof(ItemMap<SYM_BLOCK>) + (size_t)words * 4);
  }
  constexpr int BLOCK = 512;
  const int tmax = pow2_at_least(2 * cta_max);
  const size_t smem = (size_t)tmax * sizeof(int32_t);
  auto kern = k_sym_cta<BLOCK, 4>;
  const cudaError_t e = allow_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  const int grid = dev.sms * blocks_per_sm(dev, smem, BLOCK);
  kern<<<grid, BLOCK, smem, st>>>(in, list, s, ctr, u, win, win_cap, tmax, ctr_w);
  return cudaGetLastError();
}

constexpr int HEAVY_CAP = 4096;  // non-empty 32-row words per sub-range of the compact form

// accumulator: 0 or 1 = slab bitmap, 2 = compact table.  Unlike the numeric
// items, the automatic choice keeps the slab bitmap even when it holds the
// SM: a heavy column has thousands of entries or more, enough for a
// 1024-thread block, and the largest R-MAT columns (10^5 distinct rows and
// more) need dozens of compact sub-ranges, each with 2k binary searches on
// the one block that owns the column (measured: R-MAT k=64 scale 20, heavy
// symbolic 7.2 ms as a bitmap, about 13 ms compact).
cudaError_t launch_sym_heavy(const Inputs& in, const int32_t* list, const int32_t* s, const Counters* ctr, int32_t* u,
                             Window* win, int32_t* search_list, int64_t win_cap, Counters* ctr_w, int window_max,
                             int accumulator, const DupList& dup, const DeviceInfo& dev, cudaStream_t st) {
  int slab_log2 = 10;
  while (slab_log2 < SLAB_BITS && ((int64_t)1 << slab_log2) < (int64_t)in.mmax) ++slab_log2;
  const size_t w64 = (size_t)1 << (slab_log2 - 6);
  const size_t bits = w64 * 8 + ((w64 + 31) / 32) * 4 + 16;
  const size_t nsw = (size_t)1 << (slab_log2 - 10);
  const size_t smem_c = nsw * 4 + (size_t)HEAVY_CAP * 4 + nsw * 8 + 16;
  // Small slabs: 256-thread blocks, several columns in flight per SM; a slab
  // bitmap that fills the SM: one 1024-thread block.
  const bool small = bits * 2 + 4096 <= (size_t)dev.smem_per_sm / 2;
  const size_t smem = bits + (small ? sizeof(ItemMap<256>) : sizeof(ItemMap<HEAVY_BLOCK>));
  auto kern = small ? k_sym_heavy<256> : k_sym_heavy<HEAVY_BLOCK>;
  auto kern_c = k_sym_heavy_compact<256, 8>;
  const int block = small ? 256 : HEAVY_BLOCK;
  int bf = 0, bc = 0;
  if (accumulator != 2 && smem <= (size_t)dev.smem_optin) bf = resident_blocks((const void*)kern, block, smem);
  if (accumulator == 2) bc = resident_blocks((const void*)kern_c, 256, smem_c);
  if (accumulator == 2) {
    if (bc < 1) return cudaErrorInvalidConfiguration;
    // Windows end on 32-row words: a window holds at most win_target + 31 rows.
    kern_c<<<dev.sms * bc, 256, smem_c, st>>>(in, list, s, ctr, u, win, search_list, win_cap, window_max - 64,
                                             slab_log2, HEAVY_CAP, ctr_w);
    return cudaGetLastError();
  }
  if (bf < 1) return cudaErrorInvalidConfiguration;
  // Windows end on 64-row words: a window holds at most win_target + 63 rows.
  kern<<<dev.sms * bf, block, smem, st>>>(in, list, s, ctr, u, win, search_list, win_cap, window_max - 64, slab_log2,
                                          dup, ctr_w);
  return cudaGetLastError();
}

}  // namespace spk
