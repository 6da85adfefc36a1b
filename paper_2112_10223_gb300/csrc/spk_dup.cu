// spk_dup.cu -- numeric columns whose entries meet on few distinct rows (the
// partial products of a sparse product: four entries a row or more, at most
// DUP_MAX_U rows): one warp per column, Alg. 5's insert-or-add table.
//
// The table is Sec. II-C's hash table in shared memory, private to the warp:
// DUP_BUCKETS buckets of two keys (one 8-byte load reads both), linear probing
// from the bucket's first slot.  A bucket-bitmap rank (spk_numeric.cu) spends its time on the
// bitmap's width and on block barriers, and its adds are shared-memory
// compare-and-swap loops, which for doubles run at 0.9 lanes a clock per SM.
// Here almost every entry finds its row at the first load, nothing but the
// column's rows is touched, and since one input's rows are distinct, the lanes
// of one input add with plain loads and stores, input after input.  Where 32
// entries come from more than DUP_ROUNDS inputs, that many turns take longer than
// atomics: 16384 float columns of 1024 entries on 128 rows, one to an input,
// 1178 us in turns, 439 us so (1363 us as block items), two to an input 636, 248
// and 433, four 345, 187 and 277; double 1169, 477 and 826, 611, 279 and 334, 320,
// 197 and 283.  At eight to an input (four inputs) both take the same time.  The
// distinct rows, listed as they are inserted, are at the end sorted in registers
// (spk_wsort.cuh).
//
// What bounds it: issue slots (65% busy at 32 warps per SM, 125 warp
// instructions per 32 entries) and half of the shared-memory wavefronts.
// 131072 columns of 2048 entries on 128 rows, float: 2.11 -> 1.25 ms; 20011
// ragged columns of 8400 entries on 135 rows, double: 2.25 -> 1.6 ms.  Buckets of
// four keys (1.3 times the time), 1024 slots (1.2 times: 20 warps per SM) and
// eight rounds of loads in flight (1.25 times: registers) were slower.
#include <type_traits>

#include "spk_common.cuh"
#include "spk_launch.h"
#include "spk_wsort.cuh"

namespace spk {

constexpr int DUP_SLOT_BITS = 9;
constexpr int DUP_SLOTS = 1 << DUP_SLOT_BITS;
constexpr int DUP_BUCKETS = DUP_SLOTS / 2;
constexpr int DUP_MAP = 2048;                    // positions of a start-bit map
constexpr int DUP_ROUNDS = 4;                    // at most this many inputs' lanes add in turn
constexpr uint32_t DUP_EMPTY = 0xffffffffu;
static_assert(DUP_MAX_U * 2 <= DUP_SLOTS, "at most half of the slots are taken");
static_assert(DUP_ROW_BITS + DUP_SLOT_BITS <= 32, "a row and its slot share a key");
static_assert(DUP_ROW_BITS == SLAB_BITS, "columns of one slab only");

template <typename A>
struct DupSmem {
  ulonglong2 seg[WSORT_KT];        // non-empty segments: row and value addresses less their first position
  uint2 blk[DUP_MAP / 32];         // per 32 positions: start bits (kept zero), first segment
  uint2 key[DUP_BUCKETS];          // rows, DUP_EMPTY between columns
  A acc[DUP_SLOTS];                // sums, zero between columns
  uint32_t list[DUP_MAX_U + 32];   // (row, slot) in order of insertion, then sorted
  int count;                       // rows listed
};

struct DupArgs {
  const int32_t* list;     // global column ids
  const int32_t* u_arr;
  const int64_t* col_ptr;
  Outs out;
  Counters* ctr_w;
  int n;
  int kind;                // item kind of this launch (-1: all): 0 and 1, 2 float, 3 double
};

// Finds or inserts a row that its first two buckets do not hold; returns the slot.
template <typename A>
__device__ __noinline__ int dup_insert(DupSmem<A>& D, uint32_t row, uint32_t h) {
  uint32_t* keys = reinterpret_cast<uint32_t*>(D.key);
  for (int probe = 0; probe < DUP_SLOTS; ++probe) {
    const int slot = (int)((2 * h + probe) & (DUP_SLOTS - 1));
    uint32_t x = *reinterpret_cast<volatile uint32_t*>(keys + slot);
    if (x == DUP_EMPTY) {
      x = atomicCAS(keys + slot, DUP_EMPTY, row);
      if (x == DUP_EMPTY) {
        const int at = atomicAdd(&D.count, 1);
        if (at < DUP_MAX_U) D.list[at] = (row << DUP_SLOT_BITS) | (uint32_t)slot;
        return slot;
      }
    }
    if (x == row) return slot;
  }
  return -1;  // more distinct rows than the symbolic pass counted
}

// SORTED: rows strictly increasing inside every input column.
template <int DT, bool WIDE_ACC, bool SORTED, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, (DT == 1 || WIDE_ACC ? 24 : 32) / WARPS)
    k_num_dup(Inputs in, DupArgs a) {
  using V = typename std::conditional<DT == 1, double, float>::type;
  using A = typename std::conditional<DT == 1 || WIDE_ACC, double, float>::type;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  DupSmem<A>& D = reinterpret_cast<DupSmem<A>*>(sm_raw)[wid];
  for (int x = lane; x < DUP_BUCKETS; x += 32) D.key[x] = make_uint2(DUP_EMPTY, DUP_EMPTY);
  for (int x = lane; x < DUP_SLOTS; x += 32) D.acc[x] = A(0);
  for (int x = lane; x < DUP_MAP / 32; x += 32) D.blk[x].x = 0u;
  if (lane == 0) D.count = 0;
  __syncwarp();
  uint32_t* keys = reinterpret_cast<uint32_t*>(D.key);
  // Columns are handed out by a counter (heavy columns were listed first).
  int* next = &a.ctr_w->dup_next[a.kind < 0 ? 0 : a.kind];
  auto ticket = [&]() {
    int t = 0;
    if (lane == 0) t = atomicAdd(next, 1);
    return t;
  };
  int c = __shfl_sync(SPK_FULL, ticket(), 0);
  while (c < a.n) {
    const int coming = ticket();  // the next column's, on its way while this one runs
    const int g = a.list[c];
    const int q = inst_of(in, g);
    const Inst* I = in.inst + q;
    const int k = I->k, off = I->ptr_off, j = g - I->colbase;
    if (a.kind >= 0 && item_kind(I) != a.kind) {
      c = __shfl_sync(SPK_FULL, coming, 0);
      continue;
    }
    const uint32_t m = (uint32_t)I->m;
    const int u = a.u_arr[g];
    bool lost = false;
    // Bounds of inputs cb + lane and cb + lane + 32.
    auto load = [&](int cb, int (&b)[2], int (&e)[2]) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        b[h] = 0;
        e[h] = 0;
        const int i = cb + lane + 32 * h;
        if (i < k) {
          const int32_t* cp = in.cp[off + i];
          b[h] = __ldg(cp + j);
          e[h] = __ldg(cp + j + 1);
        }
      }
    };
    int nb[2], nend[2];
    load(0, nb, nend);
    for (int cb = 0; cb < k; cb += WSORT_KT) {
      const int nk = min(WSORT_KT, k - cb);
      const bool two = nk > 32;
      const int beg[2] = {nb[0], nb[1]};
      const int len[2] = {nend[0] - nb[0], nend[1] - nb[1]};
      if (cb + WSORT_KT < k) load(cb + WSORT_KT, nb, nend);  // while this chunk runs
      // Positions and table.
      const int L0 = __shfl_sync(SPK_FULL, len[0], 0);
      bool same = lane >= nk || len[0] == L0;
      if (two) same = same && (lane + 32 >= nk || len[1] == L0);
      const bool equal = __all_sync(SPK_FULL, same) && L0 >= 2 && (int64_t)L0 * nk < 65536;
      int P[2], ord[2], total;
      if (equal) {
        P[0] = lane * L0;
        P[1] = P[0] + 32 * L0;
        ord[0] = lane;
        ord[1] = lane + 32;
        total = L0 * nk;
      } else {
        const unsigned below = (1u << lane) - 1u;
        int inc = warp_incl_scan(len[0], lane);
        total = __shfl_sync(SPK_FULL, inc, 31);
        P[0] = inc - len[0];
        unsigned bal = __ballot_sync(SPK_FULL, len[0] > 0);
        ord[0] = __popc(bal & below);
        inc = warp_incl_scan(len[1], lane);
        P[1] = total + inc - len[1];
        total += __shfl_sync(SPK_FULL, inc, 31);
        ord[1] = __popc(bal);
        bal = __ballot_sync(SPK_FULL, len[1] > 0);
        ord[1] += __popc(bal & below);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (len[h] > 0) {
          const int i = off + cb + lane + 32 * h;
          const int64_t d = (int64_t)beg[h] - P[h];
          ulonglong2 x;
          x.x = reinterpret_cast<unsigned long long>(in.ri[i]) + (unsigned long long)(d * 4);
          x.y = reinterpret_cast<unsigned long long>(in.val[i]) + (unsigned long long)(d * (int64_t)sizeof(V));
          D.seg[ord[h]] = x;
        }
      const uint32_t magic = equal ? 0xFFFFFFFFu / (uint32_t)L0 + 1u : 0u;
      for (int w0 = 0; w0 < total; w0 += DUP_MAP) {
        const int n = min(DUP_MAP, total - w0);
        if (!equal) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (len[h] > 0) {
              const int p0 = P[h] - w0, p1 = p0 + len[h];
              if (p0 >= 0 && p0 < n) atomicOr(&D.blk[p0 >> 5].x, 1u << (p0 & 31));
              const int b1 = min(p1, n) - 1;
              if (p1 > 0)
                for (int b = p0 <= 0 ? 0 : (p0 + 31) >> 5; b <= b1 >> 5; ++b) D.blk[b].y = (uint32_t)ord[h];
            }
        }
        __syncwarp();
        constexpr int G = 4;
        for (int e0 = 0; e0 < n; e0 += 32 * G) {
          uint32_t r[G];
          V v[G];
          int o[G];
#pragma unroll
          for (int t = 0; t < G; ++t) {
            const int e = min(e0 + 32 * t + lane, n - 1);  // (a lane past the end repeats the last entry's row)
            if (magic) {
              o[t] = (int)__umulhi((uint32_t)(w0 + e), magic);
            } else {
              const uint2 b = D.blk[e >> 5];
              o[t] = (int)b.y + __popc(b.x & (0xfffffffeu & (0xffffffffu >> (31 - (e & 31)))));
            }
            const ulonglong2 p = D.seg[o[t]];
            r[t] = (uint32_t)__ldg(reinterpret_cast<const int32_t*>(p.x) + w0 + e);
            v[t] = __ldg(reinterpret_cast<const V*>(p.y) + w0 + e);
          }
#pragma unroll
          for (int t = 0; t < G; ++t) {
            if (e0 + 32 * t >= n) break;  // (warp-uniform)
            const bool live = e0 + 32 * t + lane < n && r[t] < m;
            const uint32_t h = (r[t] * 0x85EBCA6Bu) >> (32 - (DUP_SLOT_BITS - 1));
            const uint2 key = D.key[h];
            int slot = (int)(2 * h) + (key.y == r[t] ? 1 : 0);
            bool hit = key.x == r[t] || key.y == r[t];
            if (__any_sync(SPK_FULL, live && !hit)) {
              // The next bucket (for 3% of the rows at 128 of them), then by probing.
              const uint32_t h1 = (h + 1) & (DUP_BUCKETS - 1);
              const uint2 key1 = D.key[h1];
              if (!hit) {
                hit = key1.x == r[t] || key1.y == r[t];
                slot = (int)(2 * h1) + (key1.y == r[t] ? 1 : 0);
              }
              if (__any_sync(SPK_FULL, live && !hit)) {
                if (live && !hit) slot = dup_insert(D, r[t], h);
                lost = lost || slot < 0;
                __syncwarp();
              }
            }
            const bool add = live && slot >= 0;
            const int o0 = SORTED ? __shfl_sync(SPK_FULL, o[t], 0) : 0;
            const int o1 = SORTED ? __shfl_sync(SPK_FULL, o[t], 31) : DUP_ROUNDS;
            if (o1 - o0 < DUP_ROUNDS) {
              // One input's rows are distinct: its lanes add together.
#pragma unroll 1
              for (int x = o0; x <= o1; ++x) {
                if (add && o[t] == x) D.acc[slot] += (A)v[t];
                __syncwarp();
              }
            } else if (add) {
              atomicAdd(&D.acc[slot], (A)v[t]);
            }
          }
        }
        __syncwarp();
        if (!equal)
          for (int x = lane; x < (n + 31) >> 5; x += 32) D.blk[x].x = 0u;
        __syncwarp();
      }
    }
    // The listed rows in order, and B(:, j).
    const int got = D.count;
    const int rows = min(got, DUP_MAX_U);
    if (__any_sync(SPK_FULL, lost) || got != u) {
      if (lane == 0) atomicOr(&a.ctr_w->err, ERR_INTERNAL);  // symbolic and numeric disagree
    }
    auto sort_rows = [&](auto e_tag) {
      constexpr int E = decltype(e_tag)::value;
      uint32_t r[E];
#pragma unroll
      for (int t = 0; t < E; ++t) r[t] = 32 * t + lane < rows ? D.list[32 * t + lane] : 0xffffffffu;
      __syncwarp();
      wsort_network<E>(r, lane);
#pragma unroll
      for (int t = 0; t < E; ++t) D.list[lane * (E + 1) + t] = r[t];
      __syncwarp();
    };
    const int eb = wsort_eb<WSORT_LOW>(rows);
    if (eb == 0) sort_rows(std::integral_constant<int, 1>());
    else if (eb == 1) sort_rows(std::integral_constant<int, 2>());
    else if (eb == 2) sort_rows(std::integral_constant<int, 4>());
    else sort_rows(std::integral_constant<int, 8>());
    const int64_t out = a.col_ptr[g] - (in.col_inst ? a.col_ptr[I->colbase] : 0);
    int32_t* orow = out_row_of(a.out, q) + out;
    V* oval = static_cast<V*>(out_val_of(a.out, q)) + out;
    for (int x = lane; x < rows; x += 32) {
      const uint32_t w = D.list[x + (x >> eb)];
      const int slot = (int)(w & (DUP_SLOTS - 1));
      if (x < u) {
        orow[x] = (int32_t)(w >> DUP_SLOT_BITS);
        oval[x] = (V)D.acc[slot];
      }
      keys[slot] = DUP_EMPTY;
      D.acc[slot] = A(0);
    }
    if (got > DUP_MAX_U) {  // rows that were not listed (the inputs changed): the whole table again
      __syncwarp();
      for (int x = lane; x < DUP_SLOTS; x += 32) {
        keys[x] = DUP_EMPTY;
        D.acc[x] = A(0);
      }
    }
    __syncwarp();
    if (lane == 0) D.count = 0;
    __syncwarp();
    c = __shfl_sync(SPK_FULL, coming, 0);
  }
}

template <int DT, bool WIDE_ACC>
static cudaError_t launch_dup(const Inputs& in, const DupArgs& a, int n, const DeviceInfo& dev, cudaStream_t st) {
  constexpr int WARPS = 4;
  using A = typename std::conditional<DT == 1 || WIDE_ACC, double, float>::type;
  auto kern = in.sorted ? k_num_dup<DT, WIDE_ACC, true, WARPS> : k_num_dup<DT, WIDE_ACC, false, WARPS>;
  const size_t smem = WARPS * sizeof(DupSmem<A>);
  const int bps = resident_blocks((const void*)kern, WARPS * 32, smem);
  if (bps < 1) return cudaErrorInvalidConfiguration;
  int grid = dev.sms * bps;
  if (grid > (n + WARPS - 1) / WARPS) grid = (n + WARPS - 1) / WARPS;
  kern<<<grid, WARPS * 32, smem, st>>>(in, a);
  return cudaGetLastError();
}

cudaError_t launch_num_dup(const Inputs& in, const int32_t* list, int n, const int32_t* n_kind, const int32_t* u,
                           const int64_t* col_ptr, const Outs& out, Counters* ctr_w, const DeviceInfo& dev,
                           cudaStream_t st, int* launches) {
  *launches = 0;
  if (n <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(&ctr_w->dup_next[0], 0, sizeof(ctr_w->dup_next), st);
  DupArgs a{};
  a.list = list;
  a.u_arr = u;
  a.col_ptr = col_ptr;
  a.out = out;
  a.ctr_w = ctr_w;
  a.n = n;
  for (int q = 0; q < 4 && e == cudaSuccess; ++q) {
    if (n_kind[q] <= 0) continue;
    a.kind = n_kind[q] == n ? -1 : q;
    // Float sums of more than FP32_ACC_TERMS inputs in double.
    e = q == 0 ? launch_dup<0, false>(in, a, n_kind[q], dev, st)
        : q == 3 ? launch_dup<1, false>(in, a, n_kind[q], dev, st)
                 : launch_dup<0, true>(in, a, n_kind[q], dev, st);
    ++*launches;
  }
  return e;
}

}  // namespace spk
