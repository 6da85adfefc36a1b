// spk_wsort.cuh -- one warp sorts a light column's entries in registers.
//
// An entry's key is (row << pos_bits | position), 32 bits: the position is its
// index in the flattened column (input after input), so keys are distinct,
// equal rows end up adjacent in input order, and the value is found again
// through the position.  A column of s entries takes N = 32 E >= s keys, E one
// of 1, 2, 4, 8, 10, 12 and 16, as a bitonic network over element index
// lane * E + i: strides below E are compare-exchanges between a lane's own
// registers, the others exchange one register with another lane.  No atomics, no
// counters and no per-column table to clear, and the same work whatever the rows
// are: the order-preserving buckets of k_warp_col need an insertion sort per
// bucket, which is quadratic where rows repeat or crowd.  10 and 12 keys a lane
// are there because 16 do the work of 512 entries for 257 to 384 of them (float,
// 16 inputs, numeric: 78125 columns of 320 entries 280 -> 212 us, buckets 234;
// 65104 of 384 247 -> 205, buckets 252; symbolic 253 -> 219, filter 230).
#pragma once

#include "spk_common.cuh"

namespace spk {

constexpr int WSORT_MAX = 512;        // entries of a column
constexpr int WSORT_ROW_BITS = 23;    // rows below 2^23: 9 bits are left for the position

// Compare-exchange: a <= b afterwards.
__device__ __forceinline__ void wsort_ce(uint32_t& a, uint32_t& b) {
  const uint32_t lo = min(a, b), hi = max(a, b);
  a = lo;
  b = hi;
}

// Exchanges keys with the partner lane: the lane with `up` keeps the larger.
__device__ __forceinline__ uint32_t wsort_keep(uint32_t x, uint32_t y, bool up) {
  return (x < y) != up ? x : y;  // (keys differ, or are both past the end)
}

// Sorts a lane's E keys: Knuth's merge exchange (The Art of Computer Programming
// 3, 5.2.2, algorithm M), for any E.
template <int E, int P0, int P, int Q, int R, int D>
__device__ __forceinline__ void wsort_lane(uint32_t (&r)[E]) {
#pragma unroll
  for (int i = 0; i + D < E; ++i)
    if ((i & P) == R) wsort_ce(r[i], r[i + D]);
  if constexpr (Q != P) wsort_lane<E, P0, P, Q / 2, P, Q - P>(r);
  else if constexpr (P > 1) wsort_lane<E, P0, P / 2, P0, 0, P / 2>(r);
}

// Sorts a lane's E keys that form a bitonic sequence.  Comparing the halves
// elementwise leaves two bitonic sequences (E even); what is left at an odd
// length, 5 or 3, is sorted outright.
template <int E>
__device__ __forceinline__ void wsort_clean(uint32_t (&r)[E]) {
  constexpr int ODD = E == 10 ? 5 : E == 12 ? 3 : 1;
#pragma unroll
  for (int st = E >> 1; st >= ODD; st >>= 1) {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (i / st % 2 == 0 && i + st < E) wsort_ce(r[i], r[i + st]);
  }
#pragma unroll
  for (int h = 0; ODD > 1 && h < E; h += ODD) {
    if constexpr (ODD == 5) {
      wsort_ce(r[h], r[h + 3]);
      wsort_ce(r[h + 1], r[h + 4]);
      wsort_ce(r[h], r[h + 2]);
      wsort_ce(r[h + 1], r[h + 3]);
      wsort_ce(r[h], r[h + 1]);
      wsort_ce(r[h + 2], r[h + 4]);
      wsort_ce(r[h + 1], r[h + 2]);
      wsort_ce(r[h + 3], r[h + 4]);
      wsort_ce(r[h + 2], r[h + 3]);
    } else if constexpr (ODD == 3) {
      wsort_ce(r[h], r[h + 1]);
      wsort_ce(r[h + 1], r[h + 2]);
      wsort_ce(r[h], r[h + 1]);
    }
  }
}

// Sorts the warp's 32 E keys ascending by element index lane * E + i.  The
// merges across lanes are loops (lane masks at run time): unrolled, the
// network of 16 keys a lane alone is 36 KB of code, and warps at different
// places in it wait for instructions.
template <int E>
__device__ __forceinline__ void wsort_network(uint32_t (&r)[E], int lane) {
  if constexpr (E == 10 || E == 12) {
    wsort_lane<E, 8, 8, 8, 0, 8>(r);
  } else {
#pragma unroll
    for (int size = 2; size <= E; size <<= 1) {
      // First step of a merge: element x meets x ^ (size - 1); then strides size / 4, ..., 1.
#pragma unroll
      for (int i = 0; i < E; ++i)
        if ((i ^ (size - 1)) > i) wsort_ce(r[i], r[i ^ (size - 1)]);
#pragma unroll
      for (int st = size >> 2; st >= 1; st >>= 1) {
#pragma unroll
        for (int i = 0; i < E; ++i)
          if (!(i & st)) wsort_ce(r[i], r[i + st]);
      }
    }
  }
#pragma unroll 1
  for (int lanes = 2; lanes <= 32; lanes <<= 1) {  // runs of `lanes` lanes
    {
      const bool up = (lane & (lanes >> 1)) != 0;
      uint32_t y[E];
#pragma unroll
      for (int i = 0; i < E; ++i) y[i] = __shfl_xor_sync(SPK_FULL, r[E - 1 - i], lanes - 1);
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = wsort_keep(r[i], y[i], up);
    }
#pragma unroll 1
    for (int lm = lanes >> 2; lm >= 1; lm >>= 1) {
      const bool up = (lane & lm) != 0;
#pragma unroll
      for (int i = 0; i < E; ++i) r[i] = wsort_keep(r[i], __shfl_xor_sync(SPK_FULL, r[i], lm), up);
    }
    wsort_clean<E>(r);
  }
}

// Networks a kernel holds: 1 to 8 keys a lane, 10 and 12, 16.  Without the
// middle ones a column of more than 256 entries takes 16.
enum : int { WSORT_LOW = 1, WSORT_MID = 2, WSORT_TOP = 4, WSORT_LONG = WSORT_MID | WSORT_TOP };

// Sorted element x lies at x + (x >> eb): one pad word per E elements (an odd
// stride between lanes) or, at 10 and 12 keys a lane, per 32 (of the shifts the
// one with the fewest bank conflicts, storing and reading).
template <int SIZES>
__device__ __forceinline__ int wsort_eb(int s) {
  if (!(SIZES & WSORT_LOW) || s > 256) return (SIZES & WSORT_MID) && s <= 384 ? 5 : 4;
  return s <= 32 ? 0 : s <= 64 ? 1 : s <= 128 ? 2 : 3;
}
// Bits of a key's position, below the row.
template <int SIZES>
__device__ __forceinline__ int wsort_pb(int s) {
  return (SIZES & WSORT_LOW) && s <= 256 ? 5 + wsort_eb<SIZES>(s) : 9;
}

constexpr int WSORT_KT = 64;  // inputs per segment table, two per lane

// Per-warp shared memory.  NUMERIC: values by position, sorted keys, run starts.
struct WsortSmem {
  unsigned char* vals;  // smax values (numeric)
  uint32_t* key;        // smax + 32 words: rows by position (k > 64), then sorted keys, one pad word per E
  uint16_t* start;      // smax + 2: sorted index of each distinct row's first entry (numeric)
  ulonglong2* seg;      // WSORT_KT non-empty segments: row and value addresses less their first position
  uint2* blk;           // smax / 32 (at least 1): start bits (kept zero), first segment
};

template <typename V, bool NUMERIC>
__host__ __device__ constexpr size_t wsort_bytes(int smax) {
  return (WSORT_KT * sizeof(ulonglong2) + (size_t)(smax / 32) * sizeof(uint2) +
          (NUMERIC ? (size_t)smax * sizeof(V) : 0) + (size_t)(smax + 32) * 4 +
          (NUMERIC ? (size_t)(smax + 2) * 2 : 0) + 15) &
         ~(size_t)15;
}

template <typename V, bool NUMERIC>
__device__ __forceinline__ WsortSmem wsort_carve(unsigned char* base, int smax) {
  WsortSmem sm;
  sm.seg = reinterpret_cast<ulonglong2*>(base);
  sm.blk = reinterpret_cast<uint2*>(sm.seg + WSORT_KT);
  sm.vals = reinterpret_cast<unsigned char*>(sm.blk + smax / 32);
  sm.key = reinterpret_cast<uint32_t*>(sm.vals + (NUMERIC ? (size_t)smax * sizeof(V) : 0));
  sm.start = reinterpret_cast<uint16_t*>(sm.key + smax + 32);
  return sm;
}

// A warp that keeps several sorted columns of at most `cap` entries: one segment
// table and map, then the columns' values, keys and starts.
template <typename V>
__host__ __device__ constexpr size_t wsort_slot_bytes(int cap) {
  return ((size_t)cap * sizeof(V) + (size_t)(cap + 32) * 4 + (size_t)(cap + 2) * 2 + 15) & ~(size_t)15;
}

template <typename V>
__host__ __device__ constexpr size_t wsort_slots_bytes(int cap, int slots) {
  return WSORT_KT * sizeof(ulonglong2) + 16 * sizeof(uint2) + (size_t)slots * wsort_slot_bytes<V>(cap);
}

template <typename V>
__device__ __forceinline__ WsortSmem wsort_carve_slot(unsigned char* base, int cap, int slot) {
  WsortSmem sm;
  sm.seg = reinterpret_cast<ulonglong2*>(base);
  sm.blk = reinterpret_cast<uint2*>(sm.seg + WSORT_KT);
  sm.vals = reinterpret_cast<unsigned char*>(sm.blk + 16) + (size_t)slot * wsort_slot_bytes<V>(cap);
  sm.key = reinterpret_cast<uint32_t*>(sm.vals + (size_t)cap * sizeof(V));
  sm.start = reinterpret_cast<uint16_t*>(sm.key + cap + 32);
  return sm;
}

// One input's part of a column, and its arrays.
template <typename V>
struct WsortIn {
  int beg, len;
  const int32_t* rp;
  const V* vp;
};

// Segment table and map of the inputs this warp holds (input `lane` and, when
// two, `lane` + 32 of nk), whose entries are positions [0, total).  Returns the
// magic of e / L when all of them have L entries (then the map is not
// written), else 0.  The caller's __syncwarp publishes it.
template <typename V, bool VALS>
__device__ __forceinline__ uint32_t wsort_table(ulonglong2* seg, uint2* blk, const WsortIn<V>* s, int nk, int* total,
                                                int lane) {
  const bool two = nk > 32;
  const int L0 = __shfl_sync(SPK_FULL, s[0].len, 0);
  bool same = lane >= nk || s[0].len == L0;
  if (two) same = same && (lane + 32 >= nk || s[1].len == L0);
  const bool equal = __all_sync(SPK_FULL, same) && L0 >= 2;
  int P[2], ord[2];
  if (equal) {
    P[0] = lane * L0;
    P[1] = P[0] + 32 * L0;
    ord[0] = lane;
    ord[1] = lane + 32;
    *total = L0 * nk;
  } else {
    const unsigned below = (1u << lane) - 1u;
    int inc = warp_incl_scan(s[0].len, lane);
    *total = __shfl_sync(SPK_FULL, inc, 31);
    P[0] = inc - s[0].len;
    unsigned bal = __ballot_sync(SPK_FULL, s[0].len > 0);
    ord[0] = __popc(bal & below);
    if (two) {
      inc = warp_incl_scan(s[1].len, lane);
      P[1] = *total + inc - s[1].len;
      *total += __shfl_sync(SPK_FULL, inc, 31);
      ord[1] = __popc(bal);
      bal = __ballot_sync(SPK_FULL, s[1].len > 0);
      ord[1] += __popc(bal & below);
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if ((h == 0 || two) && s[h].len > 0) {
      const int64_t d = (int64_t)s[h].beg - P[h];
      ulonglong2 x;
      x.x = reinterpret_cast<unsigned long long>(s[h].rp) + (unsigned long long)(d * 4);
      x.y = VALS ? reinterpret_cast<unsigned long long>(s[h].vp) + (unsigned long long)(d * (int64_t)sizeof(V)) : 0ull;
      seg[ord[h]] = x;
      if (!equal) {
        atomicOr(&blk[P[h] >> 5].x, 1u << (P[h] & 31));
        for (int b = (P[h] + 31) >> 5; b <= (P[h] + s[h].len - 1) >> 5; ++b) blk[b].y = (uint32_t)ord[h];
      }
    }
  return equal ? 0xFFFFFFFFu / (uint32_t)L0 + 1u : 0u;
}

// Segment of position e.
__device__ __forceinline__ int wsort_seg(const uint2* blk, uint32_t magic, int e) {
  if (magic) return (int)__umulhi((uint32_t)e, magic);
  const uint2 b = blk[e >> 5];
  return (int)b.y + __popc(b.x & (0xfffffffeu & (0xffffffffu >> (31 - (e & 31)))));
}

// Loads the bounds of inputs cb + lane (and cb + lane + 32).
template <typename V, typename BoundsF>
__device__ __forceinline__ void wsort_bounds(WsortIn<V>* s, int cb, int nk, BoundsF& bounds, int lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    s[h] = WsortIn<V>{0, 0, nullptr, nullptr};
    if (lane + 32 * h < nk) bounds(cb + lane + 32 * h, s[h]);
  }
}

// The column's entries, sorted: bounds(i, WsortIn&) gives input i's segment and
// arrays.  Returns the number of distinct rows, or -1 when a row is not below
// m.  as_is: the keys stay in input order (rows known to be distinct, order not
// wanted).  NUMERIC: afterwards key[] holds the sorted keys, start[] the runs'
// first indexes (start[u] = s), vals[] the values by position.
template <typename V, bool NUMERIC, int E, typename BoundsF>
__device__ __forceinline__ int wsort_column(const WsortSmem& sm, int k, int s, uint32_t m, bool as_is,
                                            BoundsF& bounds, int lane) {
  constexpr int EB = E == 1 ? 0 : E == 2 ? 1 : E == 4 ? 2 : E == 8 ? 3 : E == 16 ? 4 : 5;  // wsort_eb
  constexpr int PB = E > 8 ? 9 : 5 + EB;                                                    // wsort_pb
  V* sval = reinterpret_cast<V*>(sm.vals);
  uint32_t r[E];
  bool bad = false;
  if (k <= WSORT_KT) {
    int total;
    WsortIn<V> in[2];
    wsort_bounds<V>(in, 0, k, bounds, lane);
    const uint32_t magic = wsort_table<V, NUMERIC>(sm.seg, sm.blk, in, k, &total, lane);
    __syncwarp();
    constexpr int G = E <= 8 ? E : E == 10 ? 5 : E == 12 ? 6 : 8;
#pragma unroll
    for (int t0 = 0; t0 < E; t0 += G) {
      V v[G];
#pragma unroll
      for (int x = 0; x < G; ++x) {
        const int e = min((t0 + x) * 32 + lane, s - 1);  // (a lane past the end reads the last entry)
        const ulonglong2 p = sm.seg[wsort_seg(sm.blk, magic, e)];
        r[t0 + x] = (uint32_t)__ldg(reinterpret_cast<const int32_t*>(p.x) + e);
        if constexpr (NUMERIC) v[x] = __ldg(reinterpret_cast<const V*>(p.y) + e);
      }
#pragma unroll
      for (int x = 0; x < G; ++x) {
        const int e = (t0 + x) * 32 + lane;
        if constexpr (NUMERIC) {
          if (e < s) sval[e] = v[x];
        }
        bad = bad || r[t0 + x] >= m;
        r[t0 + x] = e < s ? (r[t0 + x] << PB) | (uint32_t)e : 0xffffffffu;
      }
    }
    __syncwarp();
    if (!magic && lane < E) sm.blk[lane].x = 0u;
  } else {
    int base = 0;
#pragma unroll 1
    for (int cb = 0; cb < k; cb += WSORT_KT) {
      const int nk = min(WSORT_KT, k - cb);
      int total;
      WsortIn<V> in[2];
      wsort_bounds<V>(in, cb, nk, bounds, lane);
      const uint32_t magic = wsort_table<V, NUMERIC>(sm.seg, sm.blk, in, nk, &total, lane);
      __syncwarp();
#pragma unroll 1
      for (int e0 = 0; e0 < total; e0 += 128) {
        uint32_t x[4];
        V v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int e = min(e0 + 32 * t + lane, total - 1);
          const ulonglong2 p = sm.seg[wsort_seg(sm.blk, magic, e)];
          x[t] = (uint32_t)__ldg(reinterpret_cast<const int32_t*>(p.x) + e);
          if constexpr (NUMERIC) v[t] = __ldg(reinterpret_cast<const V*>(p.y) + e);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int e = e0 + 32 * t + lane;
          if (e < total && base + e < s) {
            bad = bad || x[t] >= m;
            sm.key[base + e] = x[t];
            if constexpr (NUMERIC) sval[base + e] = v[t];
          }
        }
      }
      base += total;
      __syncwarp();
      if (lane < E) sm.blk[lane].x = 0u;
      __syncwarp();
    }
#pragma unroll
    for (int t = 0; t < E; ++t) {
      const int e = t * 32 + lane;
      r[t] = 0xffffffffu;
      if (e < s) r[t] = (sm.key[e] << PB) | (uint32_t)e;
    }
    __syncwarp();
  }
  if (__any_sync(SPK_FULL, bad)) return -1;
  if (NUMERIC && as_is) {
#pragma unroll
    for (int t = 0; t < E; ++t) {
      const int e = t * 32 + lane;
      sm.key[e + (e >> EB)] = r[t];
    }
    __syncwarp();
    return s;
  }
  wsort_network<E>(r, lane);
  // Heads: entries whose row differs from the one before.
  const uint32_t prev = __shfl_up_sync(SPK_FULL, r[E - 1], 1);
  uint32_t heads = 0u;
  const int i0 = lane * E;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const uint32_t before = i == 0 ? prev : r[i - 1];
    const bool head = ((r[i] ^ before) >> PB) != 0u || (i == 0 && lane == 0);
    if (head && i0 + i < s) heads |= 1u << i;
  }
  const int cnt = __popc(heads);
  if constexpr (!NUMERIC) return __reduce_add_sync(SPK_FULL, cnt);
  const int inc = warp_incl_scan(cnt, lane);
  const int u = __shfl_sync(SPK_FULL, inc, 31);
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int x = i0 + i;
    sm.key[EB == 5 ? x + (x >> 5) : lane * (E + 1) + i] = r[i];  // x + (x >> EB)
  }
  int q = inc - cnt;
  if (u < s) {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if ((heads >> i) & 1u) sm.start[q++] = (uint16_t)(i0 + i);
    if (lane == 0) sm.start[u] = (uint16_t)s;
  }
  __syncwarp();
  return u;
}

// a + b = s + error, exactly (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float b, float* error) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  *error = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  return s;
}

// Sum of the run term(a), ..., term(b - 1), rounded once.  Doubles are added in
// double.  Floats are added as an unevaluated sum of three floats, because a
// double addition occupies this GPU's double units for 16 clocks a warp and a
// conversion as many: two-sum keeps the rounding error of every addition, a
// second one those of adding the errors up (Ogita, Rump and Oishi, "Accurate sum
// and dot product", 2005, their K = 3).  With u = 2^-24, what is left out is at
// most n^3 u^3 sum|terms| for n terms, below the n 2^-53 sum|terms| of a sum in
// double for n <= 724 (columns here have at most 512 entries), and nothing
// where a sum in double is exact because the partial sums fit into 53 bits.
// Sums that are not finite that way (an overflow on the way, an infinity, a NaN)
// are added again in double.
template <typename V, typename TermF>
__device__ __forceinline__ V wsort_run_sum(int a, int b, TermF&& term) {
  static_assert(WSORT_MAX <= 724, "the error bound above");
  if constexpr (sizeof(V) == 4) {
    float hi = term(a), mid = 0.0f, lo = 0.0f;
    if (b - a > 1) hi = two_sum(hi, term(a + 1), &mid);
    for (int y = a + 2; y < b; ++y) {
      float e;
      hi = two_sum(hi, term(y), &e);
      mid = two_sum(mid, e, &e);
      lo = __fadd_rn(lo, e);
    }
    float r = hi;  // (without errors as it is: minus zero stays)
    if (mid != 0.0f || lo != 0.0f) r = lo != 0.0f ? (float)((double)hi + (double)mid + (double)lo) : __fadd_rn(hi, mid);
    if (isfinite(r)) return r;
  }
  double sum = (double)term(a);
  for (int y = a + 1; y < b; ++y) sum += (double)term(y);
  return (V)sum;
}

// Writes B(:, j) from a sorted column: distinct row q's run summed by
// wsort_run_sum.  (Columns without repeated rows are copied.)
template <typename V, int SIZES>
__device__ __forceinline__ void wsort_write(const WsortSmem& sm, int s, int u, int32_t* out_row, V* out_val, int lane) {
  const int eb = wsort_eb<SIZES>(s), pb = wsort_pb<SIZES>(s);
  const uint32_t pm = (1u << pb) - 1u;
  const V* sval = reinterpret_cast<const V*>(sm.vals);
  if (u == s) {
#pragma unroll 4
    for (int q = lane; q < s; q += 32) {
      const uint32_t x = sm.key[q + (q >> eb)];
      out_row[q] = (int32_t)(x >> pb);
      out_val[q] = sval[x & pm];
    }
    return;
  }
  for (int q = lane; q < u; q += 32) {
    const int a = sm.start[q], b = sm.start[q + 1];
    const uint32_t x = sm.key[a + (a >> eb)];
    out_row[q] = (int32_t)(x >> pb);
    out_val[q] = wsort_run_sum<V>(a, b, [&](int y) { return sval[sm.key[y + (y >> eb)] & pm]; });
  }
}

// wsort_column for any s <= WSORT_MAX that the kernel's networks hold.
template <typename V, bool NUMERIC, int SIZES, typename BoundsF>
__device__ __forceinline__ int wsort_any(const WsortSmem& sm, int k, int s, uint32_t m, bool as_is, BoundsF& bounds,
                                         int lane) {
  if constexpr ((SIZES & WSORT_LOW) != 0) {
    switch (wsort_eb<WSORT_LOW>(s)) {
      case 0: return wsort_column<V, NUMERIC, 1>(sm, k, s, m, as_is, bounds, lane);
      case 1: return wsort_column<V, NUMERIC, 2>(sm, k, s, m, as_is, bounds, lane);
      case 2: return wsort_column<V, NUMERIC, 4>(sm, k, s, m, as_is, bounds, lane);
      case 3: return wsort_column<V, NUMERIC, 8>(sm, k, s, m, as_is, bounds, lane);
      default: break;
    }
  }
  if constexpr ((SIZES & WSORT_MID) != 0) {
    if (s <= 320) return wsort_column<V, NUMERIC, 10>(sm, k, s, m, as_is, bounds, lane);
    if (s <= 384) return wsort_column<V, NUMERIC, 12>(sm, k, s, m, as_is, bounds, lane);
  }
  if constexpr ((SIZES & WSORT_TOP) != 0) return wsort_column<V, NUMERIC, 16>(sm, k, s, m, as_is, bounds, lane);
  return -1;  // (not reachable)
}

}  // namespace spk
