// Queries over the compressed leaves.
//  has (Sec. 5 "Point queries"): binary search on the uncompressed heads, then
//    one pass over the leaf.
//  range_map (Sec. 3: a search for the first element, then a scan to the end
//    of the range) with f = (sum mod 2^64, count).  A query covers parts of its
//    first and last leaf and all of the leaves between them.  The parts are
//    decoded one thread per leaf (k_range_ends).  The leaves between are
//    either walked -- numbered over all queries by a prefix sum, one leaf per
//    lane of equal shares -- or, when the queries together cover more leaves
//    than the set has, every leaf is reduced once, those reductions become a
//    prefix over the leaves, and a query takes the difference at its two ends
//    (k_leaf_prefix, k_range_inner): each leaf is then decoded
//    once however often the queries overlap.
//    From one query per leaf on, every leaf is walked once with its state kept
//    at every 32nd byte, and a query looks up its two ends (k_marks,
//    k_range_marked).  Few queries take eight lanes or a warp per leaf instead of
//    one.
//  sum (App. A sum()): every leaf once.
//  map_range_length (App. A: f on at most `length` elements from the first
//    key >= start): a prefix sum of the leaves' element counts gives the leaf
//    of the last element; the rest is as for range_map.
//  range_reduce (Sec. 3 range_map with other functions): min, max, xor or
//    sum of the keys of [lo, hi) whose masked bits match a value, with the
//    count of those keys, as for range_map (the smallest match of a run of
//    leaves is the first one after its start, the keys being in order).
//  The uncompressed PMA's cells (codec 1) keep a warp per leaf.
#include <algorithm>
#include <mutex>

#include "dev_common.cuh"
#include "internal.h"
#include "leaf_thread.cuh"
#include "leaf_walk.cuh"

using namespace cpmadev;

namespace cpmaimpl {
namespace {

constexpr int kT = 256;

__device__ __forceinline__ uint64_t gtid() {
  return (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
}
__device__ __forceinline__ uint64_t gstride() { return (uint64_t)gridDim.x * blockDim.x; }

// Byte codes: a thread per query key routes it and searches its leaf
// (leafthr::leaf_has) up to the key.  Bound by instruction issue: a warp runs
// as long as its deepest search.  1e6 keys against 1e8: 136 to 141 us, 195 us when
// the leaf was decoded code by code.  (At 156 us, a block ordering its 256 keys by
// how deep each is likely to lie: 154 us, and 1.9 us more on 1e3 keys.)
__global__ void __launch_bounds__(kT) k_has(const uint64_t* __restrict__ keys, uint64_t q,
                                            const uint8_t* __restrict__ data,
                                            const uint32_t* __restrict__ used,
                                            const uint64_t* __restrict__ heads, uint64_t L,
                                            uint32_t LB, uint8_t* __restrict__ out, ull* prof) {
  ull nbytes = 0;
  for (uint64_t i = (uint64_t)blockIdx.x * kT + threadIdx.x; i < q;
       i += (uint64_t)gridDim.x * kT) {
    const uint64_t x = keys[i], j = route_leaf(heads, L, x);
    const uint32_t u = min(used[j], LB);
    out[i] = u && leafthr::leaf_has(data + j * LB, u, x) ? 1u : 0u;
    nbytes += u + 9;
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// ---- few queries: a team of lanes per leaf (leafwalk::team_run) ----

// Lanes of a team: eight, or a warp where a leaf has more than 512 bytes.
constexpr unsigned kTeam = leafwalk::kTeam, kTeamLarge = 32;
static_assert(kTeam == 8, "four teams to a warp");

template <unsigned N>
__device__ __forceinline__ unsigned team_lane() { return lane_id() & (N - 1); }
template <unsigned N>
__device__ __forceinline__ unsigned team_mask() {
  return (N < 32 ? (1u << (N & 31u)) - 1u : FULL) << (lane_id() & ~(N - 1));
}

// upper_count by a team: each step its lanes probe an entry each, so the
// search waits for 6 loads where one lane would for 18 (2e5 entries, 8 lanes).
template <unsigned N>
__device__ __forceinline__ uint64_t team_upper_count(const uint64_t* __restrict__ a, uint64_t n,
                                                     uint64_t x) {
  const unsigned tl = team_lane<N>(), m = team_mask<N>();
  uint64_t base = 0, len = n;
  while (len) {
    const uint64_t step = len / (N + 1) + 1, at = (tl + 1) * step - 1;
    const uint64_t c = __popc(__ballot_sync(m, at < len && __ldg(a + base + at) <= x));
    base += c * step;
    len = min(step - 1, len - c * step);
  }
  return base;
}

template <unsigned N>
__device__ __forceinline__ uint64_t team_route(const uint64_t* __restrict__ heads, uint64_t L,
                                               uint64_t x) {
  if (x == KEY_MAX) return heads[L];
  const uint64_t c = team_upper_count<N>(heads, L, x);
  return c ? c - 1 : 0;
}

// The lane's run with the element before it (in k.val) and the number of
// elements before it (the head included); a whole warp calls.
template <unsigned N, bool SUM = false>
__device__ __forceinline__ leafwalk::Run team_leaf(const uint8_t* leafp, uint32_t u,
                                                   uint32_t& idx) {
  const unsigned tl = team_lane<N>();
  leafwalk::Run r = leafwalk::team_run<N, SUM>(leafp, u, tl);
  __syncwarp();
  uint64_t d = r.delta;
  uint32_t n = r.codes;
#pragma unroll
  for (unsigned o = 1; o < N; o <<= 1) {
    const uint64_t y = __shfl_up_sync(FULL, d, o, N);
    const uint32_t z = __shfl_up_sync(FULL, n, o, N);
    if (tl >= o) { d += y; n += z; }
  }
  r.k.val = (u ? leafwalk::leaf_head(leafp) : 0) + (d - r.delta);
  idx = 1 + n - r.codes;
  return r;
}

// The thread-per-key kernel's work by a team per key.
template <unsigned N>
__global__ void __launch_bounds__(kT) k_has_team(const uint64_t* __restrict__ keys, uint64_t q,
                                                 const uint8_t* __restrict__ data,
                                                 const uint32_t* __restrict__ used,
                                                 const uint64_t* __restrict__ heads, uint64_t L,
                                                 uint32_t LB, uint8_t* __restrict__ out,
                                                 ull* prof) {
  ull nbytes = 0;
  const unsigned tl = team_lane<N>(), team = lane_id() / N;
  for (uint64_t i0 = (gtid() >> 5) * (32 / N); i0 < q; i0 += (gstride() >> 5) * (32 / N)) {
    const uint64_t i = i0 + team;
    uint64_t x = 0, j = 0;
    uint32_t u = 0, idx;
    if (i < q) {
      x = keys[i];
      j = team_route<N>(heads, L, x);
      u = min(used[j], LB);
    }
    __syncwarp();
    const uint8_t* leafp = data + j * LB;
    const leafwalk::Run r = team_leaf<N>(leafp, u, idx);
    bool found = u && tl == 0 && r.k.val == x;  // the head
    if (r.k.val < x && x - r.k.val <= r.delta)
      leafwalk::run_visit(leafp, u, r, [&](uint64_t v) { found |= v == x; });
    __syncwarp();
    const unsigned hit = __ballot_sync(FULL, found) & team_mask<N>();
    if (i < q && tl == 0) {
      out[i] = hit ? 1u : 0u;
      nbytes += u + 9;
    }
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// Cells (codec 1): a warp per key, 32 routed per step.
__global__ void __launch_bounds__(kT) k_has_cells(const uint64_t* __restrict__ keys, uint64_t q,
                                                  const uint8_t* __restrict__ data,
                                                  const uint32_t* __restrict__ used,
                                                  const uint64_t* __restrict__ heads, uint64_t L,
                                                  uint32_t LB, uint8_t* __restrict__ out,
                                                  ull* prof) {
  const unsigned lane = lane_id();
  ull nbytes = 0;
  uint64_t r0, r1;
  warp_share(q, gtid() >> 5, gstride() >> 5, r0, r1);
  for (uint64_t base = r0; base < r1; base += 32) {
    const uint64_t qi = base + lane;
    uint64_t xi = 0, ji = 0;
    uint32_t ui = 0;
    if (qi < r1) {
      xi = keys[qi];
      ji = route_leaf(heads, L, xi);
      ui = min(used[ji], LB);
    }
    const uint32_t nk = (uint32_t)min((uint64_t)32, r1 - base);
    uint32_t found_bits = 0;
    for (uint32_t k = 0; k < nk; k++) {
      const uint64_t x = __shfl_sync(FULL, xi, k);
      const uint64_t j = __shfl_sync(FULL, ji, k);
      const uint32_t u = __shfl_sync(FULL, ui, k);
      nbytes += u + 9;
      bool f = false;
      warp_decode(data + j * LB, u, [&](uint32_t, uint64_t val) { f |= (val == x); }, true);
      if (__any_sync(FULL, f)) found_bits |= 1u << k;
    }
    if (qi < r1) out[qi] = (found_bits >> lane) & 1u;
  }
  if (prof && lane == 0 && nbytes) atomicAdd(prof, nbytes);
}

struct RangeArgs {
  const uint64_t* lo;
  const uint64_t* hi;
  uint64_t q;
  const uint64_t* first;
  const uint64_t* off;  // q + 1 entries
  const uint8_t* data;
  const uint32_t* used;
  const uint32_t* cnt;
  uint32_t LB;
  uint64_t* sum;
  uint64_t* count;
  ull* prof;  // profiling: leaf bytes scanned (nullable)
  const uint64_t* P = nullptr;  // rank mode: elements before each leaf (L + 1)
};

// ---- the uncompressed PMA's cells (codec 1): a warp per (query, leaf) item ----
__global__ void __launch_bounds__(kT) k_range_prep(const uint64_t* __restrict__ lo,
                                                   const uint64_t* __restrict__ hi, uint64_t q,
                                                   const uint64_t* __restrict__ heads, uint64_t L,
                                                   uint64_t* __restrict__ first,
                                                   uint64_t* __restrict__ items,
                                                   uint64_t* __restrict__ sum,
                                                   uint64_t* __restrict__ count,
                                                   uint64_t init = 0) {
  for (uint64_t i = gtid(); i < q; i += gstride()) {
    const uint64_t a = lo[i], b = hi[i];
    uint64_t fl = 0, n = 0;
    if (a < b) {
      fl = route_leaf(heads, L, a);
      n = route_leaf(heads, L, b - 1) - fl + 1;
    }
    first[i] = fl;
    items[i] = n;
    sum[i] = init;
    count[i] = 0;
  }
}

// Rank of the first key >= x: elements before its leaf plus the leaf's
// elements below x (the whole warp decodes the leaf).
template <bool RAW>
__device__ __forceinline__ uint64_t rank_of(uint64_t x, const uint64_t* __restrict__ heads,
                                            const uint8_t* __restrict__ data,
                                            const uint32_t* __restrict__ used, uint64_t L,
                                            uint32_t LB, const uint64_t* __restrict__ P) {
  const uint64_t j = route_leaf(heads, L, x);
  uint32_t below = 0;
  warp_decode(data + j * LB, min(used[j], LB), [&](uint32_t, uint64_t v) { below += v < x; },
              RAW);
  return P[j] + warp_sum(below);
}

// Step 1 of the rank-space queries (warp per query): the rank range
// [r0, r1) and the leaves holding it.  KEYS: [a, b) is a key range, r0 =
// rank(a), r1 = rank(b) (r1 = r0 when a >= b).  Otherwise (map_range_length)
// a is the start key and b the length: r1 = min(r0 + b, n).
// RAW: the leaves hold cells.
template <bool KEYS, bool RAW>
__global__ void __launch_bounds__(kT) k_rank_prep(const uint64_t* __restrict__ A,
                                                  const uint64_t* __restrict__ B, uint64_t q,
                                                  const uint64_t* __restrict__ heads,
                                                  const uint8_t* __restrict__ data,
                                                  const uint32_t* __restrict__ used, uint64_t L,
                                                  uint32_t LB, const uint64_t* __restrict__ P,
                                                  uint64_t* __restrict__ r0o,
                                                  uint64_t* __restrict__ r1o,
                                                  uint64_t* __restrict__ first,
                                                  uint64_t* __restrict__ items,
                                                  uint64_t* __restrict__ sum,
                                                  uint64_t* __restrict__ count) {
  pdl_wait();
  pdl_launch();
  const unsigned lane = lane_id();
  const uint64_t gw = gtid() >> 5, nw = gstride() >> 5;
  const uint64_t n = P[L];
  for (uint64_t i = gw; i < q; i += nw) {
    const uint64_t a = A[i], b = B[i];
    const uint64_t r0 = rank_of<RAW>(a, heads, data, used, L, LB, P);
    uint64_t r1;
    if constexpr (KEYS) r1 = a < b ? rank_of<RAW>(b, heads, data, used, L, LB, P) : r0;
    else r1 = (b >= n - r0) ? n : r0 + b;
    uint64_t f = 0, it = 0;
    if (r1 > r0) {
      f = upper_count(P, L + 1, r0) - 1;
      it = upper_count(P, L + 1, r1 - 1) - f;
    }
    if (lane == 0) {
      r0o[i] = r0;
      r1o[i] = r1;
      first[i] = f;
      items[i] = it;
      if (sum) sum[i] = 0;
      if (count) count[i] = KEYS ? r1 - r0 : 0;
    }
  }
}

// range_extract: the keys of ranks [r0, r1) of every query, written from
// out[off[i]] on (entries at or past cap are dropped).  Same load-balanced
// (query, leaf) walk as k_range.
struct ExtractArgs {
  const uint64_t* r0;
  const uint64_t* r1;
  uint64_t q;
  const uint64_t* first;
  const uint64_t* item_off;  // q + 1
  const uint64_t* out_off;   // q + 1
  const uint64_t* P;
  const uint8_t* data;
  const uint32_t* used;
  uint32_t LB;
  uint64_t* out;
  uint64_t cap;
  const leafwalk::Mark* start = nullptr;  // where each query's first key lies (leaf_below)
};

template <bool RAW>
__global__ void __launch_bounds__(kT) k_extract(ExtractArgs a) {
  pdl_wait();
  const uint64_t gw = gtid() >> 5, nw = gstride() >> 5;
  const uint64_t N = a.item_off[a.q];
  const uint64_t g0 = N * gw / nw, g1 = N * (gw + 1) / nw;
  if (g0 >= g1) return;
  uint64_t qi = upper_count(a.item_off, a.q + 1, g0) - 1;
  for (uint64_t g = g0; g < g1; g++) {
    while (g >= a.item_off[qi + 1]) qi++;
    const uint64_t j = a.first[qi] + (g - a.item_off[qi]);
    const uint64_t r0 = a.r0[qi], r1 = a.r1[qi], base = a.P[j], o = a.out_off[qi];
    warp_decode(a.data + j * a.LB, min(a.used[j], a.LB), [&](uint32_t idx, uint64_t v) {
      const uint64_t r = base + idx;
      if (r >= r0 && r < r1 && o + (r - r0) < a.cap) a.out[o + (r - r0)] = v;
    }, RAW);
  }
}

// range_reduce: the functions, their identities and their atomics
template <int OP>
__device__ __forceinline__ uint64_t op_apply(uint64_t a, uint64_t b) {
  if constexpr (OP == CPMA_OP_SUM) return a + b;
  else if constexpr (OP == CPMA_OP_MIN) return a < b ? a : b;
  else if constexpr (OP == CPMA_OP_MAX) return a > b ? a : b;
  else return a ^ b;
}
template <int OP>
__host__ __device__ __forceinline__ uint64_t op_identity() {
  return OP == CPMA_OP_MIN ? ~0ull : 0ull;
}
template <int OP>
__device__ __forceinline__ void op_atomic(uint64_t* p, uint64_t v) {
  if constexpr (OP == CPMA_OP_SUM) atomicAdd((ull*)p, (ull)v);
  else if constexpr (OP == CPMA_OP_MIN) atomicMin((ull*)p, (ull)v);
  else if constexpr (OP == CPMA_OP_MAX) atomicMax((ull*)p, (ull)v);
  else atomicXor((ull*)p, (ull)v);
}

// Same load-balanced (query, leaf) walk as k_range: every leaf is read by the
// warp and filtered by range and mask.
template <int OP>
__global__ void __launch_bounds__(kT) k_range_reduce(RangeArgs a, uint64_t mask,
                                                     uint64_t value) {
  const unsigned lane = lane_id();
  const uint64_t gw = gtid() >> 5, nw = gstride() >> 5;
  const uint64_t N = a.off[a.q];
  const uint64_t g0 = N * gw / nw, g1 = N * (gw + 1) / nw;
  if (g0 >= g1) return;
  uint64_t qi = upper_count(a.off, a.q + 1, g0) - 1;
  uint64_t r = op_identity<OP>(), c = 0;
  uint64_t qend = a.off[qi + 1];
  uint64_t lo = a.lo[qi], hi = a.hi[qi], fl = a.first[qi], qoff = a.off[qi];
  for (uint64_t g = g0; g < g1;) {
    while (g >= qend) {
#pragma unroll
      for (int o = 16; o; o >>= 1) r = op_apply<OP>(r, __shfl_xor_sync(FULL, r, o));
      c = warp_sum(c);
      if (lane == 0 && c) {
        op_atomic<OP>(&a.sum[qi], r);
        atomicAdd((ull*)&a.count[qi], (ull)c);
      }
      r = op_identity<OP>();
      c = 0;
      qi++;
      qend = a.off[qi + 1];
      lo = a.lo[qi]; hi = a.hi[qi]; fl = a.first[qi]; qoff = a.off[qi];
    }
    const uint64_t j = fl + (g - qoff);
    warp_decode(a.data + j * a.LB, min(a.used[j], a.LB), [&](uint32_t, uint64_t v) {
      if (v >= lo && v < hi && (v & mask) == value) { r = op_apply<OP>(r, v); c++; }
    }, true);
    g++;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) r = op_apply<OP>(r, __shfl_xor_sync(FULL, r, o));
  c = warp_sum(c);
  if (lane == 0 && c) {
    op_atomic<OP>(&a.sum[qi], r);
    atomicAdd((ull*)&a.count[qi], (ull)c);
  }
}


// RANK: lo/hi of a query are global element ranks [r0, r1) and the end
// leaves filter by rank P[j] + index; otherwise they are keys.
template <bool RANK>
__global__ void __launch_bounds__(kT) k_range(RangeArgs a) {
  const unsigned lane = lane_id();
  const uint64_t gw = gtid() >> 5, nw = gstride() >> 5;
  const uint64_t N = a.off[a.q];
  const uint64_t g0 = N * gw / nw, g1 = N * (gw + 1) / nw;
  if (g0 >= g1) return;
  uint64_t qi = upper_count(a.off, a.q + 1, g0) - 1;
  uint64_t s = 0, c = 0;
  ull nbytes = 0;
  uint64_t qend = a.off[qi + 1];
  uint64_t lo = a.lo[qi], hi = a.hi[qi], fl = a.first[qi], qoff = a.off[qi];
  uint64_t g = g0;
  while (g < g1) {
    while (g >= qend) {
      s = warp_sum(s);
      c = warp_sum(c);
      if (lane == 0 && (s | c)) {
        atomicAdd((ull*)&a.sum[qi], (ull)s);
        atomicAdd((ull*)&a.count[qi], (ull)c);
      }
      s = 0;
      c = 0;
      qi++;
      qend = a.off[qi + 1];
      lo = a.lo[qi]; hi = a.hi[qi]; fl = a.first[qi]; qoff = a.off[qi];
    }
    const uint64_t li = g - qoff, n = qend - qoff;
    if (li > 0 && li + 1 < n) {
      // leaves strictly inside the range: no filter, chunked span sum
      const uint64_t stop = min(g1, qend - 1);  // exclusive, global item index
      uint64_t cc = 0;
      warp_span_sum(a.data, a.used, a.cnt, a.LB, fl + li, fl + (stop - qoff), s, cc, nbytes);
      if (lane == 0) c += warp_sum(cc); else warp_sum(cc);
      g = stop;
      continue;
    }
    const uint64_t j = fl + li;
    const uint32_t u = min(a.used[j], a.LB);
    nbytes += u;
    if constexpr (RANK) {
      const uint64_t r = a.P[j];
      warp_decode(a.data + j * a.LB, u, [&](uint32_t idx, uint64_t v) {
        if (r + idx >= lo && r + idx < hi) { s += v; c++; }
      }, true);
    } else {
      warp_decode(a.data + j * a.LB, u, [&](uint32_t, uint64_t v) {
        if (v >= lo && v < hi) { s += v; c++; }
      }, true);
    }
    g++;
  }
  s = warp_sum(s);
  c = warp_sum(c);
  if (lane == 0 && (s | c)) {
    atomicAdd((ull*)&a.sum[qi], (ull)s);
    atomicAdd((ull*)&a.count[qi], (ull)c);
  }
  nbytes = warp_sum(nbytes);
  if (a.prof && lane == 0 && nbytes) atomicAdd(a.prof, nbytes);
}

// ---- byte codes (codec 0): a thread per leaf ----

// The leaf arrays of one set.
struct Leaves {
  const uint8_t* data;
  const uint32_t* used;
  const uint32_t* cnt;
  const uint64_t* heads;
  uint64_t L;
  uint32_t LB;
};

// No two elements of leaf j lie further apart: the next leaf's head (an empty
// one's is that of the next with elements, or 2^64 - 1, which may itself be the
// last element of j) is not below any of them.
__device__ __forceinline__ uint64_t leaf_span(const uint64_t* __restrict__ heads, uint64_t L,
                                              uint64_t j) {
  return j + 1 < L ? __ldg(heads + j + 1) - __ldg(heads + j) : ~0ull;
}

// Last index i in [a, n) with p[i] <= x, p sorted; a when p[a] > x too.  The
// next few entries are tried first: most ranges end in their first leaf or
// the one after it.
__device__ __forceinline__ uint64_t last_from(const uint64_t* __restrict__ p, uint64_t a, uint64_t n,
                                              uint64_t x) {
  uint64_t step = 1;
#pragma unroll 1
  for (int i = 0; i < 3; i++) {
    if (a + step >= n) break;
    if (__ldg(p + a + step) > x) {
      n = a + step;
      break;
    }
    a += step;
    step <<= 1;
  }
  if (n - a <= 1) return a;
  const uint64_t c = upper_count(p + a, n - a, x);
  return c ? a + c - 1 : a;
}

// What a range query reduces: PLAIN is (sum, count) without a filter, whose
// whole groups and leaf counts need no look at single elements.
template <int OP, bool PLAIN>
struct Reduce {
  uint64_t mask, value;
  __device__ __forceinline__ void leaf(const Leaves& t, uint64_t j, uint32_t u, uint64_t& r,
                                       uint64_t& c) const {
    if constexpr (PLAIN) {
      const uint32_t m = t.cnt[j];
      r += leafwalk::leaf_sum(t.data + j * t.LB, u, m, leaf_span(t.heads, t.L, j));
      c += m;
    } else {
      if (OP == CPMA_OP_SUM && !((mask | value) >> 32) &&
          !leafwalk::any_lane(leaf_span(t.heads, t.L, j) >= 1ull << 28)) {
        leafwalk::leaf_masked_sum(t.data + j * t.LB, u, (uint32_t)mask, (uint32_t)value, r, c);
        return;
      }
      leafwalk::leaf_visit(t.data + j * t.LB, u, [&](uint64_t v) {
        if ((v & mask) == value) { r = op_apply<OP>(r, v); c++; }
      });
    }
  }
  __device__ __forceinline__ void part(const uint8_t* leafp, uint32_t u, uint64_t lo, uint64_t hi,
                                       uint64_t& r, uint64_t& c) const {
    if constexpr (PLAIN) {
      leafwalk::leaf_range_sum(leafp, u, lo, hi, r, c);
    } else {
      leafwalk::leaf_range_visit(leafp, u, lo, hi, [&](uint64_t v) {
        if ((v & mask) == value) { r = op_apply<OP>(r, v); c++; }
      });
    }
  }
};

// A range query's first and last leaf: thread i routes query i and reduces
// its part of the first leaf; the queries that reach another leaf put their
// last one on the block's list, which the first threads then take, so a warp
// runs the second decode only when 32 of them have one.  Writes the ends'
// reduction and count and the leaves strictly between (first, items).  Three
// blocks per SM for plain sums (1e5 ranges 73 us; 84 with two, 77 with four).
template <int OP, bool PLAIN>
__global__ void __launch_bounds__(kT, PLAIN ? 3 : 1) k_range_ends(const uint64_t* __restrict__ lo,
                                                   const uint64_t* __restrict__ hi, uint64_t q,
                                                   Leaves t, Reduce<OP, PLAIN> f,
                                                   uint64_t* __restrict__ first,
                                                   uint64_t* __restrict__ items,
                                                   uint64_t* __restrict__ out,
                                                   uint64_t* __restrict__ count, uint32_t* ticket, ull* prof) {
  if (ticket && gtid() == 0) *ticket = 0;
  __shared__ uint64_t s_hi[kT], s_r[kT], s_c[kT];
  __shared__ uint32_t s_leaf[kT], s_q[kT];
  __shared__ uint32_t s_n;
  ull nbytes = 0;
  const uint64_t T = blockDim.x;
  for (uint64_t base = blockIdx.x * T; base < q; base += gridDim.x * T) {
    const uint64_t i = base + threadIdx.x;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    uint64_t r = op_identity<OP>(), c = 0, fl = 0, ll = 0, a = 0, b = 0;
    if (i < q) { a = lo[i]; b = hi[i]; }
    if (a < b) {
      fl = route_leaf(t.heads, t.L, a);
      ll = last_from(t.heads, fl, t.L, b - 1);
    }
    s_c[threadIdx.x] = 0;
    if (ll > fl) {
      const uint32_t slot = atomicAdd(&s_n, 1u);
      s_q[slot] = threadIdx.x;
      s_leaf[threadIdx.x] = (uint32_t)ll;
      s_hi[threadIdx.x] = b;
    }
    if (a < b) {
      const uint32_t u = min(t.used[fl], t.LB);
      nbytes += u;
      if (u) f.part(t.data + fl * t.LB, u, a, b, r, c);
    }
    __syncthreads();
    if (threadIdx.x < s_n) {
      const uint32_t w = s_q[threadIdx.x], j = s_leaf[w];
      const uint32_t u = min(t.used[j], t.LB);
      uint64_t r2 = op_identity<OP>(), c2 = 0;
      nbytes += u;
      if (u) f.part(t.data + (uint64_t)j * t.LB, u, 0, s_hi[w], r2, c2);
      s_r[w] = r2;
      s_c[w] = c2;
    }
    __syncthreads();
    if (s_c[threadIdx.x]) {
      r = op_apply<OP>(r, s_r[threadIdx.x]);
      c += s_c[threadIdx.x];
    }
    if (i < q) {
      first[i] = fl + 1;
      items[i] = ll > fl ? ll - fl - 1 : 0;
      out[i] = r;
      count[i] = c;
    }
    __syncthreads();
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// Is this block the last of the grid to come here?  Then it sees what the
// others wrote before.
__device__ __forceinline__ bool last_block(uint32_t* ticket) {
  __shared__ uint32_t s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  const bool last = s_last != 0;
  if (last) __threadfence();
  return last;
}

// The items' offsets by the last block of the ends' kernel (64 threads) instead
// of a scan of its own: a call with few queries waits for its launches.
constexpr uint64_t kEndsScan = 1024;  // queries at most: 16 items per thread
struct EndsScan {
  uint64_t* off = nullptr;       // q + 1 entries; null: not here
  ull* done = nullptr;           // blocks done: 0 between calls
};

__device__ __forceinline__ void scan_ends(const EndsScan& z, const uint64_t* items, uint64_t q) {
  __shared__ uint64_t s_w[2];
  __shared__ uint32_t s_last;
  if (!z.off) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(z.done, 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const uint32_t per = (uint32_t)((q + 63) / 64);
  const uint64_t i0 = min(q, (uint64_t)threadIdx.x * per), i1 = min(q, i0 + per);
  uint64_t v = 0;
  for (uint64_t i = i0; i < i1; i++) v += items[i];
  const uint64_t inc = warp_incl_scan(v);
  if (lane_id() == 31) s_w[threadIdx.x >> 5] = inc;
  __syncthreads();
  uint64_t run = inc - v + (threadIdx.x >= 32 ? s_w[0] : 0ull);
  for (uint64_t i = i0; i < i1; i++) {
    z.off[i] = run;
    run += items[i];
  }
  if (threadIdx.x == 63) z.off[q] = run;
  if (threadIdx.x == 0) *z.done = 0;
}

template <int OP, unsigned N>
__device__ __forceinline__ void team_reduce(uint64_t& r, uint64_t& c) {
#pragma unroll
  for (unsigned o = N / 2; o; o >>= 1) {
    r = op_apply<OP>(r, __shfl_xor_sync(FULL, r, o));
    c += __shfl_xor_sync(FULL, c, o);
  }
}

// k_range_ends by a team per end: the two teams of a query sit side by side, a
// warp's worth takes one end after the other.
template <int OP, bool PLAIN, unsigned N>
__global__ void __launch_bounds__(kT) k_range_ends_team(const uint64_t* __restrict__ lo,
                                                        const uint64_t* __restrict__ hi, uint64_t q,
                                                        Leaves t, Reduce<OP, PLAIN> f,
                                                        uint64_t* __restrict__ first,
                                                        uint64_t* __restrict__ items,
                                                        uint64_t* __restrict__ out,
                                                        uint64_t* __restrict__ count, uint32_t* ticket, EndsScan z, ull* prof) {
  if (ticket && gtid() == 0) *ticket = 0;
  ull nbytes = 0;
  constexpr unsigned kPer = N < 32 ? 2 * N : 32;  // lanes of a query
  const unsigned tl = team_lane<N>(), mine = lane_id() / kPer;
  for (uint64_t i0 = (gtid() >> 5) * (32 / kPer); i0 < q; i0 += (gstride() >> 5) * (32 / kPer)) {
    const uint64_t i = i0 + mine;
    uint64_t a = 0, b = 0, fl = 0, ll = 0;
    if (i < q) { a = lo[i]; b = hi[i]; }
    uint64_t r = op_identity<OP>(), c = 0;
    auto take = [&](uint64_t v) {
      if (v >= a && v < b && (PLAIN || (v & f.mask) == f.value)) { r = op_apply<OP>(r, v); c++; }
    };
    auto end = [&](uint64_t j, uint32_t u) {
      const uint8_t* leafp = t.data + j * t.LB;
      uint32_t idx;
      const leafwalk::Run run = team_leaf<N>(leafp, u, idx);
      if (u && tl == 0) take(run.k.val);
      if (u && run.k.val < b && run.k.val + run.delta >= a)
        leafwalk::run_visit(leafp, u, run, take);
      __syncwarp();
      if (tl == 0) nbytes += u;
    };
    if constexpr (N < 32) {
      const bool side = (lane_id() & N) != 0u;
      uint64_t j = 0;
      if (a < b) j = team_route<N>(t.heads, t.L, side ? b - 1 : a);
      __syncwarp();
      const uint64_t other = __shfl_xor_sync(FULL, j, N);
      fl = side ? other : j;
      ll = side ? j : other;
      end(j, a < b && (!side || ll > fl) ? min(t.used[j], t.LB) : 0u);
      team_reduce<OP, N>(r, c);
      r = op_apply<OP>(r, __shfl_down_sync(FULL, r, N));
      c += __shfl_down_sync(FULL, c, N);
    } else {
      if (a < b) {
        fl = team_route<N>(t.heads, t.L, a);
        ll = team_route<N>(t.heads, t.L, b - 1);
        end(fl, min(t.used[fl], t.LB));
        if (ll > fl) end(ll, min(t.used[ll], t.LB));
      }
      __syncwarp();
      team_reduce<OP, N>(r, c);
    }
    if (lane_id() % kPer == 0 && i < q) {
      first[i] = fl + 1;
      items[i] = ll > fl ? ll - fl - 1 : 0;
      out[i] = r;
      count[i] = c;
    }
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
  scan_ends(z, items, q);
}

// The same for map_range_length: thread i takes the first length[i] elements
// from start[i] on as far as its first leaf holds them; P (elements before
// each leaf) then names the leaf of the last one and how many it gives.
__global__ void __launch_bounds__(kT) k_length_ends(const uint64_t* __restrict__ start,
                                                    const uint64_t* __restrict__ length, uint64_t q,
                                                    Leaves t, const uint64_t* __restrict__ P,
                                                    uint64_t* __restrict__ first,
                                                    uint64_t* __restrict__ items,
                                                    uint64_t* __restrict__ sum,
                                                    uint64_t* __restrict__ count, uint32_t* ticket, ull* prof) {
  pdl_wait();
  pdl_launch();
  if (ticket && gtid() == 0) *ticket = 0;
  __shared__ uint64_t s_s[kT];
  __shared__ uint32_t s_leaf[kT], s_q[kT], s_k[kT];
  __shared__ uint32_t s_n;
  ull nbytes = 0;
  const uint64_t n = P[t.L];
  const uint64_t T = blockDim.x;
  for (uint64_t base = blockIdx.x * T; base < q; base += gridDim.x * T) {
    const uint64_t i = base + threadIdx.x;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    uint64_t s = 0, c = 0, fl = 0, ll = 0, len = 0;
    if (i < q) len = length[i];
    s_s[threadIdx.x] = 0;
    if (len) {
      const uint64_t x = start[i];
      fl = ll = route_leaf(t.heads, t.L, x);
      const uint32_t u = min(t.used[fl], t.LB);
      nbytes += u;
      uint32_t below = 0, taken = 0;
      if (u) leafwalk::leaf_take_sum(t.data + fl * t.LB, u, x, len, below, taken, s);
      c = taken;
      const uint64_t r0 = P[fl] + below;              // rank of the first key >= x
      const uint64_t r1 = len >= n - r0 ? n : r0 + len;
      if (r1 > r0 + taken) {                          // more in later leaves
        ll = last_from(P, fl, t.L + 1, r1 - 1);
        const uint32_t k = (uint32_t)(r1 - P[ll]);
        const uint32_t slot = atomicAdd(&s_n, 1u);
        s_q[slot] = threadIdx.x;
        s_leaf[threadIdx.x] = (uint32_t)ll;
        s_k[threadIdx.x] = k;
        c += k;
      }
    }
    __syncthreads();
    if (threadIdx.x < s_n) {
      const uint32_t w = s_q[threadIdx.x], j = s_leaf[w];
      const uint32_t u = min(t.used[j], t.LB);
      uint32_t below, taken;
      uint64_t s2 = 0;
      nbytes += u;
      if (u) leafwalk::leaf_take_sum(t.data + (uint64_t)j * t.LB, u, 0, s_k[w], below, taken, s2);
      s_s[w] = s2;
    }
    __syncthreads();
    if (i < q) {
      first[i] = fl + 1;
      items[i] = ll > fl ? ll - fl - 1 : 0;
      sum[i] = s + s_s[threadIdx.x];
      count[i] = c;
    }
    __syncthreads();
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// k_length_ends by a team per query.
template <unsigned N>
__global__ void __launch_bounds__(kT) k_length_ends_team(
    const uint64_t* __restrict__ start, const uint64_t* __restrict__ length, uint64_t q, Leaves t,
    const uint64_t* __restrict__ P, uint64_t* __restrict__ first, uint64_t* __restrict__ items,
    uint64_t* __restrict__ sum, uint64_t* __restrict__ count, uint32_t* ticket, EndsScan z, ull* prof) {
  pdl_wait();
  pdl_launch();
  if (ticket && gtid() == 0) *ticket = 0;
  ull nbytes = 0;
  const uint64_t n = P[t.L];
  const unsigned tl = team_lane<N>(), team = lane_id() / N;
  for (uint64_t i0 = (gtid() >> 5) * (32 / N); i0 < q; i0 += (gstride() >> 5) * (32 / N)) {
    const uint64_t i = i0 + team;
    uint64_t x = 0, len = 0, fl = 0, s = 0, c = 0;
    uint32_t u = 0, idx;
    if (i < q) len = length[i];
    if (len) {
      x = start[i];
      fl = team_route<N>(t.heads, t.L, x);
      u = min(t.used[fl], t.LB);
    }
    __syncwarp();
    const uint8_t* leafp = t.data + fl * t.LB;
    leafwalk::Run run = team_leaf<N>(leafp, u, idx);
    const uint64_t head = __shfl_sync(FULL, run.k.val, 0, N);
    uint64_t below = u && tl == 0 && head < x ? 1u : 0u;
    // the run's elements below x: none, all or, for one lane, some
    if (u && run.k.val < x) {
      if (run.k.val + run.delta < x) below += run.codes;
      else leafwalk::run_visit(leafp, u, run, [&](uint64_t v) { below += v < x ? 1u : 0u; });
    }
    __syncwarp();
    team_reduce<CPMA_OP_SUM, N>(s, below);
    const uint64_t r0 = P[fl] + below;  // rank of the first key >= x
    const uint64_t r1 = len >= n - r0 ? n : r0 + len;
    // the elements of ranks [r0, r1) in two leaves: its first, and its last one
    uint64_t j = fl, ll = fl;
    for (int end = 0; end < 2; end++) {
      const uint64_t p = P[j];
      const uint64_t from = r0 > p ? r0 - p : 0, to = u ? r1 - p : 0;  // of the leaf's elements
      uint32_t at = idx;
      auto take = [&](uint64_t v) {
        if (at >= from && at < to) { s += v; c++; }
        at++;
      };
      if (u && tl == 0) {
        at = 0;
        take(run.k.val);
      }
      if (u && idx < to && idx + run.codes > from) leafwalk::run_visit(leafp, u, run, take);
      __syncwarp();
      if (tl == 0) nbytes += u;
      if (end) break;
      u = 0;
      if (len && r1 > r0 && r1 > P[fl + 1]) {  // more in later leaves
        ll = j = last_from(P, fl, t.L + 1, r1 - 1);
        u = min(t.used[j], t.LB);
      }
      __syncwarp();
      leafp = t.data + j * t.LB;
      run = team_leaf<N>(leafp, u, idx);
    }
    team_reduce<CPMA_OP_SUM, N>(s, c);
    if (tl == 0 && i < q) {
      first[i] = fl + 1;
      items[i] = ll > fl ? ll - fl - 1 : 0;
      sum[i] = s;
      count[i] = c;
    }
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
  scan_ends(z, items, q);
}

// Reductions before (min: from) each leaf, in two levels: val / cnt inside
// the tile of kT leaves, tval / tcnt over the tiles.  Unused (null) when its
// memory cannot be had; taken when the queries' inner leaves number more than
// `most`.
struct LeafPrefix {
  uint64_t* val = nullptr;   // per leaf
  uint32_t* cnt = nullptr;   // per leaf: matches before it in its tile
  uint64_t* tval = nullptr;  // per tile
  uint64_t* tcnt = nullptr;
  uint32_t* ticket = nullptr;  // blocks done, cleared by the kernel before
  uint64_t most = ~0ull;
};

// Scan of one value per thread of a block of kT by op: exclusive from the
// front (REV false) or inclusive from the back; total = all of them.
template <int OP, bool REV>
__device__ __forceinline__ uint64_t block_scan_op(uint64_t v, uint64_t* ws, uint64_t* total) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = REV ? __shfl_down_sync(FULL, x, o) : __shfl_up_sync(FULL, x, o);
    if (REV ? lane + o < 32u : lane >= (unsigned)o) x = op_apply<OP>(x, y);
  }
  if (lane == (REV ? 0u : 31u)) ws[warp] = x;
  __syncthreads();
  uint64_t carry = op_identity<OP>(), all = op_identity<OP>();
#pragma unroll
  for (unsigned w = 0; w < kT / 32; w++) {
    const uint64_t y = ws[w];
    all = op_apply<OP>(all, y);
    if (REV ? w > warp : w < warp) carry = op_apply<OP>(carry, y);
  }
  *total = all;
  __syncthreads();  // ws is reused
  if (REV) return op_apply<OP>(carry, x);
  uint64_t e = __shfl_up_sync(FULL, x, 1);
  if (lane == 0) e = op_identity<OP>();
  return op_apply<OP>(carry, e);
}

constexpr uint32_t kSumShift = 4;      // sort key of a leaf: bytes to decode / 16
constexpr uint32_t kSumBuckets = 128;  // enough for 2048-byte leaves (a multiple of 32)

// Order of the nt <= kT leaves of a tile by the bytes u to decode of each (a
// counting sort in shared memory), so the 32 leaves a warp decodes side by
// side take about the same number of steps: order[i] = the one thread i takes.
__device__ __forceinline__ void order_tile(uint32_t u, uint32_t nt, uint32_t* hist,
                                           uint32_t* order) {
  for (uint32_t i = threadIdx.x; i < kSumBuckets; i += kT) hist[i] = 0;
  __syncthreads();
  const uint32_t bkt = min(u >> kSumShift, kSumBuckets - 1);
  const uint32_t slot = threadIdx.x < nt ? atomicAdd(&hist[bkt], 1u) : 0u;
  __syncthreads();
  if (threadIdx.x < 32) {  // exclusive scan of the bucket counts
    uint32_t run = 0;
    for (uint32_t b = 0; b < kSumBuckets; b += 32) {
      const uint32_t v = hist[b + threadIdx.x];
      const uint32_t inc = warp_incl_scan(v);
      hist[b + threadIdx.x] = run + inc - v;
      run += __shfl_sync(FULL, inc, 31);
    }
  }
  __syncthreads();
  if (threadIdx.x < nt) order[hist[bkt] + slot] = threadIdx.x;
  __syncthreads();
}

// The tiles' reductions scanned in place by one block: exclusive from the
// front (min: from the back).
template <int OP>
__device__ void tile_scan(const LeafPrefix& p, uint64_t nt, uint64_t* s_ws) {
  constexpr bool REV = OP == CPMA_OP_MIN;
  // a contiguous run of tiles per thread: reduced, scanned over the block,
  // rescanned
  const uint64_t per = (nt + kT - 1) / kT;
  const uint64_t b0 = min(nt, threadIdx.x * per), b1 = min(nt, b0 + per);
  uint64_t r = op_identity<OP>(), c = 0;
  for (uint64_t b = b0; b < b1; b++) {
    r = op_apply<OP>(r, p.tval[b]);
    c += p.tcnt[b];
  }
  uint64_t all;
  uint64_t x;
  if (REV) {  // exclusive from the back: the inclusive one of the next thread
    const uint64_t inc = block_scan_op<OP, true>(r, s_ws, &all);
    __shared__ uint64_t s_inc[kT + 1];
    s_inc[threadIdx.x] = inc;
    if (threadIdx.x == 0) s_inc[kT] = op_identity<OP>();
    __syncthreads();
    x = s_inc[threadIdx.x + 1];
  } else {
    x = block_scan_op<OP, false>(r, s_ws, &all);
  }
  uint64_t y = block_scan_op<CPMA_OP_SUM, false>(c, s_ws, &all);
  for (uint64_t b = b0; b < b1; b++) {
    const uint64_t v = p.tcnt[b];
    p.tcnt[b] = y;
    y += v;
  }
  if (REV) {
    for (uint64_t b = b1; b-- > b0;) {
      const uint64_t v = p.tval[b];
      p.tval[b] = x;
      x = op_apply<OP>(x, v);
    }
  } else {
    for (uint64_t b = b0; b < b1; b++) {
      const uint64_t v = p.tval[b];
      p.tval[b] = x;
      x = op_apply<OP>(x, v);
    }
  }
}

__global__ void __launch_bounds__(kT) k_tile_scan(LeafPrefix p, uint64_t nt) {
  __shared__ uint64_t s_ws[kT / 32];
  pdl_wait();
  pdl_launch();
  tile_scan<CPMA_OP_SUM>(p, nt, s_ws);
}

// The reductions and counts of the leaves by eight lanes each, for sets of few
// leaves (sum_by_teams), to p.val and p.cnt.
template <int OP, bool PLAIN>
__global__ void __launch_bounds__(kT) k_leaf_reduce(Leaves t, Reduce<OP, PLAIN> f,
                                                    const uint64_t* __restrict__ total,
                                                    LeafPrefix p, ull* prof) {
  pdl_wait();
  pdl_launch();
  if (*total <= p.most) return;
  const unsigned tl = team_lane<kTeam>();
  ull nbytes = 0;
  for (uint64_t j0 = (gtid() >> 5) * (32 / kTeam); j0 < t.L; j0 += (gstride() >> 5) * (32 / kTeam)) {
    const uint64_t j = j0 + lane_id() / kTeam;
    const uint32_t u = j < t.L ? min(t.used[j], t.LB) : 0u;
    const uint8_t* leafp = t.data + (j < t.L ? j : 0) * t.LB;
    uint32_t idx;
    const leafwalk::Run run = team_leaf<kTeam, PLAIN>(leafp, u, idx);
    uint64_t r = op_identity<OP>(), c = 0;
    if constexpr (PLAIN) {
      if (u) {
        r = run.codes * run.k.val + run.sum + (tl == 0 ? run.k.val : 0ull);
        c = run.codes + (tl == 0 ? 1u : 0u);
      }
    } else {
      auto take = [&](uint64_t v) {
        if ((v & f.mask) == f.value) { r = op_apply<OP>(r, v); c++; }
      };
      if (u && tl == 0) take(run.k.val);
      leafwalk::run_visit(leafp, u, run, take);
      __syncwarp();
    }
    team_reduce<OP, kTeam>(r, c);
    if (tl == 0 && j < t.L) {
      p.val[j] = r;
      p.cnt[j] = (uint32_t)c;
      nbytes += u;
    }
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// Every leaf reduced once (GIVEN: k_leaf_reduce has done it), scanned inside tiles
// of kT leaves, and the tiles by the last block to finish (when the queries cover
// more than p.most leaves; otherwise nothing).
// Four blocks per SM: the lanes' scattered loads are what it waits for (plain,
// 1e8 keys: 106 us with the registers it would take, 76 us; masked sums, 5e7
// keys: 157 and 109 us).
template <int OP, bool PLAIN, bool GIVEN>
__global__ void __launch_bounds__(kT, 4) k_leaf_prefix(Leaves t, Reduce<OP, PLAIN> f,
                                                    const uint64_t* __restrict__ total,
                                                    LeafPrefix p, ull* prof) {
  __shared__ uint32_t s_hist[kSumBuckets], s_order[kT];
  __shared__ uint64_t s_r[kT], s_ws[kT / 32];
  __shared__ uint32_t s_c[kT];
  pdl_wait();
  pdl_launch();
  if (*total <= p.most) return;
  ull nbytes = 0;
  const uint64_t nt = (t.L + kT - 1) / kT;
  for (uint64_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    const uint64_t j0 = tile * kT, j = j0 + threadIdx.x;
    const uint32_t n = (uint32_t)min((uint64_t)kT, t.L - j0);
    if (!GIVEN) order_tile(threadIdx.x < n ? min(t.used[j], t.LB) : 0u, n, s_hist, s_order);
    s_r[threadIdx.x] = GIVEN && threadIdx.x < n ? p.val[j] : op_identity<OP>();
    s_c[threadIdx.x] = GIVEN && threadIdx.x < n ? p.cnt[j] : 0;
    __syncthreads();
    if (!GIVEN && threadIdx.x < n) {
      const uint32_t o = s_order[threadIdx.x];
      const uint32_t u = min(t.used[j0 + o], t.LB);
      uint64_t r = op_identity<OP>(), c = 0;
      if (u) {
        f.leaf(t, j0 + o, u, r, c);
        nbytes += u;
      }
      s_r[o] = r;
      s_c[o] = (uint32_t)c;
    }
    __syncthreads();
    uint64_t all, call;
    const uint64_t x = block_scan_op<OP, OP == CPMA_OP_MIN>(s_r[threadIdx.x], s_ws, &all);
    const uint64_t c = block_scan_op<CPMA_OP_SUM, false>((uint64_t)s_c[threadIdx.x], s_ws, &call);
    if (threadIdx.x < n) {
      p.val[j] = x;
      p.cnt[j] = (uint32_t)c;
    }
    if (threadIdx.x == 0) {
      p.tval[tile] = all;
      p.tcnt[tile] = call;
    }
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
  if (last_block(p.ticket)) tile_scan<OP>(p, nt, s_ws);
}

// The warp's equal contiguous share of N items that its lanes take one each:
// as many warps as have 32 of them, spread over the blocks, so that few items
// do not leave most lanes of every warp idle (with shares over all 9728 warps
// of the grid, the 2.4e4 inner leaves of 1e5 short scans ran 2.3 lanes a warp:
// 54 us, now 16; the 1e5 leaves that a packed neighbour query extracts 5.4
// lanes: 73 us, now 41, the start of each first leaf's walk included).
__device__ __forceinline__ void lane_share(uint64_t N, uint64_t& g0, uint64_t& g1) {
  const uint64_t w = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const uint64_t nw = max((uint64_t)1, min(gstride() >> 5, (N + 31) >> 5));
  g0 = g1 = 0;
  if (w >= nw) return;
  g0 = N * w / nw;
  g1 = N * (w + 1) / nw;
}

// The leaves strictly inside the ranges.  From the prefix: a thread per
// query.  Otherwise the (query, leaf) items in equal contiguous shares per
// warp, one leaf per lane: a lane keeps its partial while it stays on one
// query and adds it atomically when it leaves it (the functions commute); a
// warp whose lanes end on one query adds once.
template <int OP, bool PLAIN, unsigned TL>
__global__ void __launch_bounds__(kT) k_range_inner(Leaves t, Reduce<OP, PLAIN> f, uint64_t q,
                                                    const uint64_t* __restrict__ first,
                                                    const uint64_t* __restrict__ off, LeafPrefix p,
                                                    uint64_t* __restrict__ out,
                                                    uint64_t* __restrict__ count, ull* prof) {
  pdl_wait();
  const uint64_t N = off[q];
  if (N > p.most) {
    for (uint64_t i = gtid(); i < q; i += gstride()) {
      const uint64_t n = off[i + 1] - off[i];
      if (!n) continue;
      const uint64_t a = first[i], b = a + n;  // b: the query's last leaf
      const uint64_t ca = p.tcnt[a / kT] + p.cnt[a], cb = p.tcnt[b / kT] + p.cnt[b];
      if (ca == cb) continue;
      uint64_t r;
      if constexpr (OP == CPMA_OP_MIN) r = min(p.val[a], p.tval[a / kT]);
      else if constexpr (OP == CPMA_OP_MAX) r = max(p.val[b], p.tval[b / kT]);
      else if constexpr (OP == CPMA_OP_XOR)
        r = (p.val[b] ^ p.tval[b / kT]) ^ (p.val[a] ^ p.tval[a / kT]);
      else r = (p.val[b] + p.tval[b / kT]) - (p.val[a] + p.tval[a / kT]);
      out[i] = op_apply<OP>(out[i], r);
      count[i] += cb - ca;
    }
    return;
  }
  const unsigned lane = lane_id();
  if (N * kTeam * 4 <= gstride() && N * TL <= gstride()) {  // few: a team per item
    const uint64_t e0 = ((uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * (32 / TL);
    if (e0 >= N) return;
    const uint64_t e = e0 + lane / TL;
    uint64_t qi = 0, j = 0;
    uint32_t u = 0, idx;
    if (e < N) {
      qi = team_upper_count<TL>(off, q + 1, e) - 1;
      j = first[qi] + (e - off[qi]);
      u = min(t.used[j], t.LB);
    }
    __syncwarp();
    const uint8_t* leafp = t.data + j * t.LB;
    const leafwalk::Run run = team_leaf<TL>(leafp, u, idx);
    uint64_t r = op_identity<OP>(), c = 0;
    auto take = [&](uint64_t v) {
      if (PLAIN || (v & f.mask) == f.value) { r = op_apply<OP>(r, v); c++; }
    };
    if (u && team_lane<TL>() == 0) take(run.k.val);
    leafwalk::run_visit(leafp, u, run, take);
    __syncwarp();
    team_reduce<OP, TL>(r, c);
    if (team_lane<TL>() == 0 && c) {
      op_atomic<OP>(&out[qi], r);
      atomicAdd((ull*)&count[qi], (ull)c);
    }
    if (prof && team_lane<TL>() == 0 && u) atomicAdd(prof, (ull)u);
    return;
  }
  uint64_t g0, g1;
  lane_share(N, g0, g1);
  if (g0 >= g1) return;
  uint64_t qi = 0, qend = 0, qoff = 0, fl = 0;
  uint64_t r = op_identity<OP>(), c = 0;
  ull nbytes = 0;
  auto flush = [&] {
    if (c) {
      op_atomic<OP>(&out[qi], r);
      atomicAdd((ull*)&count[qi], (ull)c);
    }
    r = op_identity<OP>();
    c = 0;
  };
  for (uint64_t g = g0 + lane; g < g1; g += 32) {
    if (g >= qend) {
      flush();
      qi += upper_count(off + qi, q + 1 - qi, g) - 1;
      qoff = off[qi];
      qend = off[qi + 1];
      fl = first[qi];
    }
    const uint64_t j = fl + (g - qoff);
    const uint32_t u = min(t.used[j], t.LB);
    nbytes += u;
    if (u) f.leaf(t, j, u, r, c);
  }
  const uint64_t q0 = __shfl_sync(FULL, qi, 0);
  if (__all_sync(FULL, qi == q0 || c == 0)) {
#pragma unroll
    for (int o = 16; o; o >>= 1) r = op_apply<OP>(r, __shfl_xor_sync(FULL, r, o));
    c = warp_sum(c);
    if (lane == 0) flush();
  } else {
    flush();
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane == 0 && nbytes) atomicAdd(prof, nbytes);
}

// ---- many plain range sums: marks inside the leaves ----
//
// With a query per leaf and more, walks from the heads decode most of the set,
// and with many more decode it several times over.  Then every leaf is walked once,
// its state kept at every 32nd byte (leafwalk::Mark) and the leaves' sums and
// counts scanned, and a query is the difference of two lookups: prefix of the
// leaf, last mark below the bound, at most 32 bytes walked from there.  Bound
// by instruction issue.  Degrees of 2^20 vertices (1.4e7 edges, 1.4e5 leaves):
// 150 us, of which marking 36; 484 us walked from the heads.

// Per leaf `per` marks: [0] = its head and the sum and count before it in its
// tile, then the marks at 32, 64, ..; per tile of kT leaves tval and tcnt, as
// in LeafPrefix.
struct Marks {
  leafwalk::Mark* at = nullptr;
  uint32_t per = 0;
  LeafPrefix tiles;
};

__global__ void __launch_bounds__(kT) k_marks(Leaves t, Marks mk, ull* prof) {
  __shared__ uint32_t s_hist[kSumBuckets], s_order[kT];
  __shared__ uint64_t s_r[kT], s_h[kT], s_ws[kT / 32];
  __shared__ uint32_t s_c[kT];
  pdl_launch();
  ull nbytes = 0;
  const uint64_t nt = (t.L + kT - 1) / kT;
  for (uint64_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    const uint64_t j0 = tile * kT, j = j0 + threadIdx.x;
    const uint32_t n = (uint32_t)min((uint64_t)kT, t.L - j0);
    order_tile(threadIdx.x < n ? min(t.used[j], t.LB) : 0u, n, s_hist, s_order);
    s_r[threadIdx.x] = 0;
    s_c[threadIdx.x] = 0;
    s_h[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x < n) {
      const uint32_t o = s_order[threadIdx.x];
      const uint32_t u = min(t.used[j0 + o], t.LB);
      if (u) {
        const uint8_t* leafp = t.data + (j0 + o) * t.LB;
        leafwalk::Mark* m = mk.at + (j0 + o) * mk.per;
        uint64_t s;
        uint32_t c;
        leafwalk::leaf_marks(leafp, u, s, c,
                             [&](uint32_t i, const leafwalk::Mark& v) { m[i] = v; });
        s_r[o] = s;
        s_c[o] = c;
        s_h[o] = leafwalk::leaf_head(leafp);
        nbytes += u;
      }
    }
    __syncthreads();
    uint64_t all, call;
    const uint64_t x = block_scan_op<CPMA_OP_SUM, false>(s_r[threadIdx.x], s_ws, &all);
    const uint64_t c = block_scan_op<CPMA_OP_SUM, false>((uint64_t)s_c[threadIdx.x], s_ws, &call);
    if (threadIdx.x < n)
      mk.at[j * mk.per] = leafwalk::Mark{s_h[threadIdx.x], x, 0, (uint32_t)c, 0};
    if (threadIdx.x == 0) {
      mk.tiles.tval[tile] = all;
      mk.tiles.tcnt[tile] = call;
    }
    __syncthreads();
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// Sum and number of the set's elements < x, x's leaf being j: every element
// of the leaves before j is < x, none of those after it is.
__device__ __forceinline__ void below_marked(const Leaves& t, const Marks& mk, uint64_t j,
                                             uint64_t x, uint64_t& s, uint64_t& c) {
  const leafwalk::Mark* m = mk.at + j * mk.per;
  const leafwalk::Mark m0 = m[0];
  s = mk.tiles.tval[j / kT] + m0.sum;
  c = mk.tiles.tcnt[j / kT] + m0.cnt;
  const uint32_t u = min(t.used[j], t.LB);
  if (!u || m0.val >= x) return;
  // the last mark whose element is below x; every mark of the leaf lies at a
  // byte < u
  uint32_t a = 0, b = (u - 1u) / leafwalk::kMark;
  while (a < b) {
    const uint32_t mid = (a + b + 1u) >> 1;
    if (m[mid].val < x) a = mid;
    else b = mid - 1u;
  }
  leafwalk::Mark f = m0;
  if (a) f = m[a];
  s += a ? f.sum : f.val;
  c += a ? f.cnt : 1u;
  f.sh = a ? f.sh : 0u;
  leafwalk::below_sum(t.data + j * t.LB, u, a * leafwalk::kMark, leafwalk::walk_at(f), x, s, c);
}

__global__ void __launch_bounds__(kT) k_range_marked(const uint64_t* __restrict__ lo,
                                                     const uint64_t* __restrict__ hi, uint64_t q,
                                                     Leaves t, Marks mk,
                                                     uint64_t* __restrict__ out,
                                                     uint64_t* __restrict__ count, ull* prof) {
  pdl_wait();
  ull nbytes = 0;
  for (uint64_t i = gtid(); i < q; i += gstride()) {
    const uint64_t a = lo[i], b = hi[i];
    uint64_t s = 0, c = 0;
    if (a < b) {
      uint64_t j = route_leaf(t.heads, t.L, a), x = a;
#pragma unroll 1
      for (int e = 0; e < 2; e++) {
        uint64_t se, ce;
        below_marked(t, mk, j, x, se, ce);
        s = se - s;
        c = ce - c;
        if (e) break;
        x = b;
        j = last_from(t.heads, j, t.L, b - 1);
      }
      nbytes += 2 * leafwalk::kMark;
    }
    out[i] = s;
    count[i] = c;
  }
  nbytes = warp_sum(nbytes);
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

// Ranks of both ends of the key ranges [A, B): two lanes per query, one end
// each.  The leaves that hold the ranks come from P (elements before each
// leaf), searched from the end's own leaf on.
__global__ void __launch_bounds__(kT) k_rank_ends(const uint64_t* __restrict__ A,
                                                  const uint64_t* __restrict__ B, uint64_t q,
                                                  Leaves t, const uint64_t* __restrict__ P,
                                                  uint64_t* __restrict__ r0o,
                                                  uint64_t* __restrict__ r1o,
                                                  uint64_t* __restrict__ first,
                                                  uint64_t* __restrict__ items,
                                                  uint64_t* __restrict__ count,
                                                  leafwalk::Mark* __restrict__ start) {
  pdl_wait();
  pdl_launch();
  // whole warps stay in the loop: both lanes of a query take part in it
  for (uint64_t g = gtid() & ~31ull; g < 2 * q; g += gstride()) {
    const uint64_t e = g + lane_id(), i = e >> 1;
    uint64_t r = 0, j = 0;
    leafwalk::Mark at{0, 0, 0, 0, 0};
    if (i < q) {
      const uint64_t x = (e & 1) ? B[i] : A[i];
      j = route_leaf(t.heads, t.L, x);
      const uint32_t u = min(t.used[j], t.LB);
      r = P[j] + (u ? leafwalk::leaf_below(t.data + j * t.LB, u, x, at) : 0u);
    }
    const uint64_t r1 = __shfl_down_sync(FULL, r, 1);
    if (i < q && !(e & 1)) {
      uint64_t hi = A[i] < B[i] ? r1 : r, fl = 0, it = 0;
      if (hi > r) {
        fl = last_from(P, j, t.L + 1, r);
        it = last_from(P, fl, t.L + 1, hi - 1) - fl + 1;
      } else {
        hi = r;
      }
      r0o[i] = r;
      r1o[i] = hi;
      first[i] = fl;
      items[i] = it;
      count[i] = hi - r;
      if (start) start[i] = at;  // its byte is 0 unless fl == j
    }
  }
}

// The keys of ranks [r0, r1) of every query, one (query, leaf) item per lane:
// out[off + r - r0] = key of rank r (entries at or past cap are dropped).  A
// query's first leaf is walked from where the search for its first key ended
// (a.start, null without room for it), the others from their heads.  A
// lane stores its leaf's keys one after another; the eight bytes of
// neighbouring keys meet in the L2's lines.
__global__ void __launch_bounds__(kT) k_extract_leaf(ExtractArgs a) {
  pdl_wait();
  uint64_t g0, g1;
  lane_share(a.item_off[a.q], g0, g1);
  uint64_t qi = 0, qend = 0;
  for (uint64_t g = g0 + lane_id(); g < g1; g += 32) {
    if (g >= qend) {
      qi += upper_count(a.item_off + qi, a.q + 1 - qi, g) - 1;
      qend = a.item_off[qi + 1];
    }
    const uint64_t j = a.first[qi] + (g - a.item_off[qi]);
    const uint64_t r0 = a.r0[qi], r1 = a.r1[qi], base = a.P[j], o = a.out_off[qi];
    const uint32_t u = min(a.used[j], a.LB);
    if (!u) continue;
    if (a.cap <= o) continue;
    // element idx of the leaf goes to dst[idx] for skip <= idx < stop
    const uint64_t room = a.cap - o;
    uint64_t stop = r1 - base;
    uint32_t skip = 0;
    if (r0 >= base) {
      skip = (uint32_t)(r0 - base);
      if (stop - skip > room) stop = skip + room;
    } else {
      const uint64_t before = base - r0;  // the query's keys in earlier leaves
      if (room <= before) continue;
      stop = min(stop, room - before);
    }
    uint64_t* dst = a.out + (int64_t)(o + base - r0);
    uint32_t idx = 0, p = 8;
    const uint32_t st = (uint32_t)min(stop, (uint64_t)0xFFFFFFFFu);
    const uint8_t* leafp = a.data + j * a.LB;
    auto put = [&](uint64_t v) {
      if (idx >= skip && idx < st) dst[idx] = v;
      idx++;
    };
    leafwalk::Walk k;
    leafwalk::Mark m{0, 0, 0, 0, 0};
    if (a.start && r0 >= base) m = a.start[qi];
    if (m.sum) {  // from where the first key's search ended
      k = leafwalk::walk_at(m);
      p = (uint32_t)m.sum;
      idx = m.cnt;
    } else {
      k.val = leafwalk::leaf_head(leafp);
      put(k.val);
    }
    leafwalk::visit_from(leafp, u, p, k, put, [&] { return idx >= st; });
  }
}

__global__ void __launch_bounds__(kT, 4) k_sum(const uint8_t* __restrict__ data,
                                            const uint32_t* __restrict__ used,
                                            const uint32_t* __restrict__ cnt,
                                            const uint64_t* __restrict__ heads, uint64_t L,
                                            uint32_t LB, uint64_t* sum, uint64_t* count,
                                            ull* prof, int raw) {
  const unsigned lane = lane_id();
  const uint64_t gw = gtid() >> 5, nw = gstride() >> 5;
  const uint64_t j0 = L * gw / nw, j1 = L * (gw + 1) / nw;
  uint64_t s = 0, c = 0;
  ull nbytes = 0;
  if (raw) {
    warp_span_sum(data, used, cnt, LB, j0, j1, s, c, nbytes);
  } else {
    // the block's leaves in tiles of kT, each ordered by used bytes
    __shared__ uint32_t s_hist[kSumBuckets];
    __shared__ uint32_t s_order[kT];
    const uint64_t b0 = L * blockIdx.x / gridDim.x, b1 = L * (blockIdx.x + 1) / gridDim.x;
    for (uint64_t t0 = b0; t0 < b1; t0 += kT) {
      const uint32_t nt = (uint32_t)min((uint64_t)kT, b1 - t0);
      order_tile(threadIdx.x < nt ? min(used[t0 + threadIdx.x], LB) : 0u, nt, s_hist, s_order);
      if (threadIdx.x < nt) {
        const uint64_t jj = t0 + s_order[threadIdx.x];
        const uint32_t uu = min(used[jj], LB);
        nbytes += 8;  // its used and element counts
        if (uu) {
          const uint32_t m = cnt[jj];
          s += leafwalk::leaf_sum(data + jj * LB, uu, m, leaf_span(heads, L, jj));
          c += m;
          nbytes += uu;
        }
      }
      __syncthreads();  // s_hist and s_order are reused
    }
  }
  s = warp_sum(s);
  c = warp_sum(c);
  nbytes = warp_sum(nbytes);
  if (lane == 0 && (s | c)) {
    atomicAdd((ull*)sum, (ull)s);
    if (count) atomicAdd((ull*)count, (ull)c);
  }
  if (prof && lane == 0 && nbytes) atomicAdd(prof, nbytes + (raw ? 8ull * (j1 - j0) : 0ull));
}

// The same of byte codes by eight lanes per leaf, for sets of few leaves: bound by
// the walk of the longest run.
__global__ void __launch_bounds__(kT) k_sum_team(const uint8_t* __restrict__ data,
                                                 const uint32_t* __restrict__ used,
                                                 const uint32_t* __restrict__ cnt, uint64_t L,
                                                 uint32_t LB, uint64_t* sum, uint64_t* count,
                                                 ull* prof) {
  const unsigned tl = team_lane<kTeam>();
  uint64_t s = 0, c = 0;
  ull nbytes = 0;
  for (uint64_t j0 = (gtid() >> 5) * (32 / kTeam); j0 < L; j0 += (gstride() >> 5) * (32 / kTeam)) {
    const uint64_t j = j0 + lane_id() / kTeam;
    const uint32_t u = j < L ? min(used[j], LB) : 0u;
    uint32_t idx;
    const leafwalk::Run r = team_leaf<kTeam, true>(data + (j < L ? j : 0) * LB, u, idx);
    if (u) s += r.codes * r.k.val + r.sum + (tl == 0 ? r.k.val : 0ull);
    if (j < L && tl == 0) {
      nbytes += 8 + u;  // its used and element counts
      if (u) c += cnt[j];
    }
  }
  s = warp_sum(s);
  c = warp_sum(c);
  nbytes = warp_sum(nbytes);
  if (lane_id() == 0 && (s | c)) {
    atomicAdd((ull*)sum, (ull)s);
    if (count) atomicAdd((ull*)count, (ull)c);
  }
  if (prof && lane_id() == 0 && nbytes) atomicAdd(prof, nbytes);
}

int persistent_grid(const cpma* h) { return h->num_sms * 8; }

bool large_leaves(const cpma* h) { return h->cfg.leaf_bytes > 512; }

// Few enough queries for a team of lanes per leaf instead of a thread: a team
// spends about twice a thread's instructions on a leaf in a fraction of its time.
// Speed of teams over threads, geometric mean over sets of 300 to 1e7 keys of 1 to
// 6 bytes and short and wide queries (lowest, highest): ranges with a mask, 512-byte
// leaves, 9.8e3 queries 1.47 (1.23, 1.66), 1.5e4 1.33, 2.5e4 1.08 (0.90, 1.26), 4e4
// 0.92; plain ones 1.39, 1.28, 1.02, 0.86; scans by length 1.12, 0.99, 0.81, 0.71;
// 256-byte leaves within 0.1 of these.  2048-byte leaves, 1.5e4 and 2.5e4 queries:
// ranges 1.27 and about 1, scans by length 0.9 and 0.7.
bool few_ranges(const cpma* h, uint64_t q) { return q <= (uint64_t)h->num_sms * 160; }
bool few_scans(const cpma* h, uint64_t q) {
  return q <= (uint64_t)h->num_sms * (large_leaves(h) ? 64 : 96);
}
// A lookup is half a range.  Calls in a row over different batches of 1 to 4000 keys,
// us a call by teams / by threads, sets of 34- and 40-bit keys, of 64-bit ones and of
// edges: 256-byte leaves 6 to 8 / 6 to 9, 6 to 9 / 10 to 12, 6 to 10 / 8 to 17; 512-byte
// ones 6 to 8 / 7 to 10, 8 to 10 / 12 to 17, 7 to 12 / 9 to 27; 1024-byte ones 6 to 10 /
// 8 to 13, 6 to 12 / 17 to 27, 6 to 16 / 17 to 45; 2048-byte ones 6 to 15 / 11 to 19, 7
// to 17 / 33 to 47, 6 to 24 / 21 to 84.  7000 of them: 2048-byte leaves 20 / 19, 21 /
// 47, 30 / 83, 1024-byte ones 14 / 13, 14 / 27, 19 / 46.
bool few_lookups(const cpma* h, uint64_t q) {
  return q <= (uint64_t)h->num_sms * (large_leaves(h) ? 48 : 32);
}

// A team is a warp where a leaf has more than 512 bytes and the queries are few
// enough for that.  Speed of warps over eight lanes, 1e3, 2.5e3, 5e3, 9.7e3 queries:
// 2048-byte leaves, ranges 1.15, 1.11, 1.04, 0.94, scans by length 1.51, 1.36, 1.15,
// 0.96; 1024-byte ones 1.07, 1.02, 0.96, 0.88 and 1.30, 1.21, 1.06, 0.92.
bool warp_teams(const cpma* h, uint64_t q) {
  return large_leaves(h) && q <= (uint64_t)h->num_sms * 24;
}

// Whether a full sum takes eight lanes per leaf: while that many threads run at
// once (half of them for large leaves, where a lane's own walk is long).  Eight
// lanes / one, us: 512-byte leaves 4.3e3 of them 16.5 / 22.7, 3.9e4 (edges) 29 / 45,
// 1.2e5 43 / 28; 2048-byte ones 9.5e3 (edges) 30 / 114, 2.8e4 34 / 57, 1.4e5 100 / 91.
bool sum_by_teams(const cpma* h) {
  const uint64_t threads = (uint64_t)persistent_grid(h) * kT;
  return !h->cfg.codec && h->L * kTeam <= threads * (large_leaves(h) ? 2 : 1);
}

// Scratch of the allocation-free range_map: per-query first leaf, item count
// and item offsets, plus the partial sums of the offset scan.  It lives in the
// library's own device image, so every GPU that loads the library holds these
// 2 MiB until the process exits, and every call shares them.
constexpr uint64_t kNoAllocMaxQueries = 1ull << 16;
constexpr uint64_t kNoAllocPartials = 1024;
constexpr size_t kNoAllocBytes = 2u << 20;
static_assert((3 * kNoAllocMaxQueries + 1 + kNoAllocPartials) * 8 <= kNoAllocBytes,
              "range scratch too small");
static __device__ __align__(256) uint8_t g_range_scratch[kNoAllocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_addr[kMaxDevices] = {nullptr};

// Device address of g_range_scratch on device `dev` (which must be current).
// The host-side name of the array is only a stand-in, so the address is
// looked up once per device with cudaGetSymbolAddress and cached.
int scratch_address(int dev, uint8_t** out) {
  if (dev < 0 || dev >= kMaxDevices) return CPMA_EINVAL;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_range_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return CPMA_ECUDA;
    }
    g_scratch_addr[dev] = p;
  }
  *out = static_cast<uint8_t*>(g_scratch_addr[dev]);
  return CPMA_OK;
}

}  // namespace

namespace {

// Few enough queries for range_extract to take a warp per leaf, as for cells: a
// thread walks and stores a whole leaf in a chain that grows with its size, and
// with few leaves nothing hides it.  Warps / threads, us, lists of up to 50 and of
// 100 to 1000 keys: 512-byte leaves, 100 queries 33 / 31 and 37 / 44 (40-bit keys), 35
// / 41 and 37 / 54 (edges), 1000 41 / 35 and 49 / 46, 41 / 45 and 49 / 59; 2048-byte
// ones, 1000 47 / 46 and 56 / 92, 46 / 82 and 55 / 139, 9700 114 / 57 and 148 / 108,
// 116 / 102 and 135 / 165.  256-byte leaves by threads always.
bool extract_by_warps(const cpma* h, uint64_t q) {
  const uint64_t LB = h->cfg.leaf_bytes;
  return LB >= 512 && q <= (uint64_t)h->num_sms * LB / 128;
}

}  // namespace

int run_has(const cpma* h, const uint64_t* d_keys, uint64_t q, uint8_t* d_out, cudaStream_t st) {
  if (q == 0) return CPMA_OK;
  const bool few = !h->cfg.codec && few_lookups(h, q);
  const uint64_t per = few ? kT / (warp_teams(h, q) ? kTeamLarge : kTeam) : kT;  // keys a block
  const int grid = (int)std::max<uint64_t>(
      1, std::min<uint64_t>((q + per - 1) / per, (uint64_t)persistent_grid(h)));
  prof_begin(h, PH_HAS, st);
  const auto kern = h->cfg.codec ? k_has_cells
                    : !few       ? k_has
                    : warp_teams(h, q) ? k_has_team<kTeamLarge> : k_has_team<kTeam>;
  kern<<<grid, kT, 0, st>>>(d_keys, q, h->data, h->used, h->heads, h->L, h->cfg.leaf_bytes, d_out,
                            prof_bytes(h, PH_HAS));
  CPMA_LAUNCHED(h);
  prof_end(h, st);
  return check_cuda(cudaGetLastError());
}

namespace {

Leaves leaves_of(const cpma* h) {
  return Leaves{h->data, h->used, h->cnt, h->heads, h->L, h->cfg.leaf_bytes};
}

// Blocks of a grid of one thread per query: small batches spread over more
// SMs in blocks of two warps.
int query_block(const cpma* h, uint64_t q) { return q < (uint64_t)h->num_sms * kT ? 64 : kT; }
int query_grid(const cpma* h, uint64_t q, int block, uint64_t per_sm) {
  return (int)std::max<uint64_t>(
      1, std::min<uint64_t>((q + block - 1) / block, (uint64_t)h->num_sms * per_sm));
}

// Per leaf a reduction and a count, per tile both again.
size_t leaf_prefix_bytes(uint64_t L) { return L * 12 + (L + kT - 1) / kT * 16 + 4; }

// Grows a query buffer.
int ensure_query(cpma* h, Buf& b, size_t bytes) {
  return with_query_room(h, [&] { return ensure(h, b, bytes); });
}

// The leaf prefix's memory for this call, or none (the inner leaves are then
// walked): one query covers no leaf twice, a set without room for it under its
// memory budget does without, and so does a stream that is being captured (a
// graph would keep the address, and the memory may move with the set's size).
// A set that has been updated holds it already: the redistribution's element
// buffer, which only an update uses, and none may overlap a query.  A budget
// below what the handle holds (cpma_set_mem_budget) gives it back.
//
// The rule of the kernels: the prefix is taken when the inner leaves of all
// queries number more than the set's leaves.  Both forms decode a leaf in the
// same time, so that is where the walk starts to cost more than one pass over
// the set.  Measured at 1e8 keys (0.9e6 leaves), 1e5 ranges of 10 to 1e6
// elements (8e7 inner leaves): 9.5 ms walked, 0.19 ms with the prefix.
void* prefix_memory(cpma* h, Buf& b, size_t need, cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return nullptr;
  }
  if (h->s.E.cap >= need) return h->s.E.p;
  // Memory that a query takes of its own accord is no other handle's or
  // allocator's to get back: at most half of what the device has free.
  if (b.cap < need && !h->cfg.alloc) {
    size_t free_bytes = 0, all = 0;
    if (cudaMemGetInfo(&free_bytes, &all) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    if (need > (free_bytes + b.cap) / 2) return nullptr;
  }
  return ensure(h, b, need) == CPMA_OK ? b.p : nullptr;
}

LeafPrefix leaf_prefix(cpma* h, uint64_t q, cudaStream_t st) {
  LeafPrefix p;
  if (q < 2) return p;
  p.val = (uint64_t*)prefix_memory(h, h->s.q_pre, leaf_prefix_bytes(h->L), st);
  if (!p.val) return p;
  const uint64_t nt = (h->L + kT - 1) / kT;
  p.tval = p.val + h->L;
  p.tcnt = p.tval + nt;
  p.cnt = (uint32_t*)(p.tcnt + nt);
  p.ticket = p.cnt + h->L;
  p.most = h->L;
  return p;
}

// The marks, for at least as many plain sums as leaves: below that marking
// every leaf costs more than it saves.  Marked / walked from the heads, us, at
// a query per two leaves, per leaf, two and four per leaf: uniform 40-bit keys
// (1.9e5 leaves, ranges of 32 elements) 73 / 66, 87 / 94, 106 / 160, 151 / 312;
// edges (1.4e5 leaves, adjacent ranges) 59 / 75, 63 / 118, 78 / 180, 101 / 281.
// On small sets a few queries are done before the leaves are marked: up to 478
// leaves of 512 bytes, 100 queries 31 / 23, 1000 31 / 26 short and 32 / 38 wide ones;
// 117 leaves of 2048 bytes 35 / 25 and 35 / 35 at 2500, 35 / 44 and 35 / 57 at 9700;
// 9.5e3 of them (edges) 98 / 56 and 101 / 83, at 1.4e4 98 / 74 and 100 / 101.
// The memory they take is that of the leaves again; without room for it the
// queries walk.
uint32_t marks_per_leaf(const cpma* h) {
  return (h->cfg.leaf_bytes + leafwalk::kMark - 1) / leafwalk::kMark;
}
bool marks_pay(const cpma* h, uint64_t q) {
  return q >= h->L && q > (uint64_t)h->num_sms * (large_leaves(h) ? 48 : 4);
}
size_t marks_bytes(const cpma* h) {
  return h->L * marks_per_leaf(h) * sizeof(leafwalk::Mark) + (h->L + kT - 1) / kT * 16;
}

Marks marks_of(cpma* h, uint64_t q, cudaStream_t st) {
  Marks m;
  if (!marks_pay(h, q)) return m;
  m.at = (leafwalk::Mark*)prefix_memory(h, h->s.q_marks, marks_bytes(h), st);
  m.per = marks_per_leaf(h);
  m.tiles.tval = (uint64_t*)(m.at + h->L * m.per);
  m.tiles.tcnt = m.tiles.tval + (h->L + kT - 1) / kT;
  return m;
}

int range_marked(cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q, const Marks& m,
                 uint64_t* sum, uint64_t* count, cudaStream_t st, ull* prof) {
  const Leaves t = leaves_of(h);
  const uint64_t nt = (t.L + kT - 1) / kT;
  const unsigned g = (unsigned)std::min<uint64_t>(nt, (uint64_t)persistent_grid(h));
  k_marks<<<g, kT, 0, st>>>(t, m, prof);
  CPMA_CUDA(cudaGetLastError());
  CPMA_CUDA(launch_pdl(k_tile_scan, 1, kT, 0, st, m.tiles, nt));
  const int b = query_block(h, q);
  CPMA_CUDA(launch_pdl(k_range_marked, (unsigned)query_grid(h, q, b, 8), (unsigned)b, 0, st, lo, hi,
                       q, t, m, sum, count, prof));
  h->launches += 2;
  CPMA_LAUNCHED(h);
  return check_cuda(cudaGetLastError());
}

// What a batch of range queries keeps between its kernels.
struct RangeScratch {
  uint64_t *first, *items, *off;   // q, q, q + 1 entries
  uint64_t* partials = nullptr;    // given partials of the offset scan (else the handle's)
  uint64_t partials_cap = 0;
  ull* done = nullptr;             // EndsScan::done (none with given scratch: it outlives a call)
};

int range_scratch(cpma* h, uint64_t q, RangeScratch* r) {
  Scratch& s = h->s;
  CPMA_TRY(ensure_query(h, s.q_first, q * 8));
  CPMA_TRY(ensure_query(h, s.q_items, (q + 1) * 8));
  CPMA_TRY(ensure_query(h, s.q_off, (q + 1) * 8));
  CPMA_TRY(ensure_query(h, s.partials_q, (size_t)(2 * h->num_sms + 2) * 8));
  r->first = (uint64_t*)s.q_first.p;
  r->items = (uint64_t*)s.q_items.p;
  r->off = (uint64_t*)s.q_off.p;
  r->done = &h->d_status->query_done;
  return CPMA_OK;
}

// Whether the ends' kernel leaves the offsets (scan_ends), and with what.  Not
// in the allocation-free call: it may overlap the handle's range calls, and
// carries nothing over from one call to the next.
EndsScan ends_scan(const cpma* h, const RangeScratch& r, uint64_t q) {
  EndsScan z;
  if (r.done && few_ranges(h, q) && few_scans(h, q) && q <= kEndsScan) {
    z.off = r.off;
    z.done = r.done;
  }
  return z;
}

int scan_items(cpma* h, const RangeScratch& r, uint64_t q, cudaStream_t st) {
  if (r.partials)
    return scan_u64_given_partials(h, r.items, r.off, q, r.partials, r.partials_cap, st);
  return scan_u64_query(h, r.items, r.off, q, st);
}

// After the ends: the inner leaves of every query, added to out and count.
template <int OP, bool PLAIN>
int range_inner(cpma* h, Reduce<OP, PLAIN> f, uint64_t q, uint64_t* out, uint64_t* count,
                const RangeScratch& r, const LeafPrefix& p, cudaStream_t st, ull* prof) {
  const Leaves t = leaves_of(h);
  if (!ends_scan(h, r, q).off) CPMA_TRY(scan_items(h, r, q, st));
  const uint64_t nt = (t.L + kT - 1) / kT;
  if (p.val) {
    const unsigned g = (unsigned)std::min<uint64_t>(nt, (uint64_t)persistent_grid(h));
    const uint64_t* total = r.off + q;
    const bool teams = large_leaves(h) && sum_by_teams(h);
    if (teams) {
      CPMA_CUDA(launch_pdl(k_leaf_reduce<OP, PLAIN>, (unsigned)query_grid(h, t.L * kTeam, kT, 8),
                           kT, 0, st, t, f, total, p, prof));
      h->launches++;
    }
    CPMA_CUDA(launch_pdl(teams ? k_leaf_prefix<OP, PLAIN, true> : k_leaf_prefix<OP, PLAIN, false>,
                         g, kT, 0, st, t, f, total, p, prof));
    h->launches++;
  }
  CPMA_CUDA(launch_pdl(large_leaves(h) ? k_range_inner<OP, PLAIN, kTeamLarge>
                                       : k_range_inner<OP, PLAIN, kTeam>,
                       (unsigned)persistent_grid(h), kT, 0, st, t, f, q, r.first, r.off, p, out,
                       count, prof));
  CPMA_LAUNCHED(h);
  return check_cuda(cudaGetLastError());
}

template <int OP, bool PLAIN>
int range_leaves(cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q, uint64_t mask,
                 uint64_t value, uint64_t* out, uint64_t* count, const RangeScratch& r,
                 const LeafPrefix& p, cudaStream_t st, ull* prof) {
  const Reduce<OP, PLAIN> f{mask, value};
  if (few_ranges(h, q)) {
    const auto kern = warp_teams(h, q) ? k_range_ends_team<OP, PLAIN, kTeamLarge>
                                      : k_range_ends_team<OP, PLAIN, kTeam>;
    kern<<<query_grid(h, q * (warp_teams(h, q) ? kTeamLarge : 2 * kTeam), 64, 32), 64, 0, st>>>(
        lo, hi, q, leaves_of(h), f, r.first, r.items, out, count, p.ticket, ends_scan(h, r, q),
        prof);
  } else {
    const int b = query_block(h, q);
    k_range_ends<OP, PLAIN><<<query_grid(h, q, b, 8), b, 0, st>>>(lo, hi, q, leaves_of(h), f,
                                                                  r.first, r.items, out, count,
                                                                  p.ticket, prof);
  }
  CPMA_LAUNCHED(h);
  CPMA_CUDA(cudaGetLastError());
  return range_inner<OP, PLAIN>(h, f, q, out, count, r, p, st, prof);
}

RangeArgs raw_args(const cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q,
                   const RangeScratch& r, uint64_t* out, uint64_t* count) {
  RangeArgs a;
  a.lo = lo;
  a.hi = hi;
  a.q = q;
  a.first = r.first;
  a.off = r.off;
  a.data = h->data;
  a.used = h->used;
  a.cnt = h->cnt;
  a.LB = h->cfg.leaf_bytes;
  a.sum = out;
  a.count = count;
  a.prof = nullptr;
  return a;
}

// Cells (codec 1): route, number the items, init the outputs.
int raw_prep(cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q, uint64_t* out,
             uint64_t* count, uint64_t init, const RangeScratch& r, cudaStream_t st) {
  k_range_prep<<<query_grid(h, q, kT, 8), kT, 0, st>>>(lo, hi, q, h->heads, h->L, r.first, r.items,
                                                       out, count, init);
  CPMA_LAUNCHED(h);
  CPMA_CUDA(cudaGetLastError());
  return scan_items(h, r, q, st);
}

}  // namespace

bool release_leaf_prefix(cpma* h) {
  if (!h->s.q_pre.p && !h->s.q_marks.p) return false;
  if (cudaDeviceSynchronize() != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  release(h, h->s.q_pre);
  release(h, h->s.q_marks);
  return true;
}

int reserve_leaf_prefix(cpma* h, uint64_t q) {
  const size_t need = leaf_prefix_bytes(h->L);
  if (h->s.E.cap < need) CPMA_TRY(ensure(h, h->s.q_pre, need));
  if (!marks_pay(h, q) || h->s.E.cap >= marks_bytes(h)) return CPMA_OK;
  return ensure(h, h->s.q_marks, marks_bytes(h));
}

int run_range(const cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q, uint64_t* sum,
              uint64_t* count, cudaStream_t st) {
  if (q == 0) return CPMA_OK;
  cpma* hm = const_cast<cpma*>(h);
  RangeScratch r;
  CPMA_TRY(range_scratch(hm, q, &r));
  int rc;
  if (!h->cfg.codec) {
    const Marks m = marks_of(hm, q, st);
    if (m.at) {
      prof_begin(h, PH_RANGE, st);
      rc = range_marked(hm, lo, hi, q, m, sum, count, st, prof_bytes(h, PH_RANGE));
      prof_end(h, st);
      return rc;
    }
  }
  if (h->cfg.codec) {
    prof_begin(h, PH_RANGE_PREP, st);
    prof_add_bytes(h, PH_RANGE_PREP, 72ull * q);  // lo, hi in; first, items, sums out; scan
    CPMA_TRY(raw_prep(hm, lo, hi, q, sum, count, 0, r, st));
    prof_end(h, st);
    RangeArgs a = raw_args(h, lo, hi, q, r, sum, count);
    a.prof = prof_bytes(h, PH_RANGE);
    prof_begin(h, PH_RANGE, st);
    k_range<false><<<persistent_grid(h), kT, 0, st>>>(a);
    CPMA_LAUNCHED(h);
    rc = check_cuda(cudaGetLastError());
  } else {
    const LeafPrefix p = leaf_prefix(hm, q, st);
    prof_begin(h, PH_RANGE, st);
    rc = range_leaves<CPMA_OP_SUM, true>(hm, lo, hi, q, 0, 0, sum, count, r, p, st,
                                         prof_bytes(h, PH_RANGE));
  }
  prof_end(h, st);
  return rc;
}

int run_range_length(const cpma* h, const uint64_t* start, const uint64_t* length, uint64_t q,
                     uint64_t* sum, uint64_t* count, cudaStream_t st) {
  if (q == 0) return CPMA_OK;
  cpma* hm = const_cast<cpma*>(h);
  Scratch& s = hm->s;
  RangeScratch r;
  CPMA_TRY(range_scratch(hm, q, &r));
  if (h->cfg.codec) {
    CPMA_TRY(ensure_query(hm, s.q_lo, q * 8));
    CPMA_TRY(ensure_query(hm, s.q_hi, q * 8));
  }
  CPMA_TRY(ensure_query(hm, s.q_rank, (h->L + 1) * 8));
  uint64_t* P = (uint64_t*)s.q_rank.p;
  prof_begin(h, PH_RANGE_PREP, st);
  prof_add_bytes(h, PH_RANGE_PREP, 12ull * h->L + 88ull * q);
  CPMA_TRY(scan_u32_query(hm, h->cnt, P, h->L, st));
  if (!h->cfg.codec) {
    prof_end(h, st);
    const LeafPrefix p = leaf_prefix(hm, q, st);
    ull* prof = prof_bytes(h, PH_RANGE);
    prof_begin(h, PH_RANGE, st);
    const bool few = few_scans(h, q);
    const int b = few ? 64 : query_block(h, q);
    const int g = few ? query_grid(h, q * (warp_teams(h, q) ? kTeamLarge : kTeam), b, 32) : query_grid(h, q, b, 8);
    if (few)
      CPMA_CUDA(launch_pdl(warp_teams(h, q) ? k_length_ends_team<kTeamLarge>
                                           : k_length_ends_team<kTeam>,
                           (unsigned)g, (unsigned)b, 0, st, start, length, q, leaves_of(h), P,
                           r.first, r.items, sum, count, p.ticket, ends_scan(h, r, q), prof));
    else
      CPMA_CUDA(launch_pdl(k_length_ends, (unsigned)g, (unsigned)b, 0, st, start, length, q,
                           leaves_of(h), P, r.first, r.items, sum, count, p.ticket, prof));
    CPMA_LAUNCHED(h);
    const int rc = range_inner<CPMA_OP_SUM, true>(hm, Reduce<CPMA_OP_SUM, true>{0, 0}, q, sum,
                                                  count, r, p, st, prof);
    prof_end(h, st);
    return rc;
  }
  uint64_t* r0 = (uint64_t*)s.q_lo.p;
  uint64_t* r1 = (uint64_t*)s.q_hi.p;
  k_rank_prep<false, true><<<query_grid(h, q * 32, kT, 16), kT, 0, st>>>(
      start, length, q, h->heads, h->data, h->used, h->L, h->cfg.leaf_bytes, P, r0, r1, r.first,
      r.items, sum, count);
  CPMA_LAUNCHED(h);
  CPMA_TRY(scan_items(hm, r, q, st));
  prof_end(h, st);
  RangeArgs a = raw_args(h, r0, r1, q, r, sum, count);
  a.prof = prof_bytes(h, PH_RANGE);
  a.P = P;
  prof_begin(h, PH_RANGE, st);
  k_range<true><<<persistent_grid(h), kT, 0, st>>>(a);
  CPMA_LAUNCHED(h);
  prof_end(h, st);
  return check_cuda(cudaGetLastError());
}

int run_range_extract(const cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q,
                      uint64_t* offsets, uint64_t* out, uint64_t cap, cudaStream_t st) {
  if (q == 0) return check_cuda(cudaMemsetAsync(offsets, 0, 8, st));
  cpma* hm = const_cast<cpma*>(h);
  Scratch& s = hm->s;
  RangeScratch r;
  CPMA_TRY(range_scratch(hm, q, &r));
  CPMA_TRY(ensure_query(hm, s.q_lo, q * 8));
  CPMA_TRY(ensure_query(hm, s.q_hi, q * 8));
  CPMA_TRY(ensure_query(hm, s.q_rank, (h->L + 1) * 8));
  uint64_t* P = (uint64_t*)s.q_rank.p;
  uint64_t* r0 = (uint64_t*)s.q_lo.p;
  uint64_t* r1 = (uint64_t*)s.q_hi.p;
  // where each query's first key lies in its leaf, when there is room
  leafwalk::Mark* start = nullptr;
  const bool warps = h->cfg.codec || extract_by_warps(h, q);
  if (!warps && out && cap)
    start = (leafwalk::Mark*)prefix_memory(hm, s.q_marks, q * sizeof(leafwalk::Mark), st);
  prof_begin(h, PH_RANGE_PREP, st);
  CPMA_TRY(scan_u32_query(hm, h->cnt, P, h->L, st));
  // the counts (r1 - r0) go to `offsets` first
  if (warps) {
    CPMA_CUDA(launch_pdl(h->cfg.codec ? k_rank_prep<true, true> : k_rank_prep<true, false>,
                         (unsigned)query_grid(h, q * 32, kT, 16), kT, 0, st, lo, hi, q, h->heads,
                         h->data, h->used, h->L, h->cfg.leaf_bytes, P, r0, r1, r.first, r.items,
                         nullptr, offsets));
  } else {
    CPMA_CUDA(launch_pdl(k_rank_ends, (unsigned)query_grid(h, 2 * q, kT, 8), kT, 0, st, lo, hi, q,
                         leaves_of(h), P, r0, r1, r.first, r.items, offsets, start));
  }
  CPMA_LAUNCHED(h);
  CPMA_TRY(scan_u64_query(hm, offsets, offsets, q, st));
  const bool emit = out && cap;
  if (emit) CPMA_TRY(scan_items(hm, r, q, st));
  prof_end(h, st);
  if (!emit) return check_cuda(cudaGetLastError());
  ExtractArgs a;
  a.start = start;
  a.r0 = r0;
  a.r1 = r1;
  a.q = q;
  a.first = r.first;
  a.item_off = r.off;
  a.out_off = offsets;
  a.P = P;
  a.data = h->data;
  a.used = h->used;
  a.LB = h->cfg.leaf_bytes;
  a.out = out;
  a.cap = cap;
  prof_begin(h, PH_RANGE, st);
  CPMA_CUDA(launch_pdl(h->cfg.codec ? k_extract<true> : warps ? k_extract<false> : k_extract_leaf,
                       (unsigned)persistent_grid(h), kT, 0, st, a));
  CPMA_LAUNCHED(h);
  prof_end(h, st);
  return check_cuda(cudaGetLastError());
}

int run_range_reduce(const cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q, int op,
                     uint64_t mask, uint64_t value, uint64_t* out, uint64_t* count,
                     cudaStream_t st) {
  if (op == CPMA_OP_SUM && mask == 0 && value == 0)
    return run_range(h, lo, hi, q, out, count, st);
  if (q == 0) return CPMA_OK;
  cpma* hm = const_cast<cpma*>(h);
  RangeScratch r;
  CPMA_TRY(range_scratch(hm, q, &r));
  if (!h->cfg.codec) {
    const LeafPrefix p = leaf_prefix(hm, q, st);
    prof_begin(h, PH_RANGE, st);
    int rc;
    switch (op) {
      case CPMA_OP_SUM:
        rc = range_leaves<CPMA_OP_SUM, false>(hm, lo, hi, q, mask, value, out, count, r, p, st,
                                              nullptr);
        break;
      case CPMA_OP_MIN:
        rc = range_leaves<CPMA_OP_MIN, false>(hm, lo, hi, q, mask, value, out, count, r, p, st,
                                              nullptr);
        break;
      case CPMA_OP_MAX:
        rc = range_leaves<CPMA_OP_MAX, false>(hm, lo, hi, q, mask, value, out, count, r, p, st,
                                              nullptr);
        break;
      case CPMA_OP_XOR:
        rc = range_leaves<CPMA_OP_XOR, false>(hm, lo, hi, q, mask, value, out, count, r, p, st,
                                              nullptr);
        break;
      default: rc = CPMA_EINVAL;
    }
    prof_end(h, st);
    return rc;
  }
  uint64_t init = 0;
  switch (op) {
    case CPMA_OP_SUM: init = op_identity<CPMA_OP_SUM>(); break;
    case CPMA_OP_MIN: init = op_identity<CPMA_OP_MIN>(); break;
    case CPMA_OP_MAX: init = op_identity<CPMA_OP_MAX>(); break;
    case CPMA_OP_XOR: init = op_identity<CPMA_OP_XOR>(); break;
    default: return CPMA_EINVAL;
  }
  prof_begin(h, PH_RANGE_PREP, st);
  CPMA_TRY(raw_prep(hm, lo, hi, q, out, count, init, r, st));
  prof_end(h, st);
  const RangeArgs a = raw_args(h, lo, hi, q, r, out, count);
  prof_begin(h, PH_RANGE, st);
  const int G = persistent_grid(h);
  switch (op) {
    case CPMA_OP_SUM: k_range_reduce<CPMA_OP_SUM><<<G, kT, 0, st>>>(a, mask, value); break;
    case CPMA_OP_MIN: k_range_reduce<CPMA_OP_MIN><<<G, kT, 0, st>>>(a, mask, value); break;
    case CPMA_OP_MAX: k_range_reduce<CPMA_OP_MAX><<<G, kT, 0, st>>>(a, mask, value); break;
    default: k_range_reduce<CPMA_OP_XOR><<<G, kT, 0, st>>>(a, mask, value); break;
  }
  CPMA_LAUNCHED(h);
  prof_end(h, st);
  return check_cuda(cudaGetLastError());
}

int run_range_noalloc(const cpma* h, const uint64_t* lo, const uint64_t* hi, uint64_t q,
                      uint64_t* sum, uint64_t* count, cudaStream_t st) {
  if (q > kNoAllocMaxQueries) return CPMA_EINVAL;
  if (q == 0) return CPMA_OK;
  int dev = -1;
  CPMA_CUDA(cudaGetDevice(&dev));
  if (dev != h->device) return CPMA_EINVAL;
  uint8_t* base = nullptr;
  CPMA_TRY(scratch_address(dev, &base));
  RangeScratch r;
  r.first = reinterpret_cast<uint64_t*>(base);
  r.items = r.first + kNoAllocMaxQueries;
  r.off = r.items + kNoAllocMaxQueries;                  // q + 1 entries
  r.partials = r.off + kNoAllocMaxQueries + 1;           // kNoAllocPartials entries
  r.partials_cap = kNoAllocPartials;
  // the offset scan needs at most 2 * SMs + 1 partials: checked before any
  // launch, so a rejected call leaves the outputs untouched
  if ((uint64_t)2 * h->num_sms + 1 > kNoAllocPartials) return CPMA_EINVAL;
  // every scratch entry read below is written first on this stream: nothing
  // carries over from an earlier call
  cpma* hm = const_cast<cpma*>(h);
  if (!h->cfg.codec)
    return range_leaves<CPMA_OP_SUM, true>(hm, lo, hi, q, 0, 0, sum, count, r, LeafPrefix(), st,
                                           nullptr);
  CPMA_TRY(raw_prep(hm, lo, hi, q, sum, count, 0, r, st));
  k_range<false><<<persistent_grid(h), kT, 0, st>>>(raw_args(h, lo, hi, q, r, sum, count));
  CPMA_LAUNCHED(h);
  return check_cuda(cudaGetLastError());
}

int run_sum(const cpma* h, uint64_t* sum, uint64_t* count, cudaStream_t st) {
  CPMA_CUDA(cudaMemsetAsync(sum, 0, 8, st));
  if (count) CPMA_CUDA(cudaMemsetAsync(count, 0, 8, st));
  prof_begin(h, PH_SUM, st);
  if (sum_by_teams(h))
    k_sum_team<<<query_grid(h, h->L * kTeam, kT, 8), kT, 0, st>>>(
        h->data, h->used, h->cnt, h->L, h->cfg.leaf_bytes, sum, count, prof_bytes(h, PH_SUM));
  else
    k_sum<<<persistent_grid(h), kT, 0, st>>>(h->data, h->used, h->cnt, h->heads, h->L,
                                           h->cfg.leaf_bytes, sum, count, prof_bytes(h, PH_SUM), (int)h->cfg.codec);
  CPMA_LAUNCHED(h);
  prof_end(h, st);
  return check_cuda(cudaGetLastError());
}

}  // namespace cpmaimpl
