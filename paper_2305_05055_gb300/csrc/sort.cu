// Batch sort (Sec. 4: "an unsorted batch can be converted into a sorted batch
// in O(k log k) work") as a radix sort over 8-bit digits.
//
// One digit pass is two kernels.  Every block owns an equal contiguous run of the
// keys, in tiles of at most 4096.  It counts its keys per digit (k_digit_count),
// for itself and, by atomics, for its group of 32 blocks; every block then adds up
// the groups and the blocks of its group before it, takes its tiles in order,
// ranks each in shared memory and writes every digit's run of the tile
// contiguously behind the ones before it (k_digit_scatter).  No block waits for
// another.  (Reading the keys once and joining the tiles by decoupled look-back
// instead was slower on large batches: several hundred tiles start together, so
// each had to add up most of its predecessors' counts, 8 per round trip to the L2:
// 343 us a pass over 3e7 keys, against 42 + 182 us.)  A stable rank takes eight
// ballots per key and warp (115 instructions per 32 keys bound the scatter); where
// order among equal digits does not matter it is one atomic.
//
// Keys alone go most significant bits first, so that few passes cross memory:
// - up to 4096 keys: one block, a sorting network;
// - up to 1.25M: the OR and AND of the keys give the 8 highest bits that vary,
//   one pass by those moves the keys to 256 buckets, a block finishes each
//   (k_bucket_sort);
// - above, when more than 24 bits vary: two passes by the 16 highest of them,
//   then each block finishes the buckets that start in its 4096 keys
//   (k_window_sort), at most 6144 keys.  A bucket of more than 2048 keys (heavy
//   repeats or skew) does not fit that.  One key in 128 is counted by its bucket
//   first (k_sample): when that shows such a bucket, the passes over all varying
//   digits, lowest first, run instead, and otherwise after all if a window meets
//   one.  3e7 40-bit keys: 710 us, 1650 us for the five look-back passes; 4e6
//   R-MAT edges (six varying digits): 285, 320 and, by windows first, 540 us.
// A block finishes up to 6144 keys in shared memory in one counting pass: bins
// by the highest bits in which the keys differ, about as many as keys, one
// atomic per key, then every key's rank among the few keys of its bin.  Bins
// over kBinMost keys (repeats, clusters) send the block to digit passes in
// shared memory instead.  1e6 keys in 256 buckets: 9 us against 30 us for four
// digit passes.
//
// Keys with tags (which must move stably) take the digit passes: buckets up
// to 1.25M, all varying digits from the lowest up above.
#include <algorithm>
#include <cmath>

#include "dev_common.cuh"
#include "internal.h"

using namespace cpmadev;

namespace cpmaimpl {
namespace {

constexpr int kT = 256;
constexpr int kWarps = kT / 32;
constexpr int kItems = 16;
constexpr int kTile = kT * kItems;  // 4096 keys
// Bucket sort: one block of kBT threads, kBItems keys each, sorts a bucket of
// up to kBTile keys (spread evenly over its warps).
constexpr int kBT = 512;
constexpr int kBItems = 12;
constexpr int kBTile = kBT * kBItems;  // 6144 keys
// Batches of more than one tile and at most this many keys take the
// top-digit buckets (k / 256 keys per bucket on average, far below kBTile).
constexpr uint64_t kBucketMax = 1280ull * 1024;
// Larger batches of keys alone, and at most this many (1700 per bucket of the 16
// highest bits on average, eight standard deviations below the 2048 that fit),
// go by those bits and in windows.
constexpr uint64_t kMsdMax = 1700ull << 16;

template <bool VALS, int KT = kT, int ITEMS = kItems>
struct TileSmemT {
  uint64_t keys[KT * ITEMS];
  uint32_t vals[VALS ? KT * ITEMS : 1];  // optional 32-bit payload moved with the keys
  uint32_t wcnt[KT / 32][256];
  uint32_t dstart[256];
  uint32_t scan_tmp[8];
};

// Stable partition of the tile by digit (key >> shift) & 255.  Item j of lane
// l in warp w (j < ipw <= ITEMS) is tile element w*32*ipw + j*32 + l; the first `nvalid`
// elements are real.  On return sm.keys[0..nvalid) holds the tile sorted by
// digit (stable) and sm.dstart[d] is where digit d starts.
template <bool VALS, int KT = kT, int ITEMS = kItems>
__device__ __forceinline__ void tile_rank(const uint64_t (&key)[ITEMS], const uint32_t (&val)[ITEMS],
                                          uint32_t nvalid, int shift, TileSmemT<VALS, KT, ITEMS>& sm,
                                          uint32_t ipw = ITEMS) {
  constexpr int W = KT / 32;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < W * 256; i += KT) (&sm.wcnt[0][0])[i] = 0;
  __syncthreads();
  uint32_t rank[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; j++) {
    if ((uint32_t)j >= ipw) break;
    const uint32_t li = warp * 32 * ipw + j * 32 + lane;
    const bool valid = li < nvalid;
    const uint32_t d = (uint32_t)(key[j] >> shift) & 255u;
    const unsigned vm = __ballot_sync(FULL, valid);
    // lanes holding the same digit: one ballot per digit bit
    unsigned peers = vm, before = 0;
#pragma unroll
    for (int b = 0; b < 8; b++) {
      const bool bit = (d >> b) & 1u;
      const unsigned bb = __ballot_sync(FULL, bit);
      peers &= bit ? bb : ~bb;
    }
    if (valid) {
      before = __popc(peers & lanemask_lt());
      rank[j] = sm.wcnt[warp][d] + before;
    }
    __syncwarp();
    if (valid && before == 0) sm.wcnt[warp][d] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // per digit (threads 0..255): exclusive prefix over warps, then over digits
  {
    const int d = threadIdx.x;
    uint32_t run = 0, inc = 0;
    if (d < 256) {
#pragma unroll
      for (int w = 0; w < W; w++) {
        uint32_t c = sm.wcnt[w][d];
        sm.wcnt[w][d] = run;
        run += c;
      }
      inc = warp_incl_scan(run);
      if (lane == 31) sm.scan_tmp[warp] = inc;
    }
    __syncthreads();
    if (warp == 0) {
      uint32_t v = lane < 8 ? sm.scan_tmp[lane] : 0;
      uint32_t vi = warp_incl_scan(v);
      if (lane < 8) sm.scan_tmp[lane] = vi - v;
    }
    __syncthreads();
    if (d < 256) sm.dstart[d] = sm.scan_tmp[warp] + inc - run;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < ITEMS; j++) {
    if ((uint32_t)j >= ipw) break;
    const uint32_t li = warp * 32 * ipw + j * 32 + lane;
    if (li < nvalid) {
      const uint32_t d = (uint32_t)(key[j] >> shift) & 255u;
      const uint32_t pos = sm.dstart[d] + sm.wcnt[warp][d] + rank[j];
      sm.keys[pos] = key[j];
      if constexpr (VALS) sm.vals[pos] = val[j];
    }
  }
  __syncthreads();
}

// ---- up to kBTile keys in one block, by bins ----
constexpr uint32_t kBins = 4096;
constexpr uint32_t kBinMost = 128;  // keys of a bin ranked against each other (at most 255)
struct BinSmem {
  uint64_t keys[kBTile];
  __align__(16) uint32_t bin[kBins + 4];
  uint32_t ws[kBT / 32];
};

// Writes the n <= kBTile keys held by the block (item j of thread t; ok: which
// exist), all in [lo, lo + 2^bits), to dst in order.  false (nothing written,
// for every thread): some bin holds more than kBinMost keys.
__device__ __forceinline__ bool bin_sort(const uint64_t (&key)[kBItems], uint32_t ok, uint32_t n,
                                         uint64_t lo, uint32_t bits, BinSmem& sm,
                                         uint64_t* __restrict__ dst) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  // as many bins as keys: a power of two, 4 or 8 per thread
  const uint32_t lb = n > 2048u ? 12u : 11u, nb = 1u << lb;
  static_assert(kBT * 8 == kBins, "8 bins per thread");
  const uint32_t sh = bits > lb ? bits - lb : 0u;
  uint4* bin4 = reinterpret_cast<uint4*>(sm.bin);
  for (uint32_t i = threadIdx.x; i < nb / 4; i += kBT) bin4[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  uint32_t r[kBItems / 4] = {0u};  // places in the bins, a byte each
  bool deep = false;
#pragma unroll
  for (int j = 0; j < kBItems; j++)
    if ((ok >> j) & 1u) {
      const uint32_t at = atomicAdd(&sm.bin[(uint32_t)((key[j] - lo) >> sh)], 1u);
      deep |= at >= kBinMost;
      r[j / 4] |= at << (8 * (j % 4));
    }
  if (__syncthreads_or(deep)) return false;
  // exclusive prefix over the bins, 4 or 8 consecutive ones per thread
  const bool two = lb == 12u;
  const uint32_t i0 = threadIdx.x * (two ? 2u : 1u);
  const uint4 u = bin4[i0], v = two ? bin4[i0 + 1] : make_uint4(0u, 0u, 0u, 0u);
  const uint32_t sum = u.x + u.y + u.z + u.w + v.x + v.y + v.z + v.w;
  const uint32_t inc = warp_incl_scan(sum);
  if (lane == 31) sm.ws[warp] = inc;
  __syncthreads();
  uint32_t run = inc - sum;
  {
    const uint32_t w = lane < warp ? sm.ws[lane] : 0u;  // warp < 16
    run += __reduce_add_sync(FULL, w);
  }
  const uint4 p = make_uint4(run, run + u.x, run + u.x + u.y, run + u.x + u.y + u.z);
  bin4[i0] = p;
  if (two) {
    const uint32_t q = p.w + u.w;
    bin4[i0 + 1] = make_uint4(q, q + v.x, q + v.x + v.y, q + v.x + v.y + v.z);
  }
  if (threadIdx.x == 0) sm.bin[nb] = n;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kBItems; j++)
    if ((ok >> j) & 1u)
      sm.keys[sm.bin[(uint32_t)((key[j] - lo) >> sh)] + ((r[j / 4] >> (8 * (j % 4))) & 0xFFu)] =
          key[j];
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n; i += kBT) {
    const uint64_t x = sm.keys[i];
    const uint32_t b = (uint32_t)((x - lo) >> sh);
    const uint32_t q0 = sm.bin[b], q1 = sm.bin[b + 1];
    uint32_t at = q0;
    for (uint32_t q = q0; q < q1; q++) {
      const uint64_t y = sm.keys[q];
      at += (y < x || (y == x && q < i)) ? 1u : 0u;
    }
    dst[at] = x;
  }
  return true;
}

// Control block of one sort, zeroed before the first kernel.
struct SortCtl {
  uint32_t tot[256];       // keys per digit of the current pass
  uint32_t varying[8];     // digit p varies across the batch
  uint32_t rank[8];        // position of digit p among the varying ones
  uint32_t npass;          // number of varying digits
  uint32_t fshift;         // the field: bits [fshift, fshift + 8), the highest that vary
  uint32_t done;           // OR/AND blocks finished
  uint32_t msd;            // large batch: top 16 varying bits, then windows
  uint32_t rest;           // the passes over all digits are needed: few bits vary, or a
                           // bucket is too large for a window
  uint32_t pad;
  ull or_all, nand_all;    // OR of the keys and of their complements
};

// The thread's OR of its keys and of their complements over the batch; the
// last of the grid's blocks turns the bits that vary into the bucket field
// (the 8 highest of them), the varying digits and their number (0 when every
// key is equal); `digits`: by the digit passes whatever varies (tags).  A whole
// block must call.
__device__ __forceinline__ void vary_of(ull o, ull na, SortCtl* ctl, bool digits) {
  __shared__ ull s_or[kWarps], s_na[kWarps];
  const uint32_t olo = __reduce_or_sync(FULL, (uint32_t)o), ohi = __reduce_or_sync(FULL, (uint32_t)(o >> 32));
  const uint32_t alo = __reduce_or_sync(FULL, (uint32_t)na), ahi = __reduce_or_sync(FULL, (uint32_t)(na >> 32));
  if (lane_id() == 0) {
    s_or[threadIdx.x >> 5] = ((ull)ohi << 32) | olo;
    s_na[threadIdx.x >> 5] = ((ull)ahi << 32) | alo;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ull bo = 0, ba = 0;
    for (int w = 0; w < kWarps; w++) { bo |= s_or[w]; ba |= s_na[w]; }
    atomicOr(&ctl->or_all, bo);
    atomicOr(&ctl->nand_all, ba);
    __threadfence();
    if (atomicAdd(&ctl->done, 1u) == gridDim.x - 1) {
      __threadfence();
      const ull vary = *((volatile ull*)&ctl->or_all) & *((volatile ull*)&ctl->nand_all);
      const uint32_t hb = vary ? 64u - (uint32_t)__clzll((long long)vary) : 0u;
      ctl->fshift = hb > 8u ? hb - 8u : 0u;
      uint32_t r = 0;
      for (int p = 0; p < 8; p++) {
        const uint32_t v = ((vary >> (8 * p)) & 255u) != 0u;
        ctl->varying[p] = v;
        ctl->rank[p] = r;
        r += v;
      }
      ctl->npass = r;
      const bool msd = hb > 24u && !digits;
      ctl->msd = msd ? 1u : 0u;
      ctl->rest = msd ? 0u : 1u;
    }
  }
}

// First kernel: the bits that vary; nz words at z to zero (the passes' group
// counts, the sample's buckets).
__global__ void __launch_bounds__(kT) k_orand(const uint64_t* __restrict__ in, uint64_t k,
                                              SortCtl* ctl, bool digits, uint32_t* z, uint32_t nz) {
  pdl_wait();
  pdl_launch();
  for (uint32_t i = blockIdx.x * kT + threadIdx.x; i < nz; i += gridDim.x * kT) z[i] = 0;
  ull o = 0, na = 0;
  // eight keys per thread and step, loaded together
  const uint64_t stride = (uint64_t)gridDim.x * kT;
  uint64_t i = (uint64_t)blockIdx.x * kT + threadIdx.x;
  for (; i + 7 * stride < k; i += 8 * stride) {
    uint64_t x[8];
#pragma unroll
    for (int j = 0; j < 8; j++) x[j] = in[i + j * stride];
#pragma unroll
    for (int j = 0; j < 8; j++) { o |= x[j]; na |= ~x[j]; }
  }
  for (; i < k; i += stride) {
    const uint64_t x = in[i];
    o |= x;
    na |= ~x;
  }
  vary_of(o, na, ctl, digits);
}

// Large batches: one key in kSampleEvery, at a scattered place of each run of as
// many, counted by the 16 highest bits that vary.  `most` keys in one bucket: the
// batch takes the digit passes.
constexpr uint32_t kSampleEvery = 128, kSampleBins = 1u << 16;
__global__ void __launch_bounds__(kT) k_sample(const uint64_t* __restrict__ in, uint64_t k,
                                               SortCtl* ctl, uint32_t* bins, uint32_t most) {
  pdl_wait();
  pdl_launch();
  if (!ctl->msd) return;
  const int sh = (int)ctl->fshift - 8;
  const uint64_t n = k / kSampleEvery;
  const unsigned lane = lane_id();
  // whole warps stay in the loop
  for (uint64_t j0 = ((uint64_t)blockIdx.x * kT + threadIdx.x) & ~31ull; j0 < n;
       j0 += (uint64_t)gridDim.x * kT) {
    if (__any_sync(FULL, *((volatile uint32_t*)&ctl->rest) != 0)) return;  // decided
    const uint64_t j = j0 + lane;
    const uint32_t at = ((uint32_t)j * 0x9E3779B1u) >> 25;  // in [0, kSampleEvery)
    const bool ok = j < n;
    const uint32_t b = ok ? (uint32_t)(in[j * kSampleEvery + at] >> sh) & (kSampleBins - 1) : ~0u;
    const unsigned same = __match_any_sync(FULL, b);
    if (ok && lane == (unsigned)__ffs(same) - 1u) {
      const uint32_t c = __popc(same);
      if (atomicAdd(&bins[b], c) + c >= most) ctl->rest = 1;
    }
  }
}

// What a digit pass reads and writes.  p >= 0: digit p of the passes from the
// lowest up, which take the input, then A and B alternately, arranged so that
// the last varying one writes A (not run when the top bits and the windows
// did the sort).  kField: the input to B by the field.  kTop0, kTop1: the
// input to A by the 8 bits below the field, A to B by the field.
constexpr int kField = -1, kTop0 = -2, kTop1 = -3;
struct Pass {
  const uint64_t* in;
  const uint32_t* vin;
  uint64_t *A, *B;
  uint32_t *VA, *VB;
  uint64_t k;
  int p;
  SortCtl* ctl;
  uint32_t* grp;  // this pass's counts of digit d in blocks 32 g .. 32 g + 31, at 256 g + d
  uint32_t* cnt;  // the blocks' counts, of digit d and block b at 256 b + d
};
constexpr uint32_t kGroup = 32;
struct PassIo {
  const uint64_t* src;
  const uint32_t* vsrc;
  uint64_t* dst;
  uint32_t* vdst;
  int shift;
};
// false: nothing to do
__device__ __forceinline__ bool pass_io(const Pass& a, PassIo& io) {
  const SortCtl& c = *a.ctl;
  if (a.p == kField) {
    io = PassIo{a.in, a.vin, a.B, a.VB, (int)c.fshift};
    return c.npass != 0;
  }
  if (a.p == kTop0) {
    io = PassIo{a.in, a.vin, a.A, a.VA, (int)c.fshift - 8};
    return !c.rest;
  }
  if (a.p == kTop1) {
    io = PassIo{a.A, a.VA, a.B, a.VB, (int)c.fshift};
    return !c.rest;
  }
  if (!c.varying[a.p] || !c.rest) return false;
  const uint32_t left = c.npass - c.rank[a.p];  // passes from this one on
  io.src = left == c.npass ? a.in : (left & 1u) ? a.B : a.A;
  io.vsrc = left == c.npass ? a.vin : (left & 1u) ? a.VB : a.VA;
  io.dst = (left & 1u) ? a.A : a.B;
  io.vdst = (left & 1u) ? a.VA : a.VB;
  io.shift = 8 * a.p;
  return true;
}

// The block's keys [e0, e1), in tiles of at most 256 * ipw.  From kWholeTiles
// tiles a block on, blocks own whole tiles; below, where one tile more or less
// counts, equal shares (from a multiple of 32 keys on) in equal tiles: keys with
// tags 4e6 363 and 287 us, 4e7 the other way round by some 2 %.
constexpr uint64_t kWholeTiles = 8;
struct Share {
  uint64_t e0, e1;
  uint32_t ipw;
};
__device__ __forceinline__ Share share_of(uint64_t k) {
  Share s;
  const uint64_t b = blockIdx.x, G = gridDim.x, nt = (k + kTile - 1) / kTile;
  if (nt >= kWholeTiles * G) {
    s.e0 = nt * b / G * kTile;
    s.e1 = min(k, nt * (b + 1) / G * kTile);
    s.ipw = kItems;
    return s;
  }
  s.e0 = k * b / G & ~31ull;
  s.e1 = b + 1 == G ? k : k * (b + 1) / G & ~31ull;
  const uint64_t n = s.e1 - s.e0, step = (uint64_t)kT * ((n + kTile - 1) / kTile);
  s.ipw = step ? (uint32_t)((n + step - 1) / step) : 0u;
  return s;
}

// Keys per digit of the block, and of its group.
// (three blocks per SM run: with the 32 registers it would take, half of the eight
// loads wait for the others, 1e8 keys 128 us instead of 116)
__global__ void __launch_bounds__(kT, 3) k_digit_count(Pass a) {
  constexpr int kCopies = 4;  // histograms per block: fewer lanes on one counter
  __shared__ uint32_t hs[kCopies][256];
  pdl_wait();
  pdl_launch();
  PassIo io;
  if (!pass_io(a, io)) return;
  for (int i = threadIdx.x; i < kCopies * 256; i += kT) (&hs[0][0])[i] = 0;
  __syncthreads();
  uint32_t* h = hs[(threadIdx.x >> 5) & (kCopies - 1)];
  const Share sh = share_of(a.k);
  uint64_t i = sh.e0 + threadIdx.x;
  for (; i + 7 * kT < sh.e1; i += 8 * kT) {
    uint64_t x[8];
#pragma unroll
    for (int j = 0; j < 8; j++) x[j] = io.src[i + j * kT];
#pragma unroll
    for (int j = 0; j < 8; j++) atomicAdd(&h[(uint32_t)(x[j] >> io.shift) & 255u], 1u);
  }
  for (; i < sh.e1; i += kT) atomicAdd(&h[(uint32_t)(io.src[i] >> io.shift) & 255u], 1u);
  __syncthreads();
  static_assert(kT == 256, "a thread per digit");
  uint32_t n = 0;
#pragma unroll
  for (int q = 0; q < kCopies; q++) n += hs[q][threadIdx.x];
  a.cnt[(size_t)blockIdx.x * 256 + threadIdx.x] = n;
  if (n) atomicAdd(&a.grp[(blockIdx.x / kGroup) * 256 + threadIdx.x], n);
}

// Digit d's keys in all blocks, and in the blocks before this one.
__device__ __forceinline__ void digit_before(const Pass& a, uint32_t d, uint32_t& all,
                                             uint32_t& before) {
  const uint32_t ng = (gridDim.x + kGroup - 1) / kGroup, g0 = blockIdx.x / kGroup;
  all = before = 0;
#pragma unroll 8
  for (uint32_t g = 0; g < ng; g++) {
    const uint32_t v = a.grp[g * 256 + d];
    all += v;
    before += g < g0 ? v : 0u;
  }
#pragma unroll 8
  for (uint32_t b = g0 * kGroup; b < blockIdx.x; b++) before += a.cnt[(size_t)b * 256 + d];
}

// Partition of the tile by digit with no order among equal digits (keys
// alone): one atomic per key.
__device__ __forceinline__ void tile_rank_any(const uint64_t (&key)[kItems], uint32_t nvalid,
                                              int shift, TileSmemT<false>& sm) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  uint32_t* cnt = sm.wcnt[0];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  uint32_t rank[kItems];
#pragma unroll
  for (int j = 0; j < kItems; j++)
    if (warp * 32 * kItems + j * 32 + lane < nvalid)
      rank[j] = atomicAdd(&cnt[(uint32_t)(key[j] >> shift) & 255u], 1u);
  __syncthreads();
  const uint32_t c = cnt[threadIdx.x], inc = warp_incl_scan(c);
  if (lane == 31) sm.scan_tmp[warp] = inc;
  __syncthreads();
  uint32_t before = inc - c;
  for (unsigned w = 0; w < warp; w++) before += sm.scan_tmp[w];
  sm.dstart[threadIdx.x] = before;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kItems; j++)
    if (warp * 32 * kItems + j * 32 + lane < nvalid)
      sm.keys[sm.dstart[(uint32_t)(key[j] >> shift) & 255u] + rank[j]] = key[j];
  __syncthreads();
}

// The block's tiles in order, each ranked in shared memory and written behind
// the block's earlier keys of every digit.  WHOLE: its tiles are whole ones (with
// the items per thread known, 3e7 keys 182 us, else 195).
template <bool VALS, bool STABLE, bool WHOLE>
__global__ void __launch_bounds__(kT, 3) k_digit_scatter(Pass a) {
  static_assert(STABLE || !VALS, "tags move stably");
  extern __shared__ __align__(16) uint8_t smem_raw[];
  TileSmemT<VALS>& sm = *reinterpret_cast<TileSmemT<VALS>*>(smem_raw);
  __shared__ uint32_t s_off[256];  // where the tile's keys of a digit go, less their tile index
  __shared__ uint32_t s_ws[kWarps];
  pdl_wait();
  pdl_launch();
  PassIo io;
  if (!pass_io(a, io)) return;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const uint32_t d = threadIdx.x;
  // digit d's next position: the keys of lower digits, then those of d in
  // earlier blocks
  uint32_t t, before;
  digit_before(a, d, t, before);
  if (blockIdx.x == 0) a.ctl->tot[d] = t;
  const uint32_t inc = warp_incl_scan(t);
  if (lane == 31) s_ws[warp] = inc;
  __syncthreads();
  uint32_t run = before + inc - t;
  for (unsigned w = 0; w < warp; w++) run += s_ws[w];
  // Equal tiles where the ranks are what a tile costs (a last tile of few keys
  // would cost the block as many steps as a full one has); whole ones and a rest
  // where it is one atomic per key.
  const Share sh = share_of(a.k);
  const uint32_t ipw = STABLE && !WHOLE ? sh.ipw : (uint32_t)kItems;
  io.src += sh.e0;
  if constexpr (VALS) io.vsrc += sh.e0;
  const uint32_t n = (uint32_t)(sh.e1 - sh.e0);
  for (uint32_t base = 0; base < n; base += kT * ipw) {
    const uint32_t nvalid = min(kT * ipw, n - base);
    uint64_t key[kItems];
    uint32_t val[kItems];
#pragma unroll
    for (int j = 0; j < kItems; j++) {
      const uint32_t li = warp * 32 * ipw + j * 32 + lane;
      const bool in = (uint32_t)j < ipw && li < nvalid;
      key[j] = in ? io.src[base + li] : 0ull;
      if constexpr (VALS) val[j] = in ? io.vsrc[base + li] : 0u;
      else val[j] = 0u;
    }
    if constexpr (STABLE) tile_rank<VALS>(key, val, nvalid, io.shift, sm, ipw);
    else tile_rank_any(key, nvalid, io.shift, sm);
    s_off[d] = run - sm.dstart[d];
    run += (d < 255 ? sm.dstart[d + 1] : nvalid) - sm.dstart[d];
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nvalid; i += kT) {
      const uint64_t x = sm.keys[i];
      const uint32_t o = s_off[(uint32_t)(x >> io.shift) & 255u] + i;
      io.dst[o] = x;
      if constexpr (VALS) io.vdst[o] = sm.vals[i];
    }
    __syncthreads();  // the next tile reuses the shared arrays
  }
}

// Every key equal: no pass runs, the batch is copied to the result buffer.
__global__ void k_copy_if_no_pass(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                  const uint32_t* __restrict__ vin, uint32_t* __restrict__ vout,
                                  uint64_t k, const SortCtl* ctl) {
  pdl_wait();
  pdl_launch();
  if (ctl->npass != 0) return;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k;
       i += (uint64_t)gridDim.x * blockDim.x) {
    out[i] = in[i];
    if (vin) vout[i] = vin[i];
  }
}

// The shared memory of a block that finishes a bucket or a window.
template <bool VALS>
union FinishSmem {
  TileSmemT<VALS, kBT, kBItems> tile;
  BinSmem bins;
};

// The n <= kBTile keys at src (with their tags), all in [lo, lo + 2^bits),
// sorted into dst: by bins when there are no tags and no bin is deep, else
// stably digit by digit over the digits that vary among them.
template <bool VALS>
__device__ __forceinline__ void block_sort(const uint64_t* __restrict__ src,
                                           const uint32_t* __restrict__ vsrc,
                                           uint64_t* __restrict__ dst, uint32_t* __restrict__ vdst,
                                           uint32_t n, uint64_t lo, uint32_t bits,
                                           FinishSmem<VALS>& sm) {
  __shared__ ull s_or, s_and;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  // items per warp: the keys spread over every warp, in element order
  const uint32_t ipw = (n + 32u * (kBT / 32) - 1u) / (32u * (kBT / 32));
  uint64_t key[kBItems];
  uint32_t val[kBItems];
  uint32_t ok = 0;
  if (threadIdx.x == 0) { s_or = 0; s_and = ~0ull; }
#pragma unroll
  for (int j = 0; j < kBItems; j++) {
    const uint32_t li = warp * 32 * ipw + j * 32 + lane;
    const bool in = (uint32_t)j < ipw && li < n;
    key[j] = in ? src[li] : 0ull;
    if constexpr (VALS) val[j] = in ? vsrc[li] : 0u;
    else val[j] = 0u;
    ok |= (uint32_t)in << j;
  }
  if constexpr (!VALS)
    if (bin_sort(key, ok, n, lo, bits, sm.bins, dst)) return;
  ull o = 0, a = ~0ull;
#pragma unroll
  for (int j = 0; j < kBItems; j++)
    if ((ok >> j) & 1u) { o |= key[j]; a &= key[j]; }
  __syncthreads();
  atomicOr(&s_or, o);
  atomicAnd(&s_and, a);
  __syncthreads();
  const ull vary = s_or ^ s_and;
  for (uint32_t p = 0; p < 8; p++) {
    if (((vary >> (8 * p)) & 255u) == 0) continue;
    tile_rank<VALS, kBT, kBItems>(key, val, n, 8 * (int)p, sm.tile, ipw);
#pragma unroll
    for (int j = 0; j < kBItems; j++) {
      const uint32_t li = warp * 32 * ipw + j * 32 + lane;
      if ((ok >> j) & 1u) {
        key[j] = sm.tile.keys[li];
        if constexpr (VALS) val[j] = sm.tile.vals[li];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < kBItems; j++) {
    const uint32_t li = warp * 32 * ipw + j * 32 + lane;
    if ((ok >> j) & 1u) {
      dst[li] = key[j];
      if constexpr (VALS) vdst[li] = val[j];
    }
  }
}

// Large batches: B is in order by the top 16 varying bits; block t puts the
// buckets that start among keys [4096 t, 4096 (t + 1)) into A in full order.
constexpr uint32_t kWindowMore = kBTile - kTile;  // keys a bucket may reach past its tile
__global__ void __launch_bounds__(kBT, 2) k_window_sort(const uint64_t* __restrict__ B,
                                                        uint64_t* __restrict__ A, uint64_t k,
                                                        SortCtl* ctl) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  FinishSmem<false>& sm = *reinterpret_cast<FinishSmem<false>*>(smem_raw);
  __shared__ uint32_t s_at[2], s_rest;
  pdl_wait();
  pdl_launch();
  const int sh = (int)ctl->fshift - 8;
  // (other blocks may raise the flag meanwhile: one thread reads it)
  if (threadIdx.x == 0) s_rest = *((volatile uint32_t*)&ctl->rest);
  if (threadIdx.x < 2) s_at[threadIdx.x] = 0xFFFFFFFFu;
  __syncthreads();
  if (s_rest) return;
  // the first bucket start at or after either end of the tile, each searched
  // by half of the block
  const uint64_t t0 = (uint64_t)blockIdx.x * kTile;
  const uint32_t end = threadIdx.x / (kBT / 2), ht = threadIdx.x % (kBT / 2);
  const uint64_t from = t0 + (uint64_t)end * kTile;
  bool found = false;  // by this half
  for (uint32_t i0 = 0; i0 <= kWindowMore; i0 += kBT / 2) {
    const uint64_t i = from + i0 + ht;
    if (!found && (i == 0 || i >= k || (B[i - 1] >> sh) != (B[i] >> sh)))
      atomicMin(&s_at[end], i0 + ht);
    __syncthreads();
    found = s_at[end] != 0xFFFFFFFFu;
    if (__syncthreads_and(found)) break;
  }
  if (s_at[0] > kWindowMore || s_at[1] > kWindowMore) {
    if (threadIdx.x == 0) ctl->rest = 1;
    return;
  }
  const uint64_t b = min(k, t0 + s_at[0]), e = min(k, t0 + kTile + s_at[1]);
  if (e <= b) return;
  const uint64_t lo = B[b] >> sh, hi = B[e - 1] >> sh;  // first and last bucket
  const uint32_t bits = (uint32_t)sh + 64u - (uint32_t)__clzll((long long)(hi - lo));
  block_sort<false>(B + b, nullptr, A + b, nullptr, (uint32_t)(e - b), lo << sh, bits, sm);
}

// Bucket b of the field scatter (B[off .. off + n)), sorted (stably when there
// are tags) into the same positions of A: in shared memory when it holds at
// most kBTile keys, else (heavy repeats or skew) by a
// block-level LSD radix sort through global memory: per varying digit, one
// counting pass over the bucket, then its tiles in order, each ranked stably
// in shared memory and scattered to the running digit offsets, alternating
// between B and A (and copied to A if it ends in B).
template <bool VALS>
__global__ void __launch_bounds__(kBT, 2) k_bucket_sort(uint64_t* __restrict__ B,
                                                     uint32_t* __restrict__ VB,
                                                     uint64_t* __restrict__ A,
                                                     uint32_t* __restrict__ VA, SortCtl* ctl,
                                                     const uint64_t* __restrict__ in,
                                                     const uint32_t* __restrict__ vin,
                                                     uint64_t k) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  FinishSmem<VALS>& fsm = *reinterpret_cast<FinishSmem<VALS>*>(smem_raw);
  TileSmemT<VALS, kBT, kBItems>& sm = fsm.tile;
  __shared__ ull s_or, s_and;
  __shared__ uint32_t s_run[256];
  __shared__ uint32_t s_wt[8];
  pdl_wait();
  pdl_launch();
  if (ctl->npass == 0) {
    // every key equal: the batch as given is the result
    for (uint64_t i = (uint64_t)blockIdx.x * kBT + threadIdx.x; i < k;
         i += (uint64_t)gridDim.x * kBT) {
      A[i] = in[i];
      if constexpr (VALS) VA[i] = vin[i];
    }
    return;
  }
  const uint32_t b = blockIdx.x;
  const uint32_t n = ctl->tot[b];
  if (n == 0) return;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  // where the bucket starts: the keys of the buckets before it
  if (threadIdx.x < 256) {
    const uint32_t before = warp_sum(threadIdx.x < b ? ctl->tot[threadIdx.x] : 0u);
    if (lane == 0) s_wt[warp] = before;
  }
  __syncthreads();
  uint64_t base = 0;
#pragma unroll
  for (int w = 0; w < 8; w++) base += s_wt[w];
  const uint32_t npd = (ctl->fshift + 7u) / 8u;  // digits below the field
  if (n <= (uint32_t)kBTile) {
    block_sort<VALS>(B + base, VALS ? VB + base : nullptr, A + base, VALS ? VA + base : nullptr, n,
                     (ctl->or_all >> ctl->fshift >> 8 << 8 | b) << ctl->fshift, ctl->fshift, fsm);
    return;
  }
  if (threadIdx.x == 0) { s_or = 0; s_and = ~0ull; }
  __syncthreads();
  // ---- oversized bucket: block-level LSD through global memory ----
  {
    ull o = 0, a = ~0ull;
    for (uint32_t i = threadIdx.x; i < n; i += kBT) {
      const uint64_t x = B[base + i];
      o |= x;
      a &= x;
    }
    atomicOr(&s_or, o);
    atomicAnd(&s_and, a);
  }
  __syncthreads();
  const ull vary = s_or ^ s_and;
  uint64_t* src = B + base;
  uint64_t* dst = A + base;
  uint32_t* vsrc = VALS ? VB + base : nullptr;
  uint32_t* vdst = VALS ? VA + base : nullptr;
  bool in_a = false;
  for (uint32_t p = 0; p < npd; p++) {
    if (((vary >> (8 * p)) & 255u) == 0) continue;
    const int shift = 8 * (int)p;
    // counting pass, then exclusive offsets of the digits
    if (threadIdx.x < 256) s_run[threadIdx.x] = 0;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n; i += kBT)
      atomicAdd(&s_run[(uint32_t)(src[i] >> shift) & 255u], 1u);
    __syncthreads();
    uint32_t v = 0, inc = 0;
    if (threadIdx.x < 256) {
      v = s_run[threadIdx.x];
      inc = warp_incl_scan(v);
      if (lane == 31) s_wt[warp] = inc;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
      uint32_t wbase = 0;
      for (unsigned q = 0; q < warp; q++) wbase += s_wt[q];
      s_run[threadIdx.x] = wbase + inc - v;
    }
    __syncthreads();
    // the tiles in order: stable rank, scatter to the running offsets
    for (uint32_t t0 = 0; t0 < n; t0 += (uint32_t)kBTile) {
      const uint32_t nv = min((uint32_t)kBTile, n - t0);
      const uint32_t ipw = (nv + 32u * (kBT / 32) - 1u) / (32u * (kBT / 32));
      uint64_t key[kBItems];
      uint32_t val[kBItems];
#pragma unroll
      for (int j = 0; j < kBItems; j++) {
        const uint32_t li = warp * 32 * ipw + j * 32 + lane;
        const bool ok = (uint32_t)j < ipw && li < nv;
        key[j] = ok ? src[t0 + li] : 0ull;
        if constexpr (VALS) val[j] = ok ? vsrc[t0 + li] : 0u;
        else val[j] = 0u;
      }
      tile_rank<VALS, kBT, kBItems>(key, val, nv, shift, sm, ipw);
      for (uint32_t i = threadIdx.x; i < nv; i += kBT) {
        const uint64_t x = sm.keys[i];
        const uint32_t d = (uint32_t)(x >> shift) & 255u;
        const uint32_t o = s_run[d] + (i - sm.dstart[d]);
        dst[o] = x;
        if constexpr (VALS) vdst[o] = sm.vals[i];
      }
      __syncthreads();
      if (threadIdx.x < 256) {
        const uint32_t d = threadIdx.x;
        s_run[d] += (d < 255 ? sm.dstart[d + 1] : nv) - sm.dstart[d];
      }
      __syncthreads();
    }
    uint64_t* t = src; src = dst; dst = t;
    uint32_t* tv = vsrc; vsrc = vdst; vdst = tv;
    in_a = !in_a;
    __syncthreads();
  }
  if (!in_a) {
    for (uint32_t i = threadIdx.x; i < n; i += kBT) {
      A[base + i] = B[base + i];
      if constexpr (VALS) VA[base + i] = VB[base + i];
    }
  }
}

// Untagged batches of at most kTile keys: one block, a bitonic sorting
// network over the batch padded with 2^64-1 to n (a power of two) in shared
// memory, one compare-exchange of each pair per stage (equal keys are equal
// values, so order among them does not matter).
constexpr int kBitT = 1024;
__global__ void __launch_bounds__(kBitT) k_sort_bitonic(const uint64_t* __restrict__ in,
                                                        uint64_t* __restrict__ out, uint32_t k,
                                                        uint32_t n) {
  __shared__ uint64_t s[kTile];
  for (uint32_t i = threadIdx.x; i < n; i += kBitT) s[i] = i < k ? in[i] : ~0ull;
  __syncthreads();
  for (uint32_t size = 2; size <= n; size <<= 1) {
    for (uint32_t stride = size >> 1; stride; stride >>= 1) {
      for (uint32_t t = threadIdx.x; t < n / 2; t += kBitT) {
        const uint32_t i = 2 * t - (t & (stride - 1)), j = i + stride;  // pair t of this stage
        const uint64_t a = s[i], b = s[j];
        if ((a > b) == ((i & size) == 0)) {  // ascending runs where bit `size` of i is 0
          s[i] = b;
          s[j] = a;
        }
      }
      __syncthreads();
    }
  }
  for (uint32_t i = threadIdx.x; i < k; i += kBitT) out[i] = s[i];
}

// Tagged batches of at most kTile keys: a stable rank sort spread over many
// blocks.  Every block holds the whole batch in shared memory; P consecutive
// threads share one key, each counting over a P-th of the batch the keys
// below it and the equal keys before it, and the sum of their counts (a
// shuffle reduction) is where the key (and its tag) goes.
constexpr int kRankT = 256;
__global__ void __launch_bounds__(kRankT) k_sort_rank(const uint64_t* __restrict__ in,
                                                      uint64_t* __restrict__ out,
                                                      const uint32_t* __restrict__ vin,
                                                      uint32_t* __restrict__ vout, uint32_t k,
                                                      uint32_t P) {
  extern __shared__ __align__(16) uint64_t s_keys[];
  for (uint32_t i = threadIdx.x; i < k; i += kRankT) s_keys[i] = in[i];
  __syncthreads();
  const uint32_t g = blockIdx.x * kRankT + threadIdx.x;
  const uint32_t i = g / P, part = g % P;
  const bool valid = i < k;
  const uint64_t x = valid ? s_keys[i] : 0ull;
  const uint32_t per = (k + P - 1) / P;
  const uint32_t j0 = min(k, part * per), j1 = min(k, j0 + per);
  uint32_t r = 0;
  if (valid) {
    // equal keys count only before i: two ranges with a fixed test
    const uint32_t jm = min(max(i, j0), j1);
#pragma unroll 8
    for (uint32_t j = j0; j < jm; j++) r += s_keys[j] <= x;
#pragma unroll 8
    for (uint32_t j = jm; j < j1; j++) r += s_keys[j] < x;
  }
  for (uint32_t o = 1; o < P; o <<= 1) r += __shfl_xor_sync(FULL, r, o);
  if (valid && part == 0) {
    out[r] = x;
    vout[r] = vin[i];
  }
}

}  // namespace

namespace {
size_t ctl_bytes() { return (sizeof(SortCtl) + 255) & ~(size_t)255; }
template <bool VALS>
int& scatter_blocks_per_sm() {
  static int n = 1;
  return n;
}
template <bool VALS>
void sort_attrs() {
  static bool done = false;  // one per instantiation
  if (done) return;
  const int smem = (int)sizeof(TileSmemT<VALS>);
  cudaFuncSetAttribute(k_digit_scatter<VALS, true, false>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(k_digit_scatter<VALS, true, true>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if constexpr (!VALS)
    cudaFuncSetAttribute(k_digit_scatter<false, false, true>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(k_bucket_sort<VALS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)sizeof(FinishSmem<VALS>));
  cudaFuncSetAttribute(k_window_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)sizeof(FinishSmem<false>));
  int bps = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_digit_scatter<VALS, true, false>, kT, smem) ==
          cudaSuccess &&
      bps > 0)
    scatter_blocks_per_sm<VALS>() = bps;
  cudaGetLastError();
  done = true;
}
}  // namespace

// Blocks of a digit pass over k keys, at most: one tile each, no more than run at
// once (the scatter kernel's limit), and that many for a large batch.
template <bool VALS>
uint32_t pass_blocks_most(const cpma* h, uint64_t k) {
  const uint64_t most = (uint64_t)h->num_sms * (uint64_t)scatter_blocks_per_sm<VALS>();
  return (uint32_t)(k > kBucketMax ? most : std::min<uint64_t>((k + kTile - 1) / kTile, most));
}

// The blocks it takes: that many, or with whole tiles the fewest that give no
// block more of them.
template <bool VALS>
uint32_t pass_blocks(const cpma* h, uint64_t k) {
  const uint64_t nt = (k + kTile - 1) / kTile, most = pass_blocks_most<VALS>(h, k);
  if (nt < kWholeTiles * most) return (uint32_t)most;
  const uint64_t per = (nt + most - 1) / most;
  return (uint32_t)((nt + per - 1) / per);
}

// The sort's words in the scratch: control, group counts per pass (row 0: by the
// field or kTop0, 1: kTop1, 2 + p: digit p), sample, counts per block.  Sizes
// grow with k and are largest without tags, so that a reservation covers smaller
// and untagged batches.
struct HistLayout {
  uint32_t G, row;       // blocks, words of a row
  size_t grp, bins, cnt, bytes;
};
template <bool VALS>
HistLayout hist_layout(const cpma* h, uint64_t k) {
  HistLayout l;
  const bool large = k > kBucketMax;
  l.G = pass_blocks<VALS>(h, k);
  const uint32_t most = pass_blocks_most<VALS>(h, k);
  l.row = (most + kGroup - 1) / kGroup * 256;
  l.grp = ctl_bytes();
  l.bins = l.grp + (size_t)(large ? 10 : 1) * l.row * 4;
  l.cnt = l.bins + (large && !VALS ? kSampleBins * 4 : 0);
  l.bytes = l.cnt + (size_t)most * 256 * 4;
  return l;
}

int sort_scratch(cpma* h, uint64_t k, bool vals) {
  sort_attrs<false>();
  if (vals) sort_attrs<true>();
  if (k <= 1) return CPMA_OK;
  CPMA_TRY(ensure(h, h->s.keysA, k * 8));
  if (vals) CPMA_TRY(ensure(h, h->s.valsA, k * 4));
  if (k <= (uint64_t)kTile) return CPMA_OK;
  CPMA_TRY(ensure(h, h->s.keysB, k * 8));
  if (vals) CPMA_TRY(ensure(h, h->s.valsB, k * 4));
  return ensure(h, h->s.hist, hist_layout<false>(h, k).bytes);
}

template <bool VALS>
Pass pass_of(cpma* h, const uint64_t* d_in, const uint32_t* v_in, uint64_t k) {
  Scratch& s = h->s;
  uint8_t* ctl = reinterpret_cast<uint8_t*>(s.hist.p);
  const HistLayout l = hist_layout<VALS>(h, k);
  return Pass{d_in, v_in, (uint64_t*)s.keysA.p, (uint64_t*)s.keysB.p,
              VALS ? (uint32_t*)s.valsA.p : nullptr, VALS ? (uint32_t*)s.valsB.p : nullptr, k, 0,
              reinterpret_cast<SortCtl*>(ctl), reinterpret_cast<uint32_t*>(ctl + l.grp),
              reinterpret_cast<uint32_t*>(ctl + l.cnt)};
}

// The two kernels of a digit pass, each scheduled while the one before it
// finishes (programmatic dependent launch; each waits for it first).
template <bool VALS>
int digit_pass(cpma* h, Pass a, const HistLayout& l, int p, bool stable, cudaStream_t st) {
  const size_t smem = sizeof(TileSmemT<VALS>);
  a.p = p;
  a.grp += (size_t)(p >= 0 ? 2 + p : p == kTop1 ? 1 : 0) * l.row;
  CPMA_CUDA(launch_pdl(k_digit_count, l.G, kT, 0, st, a));
  if constexpr (VALS) stable = true;
  const bool whole = (a.k + kTile - 1) / kTile >= kWholeTiles * l.G;  // as share_of
  CPMA_CUDA(launch_pdl(!stable ? k_digit_scatter<false, false, true>
                       : whole ? k_digit_scatter<VALS, true, true>
                               : k_digit_scatter<VALS, true, false>,
                       l.G, kT, smem, st, a));
  h->launches += 2;
  return CPMA_OK;
}

// A large batch by the digits that vary, lowest first: with tags, when few
// bits vary, or when a bucket is too large for a window (the kernels return at
// once otherwise).
template <bool VALS>
int sort_digits(cpma* h, const uint64_t* d_in, const uint32_t* v_in, uint64_t k, cudaStream_t st) {
  const Pass a = pass_of<VALS>(h, d_in, v_in, k);
  const HistLayout l = hist_layout<VALS>(h, k);
  for (int p = 0; p < 8; p++) CPMA_TRY(digit_pass<VALS>(h, a, l, p, true, st));
  CPMA_CUDA(launch_pdl(k_copy_if_no_pass,
                       (unsigned)std::min<uint64_t>((uint64_t)h->num_sms * 4, (k + kT - 1) / kT),
                       kT, 0, st, d_in, a.A, v_in, a.VA, k, a.ctl));
  h->launches++;
  return CPMA_OK;
}

// most: a large batch without sort_digits (the caller looks at ctl->rest)
template <bool VALS>
int sort_impl(cpma* h, const uint64_t* d_in, const uint32_t* v_in, uint64_t k, const uint64_t** out,
              const uint32_t** vout, cudaStream_t st, bool cleared, bool most = false) {
  *out = d_in;
  if (vout) *vout = v_in;
  if (k <= 1) return CPMA_OK;
  CPMA_TRY(sort_scratch(h, k, VALS));
  uint64_t* A = (uint64_t*)h->s.keysA.p;
  uint32_t* VA = VALS ? (uint32_t*)h->s.valsA.p : nullptr;
  if (!VALS && k <= (uint64_t)kTile) {
    prof_add_bytes(h, PH_SORT, 16ull * k);
    uint32_t n = 2;
    while (n < k) n <<= 1;
    k_sort_bitonic<<<1, kBitT, 0, st>>>(d_in, A, (uint32_t)k, n);
    h->launches++;
    *out = A;
    return check_cuda(cudaGetLastError());
  }
  if (k <= (uint64_t)kTile) {
    prof_add_bytes(h, PH_SORT, 24ull * k);
    // threads per key: a power of two keeping each thread's share at 256 keys
    uint32_t P = 1;
    while (P < 32 && k > 256ull * P) P <<= 1;
    const uint32_t nb = (uint32_t)((k * P + kRankT - 1) / kRankT);
    k_sort_rank<<<nb, kRankT, k * 8, st>>>(d_in, A, v_in, VA, (uint32_t)k, P);
    h->launches++;
    *out = A;
    if (vout) *vout = VA;
    return check_cuda(cudaGetLastError());
  }
  uint64_t* B = (uint64_t*)h->s.keysB.p;
  uint32_t* VB = VALS ? (uint32_t*)h->s.valsB.p : nullptr;
  SortCtl* ctl = reinterpret_cast<SortCtl*>(h->s.hist.p);
  const HistLayout l = hist_layout<VALS>(h, k);
  const Pass a = pass_of<VALS>(h, d_in, v_in, k);
  if (!cleared) CPMA_CUDA(cudaMemsetAsync(ctl, 0, sizeof(SortCtl), st));
  // about eight keys per thread: one step of the unrolled loop
  const int ogrid = (int)std::max<uint64_t>(
      1, std::min<uint64_t>((uint64_t)h->num_sms * 8, (k + 8 * kT - 1) / (8 * kT)));
  // buckets by the 16 highest bits hold k / 65536 keys and more: no window's worth
  const bool digits = VALS || k > kMsdMax;
  CPMA_CUDA(launch_pdl(k_orand, ogrid, kT, 0, st, d_in, k, ctl, digits, a.grp,
                       (uint32_t)((l.cnt - l.grp) / 4)));
  h->launches++;
  if (k <= kBucketMax) {
    CPMA_TRY(digit_pass<VALS>(h, a, l, kField, VALS, st));
    CPMA_CUDA(launch_pdl(k_bucket_sort<VALS>, 256, kBT, sizeof(FinishSmem<VALS>), st, B, VB, A, VA,
                         ctl, d_in, v_in, k));
    h->launches++;
    // OR/AND and count reads, scatter and bucket read + write
    prof_add_bytes(h, PH_SORT, 16ull * k + (VALS ? 24ull : 16ull) * k * 2);
  } else {
    if (!digits) {
      // the mean bucket's sample and eight standard deviations, but at least
      // that of 3700 keys: a bucket of 2048 to 6144 fits its window if it starts
      // early in it, and the passes over all digits take half as long again
      const double mean = (double)(k / kSampleEvery) / kSampleBins;
      const uint32_t many = (uint32_t)std::max(29.0, mean + 8.0 * std::sqrt(mean));
      uint32_t* bins = reinterpret_cast<uint32_t*>((uint8_t*)h->s.hist.p + l.bins);
      CPMA_CUDA(launch_pdl(k_sample, (unsigned)h->num_sms * 4u, kT, 0, st, d_in, k, ctl, bins, many));
      h->launches++;
      CPMA_TRY(digit_pass<VALS>(h, a, l, kTop0, false, st));
      CPMA_TRY(digit_pass<VALS>(h, a, l, kTop1, true, st));
      CPMA_CUDA(launch_pdl(k_window_sort, (unsigned)((k + kTile - 1) / kTile), kBT,
                           sizeof(FinishSmem<false>), st, B, A, k, ctl));
      h->launches++;
      prof_add_bytes(h, PH_SORT, 72ull * k);
    } else {
      prof_add_bytes(h, PH_SORT, 8ull * k + 32ull * k * 5);  // typical: 5 varying digits
    }
    if (!most) CPMA_TRY(sort_digits<VALS>(h, d_in, v_in, k, st));
  }
  CPMA_CUDA(cudaGetLastError());
  const uint64_t* src = A;
  const uint32_t* vsrc = VA;
  *out = src;
  if (vout) *vout = vsrc;
  return CPMA_OK;
}

int sort_keys(cpma* h, const uint64_t* d_in, uint64_t k, const uint64_t** out,
              cudaStream_t st, bool cleared) {
  return sort_impl<false>(h, d_in, nullptr, k, out, nullptr, st, cleared);
}

int sort_pairs(cpma* h, const uint64_t* d_in, const uint32_t* v_in, uint64_t k,
               const uint64_t** out, const uint32_t** vout, cudaStream_t st, bool cleared) {
  return sort_impl<true>(h, d_in, v_in, k, out, vout, st, cleared);
}

uint32_t* sort_control(cpma* h, uint64_t k, uint32_t* nwords) {
  *nwords = k > (uint64_t)kTile ? (uint32_t)(sizeof(SortCtl) / 4) : 0u;
  return *nwords ? reinterpret_cast<uint32_t*>(h->s.hist.p) : nullptr;
}

int sort_keys_most(cpma* h, const uint64_t* d_in, uint64_t k, const uint64_t** out,
                   const uint32_t** over, cudaStream_t st) {
  *over = nullptr;
  CPMA_TRY(sort_impl<false>(h, d_in, nullptr, k, out, nullptr, st, false, true));
  if (k > kBucketMax) *over = &reinterpret_cast<SortCtl*>(h->s.hist.p)->rest;
  return CPMA_OK;
}

int sort_keys_rest(cpma* h, const uint64_t* d_in, uint64_t k, cudaStream_t st) {
  return sort_digits<false>(h, d_in, nullptr, k, st);
}

}  // namespace cpmaimpl
