// Thread-granular insert of a few keys into one leaf of byte codes (Sec. 4
// batch merge, Sec. 5 leaf format: an 8-byte little-endian head, then the
// deltas to the following keys as unsigned LEB128 codes, packed left, zero
// bytes after the used ones).
//
// One thread owns one leaf.  Pass A sums the leaf 16 bytes at a time with
// word-parallel arithmetic (each byte's position inside its code from the
// continuation flags of the bytes before it, then two dot products per word
// with byte weights 1 / 128 and 2^14 / 2^21), recording for every key of
// the slice the chunk it lands in; each key's chunk is then decoded byte by
// byte (by any thread: the record holds the state) to find its place: before
// the head (a new head), inside the gap that one code spans (the code is
// split), or after the last element (appended); a key equal to an element or
// to the slice key before it is skipped.  Keys sharing a gap
// form one edit: old bytes [os, oe) replaced by nl new bytes.  Every edit of
// an insert grows or keeps the size (a split code never needs more bytes
// than its two parts), so pass B rewrites the leaf in place from the end
// backwards, 16 bytes at a time: each destination chunk gathers the old
// bytes that land in it (one shift per segment between edits; a chunk wholly
// inside the segment after the last edit is one shifted 16-byte read) and is
// stored whole, before the edits' own bytes are written.  Every read of pass
// B is of a chunk at or below the one being written, so it sees old bytes
// (a delete shrinks: forward, reads at or above).
//
// The functions are __host__ __device__ so that the same code can be run on
// the host.
#pragma once
#include "leaf_walk.cuh"

namespace leafthr {

constexpr uint32_t kKeys = 4;  // slice keys per leaf on this path

// key record kinds
constexpr uint32_t kGap = 0;    // inside the gap of the code [cs, ce)
constexpr uint32_t kHead = 1;   // before the head
constexpr uint32_t kAfter = 2;  // after the last element
constexpr uint32_t kSkip = 3;   // a repeat of the slice key before it
constexpr uint32_t kChunk = 4;  // (pass A, step 1) in a code ending in the chunk at cs
constexpr uint32_t kHit = 5;    // equal to an element: the code [cs, ce) is its own

// kinds an insert leaves alone
LT_HD bool no_insert(uint32_t kind) { return kind == kSkip || kind == kHit; }

// results
constexpr uint32_t kUnchanged = 0;  // every key present: nothing written
constexpr uint32_t kWritten = 1;    // leaf rewritten in place
constexpr uint32_t kTooBig = 2;     // result exceeds the leaf: nothing written
constexpr uint32_t kLongCode = 3;   // a code of more than 4 bytes: nothing written

struct Result {
  uint32_t nb;       // new used bytes
  uint32_t newc;     // new element count
  uint32_t added;    // bit q: slice key q was added
  uint32_t wlo, whi; // byte range rewritten (kWritten)
  uint32_t E;        // edits
  uint32_t maxcode;  // longest code the edits write (bytes)
  uint64_t newhead;
};

LT_HD uint32_t leb_bytes(uint64_t d) {  // unsigned LEB128 length of d
#if defined(__CUDA_ARCH__)
  const uint32_t bl = 64u - (uint32_t)__clzll((long long)(d | 1ull));
#else
  const uint32_t bl = 64u - (uint32_t)__builtin_clzll(d | 1ull);
#endif
  return (bl + 6u) / 7u;
}

LT_HD uint32_t leb_write(uint8_t* p, uint64_t d) {
  uint32_t n = 0;
  while (d >= 128u) { p[n++] = (uint8_t)(d | 0x80u); d >>= 7; }
  p[n++] = (uint8_t)d;
  return n;
}

LT_HD uint64_t pick(const uint64_t (&y)[kKeys], uint32_t q) {
  static_assert(kKeys == 4, "four slice keys");
  return q == 0 ? y[0] : q == 1 ? y[1] : q == 2 ? y[2] : y[3];
}

// Per-thread scratch: arrays of kKeys entries at stride `rs` (key records and
// edits), so that a block's threads index shared memory without conflicts.
template <class Code>
struct ScratchT {
  uint32_t* rpos;   // key q: cs | ce << 12 | kind << 24
  uint64_t* rval;   // key q: successor value (kGap), the head (kHead), the last value (kAfter)
  Code* rcode;      // key q: value of the code [cs, ce) (kGap)
  uint32_t* epos;   // edit e: os | oe << 12 | kind << 24
  int32_t* esa;     // edit e: total size change of edits 0..e
  uint32_t* ekey;   // edit e: first key | end key << 8 | nl << 16
  uint32_t rs;
};
using Scratch = ScratchT<uint32_t>;      // leaves whose codes have at most 4 bytes
using ScratchLong = ScratchT<uint64_t>;  // any code length

// Pass A, step 1: the byte weights of one 4-byte word of codes.  cb, p1, p2
// carry the flags of the word before (bit 7 of each byte): cb = the byte is
// a continuation byte, p1 = the byte before it is one (its position g in its
// code is >= 1), p2 = g >= 2.  A byte at position g weighs 128^g in the
// value of its code, so the sum of the (partial) codes in the word is
// dp4a(pay, w01) + 2^14 dp4a(pay, w23) with w01 = 1 / 128 for g = 0 / 1 and
// w23 = 1 / 128 for g = 2 / 3 (0 elsewhere).  lc collects continuation
// bytes at position >= 3: a code of more than 4 bytes, which the 32-bit
// arithmetic does not cover.
LT_HD uint32_t word_sum(uint32_t w, uint32_t& cb, uint32_t& p1, uint32_t& p2, uint32_t& lc,
                        uint32_t& pay, uint32_t& w01, uint32_t& w23) {
  const uint32_t c = w & 0x80808080u;
  const uint32_t q1 = fshl(cb, c, 8);
  const uint32_t q2 = q1 & fshl(p1, q1, 8);
  const uint32_t q3 = q2 & fshl(p2, q2, 8);
  lc |= q3 & c;
  pay = w & 0x7F7F7F7Fu;
  w01 = ((q1 ^ 0x80808080u) >> 7) | (q1 ^ q2);
  w23 = ((q2 ^ q3) >> 7) | q3;
  cb = c;
  p1 = q1;
  p2 = q2;
  return dp4a(pay, w01, 0u) + (dp4a(pay, w23, 0u) << 14);
}

// Is x an element of the byte-code leaf of u >= 8 used bytes (bytes past them
// zero)?  The leaf is summed chunk by chunk as in pass A, to the one whose
// last element reaches x; that chunk's elements are then compared one by one,
// by all lanes of a warp together.  A leaf that turns out to hold a code of
// more than 4 bytes before x is walked instead.
LT_HD bool leaf_has(const uint8_t* leafp, uint32_t u, uint64_t x) {
  uint32_t w[4], raw[4];
  ld16(leafp, raw);
  uint64_t val = (uint64_t)raw[0] | ((uint64_t)raw[1] << 32);
  if (x <= val) return x == val;
  uint32_t carry = 0, lc = 0, cb = 0, p1 = 0, p2 = 0, g0 = 0, p0 = 0;
  for (;; p0 += 16) {
#pragma unroll
    for (int i = 0; i < 4; i++) w[i] = raw[i];
    if (p0 + 16u < u) ld16(leafp + p0 + 16u, raw);  // on its way while this one is summed
    const uint32_t cb_in = cb;
    uint32_t tsum = 0, pay = 0, w01 = 0, w23 = 0;
    if (p0) {
      tsum += word_sum(w[0], cb, p1, p2, lc, pay, w01, w23);
      tsum += word_sum(w[1], cb, p1, p2, lc, pay, w01, w23);
    }
    tsum += word_sum(w[2], cb, p1, p2, lc, pay, w01, w23);
    tsum += word_sum(w[3], cb, p1, p2, lc, pay, w01, w23);
    const uint32_t tw = ~cb & 0x80808080u;
    const uint32_t ps = pay & (tw ? ~(0xFFFFFFFFu >> clz32(tw)) : 0xFFFFFFFFu);
    const uint32_t cnew = dp4a(ps, w01, 0u) + (dp4a(ps, w23, 0u) << 14);
    lc |= tw ? 0u : 1u;
    const uint64_t vend = val + (uint32_t)(carry + tsum - cnew);
    g0 = clz32(~cb_in & 0x80808080u) >> 3;
    if (vend >= x || lc || p0 + 16u >= u) break;
    val = vend;
    carry = cnew;
  }
  if (lc) {
    bool found = false;
    leafwalk::leaf_visit(leafp, u, [&](uint64_t v) { found |= v == x; });
    return found;
  }
  // the chunk's elements relative to the one before it (zero bytes past the
  // used ones repeat the last, which is an element)
  const uint64_t dx = x - val;
  const uint32_t d = dx > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)dx;
  uint32_t cum = carry, pw = 1u << (7u * g0);
  bool found = false;
#pragma unroll
  for (int b = 0; b < 16; b++) {
    const uint32_t c = byte_of(w[b >> 2], b & 3);
    const bool code = b >= 8 || p0 != 0;  // bytes 0-7 of the leaf are the head
    cum += code ? (c & 0x7Fu) * pw : 0u;
    const bool term = code && !(c & 0x80u);
    found |= term && cum == d;
    pw = !code ? pw : (c & 0x80u) ? pw << 7 : 1u;
  }
  return found;
}

// Pass A, step 2, for key yq of the slice (rep: a repeat of the one before it),
// whose record (rpos, rval, rcode) names the chunk it lands in and the state
// that was entered with: val0 the element before it, carry0 and g0 the bits and
// byte count of the code open at its start.  The chunk is walked byte by byte
// without branches, the values relative to val0: the last terminator below the
// key, and the first that reaches it.  The record becomes the key's gap.
LT_HD void place_key(const uint8_t* leafp, uint32_t uold, uint64_t yq, bool rep, uint32_t& rpos,
                     uint64_t& rval, uint32_t& rcode) {
  const uint32_t p0 = rpos & 0xFFFu, g0 = (rpos >> 12) & 0xFFFu;
  const uint64_t val0 = rval;
  uint32_t w[4], t[4];
  leafwalk::load_chunk(leafp, p0, uold, w, t);
  const uint32_t first = p0 == 0 ? 8u : 0u;  // bytes 0-7 are the head
  if (p0 == 0) w[0] = w[1] = t[0] = t[1] = 0u;
#pragma unroll
  for (int i = 0; i < 4; i++) w[i] &= 0x7F7F7F7Fu;
  const uint32_t d = (uint32_t)(yq - val0);  // the chunk's last element reaches it
  uint32_t cum = rcode, pw = 1u << (7u * g0);
  uint32_t below = 0, cs = first - g0, at = 0, ce = 0;  // cs: relative to p0, may wrap
  bool open = true;
#pragma unroll
  for (int b = 0; b < 16; b++) {
    cum += byte_of(w[b >> 2], b & 3) * pw;
    const bool term = (t[b >> 2] & (0x80u << (8 * (b & 3)))) != 0u;
    const bool stop = term && open && cum >= d;
    const bool pass = term && open && cum < d;
    at = stop ? cum : at;
    ce = stop ? (uint32_t)b + 1u : ce;
    below = pass ? cum : below;
    cs = pass ? (uint32_t)b + 1u : cs;
    open = open && !stop;
    pw = term ? 1u : pw << 7;
    if (p0 == 0 && b == 7) pw = 1u << (7u * g0);  // the head's bytes are no codes
  }
  const uint64_t val = val0 + at;
  const uint32_t kind = rep ? kSkip : yq == val ? kHit : kGap;
  rpos = (p0 + cs) | ((p0 + ce) << 12) | (kind << 24);
  rval = val;
  rcode = at - below;
}

// The 16 bytes of the old leaf at byte offset src, bytes outside [0, LB)
// reading as zero: five 4-byte words from the 4-byte boundary at or below src
// and one byte shift (two 16-byte loads and their word selects took more).
LT_HD void chunk_at(const uint8_t* leafp, uint32_t LB, int32_t src, uint32_t (&r)[4]) {
  const int32_t base = src & ~3;
  const uint32_t s8 = 8u * (uint32_t)(src & 3);
  uint32_t W[5];
#pragma unroll
  for (int i = 0; i < 5; i++) {
    W[i] = 0u;
    if ((uint32_t)(base + 4 * i) < LB && (i < 4 || s8)) W[i] = ld4(leafp + base + 4 * i);
  }
#pragma unroll
  for (int i = 0; i < 4; i++) r[i] = fshr(W[i], W[i + 1], s8);
}

// The same for a run of chunks 16 bytes apart, downwards: of the two aligned
// blocks it spans the upper one was read for the chunk before, and is kept.
struct Block {
  uint32_t w[4] = {0u, 0u, 0u, 0u};
  int32_t at = -64;
};

LT_HD void block_at(const uint8_t* leafp, uint32_t LB, int32_t at, const Block& kept,
                    uint32_t (&r)[4]) {
  if (at == kept.at) {
#pragma unroll
    for (int i = 0; i < 4; i++) r[i] = kept.w[i];
  } else if ((uint32_t)at < LB) {
    ld16(leafp + at, r);
  } else {
#pragma unroll
    for (int i = 0; i < 4; i++) r[i] = 0u;
  }
}

LT_HD void next_chunk_at(const uint8_t* leafp, uint32_t LB, int32_t src, Block& kept,
                         uint32_t (&r)[4]) {
  const int32_t base = src & ~15;
  const uint32_t s = (uint32_t)src & 15u;
  uint32_t lo[4], hi[4] = {0u, 0u, 0u, 0u};
  block_at(leafp, LB, base, kept, lo);
  if (s) block_at(leafp, LB, base + 16, kept, hi);
  const bool two = (s & 8u) != 0u, one = (s & 4u) != 0u;
  const uint32_t y[6] = {two ? lo[2] : lo[0], two ? lo[3] : lo[1], two ? hi[0] : lo[2],
                         two ? hi[1] : lo[3], two ? hi[2] : hi[0], two ? hi[3] : hi[1]};
  uint32_t z[5];
#pragma unroll
  for (int i = 0; i < 5; i++) z[i] = one ? y[i + 1] : y[i];
#pragma unroll
  for (int i = 0; i < 4; i++) r[i] = fshr(z[i], z[i + 1], 8u * (s & 3u));
  kept.at = base;
#pragma unroll
  for (int i = 0; i < 4; i++) kept.w[i] = lo[i];
}

// r with the bytes [a, b) of x in place of its own.
LT_HD void take_bytes(uint32_t (&r)[4], const uint32_t (&x)[4], uint32_t a, uint32_t b) {
  const uint32_t m16 = (b >= 16u ? 0xFFFFu : ((1u << b) - 1u)) & ~((1u << a) - 1u);
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const uint32_t m = bmask4((m16 >> (4 * i)) & 0xFu);
    r[i] = (r[i] & ~m) | (x[i] & m);
  }
}

// Pass B: destination bounds [dlo, dhi) and shift sa of segment e (-1 .. E-1):
// the old bytes [oe_e, os_{e+1}) moved by sa_e (oe_{-1} = 0, os_E = uold,
// sa_{-1} = 0).
template <class SC>
LT_HD void seg_bounds(const SC& S, uint32_t E, uint32_t uold, uint32_t os0, int e,
                      int32_t& dlo, int32_t& dhi, int32_t& sa) {
  uint32_t lo = 0u, hi = os0;
  sa = 0;
  if (e >= 0) {
    lo = (S.epos[e * S.rs] >> 12) & 0xFFFu;
    hi = (e + 1 < (int)E) ? (S.epos[(e + 1) * S.rs] & 0xFFFu) : uold;
    sa = S.esa[e * S.rs];
  }
  dlo = (int32_t)lo + sa;
  dhi = (int32_t)hi + sa;
}

// Pass A: a record for every slice key (kind, code bytes, values; see
// Scratch).  Returns kWritten when every key is placed (nothing is written),
// else kLongCode (the leaf holds a code of more than 4 bytes).  head
// receives the leaf's first element.
constexpr uint32_t kPlaced = kWritten;

// Step 1: keys before, at and after the leaf's elements get their records, the
// others (kChunk) the chunk that takes them.
LT_HD uint32_t pass_a_sum(const uint8_t* leafp, uint32_t uold, const uint64_t (&y)[kKeys],
                          uint32_t s, const Scratch& S, uint64_t& head) {
  uint32_t w[4];
  ld16(leafp, w);
  head = (uint64_t)w[0] | ((uint64_t)w[1] << 32);
  uint32_t k = 0;
  while (k < s && pick(y, k) <= head) {
    const uint64_t x = pick(y, k);
    const bool rep = k > 0 && pick(y, k - 1) == x;
    const uint32_t kind = rep ? kSkip : x == head ? kHit : kHead;
    S.rpos[k * S.rs] = 0u | (8u << 12) | (kind << 24);
    S.rval[k * S.rs] = head;
    S.rcode[k * S.rs] = 0u;
    k++;
  }
  // chunk sums over the whole leaf (a warp's threads then take the
  // same number of steps); every key gets the chunk (p0, entry state) of
  // the code it falls in, or stays for the end
  uint64_t ycur = k < s ? pick(y, k) : ~0ull;
  uint64_t val = head;
  uint32_t carry = 0, lc = 0, cb = 0, p1 = 0, p2 = 0;
  // (bytes past the used ones are zero: packed left)
  auto chunk = [&](uint32_t p0, const uint32_t (&w)[4]) {
    const uint32_t cb_in = cb;    // flags of the last word before p0
    uint32_t tsum = 0, pay = 0, w01 = 0, w23 = 0;
    if (p0) {
      tsum += word_sum(w[0], cb, p1, p2, lc, pay, w01, w23);
      tsum += word_sum(w[1], cb, p1, p2, lc, pay, w01, w23);
    }
    tsum += word_sum(w[2], cb, p1, p2, lc, pay, w01, w23);
    tsum += word_sum(w[3], cb, p1, p2, lc, pay, w01, w23);
    // the code still open at the chunk end: the bytes of the last word after
    // its last terminator (a code of at most 4 bytes has one there)
    const uint32_t tw = ~cb & 0x80808080u;
    const uint32_t ps = pay & (tw ? ~(0xFFFFFFFFu >> clz32(tw)) : 0xFFFFFFFFu);
    const uint32_t cnew = dp4a(ps, w01, 0u) + (dp4a(ps, w23, 0u) << 14);
    lc |= tw ? 0u : 1u;
    const uint64_t vend = val + (uint32_t)(carry + tsum - cnew);
    if (vend >= ycur) {
      // bytes of the code open at p0 (trailing continuation bytes before it)
      const uint32_t g0 = clz32(~cb_in & 0x80808080u) >> 3;
      while (k < s && ycur <= vend) {
        S.rpos[k * S.rs] = p0 | (g0 << 12) | (kChunk << 24);
        S.rval[k * S.rs] = val;
        S.rcode[k * S.rs] = carry;
        k++;
        ycur = k < s ? pick(y, k) : ~0ull;
      }
    }
    val = vend;
    carry = cnew;
  };
  // 32 bytes at a time: a lane's loads hit lines of their own, so their number
  // counts
  const bool wide = (reinterpret_cast<uintptr_t>(leafp) & 31u) == 0;
  uint32_t w2[4];
  for (uint32_t p0 = 0; p0 < uold; p0 += 32) {
    const bool two = p0 + 16u < uold;
    if (wide && two) {
      leafwalk::ld32(leafp + p0, w, w2);
    } else {
      if (p0) ld16(leafp + p0, w);
      if (two) ld16(leafp + p0 + 16u, w2);
    }
    chunk(p0, w);
    if (two) chunk(p0 + 16u, w2);
  }
  if (lc) return kLongCode;
  const uint64_t lastv = val;
  for (; k < s; k++) {
    const uint64_t x = pick(y, k);
    const bool rep = k > 0 && pick(y, k - 1) == x;
    S.rpos[k * S.rs] = uold | (uold << 12) | ((rep ? kSkip : kAfter) << 24);
    S.rval[k * S.rs] = lastv;
    S.rcode[k * S.rs] = 0u;
  }
  return kPlaced;
}

LT_HD uint32_t pass_a(const uint8_t* leafp, uint32_t uold, const uint64_t (&y)[kKeys], uint32_t s,
                      const Scratch& S, uint64_t& head) {
  const uint32_t res = pass_a_sum(leafp, uold, y, s, S, head);
  if (res != kPlaced) return res;
  // step 2: exact gaps inside the recorded chunks
  for (uint32_t q = 0; q < s; q++) {
    if ((S.rpos[q * S.rs] >> 24) != kChunk) continue;
    place_key(leafp, uold, pick(y, q), q > 0 && pick(y, q - 1) == pick(y, q), S.rpos[q * S.rs],
              S.rval[q * S.rs], S.rcode[q * S.rs]);
  }
  return kPlaced;
}

// The same for leaves with codes of any length, eight bytes at a time with
// 64-bit values (the leaf walk's groups: Walk carries the element before the
// group and the code open at it).  Always kPlaced.
LT_HD uint32_t pass_a(const uint8_t* leafp, uint32_t uold, const uint64_t (&y)[kKeys], uint32_t s,
                      const ScratchLong& S, uint64_t& head) {
  uint32_t w[4], t[4], raw[4];
  ld16(leafp, raw);
  head = (uint64_t)raw[0] | ((uint64_t)raw[1] << 32);
  uint32_t k = 0;
  while (k < s && pick(y, k) <= head) {
    const uint64_t x = pick(y, k);
    const bool rep = k > 0 && pick(y, k - 1) == x;
    const uint32_t kind = rep ? kSkip : x == head ? kHit : kHead;
    S.rpos[k * S.rs] = 0u | (8u << 12) | (kind << 24);
    S.rval[k * S.rs] = head;
    S.rcode[k * S.rs] = 0u;
    k++;
  }
  // step 1: every key gets the group that reaches it and the walk's state there
  uint64_t ycur = k < s ? pick(y, k) : ~0ull;
  leafwalk::Walk c;
  c.val = head;
  auto group = [&](uint32_t p0, int i) {
    const leafwalk::Walk c0 = c;
    uint32_t T;
    uint64_t ss;
    leafwalk::group_sum(w[i], w[i + 1], t[i], t[i + 1], c, T, ss);
    while (k < s && ycur <= c.val) {
      S.rpos[k * S.rs] = p0 | ((c0.sh / 7u) << 12) | (kChunk << 24);
      S.rval[k * S.rs] = c0.val;
      S.rcode[k * S.rs] = c0.acc;
      k++;
      ycur = k < s ? pick(y, k) : ~0ull;
    }
  };
  for (uint32_t p0 = 0; p0 < uold && k < s; p0 += 16) {
    leafwalk::next_chunk(leafp, p0, uold, raw, w, t);
    if (p0) group(p0, 0);
    if (p0 + 8u < uold) group(p0 + 8u, 2);
  }
  // step 2: exact gaps inside the recorded groups
  for (uint32_t q = 0; q < k; q++) {
    const uint32_t rp = S.rpos[q * S.rs];
    if ((rp >> 24) != kChunk) continue;  // placed (head keys, or by an earlier group)
    const uint32_t p0 = rp & 0xFFFu, g0 = (rp >> 12) & 0xFFFu;
    uint64_t val = S.rval[q * S.rs], acc = S.rcode[q * S.rs];
    uint32_t sh = 7u * g0, cs = p0 - g0;
    uint32_t q1 = q + 1;
    while (q1 < k && S.rpos[q1 * S.rs] == rp) q1++;
    uint64_t yc = pick(y, q);
    uint32_t qq = q;
    for (uint32_t b = 0; b < 8u && p0 + b < uold && qq < q1; b++) {
      const uint32_t ch = leafp[p0 + b];
      acc |= (uint64_t)(ch & 0x7Fu) << sh;
      if (ch & 0x80u) {
        sh += 7u;
        continue;
      }
      val += acc;
      const uint32_t ce = p0 + b + 1u;
      while (qq < q1 && yc <= val) {
        const bool rep = qq > 0 && pick(y, qq - 1) == yc;
        const uint32_t kind = rep ? kSkip : yc == val ? kHit : kGap;
        S.rpos[qq * S.rs] = cs | (ce << 12) | (kind << 24);
        S.rval[qq * S.rs] = val;
        S.rcode[qq * S.rs] = acc;
        qq++;
        if (qq < q1) yc = pick(y, qq);
      }
      acc = 0;
      sh = 0;
      cs = ce;
    }
    q = q1 - 1;
  }
  for (; k < s; k++) {
    const uint64_t x = pick(y, k);
    const bool rep = k > 0 && pick(y, k - 1) == x;
    S.rpos[k * S.rs] = uold | (uold << 12) | ((rep ? kSkip : kAfter) << 24);
    S.rval[k * S.rs] = c.val;
    S.rcode[k * S.rs] = 0u;
  }
  return kPlaced;
}

// The edits of inserting the sorted slice y[0..s) (1 <= s <= kKeys, repeats
// allowed), placed by pass A, into the leaf at leafp (uold >= 8 used bytes, m
// elements, LB bytes, 16-byte aligned).  Returns one of the results above
// and writes nothing; kWritten means the leaf is to be rewritten (R.wlo ..
// R.whi, the R.E edits in S).
template <class SC>
LT_HD uint32_t plan_insert(uint32_t LB, uint32_t uold, uint32_t m, const uint64_t (&y)[kKeys],
                           uint32_t s, uint64_t head, const SC& S, Result& R) {
  // ---- edits: new keys grouped by the gap they fall in ----
  uint32_t E = 0, nn = 0, added = 0, mc = 0;
  int32_t tot = 0;
  uint64_t newhead = head;
  for (uint32_t q = 0; q < s;) {
    const uint32_t rp = S.rpos[q * S.rs];
    const uint32_t kind = rp >> 24;
    if (no_insert(kind)) { q++; continue; }
    // keys q..q1 (kSkip ones among them are repeats) share this gap
    const uint32_t os = rp & 0xFFFu, oe = (rp >> 12) & 0xFFFu;
    const uint64_t rv = S.rval[q * S.rs];
    uint64_t prev = pick(y, q);
    uint32_t nl, cl = 0;
    if (kind == kHead) { nl = 8u; newhead = prev; }
    else if (kind == kGap) nl = cl = leb_bytes(prev - (rv - S.rcode[q * S.rs]));
    else nl = cl = leb_bytes(prev - rv);
    mc = mc > cl ? mc : cl;
    added |= 1u << q;
    nn++;
    uint32_t q1 = q + 1;
    for (; q1 < s; q1++) {
      const uint32_t rp1 = S.rpos[q1 * S.rs];
      if ((rp1 & 0xFFFu) != os) break;
      if (no_insert(rp1 >> 24)) continue;
      const uint64_t x = pick(y, q1);
      cl = leb_bytes(x - prev);
      mc = mc > cl ? mc : cl;
      nl += cl;
      prev = x;
      added |= 1u << q1;
      nn++;
    }
    if (kind != kAfter) {  // the old successor (head or code end)
      cl = leb_bytes(rv - prev);
      mc = mc > cl ? mc : cl;
      nl += cl;
    }
    tot += (int32_t)nl - (int32_t)(oe - os);
    S.epos[E * S.rs] = os | (oe << 12) | (kind << 24);
    S.esa[E * S.rs] = tot;
    S.ekey[E * S.rs] = q | (q1 << 8) | (nl << 16);
    E++;
    q = q1;
  }
  R.added = added;
  R.maxcode = mc;
  R.newc = m + nn;
  R.nb = (uint32_t)((int32_t)uold + tot);
  R.newhead = newhead;
  R.E = E;
  if (nn == 0) return kUnchanged;
  if (R.nb > LB) return kTooBig;
  R.wlo = (S.epos[0] & 0xFFFu) & ~15u;
  R.whi = (R.nb + 15u) & ~15u;
  return kWritten;
}

// Chunk o of the rewritten leaf from segment cur (destination [slo, shi), shift
// ssa) and, where it starts inside the chunk, the ones before it.  Bytes of
// edits are left as they fall (their own bytes are written last); bytes past
// the new used ones (shi of the last segment) are zero.
// kept: null, or the block read for the chunk after this one (next_chunk_at).
template <class SC>
LT_HD void build_chunk(const uint8_t* leafp, uint32_t LB, uint32_t uold, const SC& S, uint32_t E,
                       uint32_t os0, int cur, int32_t slo, int32_t shi, int32_t ssa, int32_t o,
                       Block* kept, uint32_t (&r)[4]) {
  if (kept) next_chunk_at(leafp, LB, o - ssa, *kept, r);
  else chunk_at(leafp, LB, o - ssa, r);
  if (o + 16 > shi && cur + 1 == (int)E) {
    const uint32_t zero[4] = {0u, 0u, 0u, 0u};
    take_bytes(r, zero, shi > o ? (uint32_t)(shi - o) : 0u, 16u);
  }
  while (slo > o && cur >= 0) {
    cur--;
    seg_bounds(S, E, uold, os0, cur, slo, shi, ssa);
    if (shi <= o) break;  // wholly below this chunk: so are the earlier ones
    uint32_t x[4];
    chunk_at(leafp, LB, o - ssa, x);
    take_bytes(r, x, 0u, shi - o < 16 ? (uint32_t)(shi - o) : 16u);
  }
}

// Pass B by one thread: the chunks R.wlo .. R.whi of the leaf from the end
// backwards, each built from the segments that land in it and stored whole.
// Every chunk is one shifted read, whatever segment it lies in; the one an
// edit falls into merges a second (with one or two keys in most leaves, some
// lane of every warp is at such a chunk in every step, so that is all a step
// may cost).  1e6 keys into 1e8, the kernel: 290 us gathering those chunks
// segment by segment, 254 so; 230 then became 197 with one 16-byte load per
// chunk instead of five words (32 lanes' loads hit 32 lines; the deletes' way,
// forwards, gained nothing: 189 and 193).
template <class SC>
LT_HD void rewrite_leaf(uint8_t* leafp, uint32_t LB, uint32_t uold, const SC& S,
                        const Result& R) {
  const uint32_t E = R.E;
  const uint32_t os0 = S.epos[0] & 0xFFFu;
  int cur = (int)E - 1;  // the highest segment not wholly above chunk o
  int32_t slo, shi, ssa;
  seg_bounds(S, E, uold, os0, cur, slo, shi, ssa);
  Block kept;
  for (int32_t o = (int32_t)R.whi - 16; o >= (int32_t)R.wlo; o -= 16) {
    while (cur >= 0 && slo >= o + 16) {
      cur--;
      seg_bounds(S, E, uold, os0, cur, slo, shi, ssa);
    }
    uint32_t r[4];
    build_chunk(leafp, LB, uold, S, E, os0, cur, slo, shi, ssa, o, &kept, r);
    st16(leafp + o, r);
  }
}

// The edits' own bytes (new head, split codes), after the chunks are stored.
template <class SC>
LT_HD void write_edits(uint8_t* leafp, const uint64_t (&y)[kKeys], const SC& S,
                       const Result& R) {
  for (uint32_t e = 0; e < R.E; e++) {
    const uint32_t ep = S.epos[e * S.rs], ek = S.ekey[e * S.rs];
    const uint32_t kind = ep >> 24, os = ep & 0xFFFu;
    const uint32_t q0 = ek & 0xFFu, q1 = (ek >> 8) & 0xFFu;
    const int32_t sb = e ? S.esa[(e - 1) * S.rs] : 0;
    uint8_t* p = leafp + (int32_t)os + sb;
    const uint64_t rv = S.rval[q0 * S.rs];
    uint64_t prev = pick(y, q0);
    if (kind == kHead) {
#pragma unroll
      for (int i = 0; i < 8; i++) p[i] = (uint8_t)(prev >> (8 * i));
      p += 8;
    } else if (kind == kGap) {
      p += leb_write(p, prev - (rv - S.rcode[q0 * S.rs]));
    } else {
      p += leb_write(p, prev - rv);
    }
    for (uint32_t q = q0 + 1; q < q1; q++) {
      if (no_insert(S.rpos[q * S.rs] >> 24)) continue;
      const uint64_t x = pick(y, q);
      p += leb_write(p, x - prev);
      prev = x;
    }
    if (kind != kAfter) leb_write(p, rv - prev);
  }
}

// ---------------------------------------------------------------------------
// Delete.  Keys equal to elements (kHit) whose codes are adjacent form a run;
// a run's edit replaces the codes of its elements and of the element after
// it (the successor) by one code: successor minus the element before the run
// (Sec. 3: the neighbours of a removed key become neighbours), or, for a run
// that starts at the head, the successor as the new 8-byte head; a run that
// reaches the last element just goes.  Such an edit never grows the leaf
// (the merged delta needs no more bytes than the two it replaces), so the
// rewrite runs forward.
// ---------------------------------------------------------------------------

// Unsigned LEB128 code at p (at most 10 bytes): value, and its length in len.
LT_HD uint64_t leb_read(const uint8_t* p, uint32_t& len) {
  uint64_t v = 0;
  uint32_t n = 0;
  for (;;) {
    const uint32_t c = p[n];
    v |= (uint64_t)(c & 0x7Fu) << (7u * n);
    n++;
    if (!(c & 0x80u) || n == 10u) break;
  }
  len = n;
  return v;
}

// The edits of deleting the sorted slice y[0..s) (1 <= s <= kKeys, repeats
// allowed), placed by pass A, from the leaf (as plan_insert).  R.added: bit q =
// slice key q was removed; R.wlo .. R.whi covers the old used bytes from the
// first edit on, so the bytes freed at the end are cleared.
template <class SC>
LT_HD uint32_t plan_delete(const uint8_t* leafp, uint32_t uold, uint32_t m,
                           const uint64_t (&y)[kKeys], uint32_t s, uint64_t head, const SC& S,
                           Result& R) {
  uint32_t E = 0, nn = 0, removed = 0;
  int32_t tot = 0;
  uint64_t newhead = head;
  for (uint32_t q = 0; q < s;) {
    const uint32_t rp = S.rpos[q * S.rs];
    if ((rp >> 24) != kHit) { q++; continue; }
    const uint32_t os = rp & 0xFFFu;
    uint32_t ce = (rp >> 12) & 0xFFFu;
    const uint64_t pred = S.rval[q * S.rs] - S.rcode[q * S.rs];  // unused when os == 0
    uint64_t lastv = S.rval[q * S.rs];
    removed |= 1u << q;
    nn++;
    uint32_t q1 = q + 1;
    for (; q1 < s; q1++) {
      const uint32_t r1 = S.rpos[q1 * S.rs], k1 = r1 >> 24;
      if (k1 == kSkip) continue;          // a repeat
      if ((r1 & 0xFFFu) != ce) break;     // beyond the successor's code
      if (k1 != kHit) continue;           // absent, in the gap before the successor
      ce = (r1 >> 12) & 0xFFFu;           // the successor itself goes: the run grows
      lastv = S.rval[q1 * S.rs];
      removed |= 1u << q1;
      nn++;
    }
    uint32_t oe = uold, nl = 0;
    uint64_t nv = 0;
    if (ce < uold) {  // the successor's code: right after the run
      uint32_t dl;
      const uint64_t succ = lastv + leb_read(leafp + ce, dl);
      oe = ce + dl;
      if (os == 0) {
        nl = 8u;
        nv = succ;
        newhead = succ;
      } else {
        nv = succ - pred;
        nl = leb_bytes(nv);
      }
    }
    tot += (int32_t)nl - (int32_t)(oe - os);
    S.epos[E * S.rs] = os | (oe << 12) | ((os == 0 ? kHead : kGap) << 24);
    S.esa[E * S.rs] = tot;
    S.ekey[E * S.rs] = q | (q1 << 8) | (nl << 16);
    S.rval[q * S.rs] = nv;  // what the edit writes (the record is used up)
    E++;
    q = q1;
  }
  R.added = removed;
  R.maxcode = 0;
  R.newc = m - nn;
  R.nb = (uint32_t)((int32_t)uold + tot);
  R.newhead = R.newc ? newhead : ~0ull;
  R.E = E;
  if (nn == 0) return kUnchanged;
  R.wlo = (S.epos[0] & 0xFFFu) & ~15u;
  R.whi = (uold + 15u) & ~15u;
  return kWritten;
}

// Pass B of a delete by one thread: the chunks R.wlo .. R.whi from the front
// (every shift is <= 0, so a chunk's sources lie at or above it: not yet
// written), each built as in rewrite_leaf; the chunks past the new used bytes
// are cleared.
template <class SC>
LT_HD void rewrite_forward(uint8_t* leafp, uint32_t LB, uint32_t uold, const SC& S,
                           const Result& R) {
  const uint32_t E = R.E;
  const uint32_t os0 = S.epos[0] & 0xFFFu;
  int cur = -1;  // the highest segment that starts at or before the chunk's end
  int32_t slo = 0, shi = (int32_t)os0, ssa = 0;
  for (int32_t o = (int32_t)R.wlo; o < (int32_t)R.whi; o += 16) {
    while (cur + 1 < (int)E) {
      int32_t lo2, hi2, sa2;
      seg_bounds(S, E, uold, os0, cur + 1, lo2, hi2, sa2);
      if (lo2 >= o + 16) break;
      cur++;
      slo = lo2;
      shi = hi2;
      ssa = sa2;
    }
    uint32_t r[4];
    build_chunk(leafp, LB, uold, S, E, os0, cur, slo, shi, ssa, o, nullptr, r);
    st16(leafp + o, r);
  }
}

// The delete edits' own bytes: a new head, or the merged code.
template <class SC>
LT_HD void write_delete_edits(uint8_t* leafp, const SC& S, const Result& R) {
  for (uint32_t e = 0; e < R.E; e++) {
    const uint32_t ep = S.epos[e * S.rs], ek = S.ekey[e * S.rs];
    const uint32_t nl = ek >> 16;
    if (!nl) continue;
    const uint32_t q0 = ek & 0xFFu, os = ep & 0xFFFu;
    const int32_t sb = e ? S.esa[(e - 1) * S.rs] : 0;
    uint8_t* p = leafp + (int32_t)os + sb;
    const uint64_t nv = S.rval[q0 * S.rs];
    if ((ep >> 24) == kHead) {
#pragma unroll
      for (int i = 0; i < 8; i++) p[i] = (uint8_t)(nv >> (8 * i));
    } else {
      leb_write(p, nv);
    }
  }
}

// Pass A and the edits (DEL: of the delete) by one thread.
template <bool DEL, class SC>
LT_HD uint32_t plan(const uint8_t* leafp, uint32_t LB, uint32_t uold, uint32_t m,
                    const uint64_t (&y)[kKeys], uint32_t s, const SC& S, Result& R) {
  uint64_t head;
  const uint32_t res = pass_a(leafp, uold, y, s, S, head);
  if (res != kPlaced) return res;
  return DEL ? plan_delete(leafp, uold, m, y, s, head, S, R)
             : plan_insert(LB, uold, m, y, s, head, S, R);
}

template <class SC>
LT_HD uint32_t delete_leaf(uint8_t* leafp, uint32_t LB, uint32_t uold, uint32_t m,
                           const uint64_t (&y)[kKeys], uint32_t s, const SC& S,
                           Result& R) {
  const uint32_t res = plan<true>(leafp, LB, uold, m, y, s, S, R);
  if (res == kWritten) {
    rewrite_forward(leafp, LB, uold, S, R);
    write_delete_edits(leafp, S, R);
  }
  return res;
}

// All of it by one thread: returns one of the results above; the leaf is
// written only for kWritten.
template <class SC>
LT_HD uint32_t insert_leaf(uint8_t* leafp, uint32_t LB, uint32_t uold, uint32_t m,
                           const uint64_t (&y)[kKeys], uint32_t s, const SC& S,
                           Result& R) {
  const uint32_t res = plan<false>(leafp, LB, uold, m, y, s, S, R);
  if (res == kWritten) {
    rewrite_leaf(leafp, LB, uold, S, R);
    write_edits(leafp, y, S, R);
  }
  return res;
}

}  // namespace leafthr
