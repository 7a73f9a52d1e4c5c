// One thread's walk over a byte-code leaf (Sec. 5 leaf format: an 8-byte
// little-endian head, then the deltas to the following keys as unsigned
// LEB128 codes, packed left), eight bytes ("a group") at a time.
//
// Inside a group each byte adds its payload times 128^(bytes before it in its
// code) to acc, and acc is not cleared at a terminator: at the k-th terminator
// of the group it holds the bits of every code closed so far in the group
// (plus the open code carried in), so the element closed there is val + acc.
// A group of T terminators therefore adds T * val + sum_k acc_k to a sum of
// elements, val moves on by the acc of its last terminator, and acc keeps only
// the open code's bits.  While no code has more than 4 bytes everything in a
// group fits 32 bits (at most 11 payload bytes feed it and sum_k acc_k <
// 9 * 2^28); a group that a longer code touches -- four continuation bytes in
// a row end in it, or the code carried in has four already -- takes 64 bits,
// byte by byte for codes of 5 bytes (edges u << 32 | v), code by code for
// longer ones (64-bit hashes).  The lanes of a warp agree on the form (a vote
// per group): a set whose codes are all short never pays for the others.
// 1e5 scans of 64-bit keys: 172 us byte by byte, 137 us code by code; degrees
// of 2^20 vertices: 484 and 536 us, so codes of 5 bytes stay byte by byte.
//
// Which bytes end a code is passed in (term flags, bit 7 of each byte), so
// bytes past the leaf's used ones are neither codes nor terminators.
//
// The functions are __host__ __device__ so that the same code can be run on
// the host.
#pragma once
#include "leaf_bits.cuh"

namespace leafwalk {

using leafthr::bmask4;
using leafthr::byte_of;
using leafthr::fshl;
using leafthr::ld16;
using leafthr::popc;

constexpr uint32_t kFlags = 0x80808080u;

struct Walk {
  uint64_t val = 0;  // the last element closed
  uint64_t acc = 0;  // bits of the open code
  uint32_t sh = 0;   // 7 * its bytes
  uint32_t c = 0;    // continuation flags of the word before
  uint32_t y = 0;    // c with the byte before it a continuation byte too
};

LT_HD bool any_lane(bool p) {
#if defined(__CUDA_ARCH__)
  return __any_sync(__activemask(), p);
#else
  return p;
#endif
}

// The longest codes that touch the group (wa, wb), over the lanes: 0 = at most
// 4 bytes, 1 = 5, 2 = more.  Moves the flags carried in k on.
LT_HD int group_form(uint32_t wa, uint32_t wb, Walk& k) {
  const uint32_t ca = wa & kFlags, cb = wb & kFlags;
  const uint32_t ya = ca & fshl(k.c, ca, 8), yb = cb & fshl(ca, cb, 8);
  const uint32_t za = ya & fshl(k.y, ya, 16), zb = yb & fshl(ya, yb, 16);  // 4 in a row
  const uint32_t z5 = (za & k.c) | (zb & ca);
  k.c = cb;
  k.y = yb;
  if (!any_lane((za | zb) != 0u || k.sh >= 28u)) return 0;
  return any_lane(z5 != 0u || k.sh > 28u) ? 2 : 1;
}

// The group in 32 bits, byte by byte (form 0): step(acc) after each code closed.
template <class D>
LT_HD void short_codes(uint32_t pa, uint32_t pb, uint32_t ta, uint32_t tb, Walk& k, D&& done) {
  uint32_t acc = (uint32_t)k.acc, pw = 1u << k.sh, r = 0;
#pragma unroll
  for (int b = 0; b < 8; b++) {
    acc += byte_of(b < 4 ? pa : pb, b & 3) * pw;
    const bool term = ((b < 4 ? ta : tb) & (0x80u << (8 * (b & 3)))) != 0u;
    if (term) done(acc);
    r = term ? acc : r;
    pw = term ? 1u : pw << 7;
  }
  k.val += r;
  k.acc = acc - r;
  k.sh = 31u - leafthr::clz32(pw);
}

// The same with a 64-bit sum of 32-bit products, for codes of up to 5 bytes
// (form 1).
template <class D>
LT_HD void medium_codes(uint32_t pa, uint32_t pb, uint32_t ta, uint32_t tb, Walk& k, D&& done) {
  uint64_t acc = k.acc, r = 0;
  uint32_t pw = 1u << k.sh;
#pragma unroll
  for (int b = 0; b < 8; b++) {
    acc += (uint64_t)byte_of(b < 4 ? pa : pb, b & 3) * pw;
    const bool term = ((b < 4 ? ta : tb) & (0x80u << (8 * (b & 3)))) != 0u;
    if (term) done(acc);
    r = term ? acc : r;
    pw = term ? 1u : pw << 7;
  }
  k.val += r;
  k.acc = acc - r;
  k.sh = 31u - leafthr::clz32(pw);
}

// Codes of any length (form 2): the payloads packed to 56 bits once, then one
// step per code closed -- codes this long leave few in a group.  done(acc)
// after each, acc its element less the val the group was entered with.
template <class D>
LT_HD void long_codes(uint32_t pa, uint32_t pb, uint32_t ta, uint32_t tb, Walk& k, D&& done) {
  using leafthr::dp4a;
  const uint32_t lo = dp4a(pa, 0x00008001u, 0u) + (dp4a(pa, 0x80010000u, 0u) << 14);
  const uint32_t hi = dp4a(pb, 0x00008001u, 0u) + (dp4a(pb, 0x80010000u, 0u) << 14);
  const uint64_t v = (uint64_t)lo | ((uint64_t)hi << 28);
  // terminators as bits 0..7
  uint32_t t = ((((ta >> 7) * 0x01020408u) >> 24) & 0xFu) |
               (((((tb >> 7) * 0x01020408u) >> 24) & 0xFu) << 4);
  uint64_t acc = k.acc, cum = 0;
  uint32_t sh = k.sh & 63u, pos = 0;
  while (t) {
    const uint32_t e = 7u * leafthr::ctz32(t) + 7u;
    cum += acc | (((v >> pos) & ((1ull << (e - pos)) - 1ull)) << sh);
    done(cum);
    acc = 0;
    sh = 0;
    pos = e;
    t &= t - 1u;
  }
  k.val += cum;
  k.acc = acc | ((v >> pos) << sh);
  k.sh = sh + 56u - pos;
}

// The group (wa, wb) with terminators ta, tb: T = elements closed, ss = the
// sum of (element - val), each against the val the group was entered with,
// which k.val then leaves behind.
LT_HD void group_sum(uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb, Walk& k, uint32_t& T,
                     uint64_t& ss) {
  const uint32_t pa = wa & 0x7F7F7F7Fu, pb = wb & 0x7F7F7F7Fu;
  T = popc(ta) + popc(tb);
  const int form = group_form(wa, wb, k);
  if (form == 0) {
    uint32_t s32 = 0;
    short_codes(pa, pb, ta, tb, k, [&](uint32_t acc) { s32 += acc; });
    ss = s32;
  } else {
    uint64_t s64 = 0;
    if (form == 1) medium_codes(pa, pb, ta, tb, k, [&](uint64_t acc) { s64 += acc; });
    else long_codes(pa, pb, ta, tb, k, [&](uint64_t acc) { s64 += acc; });
    ss = s64;
  }
}

// The same group, f(element) called for each element it closes, in order.
template <class F>
LT_HD void group_visit(uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb, Walk& k, F&& f) {
  const uint32_t pa = wa & 0x7F7F7F7Fu, pb = wb & 0x7F7F7F7Fu;
  const uint64_t v = k.val;
  const int form = group_form(wa, wb, k);
  if (form == 0) short_codes(pa, pb, ta, tb, k, [&](uint32_t acc) { f(v + acc); });
  else if (form == 1) medium_codes(pa, pb, ta, tb, k, [&](uint64_t acc) { f(v + acc); });
  else long_codes(pa, pb, ta, tb, k, [&](uint64_t acc) { f(v + acc); });
}

// The 16 bytes of the leaf at p0 (zero past the u used ones) and which of
// them end a code.
LT_HD void load_chunk(const uint8_t* leafp, uint32_t p0, uint32_t u, uint32_t (&w)[4],
                      uint32_t (&t)[4]) {
  ld16(leafp + p0, w);
  if (p0 + 16u > u) {
    const uint32_t keep = u > p0 ? (1u << (u - p0)) - 1u : 0u;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const uint32_t m = bmask4((keep >> (4 * i)) & 0xFu);
      w[i] &= m;
      t[i] = ~w[i] & kFlags & m;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; i++) t[i] = ~w[i] & kFlags;
  }
}

// load_chunk for a loop over the leaf: w holds the raw chunk at p0, and the
// next one is loaded before this one is decoded.
LT_HD void next_chunk(const uint8_t* leafp, uint32_t p0, uint32_t u, uint32_t (&raw)[4],
                      uint32_t (&w)[4], uint32_t (&t)[4]) {
#pragma unroll
  for (int i = 0; i < 4; i++) w[i] = raw[i];
  if (p0 + 16u < u) ld16(leafp + p0 + 16u, raw);
  if (p0 + 16u > u) {
    const uint32_t keep = u > p0 ? (1u << (u - p0)) - 1u : 0u;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const uint32_t m = bmask4((keep >> (4 * i)) & 0xFu);
      w[i] &= m;
      t[i] = ~w[i] & kFlags & m;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; i++) t[i] = ~w[i] & kFlags;
  }
}

LT_HD uint64_t leaf_head(const uint8_t* leafp) {
  uint32_t w[4];
  ld16(leafp, w);
  return (uint64_t)w[0] | ((uint64_t)w[1] << 32);
}

// 32 bytes at p (32-byte aligned) in one load.
LT_HD void ld32(const uint8_t* p, uint32_t (&a)[4], uint32_t (&b)[4]) {
#if defined(__CUDA_ARCH__)
  const ulonglong4_32a v = *reinterpret_cast<const ulonglong4_32a*>(p);
  a[0] = (uint32_t)v.x; a[1] = (uint32_t)(v.x >> 32);
  a[2] = (uint32_t)v.y; a[3] = (uint32_t)(v.y >> 32);
  b[0] = (uint32_t)v.z; b[1] = (uint32_t)(v.z >> 32);
  b[2] = (uint32_t)v.w; b[3] = (uint32_t)(v.w >> 32);
#else
  ld16(p, a);
  ld16(p + 16, b);
#endif
}

// ---- sum of a whole leaf ----
//
// With m elements, head h, and for every byte b of codes its payload p_b, the
// bytes g_b before it in its code and the terminators R_b at or after it, the
// sum of the elements is m h + sum_b p_b 128^g_b R_b: a byte counts in every
// element from its own on.  While no code has more than 4 bytes that is four
// sums of byte products,
//   A0 + 127 A1 + (128^2 - 128) A2 + (128^3 - 128^2) A3,
//   Ai = sum of p_b R_b over the bytes with g_b >= i,
// each a dp4a per word that accumulates in 32 bits over the leaf (p R < 2^15,
// at most 2040 bytes), with no carry from byte to byte but the continuation
// flags: 24 integer operations per word, and neither elements nor 64-bit
// values inside the loop.  R_b fits a byte when the leaf has at most 255
// codes; with more, R_b = (codes from the 128-byte block on) - (terminators of
// the block before b), the first times the block's plain sum (four more dp4a
// per word).
//
// The leaf's first codes tell a set with codes over 4 bytes: such leaves are
// walked group by group instead.  One whose first long code comes later is
// walked after all.
//
// Measured on a full scan of 1e8 keys (0.9e6 leaves of 512 bytes, 250 used):
// 70 us against 114 us for a loop over the bytes with a running value
// (9 operations a byte), which the integer ALU pipe bounded.  87 us with all
// four planes; 83 with the two or three that the leaf's span allows; 79 with
// 32-byte loads (each lane's loads hit a line of their own, so their number
// counts); 70 with the next 32 bytes on their way and 64 registers.

// Bit 7 of each byte -> 0x00 / 0xFF.
LT_HD uint32_t spread(uint32_t q) {
#if defined(__CUDA_ARCH__)
  uint32_t r;
  asm("prmt.b32 %0, %1, %1, 0xBA98;" : "=r"(r) : "r"(q));  // sign of each byte
  return r;
#else
  return ((q & kFlags) >> 7) * 0xFFu;
#endif
}

LT_HD uint32_t top_byte4(uint32_t x) {  // its top byte in all four
#if defined(__CUDA_ARCH__)
  return __byte_perm(x, 0u, 0x3333u);
#else
  return (x >> 24) * 0x01010101u;
#endif
}

// What one word of codes leaves to the next: flags (continuation, and byte
// index in its code >= 1, 2), and whether a code of more than 4 bytes was met.
struct WordFlags {
  uint32_t c = 0, q1 = 0, q2 = 0, lng = 0;
};

// Masks of the word's bytes with g >= 1, 2, 3 (those of the first N planes), and
// its terminators as bytes 0 / 1 prefix-summed (inclusive).  With N < 4 no code
// has more than N bytes.
template <int N>
LT_HD void word_masks(uint32_t w, WordFlags& f, uint32_t& m1, uint32_t& m2, uint32_t& m3,
                      uint32_t& P) {
  const uint32_t c = w & kFlags;
  const uint32_t q1 = fshl(f.c, c, 8);
  const uint32_t q2 = N > 2 ? q1 & fshl(f.q1, q1, 8) : 0u;
  const uint32_t q3 = N > 3 ? q2 & fshl(f.q2, q2, 8) : 0u;
  if (N > 3) f.lng |= q3 & c;
  f.c = c;
  f.q1 = q1;
  f.q2 = q2;
  m1 = spread(q1);
  m2 = N > 2 ? spread(q2) : 0u;
  m3 = N > 3 ? spread(q3) : 0u;
  P = (~(w >> 7) & 0x01010101u) * 0x01010101u;
}

LT_HD uint64_t plane_sum(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3) {
  return a0 + 127ull * a1 + 16256ull * a2 + 2080768ull * a3;
}

// Leaf of m - 1 <= 255 codes, none over N bytes if N < 4.  false: it has a code
// of more than 4 bytes.
template <int N>
LT_HD bool sum_few(const uint8_t* leafp, uint32_t u, uint32_t m, uint64_t& s) {
  WordFlags f;
  uint32_t R = (m - 1u) * 0x01010101u;  // R of the next byte, in all four
  uint32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;
  auto word = [&](uint32_t w) {
    uint32_t m1, m2, m3, P;
    word_masks<N>(w, f, m1, m2, m3, P);
    const uint32_t r = R - (P << 8);  // bytes past the last code go below zero:
    R -= top_byte4(P);                // they borrow upwards only, and are zero
    const uint32_t p = w & 0x7F7F7F7Fu;
    a0 = leafthr::dp4a(p, r, a0);
    a1 = leafthr::dp4a(p, r & m1, a1);
    if (N > 2) a2 = leafthr::dp4a(p, r & m2, a2);
    if (N > 3) a3 = leafthr::dp4a(p, r & m3, a3);
  };
  uint32_t w[4], w2[4];
  // 32 bytes (one sector) per step: both halves are loaded before either is
  // decoded, so each sector is requested once
  const bool wide = (reinterpret_cast<uintptr_t>(leafp) & 31u) == 0;
  uint32_t n1[4], n2[4];
  auto load = [&](uint32_t p0) {
    if (p0 >= u) return;
    const bool two = p0 + 16u < u;
    if (wide && two) {
      ld32(leafp + p0, n1, n2);
    } else {
      ld16(leafp + p0, n1);
      if (two) ld16(leafp + p0 + 16u, n2);
    }
  };
  load(0);
  for (uint32_t p0 = 0; p0 < u; p0 += 32) {
    const bool two = p0 + 16u < u;
#pragma unroll
    for (int i = 0; i < 4; i++) { w[i] = n1[i]; w2[i] = n2[i]; }
    load(p0 + 32u);
    if (p0) {
      word(w[0]);
      word(w[1]);
    } else {
      s = m * ((uint64_t)w[0] | ((uint64_t)w[1] << 32));
    }
    word(w[2]);
    word(w[3]);
    if (two) {
#pragma unroll
      for (int i = 0; i < 4; i++) word(w2[i]);
    }
  }
  s += plane_sum(a0, a1, a2, a3);
  return f.lng == 0u;
}

// The same for any number of codes, in blocks of 128 bytes.
LT_HD bool sum_many(const uint8_t* leafp, uint32_t u, uint32_t m, uint64_t& s) {
  WordFlags f;
  const uint64_t h = leaf_head(leafp);
  s = m * h;
  uint32_t before = 0;  // codes before the block
  for (uint32_t b0 = 0; b0 < u; b0 += 128) {
    uint32_t B = 0;  // terminators of the block before the next byte, in all four
    uint32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0, d0 = 0, d1 = 0, d2 = 0, d3 = 0;
    const uint32_t be = b0 + 128u < u ? b0 + 128u : u;
    for (uint32_t p0 = b0; p0 < be; p0 += 16) {
      uint32_t w[4];
      ld16(leafp + p0, w);
#pragma unroll
      for (int i = 0; i < 4; i++) {
        if (i < 2 && p0 == 0) continue;  // the head
        uint32_t m1, m2, m3, P;
        word_masks<4>(w[i], f, m1, m2, m3, P);
        const uint32_t r = B + (P << 8);
        B += top_byte4(P);
        const uint32_t p = w[i] & 0x7F7F7F7Fu;
        a0 = leafthr::dp4a(p, r, a0);
        a1 = leafthr::dp4a(p, r & m1, a1);
        a2 = leafthr::dp4a(p, r & m2, a2);
        a3 = leafthr::dp4a(p, r & m3, a3);
        d0 = leafthr::dp4a(p, 0x01010101u, d0);
        d1 = leafthr::dp4a(p, m1 & 0x01010101u, d1);
        d2 = leafthr::dp4a(p, m2 & 0x01010101u, d2);
        d3 = leafthr::dp4a(p, m3 & 0x01010101u, d3);
      }
    }
    s += (uint64_t)(m - 1u - before) * plane_sum(d0, d1, d2, d3) - plane_sum(a0, a1, a2, a3);
    before += B & 0xFFu;
  }
  return f.lng == 0u;
}

// Sum of the elements of a leaf of u >= 8 used bytes.
LT_HD uint64_t sum_walked(const uint8_t* leafp, uint32_t u) {
  Walk k;
  k.val = leaf_head(leafp);
  uint64_t s = k.val;
  uint32_t raw[4];
  ld16(leafp, raw);
  for (uint32_t p0 = 0; p0 < u; p0 += 16) {
    uint32_t w[4], t[4], T;
    uint64_t ss, v;
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0) {  // bytes 0-7 are the head
      v = k.val;
      group_sum(w[0], w[1], t[0], t[1], k, T, ss);
      s += T * v + ss;
    }
    v = k.val;
    group_sum(w[2], w[3], t[2], t[3], k, T, ss);
    s += T * v + ss;
  }
  return s;
}

// Do four continuation bytes in a row end among the leaf's first 24 bytes of
// codes (words a, b, c)?
LT_HD bool long_in(uint32_t a, uint32_t b, const uint32_t (&c)[4]) {
  const uint32_t x[6] = {a, b, c[0], c[1], c[2], c[3]};
  uint32_t f = 0, y = 0, z = 0;
#pragma unroll
  for (int i = 0; i < 6; i++) {
    const uint32_t fi = x[i] & kFlags, yi = fi & fshl(f, fi, 8);
    z |= yi & fshl(y, yi, 16);
    f = fi;
    y = yi;
  }
  return z != 0u;
}

// The same for a leaf of m elements, whose bytes past u are zero; span: no two
// of its elements lie further apart (the next leaf's head less its own), which
// bounds its codes: below 2^21 they have at most 3 bytes, below 2^14 two, and
// the planes of the others are left out for a warp of such leaves.
LT_HD uint64_t leaf_sum(const uint8_t* leafp, uint32_t u, uint32_t m, uint64_t span) {
  if (!any_lane(m > 256u || span >= 1ull << 21)) {
    uint64_t s = 0;
    if (any_lane(span >= 1ull << 14)) sum_few<3>(leafp, u, m, s);
    else sum_few<2>(leafp, u, m, s);
    return s;
  }
  uint32_t w[4], w2[4] = {0u, 0u, 0u, 0u};
  ld16(leafp, w);
  if (u > 16u) ld16(leafp + 16, w2);
  uint64_t s;
  if (!any_lane(long_in(w[2], w[3], w2))) {
    const bool ok = any_lane(m > 256u) ? sum_many(leafp, u, m, s) : sum_few<4>(leafp, u, m, s);
    if (ok) return s;
  }
  return sum_walked(leafp, u);
}

// The walk's state at a byte of the leaf.
struct alignas(16) Mark {
  uint64_t val;  // the last element closed before it
  uint64_t sum;  // the sum of those elements, the head included (or as said)
  uint64_t acc;  // the open code, as in Walk
  uint32_t cnt;
  uint32_t sh;
};

// The flags carried in follow from the open code's bytes.
LT_HD Walk walk_at(const Mark& m) {
  Walk k;
  k.val = m.val;
  k.acc = m.acc;
  k.sh = m.sh;
  const uint32_t n = m.sh / 7u;  // continuation bytes right before it
  k.c = n >= 4u ? kFlags : n ? kFlags << (8u * (4u - n)) : 0u;
  k.y = n >= 5u ? kFlags : n > 1u ? kFlags << (8u * (5u - n)) : 0u;
  return k;
}

// Chunks of 16 bytes whose elements are all below x, passed over whole: k and
// n (the elements closed) move past them, raw holds the chunk at the byte
// returned, where the walk goes on.  From the leaf's start, raw its first
// chunk.  With codes of up to 5 bytes a chunk is five sums of byte products
// (payloads at position 0 to 4 of their code), no step per byte: about 110
// operations, 150 by groups of 8 while codes are short and 220 when a lane has
// a longer one.  (Not before a loop over the range itself, as in
// leaf_range_sum: a warp then takes its longest skip and its longest range one
// after the other; 1e5 ranges 189 -> 200 us.)  It stops before a chunk with a code of more than 5 bytes, and
// before the last, partial one.
LT_HD uint32_t skip_below(const uint8_t* leafp, uint32_t u, uint64_t x, Walk& k, uint32_t& n,
                          uint32_t (&raw)[4]) {
  using leafthr::dp4a;
  uint32_t c = 0, q1 = 0, q2 = 0, q3 = 0, lng = 0, p0 = 0;
  for (; p0 + 16u <= u; p0 += 16u) {
    uint32_t next[4] = {0u, 0u, 0u, 0u};
    if (p0 + 16u < u) ld16(leafp + p0 + 16u, next);  // on its way while this one is summed
    uint32_t s01 = 0, s23 = 0, s4 = 0, conts = 0, pay = 0, w01 = 0, w23 = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      if (i < 2 && p0 == 0) continue;  // the head
      const uint32_t cw = raw[i] & kFlags;
      const uint32_t b1 = fshl(c, cw, 8);  // position in its code >= 1, .. >= 4
      const uint32_t b2 = b1 & fshl(q1, b1, 8);
      const uint32_t b3 = b2 & fshl(q2, b2, 8);
      const uint32_t b4 = b3 & fshl(q3, b3, 8);
      lng |= b4 & cw;
      pay = raw[i] & 0x7F7F7F7Fu;
      w01 = ((~b1 & kFlags) >> 7) | (b1 ^ b2);
      w23 = ((b2 ^ b3) >> 7) | (b3 ^ b4);
      s01 = dp4a(pay, w01, s01);
      s23 = dp4a(pay, w23, s23);
      s4 = dp4a(pay, b4 >> 7, s4);
      conts += popc(cw);
      c = cw;
      q1 = b1;
      q2 = b2;
      q3 = b3;
    }
    // the open code: it starts in the last word, or lng is set
    const uint32_t tw = ~c & kFlags;
    const uint32_t ps = pay & (tw ? ~(0xFFFFFFFFu >> leafthr::clz32(tw)) : 0xFFFFFFFFu);
    const uint32_t open = dp4a(ps, w01, 0u) + (dp4a(ps, w23, 0u) << 14);
    const uint64_t end =
        k.val + (k.acc + s01 + ((uint64_t)s23 << 14) + ((uint64_t)s4 << 28) - open);
    if (lng || end >= x) break;
    n += (p0 ? 16u : 8u) - conts;
    k.val = end;
    k.acc = open;
    k.sh = tw ? 7u * (leafthr::clz32(tw) >> 3) : 28u;
    k.c = c;
    k.y = c & q1;
#pragma unroll
    for (int i = 0; i < 4; i++) raw[i] = next[i];
  }
  return p0;
}

// f(element) for every element of a leaf of u >= 8 used bytes, in order.
template <class F>
LT_HD void leaf_visit(const uint8_t* leafp, uint32_t u, F&& f) {
  Walk k;
  k.val = leaf_head(leafp);
  f(k.val);
  uint32_t raw[4];
  ld16(leafp, raw);
  for (uint32_t p0 = 0; p0 < u; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0) group_visit(w[0], w[1], t[0], t[1], k, f);
    group_visit(w[2], w[3], t[2], t[3], k, f);
  }
}

// Adds to s and c the sum and the number of the elements v of a leaf of u >= 8
// used bytes, none of whose codes has more than 4, with (v & mask) == value, a
// mask of the low 32 bits: no look at the codes' lengths, and per element the
// low word compared and 32 bits added.
LT_HD void leaf_masked_sum(const uint8_t* leafp, uint32_t u, uint32_t mask, uint32_t value,
                           uint64_t& s, uint64_t& c) {
  Walk k;
  k.val = leaf_head(leafp);
  if (((uint32_t)k.val & mask) == value) { s += k.val; c++; }
  auto group = [&](uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb) {
    const uint64_t v = k.val;
    uint32_t n = 0, s32 = 0;
    short_codes(wa & 0x7F7F7F7Fu, wb & 0x7F7F7F7Fu, ta, tb, k, [&](uint32_t acc) {
      if ((((uint32_t)v + acc) & mask) == value) { n++; s32 += acc; }
    });
    s += n * v + s32;
    c += n;
  };
  uint32_t raw[4];
  ld16(leafp, raw);
  for (uint32_t p0 = 0; p0 < u; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0) group(w[0], w[1], t[0], t[1]);
    group(w[2], w[3], t[2], t[3]);
  }
}

// f(element) for the elements that the walk k closes from byte p (a multiple
// of 8, past the head) on, until done() holds after a group.
template <class F, class D>
LT_HD void visit_from(const uint8_t* leafp, uint32_t u, uint32_t p, Walk k, F&& f, D&& done) {
  uint32_t p0 = p & ~15u;
  uint32_t raw[4];
  if (p0 < u) ld16(leafp + p0, raw);
  for (; p0 < u && !done(); p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0 >= p) group_visit(w[0], w[1], t[0], t[1], k, f);
    if (!done()) group_visit(w[2], w[3], t[2], t[3], k, f);
  }
}

// f(element) for the elements v with lo <= v < hi of a leaf of u >= 8 used
// bytes, in order.
template <class F>
LT_HD void leaf_range_visit(const uint8_t* leafp, uint32_t u, uint64_t lo, uint64_t hi, F&& f) {
  Walk k;
  k.val = leaf_head(leafp);
  if (k.val >= hi) return;
  uint32_t p = 8;
  if (k.val >= lo) {
    f(k.val);
  } else {
    uint32_t raw[4], n = 0;
    ld16(leafp, raw);
    p = skip_below(leafp, u, lo, k, n, raw);
    if (!p) p = 8;
  }
  uint64_t last = k.val;
  visit_from(leafp, u, p, k, [&](uint64_t v) {
    if (v >= lo && v < hi) f(v);
    last = v;
  }, [&] { return last >= hi; });
}

// A group set aside: the walk as it was before it, and its words.  The few
// groups that a bound falls into are decoded after the loop over the leaf, by
// all lanes of a warp together, instead of inside it, where each lane would
// stop the others at its own step.
struct Held {
  Walk k;
  uint32_t wa, wb, ta, tb;
};

// Sum and count of the elements v with lo <= v < hi of a leaf of u >= 8 used
// bytes, added to s and c.
LT_HD void leaf_range_sum(const uint8_t* leafp, uint32_t u, uint64_t lo, uint64_t hi, uint64_t& s,
                          uint64_t& c) {
  Walk k;
  k.val = leaf_head(leafp);
  if (k.val >= hi) return;
  bool open = k.val >= lo;  // every later element is >= lo
  if (open) { s += k.val; c++; }
  Held a, b;
  uint32_t held = 0;
  bool done = false;
  auto step = [&](uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb) {
    const Walk k0 = k;
    uint32_t T;
    uint64_t ss;
    group_sum(wa, wb, ta, tb, k, T, ss);
    if ((!open && k.val >= lo) || k.val >= hi) {  // at most two such groups
      const Held g{k0, wa, wb, ta, tb};
      if (!held) a = g;
      else b = g;
      held++;
      open = true;
      done = k.val >= hi;
    } else if (open) {
      s += T * k0.val + ss;
      c += T;
    }
  };
  uint32_t raw[4];
  ld16(leafp, raw);
  for (uint32_t p0 = 0; p0 < u && !done; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0) step(w[0], w[1], t[0], t[1]);
    if (!done) step(w[2], w[3], t[2], t[3]);
  }
  auto take = [&](uint64_t v) {
    if (v >= lo && v < hi) { s += v; c++; }
  };
  if (held) group_visit(a.wa, a.wb, a.ta, a.tb, a.k, take);
  if (held > 1) group_visit(b.wa, b.wb, b.ta, b.tb, b.k, take);
}

// The first `most` elements >= lo of a leaf of u >= 8 used bytes: below = the
// elements < lo, taken and s = how many were taken and their sum.
LT_HD void leaf_take_sum(const uint8_t* leafp, uint32_t u, uint64_t lo, uint64_t most,
                         uint32_t& below, uint32_t& taken, uint64_t& s) {
  Walk k;
  k.val = leaf_head(leafp);
  below = taken = 0;
  s = 0;
  auto take = [&](uint64_t v) {
    if (v < lo) below++;
    else if (taken < most) { s += v; taken++; }
  };
  take(k.val);
  uint32_t p = 8;  // the next group's byte
  uint32_t raw[4];
  ld16(leafp, raw);
  if (k.val < lo) {
    const uint32_t p0 = skip_below(leafp, u, lo, k, below, raw);
    if (p0) p = p0;
  }
  // up to the group that reaches lo, counted; that group; then whole groups
  // while they fit; then the group that does not
  Held g;
  bool have = false;
  auto before = [&](uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb) {
    g = Held{k, wa, wb, ta, tb};
    uint32_t T;
    uint64_t ss;
    group_sum(wa, wb, ta, tb, k, T, ss);
    have = k.val >= lo;
    if (!have) below += T;
    p += 8;
  };
  for (uint32_t p0 = p & ~15u; p < u && k.val < lo; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0 == p) before(w[0], w[1], t[0], t[1]);
    if (p < u && k.val < lo) before(w[2], w[3], t[2], t[3]);
  }
  if (have) group_visit(g.wa, g.wb, g.ta, g.tb, g.k, take);
  have = false;
  auto within = [&](uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb) {
    g = Held{k, wa, wb, ta, tb};
    uint32_t T;
    uint64_t ss;
    group_sum(wa, wb, ta, tb, k, T, ss);
    have = taken + T > most;
    if (!have) {
      s += T * g.k.val + ss;
      taken += T;
    }
    p += 8;
  };
  if (p < u) ld16(leafp + (p & ~15u), raw);
  for (uint32_t p0 = p & ~15u; p < u && !have && taken < most; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0 == p) within(w[0], w[1], t[0], t[1]);
    if (p < u && !have && taken < most) within(w[2], w[3], t[2], t[3]);
  }
  if (have) group_visit(g.wa, g.wb, g.ta, g.tb, g.k, take);
}

// Elements < x of a leaf of u >= 8 used bytes.  at = where the first element
// >= x is closed, if the leaf has one past its head: the state before its
// group of 8 bytes, `sum` the group's byte and `cnt` the elements before it;
// else the byte is 0.
LT_HD uint32_t leaf_below(const uint8_t* leafp, uint32_t u, uint64_t x, Mark& at) {
  Walk k;
  k.val = leaf_head(leafp);
  at = Mark{0, 0, 0, 0, 0};
  if (k.val >= x) return 0;
  uint32_t n = 1, p = 0;
  Held g;
  bool have = false;
  auto step = [&](uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb) {
    g = Held{k, wa, wb, ta, tb};
    uint32_t T;
    uint64_t ss;
    group_sum(wa, wb, ta, tb, k, T, ss);
    have = k.val >= x;
    if (!have) n += T;
  };
  uint32_t raw[4];
  ld16(leafp, raw);
  uint32_t p0 = skip_below(leafp, u, x, k, n, raw);
  for (; p0 < u && !have; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    p = p0;
    if (p0) step(w[0], w[1], t[0], t[1]);
    if (!have) {
      p = p0 + 8u;
      step(w[2], w[3], t[2], t[3]);
    }
  }
  if (have) {
    at = Mark{g.k.val, p, g.k.acc, n, g.k.sh};
    group_visit(g.wa, g.wb, g.ta, g.tb, g.k, [&](uint64_t v) { n += v < x ? 1u : 0u; });
  }
  return n;
}

// ---- a leaf walked by a team of lanes ----
//
// One lane walks a leaf in some 30 steps that wait for one another; with few
// queries on the GPU that chain is what a call waits for.  Here each of N lanes
// (eight, or a warp for leaves of more than 512 bytes) takes an equal run of
// 16-byte chunks: it enters with the code open at
// its first byte (found by walking the chunk before from any state: every code
// has at most 10 bytes, so one ends in it), sums its deltas, learns from a scan
// over the team the element before its run, and then visits its elements.
constexpr uint32_t kTeam = 8;

struct Run {
  Walk k;               // at byte b0; val 0 until the scan over the team
  uint32_t b0, b1;      // the lane's bytes
  uint64_t delta = 0;   // what its codes add up to
  uint64_t sum = 0;     // SUM: its elements', less the element before the run
  uint32_t codes = 0;
};

// Lane tl's run (of N) of a leaf of u used bytes (0: no leaf).
template <uint32_t N = kTeam, bool SUM = false>
LT_HD Run team_run(const uint8_t* leafp, uint32_t u, uint32_t tl) {
  const uint32_t per = 16u * (((u + 15u) / 16u + N - 1u) / N);
  Run r;
  r.b0 = per * tl;
  r.b1 = r.b0 + per < u ? r.b0 + per : u;
  uint32_t w[4], t[4], T;
  uint64_t ss;
  Walk k;
  if (tl && r.b0 < u) {
    load_chunk(leafp, r.b0 - 16u, u, w, t);
    if (r.b0 > 16u) group_sum(w[0], w[1], t[0], t[1], k, T, ss);  // else the head
    group_sum(w[2], w[3], t[2], t[3], k, T, ss);
    k.val = 0;
  }
  r.k = k;
  for (uint32_t p0 = r.b0; p0 < r.b1; p0 += 16) {
    load_chunk(leafp, p0, u, w, t);
    uint64_t v = k.val;
    if (p0) {
      group_sum(w[0], w[1], t[0], t[1], k, T, ss);
      r.codes += T;
      if (SUM) r.sum += T * v + ss;
    }
    v = k.val;
    group_sum(w[2], w[3], t[2], t[3], k, T, ss);
    r.codes += T;
    if (SUM) r.sum += T * v + ss;
  }
  r.delta = k.val;
  return r;
}

// f(element) for the run's elements (its k.val set), the head not among them.
template <class F>
LT_HD void run_visit(const uint8_t* leafp, uint32_t u, const Run& r, F&& f) {
  Walk k = r.k;
  for (uint32_t p0 = r.b0; p0 < r.b1; p0 += 16) {
    uint32_t w[4], t[4];
    load_chunk(leafp, p0, u, w, t);
    if (p0) group_visit(w[0], w[1], t[0], t[1], k, f);
    group_visit(w[2], w[3], t[2], t[3], k, f);
  }
}

// ---- marks: the walk's state at every kMark-th byte of a leaf ----
//
// For many queries on one leaf the walk is done once and kept at every 32nd
// byte: a query then starts at the last mark whose element is below its bound
// and walks at most 32 bytes instead of half the leaf.  (Every 64th byte:
// degrees of 2^20 vertices 192 us instead of 150.)
constexpr uint32_t kMark = 32;

// Walks a leaf of u >= 8 used bytes: put(i, its state at byte kMark * i) for
// 0 < kMark * i < u; s and c = the sum and the number of its elements.
template <class F>
LT_HD void leaf_marks(const uint8_t* leafp, uint32_t u, uint64_t& s, uint32_t& c, F&& put) {
  Walk k;
  k.val = leaf_head(leafp);
  s = k.val;
  c = 1;
  uint32_t raw[4];
  ld16(leafp, raw);
  for (uint32_t p0 = 0; p0 < u; p0 += 16) {
    uint32_t w[4], t[4], T;
    uint64_t ss, v;
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0) {  // bytes 0-7 are the head
      if (p0 % kMark == 0) put(p0 / kMark, Mark{k.val, s, k.acc, c, k.sh});
      v = k.val;
      group_sum(w[0], w[1], t[0], t[1], k, T, ss);
      s += T * v + ss;
      c += T;
    }
    v = k.val;
    group_sum(w[2], w[3], t[2], t[3], k, T, ss);
    s += T * v + ss;
    c += T;
  }
}

// Adds the sum and the number of the elements < x that the walk k closes from
// byte p (a multiple of 16) on to s and c.  k.val < x.  With this few groups
// to go each is compared element by element, instead of being summed whole and
// the last one decoded again.
LT_HD void below_sum(const uint8_t* leafp, uint32_t u, uint32_t p, Walk k, uint64_t x, uint64_t& s,
                     uint64_t& c) {
  auto step = [&](uint32_t wa, uint32_t wb, uint32_t ta, uint32_t tb) {
    const uint32_t pa = wa & 0x7F7F7F7Fu, pb = wb & 0x7F7F7F7Fu;
    const uint64_t v = k.val, d = x - v;  // elements val + acc with acc < d
    uint32_t n = 0;
    uint64_t ss = 0;
    const int form = group_form(wa, wb, k);
    if (form == 0) {
      const uint32_t d32 = d >> 32 ? 0xFFFFFFFFu : (uint32_t)d;
      uint32_t s32 = 0;
      short_codes(pa, pb, ta, tb, k, [&](uint32_t acc) {
        if (acc < d32) { n++; s32 += acc; }
      });
      ss = s32;
    } else {
      auto take = [&](uint64_t acc) {
        if (acc < d) { n++; ss += acc; }
      };
      if (form == 1) medium_codes(pa, pb, ta, tb, k, take);
      else long_codes(pa, pb, ta, tb, k, take);
    }
    s += n * v + ss;
    c += n;
  };
  uint32_t raw[4];
  if (p < u) ld16(leafp + p, raw);
  for (uint32_t p0 = p; p0 < u && k.val < x; p0 += 16) {
    uint32_t w[4], t[4];
    next_chunk(leafp, p0, u, raw, w, t);
    if (p0) step(w[0], w[1], t[0], t[1]);
    if (k.val < x) step(w[2], w[3], t[2], t[3]);
  }
}

}  // namespace leafwalk
