// Word and byte operations of the per-leaf code, for the device and (the same
// results) the host.
#pragma once
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define LT_HD __host__ __device__ __forceinline__
#else
#define LT_HD inline
#endif

namespace leafthr {

LT_HD uint32_t fshr(uint32_t lo, uint32_t hi, uint32_t sh) {  // low word of (hi:lo) >> sh, sh < 32
#if defined(__CUDA_ARCH__)
  return __funnelshift_r(lo, hi, sh);
#else
  return sh ? (lo >> sh) | (hi << (32u - sh)) : lo;
#endif
}

LT_HD uint32_t fshl(uint32_t lo, uint32_t hi, uint32_t sh) {  // high word of (hi:lo) << sh, 0 < sh < 32
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, sh);
#else
  return (hi << sh) | (lo >> (32u - sh));
#endif
}

LT_HD uint32_t dp4a(uint32_t a, uint32_t b, uint32_t c) {  // c + sum of the four byte products
#if defined(__CUDA_ARCH__)
  return __dp4a(a, b, c);
#else
  for (int i = 0; i < 4; i++) c += ((a >> (8 * i)) & 0xFFu) * ((b >> (8 * i)) & 0xFFu);
  return c;
#endif
}

LT_HD uint32_t clz32(uint32_t x) {  // leading zeros, 32 for x == 0
#if defined(__CUDA_ARCH__)
  return (uint32_t)__clz((int)x);
#else
  return x ? (uint32_t)__builtin_clz(x) : 32u;
#endif
}

LT_HD uint32_t ctz32(uint32_t x) {  // trailing zeros, x != 0
#if defined(__CUDA_ARCH__)
  return (uint32_t)__ffs((int)x) - 1u;
#else
  return (uint32_t)__builtin_ctz(x);
#endif
}

LT_HD void ld16(const uint8_t* p, uint32_t (&w)[4]) {
#if defined(__CUDA_ARCH__)
  const uint4 v = *reinterpret_cast<const uint4*>(p);
  w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
#else
  memcpy(w, p, 16);
#endif
}

LT_HD uint32_t ld4(const uint8_t* p) {
#if defined(__CUDA_ARCH__)
  return *reinterpret_cast<const uint32_t*>(p);
#else
  uint32_t v;
  memcpy(&v, p, 4);
  return v;
#endif
}

LT_HD void st16(uint8_t* p, const uint32_t (&w)[4]) {
#if defined(__CUDA_ARCH__)
  *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
#else
  memcpy(p, w, 16);
#endif
}

LT_HD uint32_t popc(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return (uint32_t)__popc(x);
#else
  return (uint32_t)__builtin_popcount(x);
#endif
}

LT_HD uint32_t bmask4(uint32_t b4) {  // 4 bits -> 0x00 / 0xFF bytes
  return ((b4 * 0x00204081u) & 0x01010101u) * 0xFFu;
}

LT_HD uint32_t byte_of(uint32_t v, int i) {  // byte i of v, zero-extended
#if defined(__CUDA_ARCH__)
  return __byte_perm(v, 0u, 0x4440u + (uint32_t)i);
#else
  return (v >> (8 * i)) & 0xFFu;
#endif
}

}  // namespace leafthr
