// bitplane.cuh -- bit-plane arithmetic of the partition pass: one thread holds
// 32 consecutive elements of a tile, and plane j is the 32-bit word of their
// digit bits b_j (bit i = element i).  In this form a stable 1-bit split of
// 32 elements moves whole planes by shifts and masks: no element is loaded,
// ranked or stored per level.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace wtk {

#define WT_HD __host__ __device__ __forceinline__

// x rotated right by s (mod 32)
WT_HD uint32_t rotr32(uint32_t x, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(x, x, (uint32_t)s);
#else
  const uint32_t k = (uint32_t)s & 31u;
  return k ? (x >> k) | (x << (32 - k)) : x;
#endif
}

WT_HD uint32_t byte_perm(uint32_t a, uint32_t b, uint32_t sel) {
#ifdef __CUDA_ARCH__
  return __byte_perm(a, b, sel);
#else
  uint32_t r = 0;
  for (int i = 0; i < 4; i++) {
    const uint32_t k = (sel >> (4 * i)) & 7u;
    r |= (((k < 4 ? a >> (8 * k) : b >> (8 * (k - 4)))) & 0xffu) << (8 * i);
  }
  return r;
#endif
}

// Four registers of eight nibbles, R[q] nibble k = the top four bits of the
// digit of element 4k + q, to four planes: a 4 x 4 bit transpose of every
// nibble column in two exchange steps; plane 0 is the digit's top bit.
WT_HD void nibbles_to_planes(const uint32_t R[4], uint32_t p[4]) {
  const uint32_t m2 = 0x33333333u, m1 = 0x55555555u;
  const uint32_t a0 = (R[0] & m2) | ((R[2] & m2) << 2), a2 = ((R[0] >> 2) & m2) | (R[2] & ~m2);
  const uint32_t a1 = (R[1] & m2) | ((R[3] & m2) << 2), a3 = ((R[1] >> 2) & m2) | (R[3] & ~m2);
  p[3] = (a0 & m1) | ((a1 & m1) << 1);
  p[2] = ((a0 >> 1) & m1) | (a1 & ~m1);
  p[1] = (a2 & m1) | ((a3 & m1) << 1);
  p[0] = ((a2 >> 1) & m1) | (a3 & ~m1);
}

// Planes of the top digit bits (below bit rbits) of 32 elements of 1, 2 or 4
// bytes, given as the 8, 16 or 32 words that hold them; load(i) returns four
// words from word 4i on.  Planes past the digit hold other bits of the
// elements: the caller clears them.
template <int EW, typename Load>
WT_HD void planes_of(Load&& load, int rbits, uint32_t p[4]) {
  const int s = rbits - 4;  // negative: the digit sits below a nibble's top
  uint32_t R[4];
  if (EW == 1) {
    uint32_t z[4];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      uint32_t w[4];
      load(i, w);
#pragma unroll
      for (int k = 0; k < 2; k++)
        z[2 * i + k] = (rotr32(w[2 * k], s) & 0x0F0F0F0Fu) + 16u * (rotr32(w[2 * k + 1], s) & 0x0F0F0F0Fu);
    }
    // byte q of z[i] = nibbles 2i, 2i+1 of R[q]: a 4 x 4 byte transpose
    const uint32_t t0 = byte_perm(z[0], z[1], 0x5140), t1 = byte_perm(z[2], z[3], 0x5140);
    const uint32_t t2 = byte_perm(z[0], z[1], 0x7362), t3 = byte_perm(z[2], z[3], 0x7362);
    R[0] = byte_perm(t0, t1, 0x5410);
    R[1] = byte_perm(t0, t1, 0x7632);
    R[2] = byte_perm(t2, t3, 0x5410);
    R[3] = byte_perm(t2, t3, 0x7632);
  } else if (EW == 2) {
    uint32_t e[2][2] = {{0, 0}, {0, 0}};  // [elements 0-15 or 16-31][word parity]
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint32_t w[4];
      load(i, w);
#pragma unroll
      for (int k = 0; k < 4; k++)
        e[i >> 1][k & 1] += (rotr32(w[k], s) & 0x000F000Fu) << (8 * (i & 1) + 4 * (k >> 1));
    }
    R[0] = byte_perm(e[0][0], e[1][0], 0x5410);
    R[1] = byte_perm(e[0][0], e[1][0], 0x7632);
    R[2] = byte_perm(e[0][1], e[1][1], 0x5410);
    R[3] = byte_perm(e[0][1], e[1][1], 0x7632);
  } else {
    R[0] = R[1] = R[2] = R[3] = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
      uint32_t w[4];
      load(i, w);
#pragma unroll
      for (int q = 0; q < 4; q++) R[q] += (rotr32(w[q], s) & 0xFu) << (4 * i);
    }
  }
  nibbles_to_planes(R, p);
}

// the low n bits set, 0 <= n <= 32
WT_HD uint32_t low_mask(uint32_t n) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(r) : "r"(n));
  return r;
#else
  return n >= 32 ? ~0u : (1u << n) - 1u;
#endif
}

WT_HD int pop32(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __popc(x);
#else
  return __builtin_popcount(x);
#endif
}

// The moves of a compress within each byte (after Hacker's Delight, 2nd
// edition, section 7-4, on four bytes at once): the bits at the set positions of
// m to their byte's high end, in order, in conditional shifts by 1, 2 and 4.  A
// shift to the left of the bits t of x, whose places are free, is the
// multiplication-addition x + t (2^s - 1): half of the work goes to the
// multipliers instead of the logic pipe that bounds the pass.
struct ByteCompress {
  uint32_t m, mv[3];
};

// The moves for the bits at m (c1) and for the others (c0).  Bit i of a byte
// has 7 - i bits above it, so whether the zeros above it are odd in number
// gives the same of the ones: one prefix parity serves both first shifts.
WT_HD void byte_compress_plans(uint32_t m, ByteCompress& c0, ByteCompress& c1) {
  const uint32_t mk0 = (m >> 1) & 0x7F7F7F7Fu;
  uint32_t par = mk0 ^ ((mk0 >> 1) & 0x7F7F7F7Fu);
  par ^= (par >> 2) & 0x3F3F3F3Fu;
  par ^= (par >> 4) & 0x0F0F0F0Fu;
#pragma unroll
  for (int h = 0; h < 2; h++) {
    ByteCompress& c = h ? c1 : c0;
    uint32_t x = h ? m : ~m, mk = h ? (~m >> 1) & 0x7F7F7F7Fu : mk0;
    c.m = x;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      uint32_t mp = h ? par ^ 0x55555555u : par;
      if (i) {
        mp = mk ^ ((mk >> 1) & 0x7F7F7F7Fu);
        mp ^= (mp >> 2) & 0x3F3F3F3Fu;
        mp ^= (mp >> 4) & 0x0F0F0F0Fu;
      }
      const uint32_t mv = mp & x;
      c.mv[i] = mv;
      x += mv * ((1u << (1 << i)) - 1u);
      mk &= ~mp;
    }
  }
}

WT_HD uint32_t byte_compress(const ByteCompress& c, uint32_t x) {
  x &= c.m;
#pragma unroll
  for (int i = 0; i < 3; i++) x += (x & c.mv[i]) * ((1u << (1 << i)) - 1u);
  return x;
}

WT_HD uint32_t reverse32(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __brev(x);
#else
  uint32_t r = 0;
  for (int i = 0; i < 32; i++) r |= ((x >> i) & 1u) << (31 - i);
  return r;
#endif
}

// The stable split of 32 elements by plane b, the first element in the top bit
// here: the planes x[0..N) with the zeros' bits first (on top), the ones' bits
// after them.  Each byte is split by itself, then its two pieces move up by the
// bits of the other kind above it.  (Fewer than 32 elements: the bits past them
// set in every plane keep them behind the others.)
template <int N>
WT_HD void split_planes(uint32_t b, uint32_t* x) {
  ByteCompress c0, c1;
  byte_compress_plans(b, c0, c1);
  // zeros per byte; zeros above each byte, and ones
  uint32_t n = ~b - ((~b >> 1) & 0x55555555u);
  n = (n & 0x33333333u) + ((n >> 2) & 0x33333333u);
  n = (n + (n >> 4)) & 0x0F0F0F0Fu;
  const uint32_t q = n * 0x01010101u, z = q >> 24;
  const uint32_t zeros = z * 0x01010101u - q, ones = 0x00081018u - zeros;
  uint32_t fz[3], fo[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    fz[k] = low_mask((ones >> (8 * k)) & 31u);
    fo[k] = low_mask((zeros >> (8 * k)) & 31u);
  }
#pragma unroll
  for (int i = 0; i < N; i++) {
    uint32_t l = byte_compress(c0, x[i]), h = byte_compress(c1, x[i]);
    const uint32_t l0 = l, h0 = h;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      l += (l0 & (0xffu << (8 * k))) * fz[k];
      h += (h0 & (0xffu << (8 * k))) * fo[k];
    }
#ifdef __CUDA_ARCH__
    x[i] = l | __funnelshift_rc(h, 0u, z);
#else
    x[i] = l | (z < 32 ? h >> z : 0u);
#endif
  }
}

// Elements of every key among the valid ones (key bit j = plane j), two
// 16-bit counts a word: word k holds keys 2k (low half) and 2k + 1.
WT_HD void key_counts(const uint32_t p[4], uint32_t v, uint32_t c[8]) {
  const uint32_t a0 = ~p[0] & v, a1 = p[0] & v;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const uint32_t m = ((k & 1) ? p[1] : ~p[1]) & ((k & 2) ? p[2] : ~p[2]) & ((k & 4) ? p[3] : ~p[3]);
    c[k] = (uint32_t)pop32(m & a0) + ((uint32_t)pop32(m & a1) << 16);
  }
}

}  // namespace wtk
