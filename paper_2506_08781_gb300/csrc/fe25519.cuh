// Arithmetic in F_p, p = 2^255 - 19 (the edwards25519 base field), as eight 32-bit limbs,
// little-endian.  Elements are kept "lazy": any value in [0, 2^256) that is congruent to
// the element; fe_canon() gives the unique representative in [0, p).
#pragma once
#include <cstdint>

namespace poslo {

struct fe { uint32_t v[8]; };

__device__ __forceinline__ fe fe_zero() { fe r; for (int i = 0; i < 8; ++i) r.v[i] = 0; return r; }
__device__ __forceinline__ fe fe_one() { fe r = fe_zero(); r.v[0] = 1; return r; }

__device__ __forceinline__ fe fe_const(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t a4,
                                       uint32_t a5, uint32_t a6, uint32_t a7) {
  fe r; r.v[0] = a0; r.v[1] = a1; r.v[2] = a2; r.v[3] = a3; r.v[4] = a4; r.v[5] = a5; r.v[6] = a6; r.v[7] = a7;
  return r;
}

// d = -121665/121666 and 2d, sqrt(-1) = 2^((p-1)/4)  (RFC 8032 Sec. 5.1).
__device__ __forceinline__ fe fe_d() {
  return fe_const(0x135978a3u, 0x75eb4dcau, 0x4141d8abu, 0x00700a4du, 0x7779e898u, 0x8cc74079u, 0x2b6ffe73u, 0x52036ceeu);
}
__device__ __forceinline__ fe fe_d2() {
  return fe_const(0x26b2f159u, 0xebd69b94u, 0x8283b156u, 0x00e0149au, 0xeef3d130u, 0x198e80f2u, 0x56dffce7u, 0x2406d9dcu);
}
__device__ __forceinline__ fe fe_dinv() {   // 1/d
  return fe_const(0xcdc9f843u, 0x25e0f276u, 0x4279542eu, 0x0b5dd698u, 0xcdb9cf66u, 0x2b162114u, 0x14d5ce43u, 0x40907ed2u);
}
__device__ __forceinline__ fe fe_sqrtm1() {
  return fe_const(0x4a0ea0b0u, 0xc4ee1b27u, 0xad2fe478u, 0x2f431806u, 0x3dfbd7a7u, 0x2b4d0099u, 0x4fc1df0bu, 0x2b832480u);
}

// r = a + b, folding the carry out of bit 256 twice (2^256 = 38).  After a second carry the
// value is below 38, so the second fold cannot carry out of the lowest limb.
__device__ __forceinline__ fe fe_add(const fe& a, const fe& b) {
  fe r;
  uint32_t c;
  asm("add.cc.u32 %0, %9, %17;\n\t"
      "addc.cc.u32 %1, %10, %18;\n\t"
      "addc.cc.u32 %2, %11, %19;\n\t"
      "addc.cc.u32 %3, %12, %20;\n\t"
      "addc.cc.u32 %4, %13, %21;\n\t"
      "addc.cc.u32 %5, %14, %22;\n\t"
      "addc.cc.u32 %6, %15, %23;\n\t"
      "addc.cc.u32 %7, %16, %24;\n\t"
      "addc.u32 %8, 0, 0;"
      : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
        "=r"(r.v[7]), "=r"(c)
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]), "r"(a.v[7]),
        "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]), "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
  const uint32_t k = c * 38u;
  asm("add.cc.u32 %0, %0, %9;\n\t"
      "addc.cc.u32 %1, %1, 0;\n\t"
      "addc.cc.u32 %2, %2, 0;\n\t"
      "addc.cc.u32 %3, %3, 0;\n\t"
      "addc.cc.u32 %4, %4, 0;\n\t"
      "addc.cc.u32 %5, %5, 0;\n\t"
      "addc.cc.u32 %6, %6, 0;\n\t"
      "addc.cc.u32 %7, %7, 0;\n\t"
      "addc.u32 %8, 0, 0;"
      : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]), "+r"(r.v[6]),
        "+r"(r.v[7]), "=r"(c)
      : "r"(k));
  r.v[0] += c * 38u;
  return r;
}

// r = a - b: on a borrow out of bit 256 the wrapped value is 2^256 too large, i.e. 38 too
// large mod p, so 38 is subtracted.  After a second borrow the value is at least 2^256 - 38, so
// the second subtraction cannot borrow from the lowest limb.
__device__ __forceinline__ fe fe_sub(const fe& a, const fe& b) {
  fe r;
  uint32_t bo;
  asm("sub.cc.u32 %0, %9, %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32 %8, 0, 0;"
      : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
        "=r"(r.v[7]), "=r"(bo)
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]), "r"(a.v[7]),
        "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]), "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
  const uint32_t k = bo & 38u;   // bo is 0 or 0xffffffff
  asm("sub.cc.u32 %0, %0, %9;\n\t"
      "subc.cc.u32 %1, %1, 0;\n\t"
      "subc.cc.u32 %2, %2, 0;\n\t"
      "subc.cc.u32 %3, %3, 0;\n\t"
      "subc.cc.u32 %4, %4, 0;\n\t"
      "subc.cc.u32 %5, %5, 0;\n\t"
      "subc.cc.u32 %6, %6, 0;\n\t"
      "subc.cc.u32 %7, %7, 0;\n\t"
      "subc.u32 %8, 0, 0;"
      : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]), "+r"(r.v[6]),
        "+r"(r.v[7]), "=r"(bo)
      : "r"(k));
  r.v[0] -= bo & 38u;
  return r;
}

// r = a + b, or a - b when neg: a + (b ^ m) + (m & 1) with m = neg ? ~0 : 0, one chain for both.
// The carry out means "above 2^256" for a sum and "no borrow" for a difference; 38 is added or
// subtracted accordingly, at most twice (fe_add, fe_sub).
__device__ __forceinline__ fe fe_addsub(const fe& a, const fe& b, bool neg) {
  const uint32_t m = neg ? 0xffffffffu : 0u;
  fe r;
  uint32_t c;
  asm("add.cc.u32 %0, %9, %9;\n\t"   // carry in: bit 31 of m
      "addc.cc.u32 %0, %10, %18;\n\t"
      "addc.cc.u32 %1, %11, %19;\n\t"
      "addc.cc.u32 %2, %12, %20;\n\t"
      "addc.cc.u32 %3, %13, %21;\n\t"
      "addc.cc.u32 %4, %14, %22;\n\t"
      "addc.cc.u32 %5, %15, %23;\n\t"
      "addc.cc.u32 %6, %16, %24;\n\t"
      "addc.cc.u32 %7, %17, %25;\n\t"
      "addc.u32 %8, 0, 0;"
      : "=&r"(r.v[0]), "=&r"(r.v[1]), "=&r"(r.v[2]), "=&r"(r.v[3]), "=&r"(r.v[4]), "=&r"(r.v[5]), "=&r"(r.v[6]),
        "=&r"(r.v[7]), "=&r"(c)
      : "r"(m), "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]),
        "r"(a.v[7]), "r"(b.v[0] ^ m), "r"(b.v[1] ^ m), "r"(b.v[2] ^ m), "r"(b.v[3] ^ m), "r"(b.v[4] ^ m),
        "r"(b.v[5] ^ m), "r"(b.v[6] ^ m), "r"(b.v[7] ^ m));
  // fold: +38 (sum with carry), -38 (difference with borrow) or nothing, as a signed 256-bit word
  const uint32_t hit = (c ^ m) & 1u;               // 1: a fold is due
  const uint32_t k = ((38u ^ m) - m) & (0u - hit);  // 38, -38 or 0
  const uint32_t x = m & (0u - hit);                // its upper words
  asm("add.cc.u32 %0, %0, %9;\n\t"
      "addc.cc.u32 %1, %1, %10;\n\t"
      "addc.cc.u32 %2, %2, %10;\n\t"
      "addc.cc.u32 %3, %3, %10;\n\t"
      "addc.cc.u32 %4, %4, %10;\n\t"
      "addc.cc.u32 %5, %5, %10;\n\t"
      "addc.cc.u32 %6, %6, %10;\n\t"
      "addc.cc.u32 %7, %7, %10;\n\t"
      "addc.u32 %8, 0, 0;"
      : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]), "+r"(r.v[6]),
        "+r"(r.v[7]), "=&r"(c)
      : "r"(k), "r"(x));
  r.v[0] += ((38u ^ m) - m) & (0u - ((c ^ x) & 1u) & (0u - hit));
  return r;
}

// Products (the IMAD pipe's work).  A 32 x 32 -> 64 bit product added to a register pair with
// carry in and out, written as the PTX pair mad.lo.cc / madc.hi.cc on the pair's two words, is
// one wide multiply-add: half the issue rate of a 32-bit IMAD and two thirds of the separate
// low and high products.  A pair starts at an even word, so a product a_i b_j with i + j even
// goes to the accumulator E, one with i + j odd to O, which is kept one word lower:
// a b = E + 2^32 O.  A row of products by one b_j over every other a_i is one carry chain; its
// carry out starts the next word.
//
// Measured on GB300 (cycles per operation and SM quarter with 8 warps on it / with one):
// squaring 222 / 352, product 340 / 530, where rows of 64-bit partial sums in C (a wide
// product and the addition of a word and a carry each) took 267 / 448 and 410 / 640.  44 (72)
// wide products of 4 cycles each are 176 (288) cycles: the pipe is 85 % busy, the rest are
// register-port conflicts and the few carry additions that issue on the same pipe.
// The paper's GPU code used 4x64-bit words with add.cc.u64 (Sec. 7.4, "Finite Field Arithmetic
// with PTX Instructions"); on NVIDIA parts a 64-bit multiply is itself emulated with 32-bit
// IMADs, so 32-bit limbs are the native width here.

__device__ __forceinline__ void fe_wide0(uint32_t* x, uint32_t a, uint32_t b) {
  const uint64_t p = (uint64_t)a * b;
  x[0] = (uint32_t)p;
  x[1] = (uint32_t)(p >> 32);
}

// x[0..2n) += (a0, a1, ...) * b, one wide product per pair of words; the carry out goes to c
// (widec) or cannot occur (wide: the last pair holds at most a carry before the product).
__device__ __forceinline__ void fe_widec1(uint32_t* x, uint32_t a0, uint32_t b, uint32_t& c) {
  asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\t"
      "madc.hi.cc.u32 %1, %3, %4, %1;\n\t"
      "addc.u32 %2, 0, 0;"
      : "+r"(x[0]), "+r"(x[1]), "=r"(c)
      : "r"(a0), "r"(b));
}
__device__ __forceinline__ void fe_wide1(uint32_t* x, uint32_t a0, uint32_t b) {
  asm("mad.lo.cc.u32 %0, %2, %3, %0;\n\t"
      "madc.hi.u32 %1, %2, %3, %1;"
      : "+r"(x[0]), "+r"(x[1])
      : "r"(a0), "r"(b));
}
__device__ __forceinline__ void fe_widec2(uint32_t* x, uint32_t a0, uint32_t a1, uint32_t b, uint32_t& c) {
  asm("mad.lo.cc.u32 %0, %5, %7, %0;\n\t"
      "madc.hi.cc.u32 %1, %5, %7, %1;\n\t"
      "madc.lo.cc.u32 %2, %6, %7, %2;\n\t"
      "madc.hi.cc.u32 %3, %6, %7, %3;\n\t"
      "addc.u32 %4, 0, 0;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "=r"(c)
      : "r"(a0), "r"(a1), "r"(b));
}
__device__ __forceinline__ void fe_wide2(uint32_t* x, uint32_t a0, uint32_t a1, uint32_t b) {
  asm("mad.lo.cc.u32 %0, %4, %6, %0;\n\t"
      "madc.hi.cc.u32 %1, %4, %6, %1;\n\t"
      "madc.lo.cc.u32 %2, %5, %6, %2;\n\t"
      "madc.hi.u32 %3, %5, %6, %3;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3])
      : "r"(a0), "r"(a1), "r"(b));
}
__device__ __forceinline__ void fe_widec3(uint32_t* x, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t b,
                                           uint32_t& c) {
  asm("mad.lo.cc.u32 %0, %7, %10, %0;\n\t"
      "madc.hi.cc.u32 %1, %7, %10, %1;\n\t"
      "madc.lo.cc.u32 %2, %8, %10, %2;\n\t"
      "madc.hi.cc.u32 %3, %8, %10, %3;\n\t"
      "madc.lo.cc.u32 %4, %9, %10, %4;\n\t"
      "madc.hi.cc.u32 %5, %9, %10, %5;\n\t"
      "addc.u32 %6, 0, 0;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]), "=r"(c)
      : "r"(a0), "r"(a1), "r"(a2), "r"(b));
}
__device__ __forceinline__ void fe_wide3(uint32_t* x, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t b) {
  asm("mad.lo.cc.u32 %0, %6, %9, %0;\n\t"
      "madc.hi.cc.u32 %1, %6, %9, %1;\n\t"
      "madc.lo.cc.u32 %2, %7, %9, %2;\n\t"
      "madc.hi.cc.u32 %3, %7, %9, %3;\n\t"
      "madc.lo.cc.u32 %4, %8, %9, %4;\n\t"
      "madc.hi.u32 %5, %8, %9, %5;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5])
      : "r"(a0), "r"(a1), "r"(a2), "r"(b));
}
__device__ __forceinline__ void fe_widec4(uint32_t* x, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                           uint32_t b, uint32_t& c) {
  asm("mad.lo.cc.u32 %0, %9, %13, %0;\n\t"
      "madc.hi.cc.u32 %1, %9, %13, %1;\n\t"
      "madc.lo.cc.u32 %2, %10, %13, %2;\n\t"
      "madc.hi.cc.u32 %3, %10, %13, %3;\n\t"
      "madc.lo.cc.u32 %4, %11, %13, %4;\n\t"
      "madc.hi.cc.u32 %5, %11, %13, %5;\n\t"
      "madc.lo.cc.u32 %6, %12, %13, %6;\n\t"
      "madc.hi.cc.u32 %7, %12, %13, %7;\n\t"
      "addc.u32 %8, 0, 0;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]), "+r"(x[6]), "+r"(x[7]), "=r"(c)
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b));
}
__device__ __forceinline__ void fe_wide4(uint32_t* x, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b) {
  asm("mad.lo.cc.u32 %0, %8, %12, %0;\n\t"
      "madc.hi.cc.u32 %1, %8, %12, %1;\n\t"
      "madc.lo.cc.u32 %2, %9, %12, %2;\n\t"
      "madc.hi.cc.u32 %3, %9, %12, %3;\n\t"
      "madc.lo.cc.u32 %4, %10, %12, %4;\n\t"
      "madc.hi.cc.u32 %5, %10, %12, %5;\n\t"
      "madc.lo.cc.u32 %6, %11, %12, %6;\n\t"
      "madc.hi.u32 %7, %11, %12, %7;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]), "+r"(x[6]), "+r"(x[7])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b));
}

// t[0..15] = E + 2^32 O.
__device__ __forceinline__ void fe_merge(uint32_t t[16], const uint32_t E[16], const uint32_t O[15]) {
  t[0] = E[0];
  asm("add.cc.u32 %0, %15, %30;\n\t"
      "addc.cc.u32 %1, %16, %31;\n\t"
      "addc.cc.u32 %2, %17, %32;\n\t"
      "addc.cc.u32 %3, %18, %33;\n\t"
      "addc.cc.u32 %4, %19, %34;\n\t"
      "addc.cc.u32 %5, %20, %35;\n\t"
      "addc.cc.u32 %6, %21, %36;\n\t"
      "addc.cc.u32 %7, %22, %37;\n\t"
      "addc.cc.u32 %8, %23, %38;\n\t"
      "addc.cc.u32 %9, %24, %39;\n\t"
      "addc.cc.u32 %10, %25, %40;\n\t"
      "addc.cc.u32 %11, %26, %41;\n\t"
      "addc.cc.u32 %12, %27, %42;\n\t"
      "addc.cc.u32 %13, %28, %43;\n\t"
      "addc.u32 %14, %29, %44;"
      : "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]), "=&r"(t[6]), "=&r"(t[7]), "=&r"(t[8]),
        "=&r"(t[9]), "=&r"(t[10]), "=&r"(t[11]), "=&r"(t[12]), "=&r"(t[13]), "=&r"(t[14]), "=&r"(t[15])
      : "r"(E[1]), "r"(E[2]), "r"(E[3]), "r"(E[4]), "r"(E[5]), "r"(E[6]), "r"(E[7]), "r"(E[8]), "r"(E[9]),
        "r"(E[10]), "r"(E[11]), "r"(E[12]), "r"(E[13]), "r"(E[14]), "r"(E[15]), "r"(O[0]), "r"(O[1]), "r"(O[2]),
        "r"(O[3]), "r"(O[4]), "r"(O[5]), "r"(O[6]), "r"(O[7]), "r"(O[8]), "r"(O[9]), "r"(O[10]), "r"(O[11]),
        "r"(O[12]), "r"(O[13]), "r"(O[14]));
}

// r = t mod p for a product t: 2^256 = 38 folds the upper half (four even and four odd wide
// products, as above), then 2^255 = 19 the bits above 255, which leaves r below 2^255 + 2^13.
__device__ __forceinline__ fe fe_fold512(const uint32_t t[16]) {
  uint32_t E[8], O[8], top;
#pragma unroll
  for (int k = 0; k < 8; ++k) E[k] = t[k];
#pragma unroll
  for (int k = 0; k < 4; ++k) fe_wide0(O + 2 * k, t[9 + 2 * k], 38u);
  fe_widec4(E, t[8], t[10], t[12], t[14], 38u, top);
  asm("add.cc.u32 %0, %0, %8;\n\t"
      "addc.cc.u32 %1, %1, %9;\n\t"
      "addc.cc.u32 %2, %2, %10;\n\t"
      "addc.cc.u32 %3, %3, %11;\n\t"
      "addc.cc.u32 %4, %4, %12;\n\t"
      "addc.cc.u32 %5, %5, %13;\n\t"
      "addc.cc.u32 %6, %6, %14;\n\t"
      "addc.u32 %7, %7, %15;"
      : "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(top)
      : "r"(O[0]), "r"(O[1]), "r"(O[2]), "r"(O[3]), "r"(O[4]), "r"(O[5]), "r"(O[6]), "r"(O[7]));
  const uint32_t h = __funnelshift_l(E[7], top, 1);   // bits 255 and up, below 2^8
  E[7] &= 0x7fffffffu;
  fe r;
  asm("mad.lo.cc.u32 %0, %8, 19, %9;\n\t"
      "addc.cc.u32 %1, %10, 0;\n\t"
      "addc.cc.u32 %2, %11, 0;\n\t"
      "addc.cc.u32 %3, %12, 0;\n\t"
      "addc.cc.u32 %4, %13, 0;\n\t"
      "addc.cc.u32 %5, %14, 0;\n\t"
      "addc.cc.u32 %6, %15, 0;\n\t"
      "addc.u32 %7, %16, 0;"
      : "=&r"(r.v[0]), "=&r"(r.v[1]), "=&r"(r.v[2]), "=&r"(r.v[3]), "=&r"(r.v[4]), "=&r"(r.v[5]), "=&r"(r.v[6]),
        "=&r"(r.v[7])
      : "r"(h), "r"(E[0]), "r"(E[1]), "r"(E[2]), "r"(E[3]), "r"(E[4]), "r"(E[5]), "r"(E[6]), "r"(E[7]));
  return r;
}

__device__ __forceinline__ void fe_mul512(uint32_t t[16], const uint32_t* a, const uint32_t* b) {
  uint32_t E[16], O[16];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    fe_wide0(E + 2 * k, a[2 * k], b[0]);
    fe_wide0(O + 2 * k, a[2 * k + 1], b[0]);
  }
  E[8] = 0;
#pragma unroll
  for (int j = 1; j < 8; j += 2) {
    fe_widec4(O + j - 1, a[0], a[2], a[4], a[6], b[j], O[j + 7]);
    E[j + 8] = 0;
    fe_wide4(E + j + 1, a[1], a[3], a[5], a[7], b[j]);
    if (j == 7) break;
    fe_widec4(E + j + 1, a[0], a[2], a[4], a[6], b[j + 1], E[j + 9]);
    O[j + 8] = 0;
    fe_wide4(O + j + 1, a[1], a[3], a[5], a[7], b[j + 1]);
  }
  fe_merge(t, E, O);
}

__device__ __forceinline__ fe fe_mul(const fe& a, const fe& b) {
  uint32_t t[16];
  fe_mul512(t, a.v, b.v);
  return fe_fold512(t);
}

// a^2: the 28 cross products a_i a_j (i < j) in rows by a_i, doubled by a funnel shift, then the
// 8 squares a_i^2 at word 2i in one chain.
__device__ __forceinline__ void fe_sq512(uint32_t t[16], const uint32_t* a) {
  uint32_t E[16], O[15];
  fe_wide0(O, a[0], a[1]);
  fe_wide0(O + 2, a[0], a[3]);
  fe_wide0(O + 4, a[0], a[5]);
  fe_wide0(O + 6, a[0], a[7]);
  E[0] = E[1] = 0;
  fe_wide0(E + 2, a[0], a[2]);
  fe_wide0(E + 4, a[0], a[4]);
  fe_wide0(E + 6, a[0], a[6]);
  fe_widec3(O + 2, a[2], a[4], a[6], a[1], O[8]);
  E[8] = E[9] = 0;
  fe_wide3(E + 4, a[3], a[5], a[7], a[1]);
  O[9] = 0;
  fe_wide3(O + 4, a[3], a[5], a[7], a[2]);
  fe_widec2(E + 6, a[4], a[6], a[2], E[10]);
  fe_widec2(O + 6, a[4], a[6], a[3], O[10]);
  E[11] = 0;
  fe_wide2(E + 8, a[5], a[7], a[3]);
  O[11] = 0;
  fe_wide2(O + 8, a[5], a[7], a[4]);
  fe_widec1(E + 10, a[6], a[4], E[12]);
  fe_widec1(O + 10, a[6], a[5], O[12]);
  E[13] = 0;
  fe_wide1(E + 12, a[7], a[5]);
  O[13] = 0;
  fe_wide1(O + 12, a[7], a[6]);
  E[14] = E[15] = 0; O[14] = 0;
  fe_merge(t, E, O);
#pragma unroll
  for (int k = 15; k > 0; --k) t[k] = __funnelshift_l(t[k - 1], t[k], 1);
  t[0] = 0;
  asm("mad.lo.cc.u32 %0, %16, %16, %0;\n\t"
      "madc.hi.cc.u32 %1, %16, %16, %1;\n\t"
      "madc.lo.cc.u32 %2, %17, %17, %2;\n\t"
      "madc.hi.cc.u32 %3, %17, %17, %3;\n\t"
      "madc.lo.cc.u32 %4, %18, %18, %4;\n\t"
      "madc.hi.cc.u32 %5, %18, %18, %5;\n\t"
      "madc.lo.cc.u32 %6, %19, %19, %6;\n\t"
      "madc.hi.cc.u32 %7, %19, %19, %7;\n\t"
      "madc.lo.cc.u32 %8, %20, %20, %8;\n\t"
      "madc.hi.cc.u32 %9, %20, %20, %9;\n\t"
      "madc.lo.cc.u32 %10, %21, %21, %10;\n\t"
      "madc.hi.cc.u32 %11, %21, %21, %11;\n\t"
      "madc.lo.cc.u32 %12, %22, %22, %12;\n\t"
      "madc.hi.cc.u32 %13, %22, %22, %13;\n\t"
      "madc.lo.cc.u32 %14, %23, %23, %14;\n\t"
      "madc.hi.u32 %15, %23, %23, %15;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]),
        "+r"(t[8]), "+r"(t[9]), "+r"(t[10]), "+r"(t[11]), "+r"(t[12]), "+r"(t[13]), "+r"(t[14]), "+r"(t[15])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]));
}

__device__ __forceinline__ fe fe_sq(const fe& a) {
  uint32_t t[16];
  fe_sq512(t, a.v);
  return fe_fold512(t);
}

// n successive squarings; the loop is kept rolled so the exponentiation chains of the
// inversion and square root stay small in the instruction cache.
__device__ __forceinline__ fe fe_sqn(fe a, int n) {
#pragma unroll 1
  for (int i = 0; i < n; ++i) a = fe_sq(a);
  return a;
}

// Unique representative in [0, p): subtract p while the value is >= p (at most twice for
// a value below 2^256 = 2p + 38).
__device__ __forceinline__ fe fe_canon(fe a) {
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    fe r;
    uint32_t bo;
    asm("sub.cc.u32 %0, %9, 0xffffffed;\n\t"
        "subc.cc.u32 %1, %10, 0xffffffff;\n\t"
        "subc.cc.u32 %2, %11, 0xffffffff;\n\t"
        "subc.cc.u32 %3, %12, 0xffffffff;\n\t"
        "subc.cc.u32 %4, %13, 0xffffffff;\n\t"
        "subc.cc.u32 %5, %14, 0xffffffff;\n\t"
        "subc.cc.u32 %6, %15, 0xffffffff;\n\t"
        "subc.cc.u32 %7, %16, 0x7fffffff;\n\t"
        "subc.u32 %8, 0, 0;"
        : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
          "=r"(r.v[7]), "=r"(bo)
        : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]),
          "r"(a.v[7]));
    // keep r when no borrow (a >= p)
#pragma unroll
    for (int i = 0; i < 8; ++i) a.v[i] = bo ? a.v[i] : r.v[i];
  }
  return a;
}

__device__ __forceinline__ bool fe_is_zero(const fe& a) {
  const fe c = fe_canon(a);
  uint32_t o = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) o |= c.v[i];
  return o == 0;
}

__device__ __forceinline__ bool fe_eq(const fe& a, const fe& b) { return fe_is_zero(fe_sub(a, b)); }

__device__ __forceinline__ fe fe_neg(const fe& a) { return fe_sub(fe_zero(), a); }

__device__ __forceinline__ fe fe_select(const fe& a, const fe& b, bool pick_b) {
  fe r;
#pragma unroll
  for (int i = 0; i < 8; ++i) r.v[i] = pick_b ? b.v[i] : a.v[i];
  return r;
}

// z^((p-5)/8) = z^(2^252 - 3) by the chain z^2, z^9, z^11, z^(2^5 - 1), then eight stages of
// "n squarings, one product": exponents 2^k - 1 for k = 10, 20, 40, 50, 100, 200, 250 and last
// 2^252 - 3.  A stage multiplies by the value it started from, by z^(2^10 - 1) (to reach 50), by
// z^(2^50 - 1) (250) or by z (last).  One loop instead of a call per stage: the decoding runs as
// one copy each of the squaring and the product (a few KB of code instead of 48), which a
// launch of few points fetches from a cold instruction cache.  The factors are indexed at run
// time and so live in local memory, read eight times, instead of 24 registers held through
// every squaring.
__device__ __forceinline__ fe fe_pow_p58(const fe& z) {
  const fe z2 = fe_sq(z);
  const fe z9 = fe_mul(fe_sqn(z2, 2), z);
  fe cur = fe_mul(fe_sq(fe_mul(z9, z2)), z9);   // 2^5 - 1
  // what a stage multiplies by: 0 the value it started from, 1 z^(2^10 - 1), 2 z^(2^50 - 1), 3 z
  fe keep[4];
  keep[3] = z;
#pragma unroll 1
  for (int k = 0; k < 8; ++k) {
    // squarings of the stages: 5, 10, 20, 10, 50, 100, 50, 2 (one byte each)
    const int n = (int)(0x023264320a140a05ull >> (8 * k) & 0xff);
    keep[0x00020010u >> (4 * k) & 3] = cur;
    cur = fe_mul(fe_sqn(cur, n), keep[0x32021010u >> (4 * k) & 3]);
  }
  return cur;
}

// z^-1 mod p (0 -> 0) by division steps (D. J. Bernstein, B.-Y. Yang, "Fast constant-time gcd
// computation and modular inversion", TCHES 2019): from (delta, f, g) = (1, p, z), a step is
//   (1 - delta, g, (g - f) / 2)        if delta > 0 and g is odd,
//   (1 + delta, f, (g + (g mod 2) f) / 2)  otherwise,
// and after at most (49 * 255 + 57) / 17 < 741 of them g = 0 and f = +-1.  The steps look only
// at the low bits, so 30 at a time run on one word each of f and g and are collected in a
// matrix (u v; q r) of entries at most 2^30, which then moves f, g (exactly) and the
// coefficients d, e with d z = f, e z = g (mod p): (u d + v e + m p) / 2^30, with m chosen to
// make the division exact.  Numbers are nine signed limbs of 30 bits; in them p is 2^15 at limb
// 8 and -19 at limb 0.  |m| <= 2^29, so d and e grow by at most p / 2 a batch.  (Signed limbs of
// 30 bits with 30 steps collected in a matrix are also how libsecp256k1's modinv32 lays this out.)
// One thread's chain: about 20 batches of some 1,500 cycles, where the 255 squarings and 11
// products of z^(p-2) took 95,000 cycles.
static __device__ __noinline__ fe fe_inv(const fe& z) {
  constexpr int32_t M = (1 << 30) - 1;
  constexpr uint32_t kInv19 = 678152731u;   // 19^-1 mod 2^30
  static_assert(((uint64_t)kInv19 * 19u & (uint32_t)M) == 1u, "inverse of 19 mod 2^30");
  const fe a = fe_canon(z);
  int32_t f[9], g[9], d[9], e[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    f[k] = M;
    d[k] = 0;
    e[k] = 0;
    // bits 30k .. 30k + 29 of a: word k - 1 or k on, offset 30k mod 32
    const int w = (30 * k) >> 5, o = (30 * k) & 31;
    const uint32_t hi = w + 1 < 8 ? a.v[w + 1] : 0u;
    g[k] = (int32_t)(__funnelshift_r(a.v[w], hi, o) & (uint32_t)M);
  }
  f[0] = M + 1 - 19;
  f[8] = 0x7fff;
  e[0] = 1;
  int32_t delta = 1;
#pragma unroll 1
  for (int batch = 0; batch < 25; ++batch) {
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) any |= (uint32_t)g[k];
    if (any == 0) break;
    uint32_t f0 = (uint32_t)f[0] | (uint32_t)f[1] << 30, g0 = (uint32_t)g[0] | (uint32_t)g[1] << 30;
    int32_t u = 1, v = 0, q = 0, r = 1;
#pragma unroll 6
    for (int i = 0; i < 30; ++i) {
      const int32_t odd = -(int32_t)(g0 & 1u);
      const bool swap = odd != 0 && delta > 0;
      const uint32_t tf = swap ? 0u - f0 : f0;
      const int32_t tu = swap ? -u : u, tv = swap ? -v : v;
      f0 = swap ? g0 : f0;
      u = (swap ? q : u) << 1;
      v = (swap ? r : v) << 1;
      g0 = (g0 + (tf & (uint32_t)odd)) >> 1;
      q += tu & odd;
      r += tv & odd;
      delta = (swap ? -delta : delta) + 1;
    }
    int64_t cf = (int64_t)u * f[0] + (int64_t)v * g[0], cg = (int64_t)q * f[0] + (int64_t)r * g[0];
    int64_t cd = (int64_t)u * d[0] + (int64_t)v * e[0], ce = (int64_t)q * d[0] + (int64_t)r * e[0];
    // m = cd / 19 mod 2^30 as a signed 30-bit number: cd - 19 m = 0 mod 2^30
    const int32_t md = (int32_t)((uint32_t)cd * kInv19 << 2) >> 2, me = (int32_t)((uint32_t)ce * kInv19 << 2) >> 2;
    cd -= (int64_t)19 * md;
    ce -= (int64_t)19 * me;
    cf >>= 30; cg >>= 30; cd >>= 30; ce >>= 30;
#pragma unroll
    for (int k = 1; k < 9; ++k) {
      cf += (int64_t)u * f[k] + (int64_t)v * g[k];
      cg += (int64_t)q * f[k] + (int64_t)r * g[k];
      cd += (int64_t)u * d[k] + (int64_t)v * e[k];
      ce += (int64_t)q * d[k] + (int64_t)r * e[k];
      if (k == 8) {
        cd += (int64_t)md << 15;
        ce += (int64_t)me << 15;
      }
      f[k - 1] = (int32_t)cf & M; g[k - 1] = (int32_t)cg & M;
      d[k - 1] = (int32_t)cd & M; e[k - 1] = (int32_t)ce & M;
      cf >>= 30; cg >>= 30; cd >>= 30; ce >>= 30;
    }
    f[8] = (int32_t)cf; g[8] = (int32_t)cg; d[8] = (int32_t)cd; e[8] = (int32_t)ce;
  }
  // +-d + 16 p (|d| <= 13 p), carried into non-negative limbs below 2^260
  const bool neg = f[8] < 0;
  int32_t c = -16 * 19;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    c += (neg ? -d[k] : d[k]) + (k == 8 ? 1 << 19 : 0);
    d[k] = k < 8 ? c & M : c;
    c >>= 30;
  }
  fe x;
#pragma unroll
  for (int k = 0; k < 8; ++k) x.v[k] = (uint32_t)d[k] >> (2 * k) | (uint32_t)d[k + 1] << (30 - 2 * k);
  // 2^255 = 19 for the bits above
  uint32_t cc = 19u * ((uint32_t)d[8] >> 15);
  x.v[7] &= 0x7fffffffu;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint64_t t = (uint64_t)x.v[k] + cc;
    x.v[k] = (uint32_t)t;
    cc = (uint32_t)(t >> 32);
  }
  return x;
}

__device__ __forceinline__ uint32_t fe_parity(const fe& a) { return fe_canon(a).v[0] & 1u; }

}  // namespace poslo
