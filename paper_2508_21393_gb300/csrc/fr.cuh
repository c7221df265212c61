// BLS12-381 scalar field F_r, 8 x 32-bit little-endian limbs, Montgomery
// arithmetic with R = 2^256 (host and device).
//
// The field is the one Sec. V fixes for the protocol (BLS12-381, |F| ~ 2^254):
//   r = 0x73eda753299d7d483339d80809a1d80553bda402fffe5bfeffffffff00000001.
// r < 2^255, so a sum of two reduced elements never overflows 256 bits.
// Limb constants below were derived from r by modular exponentiation:
//   R1 = 2^256 mod r, R2 = 2^512 mod r, R3 = 2^768 mod r, n' = -r^-1 mod 2^32.
//
// Representations used by the prover:
//   canonical      x in [0, r)                 (ABI, proofs, transcript)
//   Montgomery     x.R mod r                   (device arithmetic)
//   double-Mont.   x.R^2 mod r                 (eq-table weights of the int16
//                  fold: one REDC of sum(E.R^2 . p) lands in Montgomery form)
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define VL_HD __host__ __device__ __forceinline__
#else
#define VL_HD inline
#endif

namespace vl {

// 16-byte aligned: elements move as two 16-byte loads or stores.
struct alignas(16) Fr {
  uint32_t v[8];
};

VL_HD constexpr uint32_t r_limb(int i) {
  return i == 0 ? 0x00000001u : i == 1 ? 0xffffffffu : i == 2 ? 0xfffe5bfeu
       : i == 3 ? 0x53bda402u : i == 4 ? 0x09a1d805u : i == 5 ? 0x3339d808u
       : i == 6 ? 0x299d7d48u : 0x73eda753u;
}
VL_HD constexpr uint32_t r1_limb(int i) {  // R mod r  (Montgomery form of 1)
  return i == 0 ? 0xfffffffeu : i == 1 ? 0x00000001u : i == 2 ? 0x00034802u
       : i == 3 ? 0x5884b7fau : i == 4 ? 0xecbc4ff5u : i == 5 ? 0x998c4fefu
       : i == 6 ? 0xacc5056fu : 0x1824b159u;
}
VL_HD constexpr uint32_t r2_limb(int i) {  // R^2 mod r
  return i == 0 ? 0xf3f29c6du : i == 1 ? 0xc999e990u : i == 2 ? 0x87925c23u
       : i == 3 ? 0x2b6cedcbu : i == 4 ? 0x7254398fu : i == 5 ? 0x05d31496u
       : i == 6 ? 0x9f59ff11u : 0x0748d9d9u;
}
VL_HD constexpr uint32_t r3_limb(int i) {  // R^3 mod r
  return i == 0 ? 0x439b73afu : i == 1 ? 0xc62c1807u : i == 2 ? 0x8cf06990u
       : i == 3 ? 0x1b3e0d18u : i == 4 ? 0xc7b5f418u : i == 5 ? 0x73d13c71u
       : i == 6 ? 0xc8db33e9u : 0x6e2a5bb9u;
}
static constexpr uint32_t NPRIME = 0xffffffffu;  // -r^-1 mod 2^32 (r = 1 mod 2^32)

VL_HD void cond_sub_r(uint32_t (&t)[8], uint32_t hi);

VL_HD Fr fr_zero() { Fr z; for (int i = 0; i < 8; i++) z.v[i] = 0; return z; }
VL_HD Fr fr_small(uint32_t x) { Fr z = fr_zero(); z.v[0] = x; return z; }
VL_HD Fr fr_r1() { Fr z; for (int i = 0; i < 8; i++) z.v[i] = r1_limb(i); return z; }
VL_HD Fr fr_r2() { Fr z; for (int i = 0; i < 8; i++) z.v[i] = r2_limb(i); return z; }
VL_HD Fr fr_r3() { Fr z; for (int i = 0; i < 8; i++) z.v[i] = r3_limb(i); return z; }

VL_HD bool fr_is_zero(const Fr& a) {
  uint32_t o = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) o |= a.v[i];
  return o == 0;
}

VL_HD bool fr_eq(const Fr& a, const Fr& b) {
  uint32_t o = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) o |= a.v[i] ^ b.v[i];
  return o == 0;
}

#if defined(__CUDACC__)
// Device arithmetic on carry chains (PTX add.cc / mad.cc).  The C forms below
// (64-bit temporaries, used on the host) spend about three ALU instructions
// per limb on carries; with the flag kept in the condition code a limb costs
// one instruction, and a product's mad.lo.cc / madc.hi.cc pair on an aligned
// pair of words one wide multiply-add.  Measured on a GB300 (152 x 8 CTAs of
// 256 threads): additions 354 -> 832 G/s, subtractions 425 -> 868 G/s,
// Montgomery products 45.5 -> 63.9 G/s (of 78.7 G/s if the wide multiply-adds
// of a textbook product were all that ran).

// d = a + b mod 2^256.
__device__ __forceinline__ void add8(uint32_t (&d)[8], const uint32_t (&a)[8], const uint32_t (&b)[8]) {
  asm("add.cc.u32 %0, %8, %16; addc.cc.u32 %1, %9, %17; addc.cc.u32 %2, %10, %18; addc.cc.u32 %3, %11, %19;\n\t"
      "addc.cc.u32 %4, %12, %20; addc.cc.u32 %5, %13, %21; addc.cc.u32 %6, %14, %22; addc.u32 %7, %15, %23;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]), "r"(b[1]),
        "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
}

// d = a - b mod 2^256; returns 0xffffffff if it wrapped, else 0.
__device__ __forceinline__ uint32_t sub8(uint32_t (&d)[8], const uint32_t (&a)[8], const uint32_t (&b)[8]) {
  uint32_t w;
  asm("sub.cc.u32 %0, %9, %17; subc.cc.u32 %1, %10, %18; subc.cc.u32 %2, %11, %19; subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21; subc.cc.u32 %5, %14, %22; subc.cc.u32 %6, %15, %23; subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32 %8, 0, 0;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(w)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]), "r"(b[1]),
        "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  return w;
}

// A running product or reduction is kept as two arrays, value = e + 2^32 o:
// e[2i], e[2i+1] and o[2i], o[2i+1] are the aligned word pairs that wide
// multiply-adds by the even and the odd limbs of the other factor land on.

// o += a_odd b, e += a_even b (first row: e, o overwritten).
__device__ __forceinline__ void mul_row0(uint32_t (&e)[8], uint32_t (&o)[8], const uint32_t (&a)[8], uint32_t b) {
  asm("mul.lo.u32 %0, %8, %12; mul.hi.u32 %1, %8, %12; mul.lo.u32 %2, %9, %12; mul.hi.u32 %3, %9, %12;\n\t"
      "mul.lo.u32 %4, %10, %12; mul.hi.u32 %5, %10, %12; mul.lo.u32 %6, %11, %12; mul.hi.u32 %7, %11, %12;"
      : "=&r"(e[0]), "=&r"(e[1]), "=&r"(e[2]), "=&r"(e[3]), "=&r"(e[4]), "=&r"(e[5]), "=&r"(e[6]), "=&r"(e[7])
      : "r"(a[0]), "r"(a[2]), "r"(a[4]), "r"(a[6]), "r"(b));
  asm("mul.lo.u32 %0, %8, %12; mul.hi.u32 %1, %8, %12; mul.lo.u32 %2, %9, %12; mul.hi.u32 %3, %9, %12;\n\t"
      "mul.lo.u32 %4, %10, %12; mul.hi.u32 %5, %10, %12; mul.lo.u32 %6, %11, %12; mul.hi.u32 %7, %11, %12;"
      : "=&r"(o[0]), "=&r"(o[1]), "=&r"(o[2]), "=&r"(o[3]), "=&r"(o[4]), "=&r"(o[5]), "=&r"(o[6]), "=&r"(o[7])
      : "r"(a[1]), "r"(a[3]), "r"(a[5]), "r"(a[7]), "r"(b));
}

// Add m r with m = -e[0] (r = 1 mod 2^32, so n' = -1), which makes e[0] zero.
// r's lowest limb is 1: its product with m is an addition.
__device__ __forceinline__ void redc_row(uint32_t (&e)[8], uint32_t (&o)[8]) {
  const uint32_t m = 0u - e[0];
  asm("mad.lo.cc.u32 %0, %8, %9, %0; madc.hi.cc.u32 %1, %8, %9, %1; madc.lo.cc.u32 %2, %8, %10, %2;\n\t"
      "madc.hi.cc.u32 %3, %8, %10, %3; madc.lo.cc.u32 %4, %8, %11, %4; madc.hi.cc.u32 %5, %8, %11, %5;\n\t"
      "madc.lo.cc.u32 %6, %8, %12, %6; madc.hi.u32 %7, %8, %12, %7;"
      : "+&r"(o[0]), "+&r"(o[1]), "+&r"(o[2]), "+&r"(o[3]), "+&r"(o[4]), "+&r"(o[5]), "+&r"(o[6]), "+&r"(o[7])
      : "r"(m), "r"(r_limb(1)), "r"(r_limb(3)), "r"(r_limb(5)), "r"(r_limb(7)));
  asm("add.cc.u32 %0, %0, %9; addc.cc.u32 %1, %1, 0; madc.lo.cc.u32 %2, %9, %10, %2;\n\t"
      "madc.hi.cc.u32 %3, %9, %10, %3; madc.lo.cc.u32 %4, %9, %11, %4; madc.hi.cc.u32 %5, %9, %11, %5;\n\t"
      "madc.lo.cc.u32 %6, %9, %12, %6; madc.hi.cc.u32 %7, %9, %12, %7; addc.u32 %8, %8, 0;"
      : "+&r"(e[0]), "+&r"(e[1]), "+&r"(e[2]), "+&r"(e[3]), "+&r"(e[4]), "+&r"(e[5]), "+&r"(e[6]), "+&r"(e[7]), "+&r"(o[7])
      : "r"(m), "r"(r_limb(2)), "r"(r_limb(4)), "r"(r_limb(6)));
}

// Drop the zero word e[0] (the value moves down by 2^32: o becomes the even
// array with e[1] added at its bottom, e[2..7] the odd one) and add a b.
__device__ __forceinline__ void mul_row(uint32_t (&e)[8], uint32_t (&o)[8], const uint32_t (&a)[8], uint32_t b) {
  uint32_t n[8];
  asm("add.cc.u32 %8, %8, %9; madc.lo.cc.u32 %0, %16, %20, %10; madc.hi.cc.u32 %1, %16, %20, %11;\n\t"
      "madc.lo.cc.u32 %2, %17, %20, %12; madc.hi.cc.u32 %3, %17, %20, %13; madc.lo.cc.u32 %4, %18, %20, %14;\n\t"
      "madc.hi.cc.u32 %5, %18, %20, %15; madc.lo.cc.u32 %6, %19, %20, 0; madc.hi.u32 %7, %19, %20, 0;"
      : "=&r"(n[0]), "=&r"(n[1]), "=&r"(n[2]), "=&r"(n[3]), "=&r"(n[4]), "=&r"(n[5]), "=&r"(n[6]), "=&r"(n[7]),
        "+&r"(o[0])
      : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(a[1]), "r"(a[3]), "r"(a[5]),
        "r"(a[7]), "r"(b));
  asm("mad.lo.cc.u32 %0, %9, %13, %0; madc.hi.cc.u32 %1, %9, %13, %1; madc.lo.cc.u32 %2, %10, %13, %2;\n\t"
      "madc.hi.cc.u32 %3, %10, %13, %3; madc.lo.cc.u32 %4, %11, %13, %4; madc.hi.cc.u32 %5, %11, %13, %5;\n\t"
      "madc.lo.cc.u32 %6, %12, %13, %6; madc.hi.cc.u32 %7, %12, %13, %7; addc.u32 %8, %8, 0;"
      : "+&r"(o[0]), "+&r"(o[1]), "+&r"(o[2]), "+&r"(o[3]), "+&r"(o[4]), "+&r"(o[5]), "+&r"(o[6]), "+&r"(o[7]), "+&r"(n[7])
      : "r"(a[0]), "r"(a[2]), "r"(a[4]), "r"(a[6]), "r"(b));
#pragma unroll
  for (int j = 0; j < 8; j++) {
    e[j] = o[j];
    o[j] = n[j];
  }
}

// Drop the zero word e[0] and run the next reduction row: the carry of the
// drop goes straight into the row's odd chain.
__device__ __forceinline__ void redc_next(uint32_t (&e)[8], uint32_t (&o)[8]) {
  uint32_t n[8], m;
  asm("add.cc.u32 %8, %8, %10; sub.u32 %9, 0, %8; madc.lo.cc.u32 %0, %9, %17, %11;\n\t"
      "madc.hi.cc.u32 %1, %9, %17, %12; madc.lo.cc.u32 %2, %9, %18, %13; madc.hi.cc.u32 %3, %9, %18, %14;\n\t"
      "madc.lo.cc.u32 %4, %9, %19, %15; madc.hi.cc.u32 %5, %9, %19, %16; madc.lo.cc.u32 %6, %9, %20, 0;\n\t"
      "madc.hi.u32 %7, %9, %20, 0;"
      : "=&r"(n[0]), "=&r"(n[1]), "=&r"(n[2]), "=&r"(n[3]), "=&r"(n[4]), "=&r"(n[5]), "=&r"(n[6]), "=&r"(n[7]),
        "+&r"(o[0]), "=&r"(m)
      : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(r_limb(1)), "r"(r_limb(3)),
        "r"(r_limb(5)), "r"(r_limb(7)));
  asm("add.cc.u32 %0, %0, %9; addc.cc.u32 %1, %1, 0; madc.lo.cc.u32 %2, %9, %10, %2;\n\t"
      "madc.hi.cc.u32 %3, %9, %10, %3; madc.lo.cc.u32 %4, %9, %11, %4; madc.hi.cc.u32 %5, %9, %11, %5;\n\t"
      "madc.lo.cc.u32 %6, %9, %12, %6; madc.hi.cc.u32 %7, %9, %12, %7; addc.u32 %8, %8, 0;"
      : "+&r"(o[0]), "+&r"(o[1]), "+&r"(o[2]), "+&r"(o[3]), "+&r"(o[4]), "+&r"(o[5]), "+&r"(o[6]), "+&r"(o[7]), "+&r"(n[7])
      : "r"(m), "r"(r_limb(2)), "r"(r_limb(4)), "r"(r_limb(6)));
#pragma unroll
  for (int j = 0; j < 8; j++) {
    e[j] = o[j];
    o[j] = n[j];
  }
}

// o + e / 2^32 for e[0] = 0 (a value below 2^256).
__device__ __forceinline__ Fr join_rows(const uint32_t (&e)[8], const uint32_t (&o)[8]) {
  const uint32_t s[8] = {e[1], e[2], e[3], e[4], e[5], e[6], e[7], 0u};
  Fr x;
  add8(x.v, o, s);
  return x;
}

// w += a b for a 17-limb accumulator (512-bit products, unreduced; up to 2^34
// of them): half a Montgomery product's multiply-adds.  A sum of products
// is reduced once at its end (wide_redc).
__device__ __forceinline__ void wide_mac(uint32_t (&w)[17], const Fr& a, const Fr& b) {
  uint32_t e[8], o[8];
  asm("mul.lo.u32 %0, %8, %12; mul.hi.u32 %1, %8, %12; mul.lo.u32 %2, %9, %12; mul.hi.u32 %3, %9, %12;\n\t"
      "mul.lo.u32 %4, %10, %12; mul.hi.u32 %5, %10, %12; mul.lo.u32 %6, %11, %12; mul.hi.u32 %7, %11, %12;"
      : "=&r"(o[0]), "=&r"(o[1]), "=&r"(o[2]), "=&r"(o[3]), "=&r"(o[4]), "=&r"(o[5]), "=&r"(o[6]), "=&r"(o[7])
      : "r"(a.v[1]), "r"(a.v[3]), "r"(a.v[5]), "r"(a.v[7]), "r"(b.v[0]));
#pragma unroll
  for (int j = 0; j < 8; j++) e[j] = w[j];
  asm("mad.lo.cc.u32 %0, %9, %13, %0; madc.hi.cc.u32 %1, %9, %13, %1; madc.lo.cc.u32 %2, %10, %13, %2;\n\t"
      "madc.hi.cc.u32 %3, %10, %13, %3; madc.lo.cc.u32 %4, %11, %13, %4; madc.hi.cc.u32 %5, %11, %13, %5;\n\t"
      "madc.lo.cc.u32 %6, %12, %13, %6; madc.hi.cc.u32 %7, %12, %13, %7; addc.u32 %8, %8, 0;"
      : "+&r"(e[0]), "+&r"(e[1]), "+&r"(e[2]), "+&r"(e[3]), "+&r"(e[4]), "+&r"(e[5]), "+&r"(e[6]), "+&r"(e[7]),
        "+&r"(o[7])
      : "r"(a.v[0]), "r"(a.v[2]), "r"(a.v[4]), "r"(a.v[6]), "r"(b.v[0]));
  w[0] = e[0];
#pragma unroll
  for (int i = 1; i < 8; i++) {
    mul_row(e, o, a.v, b.v[i]);
    w[i] = e[0];
  }
  const Fr hi = join_rows(e, o);
  asm("add.cc.u32 %0, %0, %9; addc.cc.u32 %1, %1, %10; addc.cc.u32 %2, %2, %11; addc.cc.u32 %3, %3, %12;\n\t"
      "addc.cc.u32 %4, %4, %13; addc.cc.u32 %5, %5, %14; addc.cc.u32 %6, %6, %15; addc.cc.u32 %7, %7, %16;\n\t"
      "addc.u32 %8, %8, 0;"
      : "+&r"(w[8]), "+&r"(w[9]), "+&r"(w[10]), "+&r"(w[11]), "+&r"(w[12]), "+&r"(w[13]), "+&r"(w[14]), "+&r"(w[15]),
        "+&r"(w[16])
      : "r"(hi.v[0]), "r"(hi.v[1]), "r"(hi.v[2]), "r"(hi.v[3]), "r"(hi.v[4]), "r"(hi.v[5]), "r"(hi.v[6]),
        "r"(hi.v[7]));
}

// (t + m r) / 2^256 for the m that makes it whole, t < 2^256: in [0, r].
__device__ __forceinline__ Fr redc_low(const uint32_t (&t)[8]) {
  uint32_t e[8], o[8];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    e[j] = t[j];
    o[j] = 0;
  }
  redc_row(e, o);
#pragma unroll
  for (int i = 1; i < 8; i++) redc_next(e, o);
  return join_rows(e, o);
}

// The Montgomery reduction of a sum of n products of reduced elements, as
// eight 64-bit columns (the ninth limb on top of the last column): below
// (0.46 n + 1) r, to be added to other such sums and reduced by redc_columns.
__device__ __forceinline__ void wide_redc(const uint32_t (&w)[17], unsigned long long (&col)[8]) {
  uint32_t lo[8], hi[8], top;
#pragma unroll
  for (int j = 0; j < 8; j++) lo[j] = w[j];
  const Fr x = redc_low(lo);
  asm("add.cc.u32 %0, %9, %17; addc.cc.u32 %1, %10, %18; addc.cc.u32 %2, %11, %19; addc.cc.u32 %3, %12, %20;\n\t"
      "addc.cc.u32 %4, %13, %21; addc.cc.u32 %5, %14, %22; addc.cc.u32 %6, %15, %23; addc.cc.u32 %7, %16, %24;\n\t"
      "addc.u32 %8, %25, 0;"
      : "=&r"(hi[0]), "=&r"(hi[1]), "=&r"(hi[2]), "=&r"(hi[3]), "=&r"(hi[4]), "=&r"(hi[5]), "=&r"(hi[6]),
        "=&r"(hi[7]), "=&r"(top)
      : "r"(x.v[0]), "r"(x.v[1]), "r"(x.v[2]), "r"(x.v[3]), "r"(x.v[4]), "r"(x.v[5]), "r"(x.v[6]), "r"(x.v[7]),
        "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]), "r"(w[16]));
#pragma unroll
  for (int j = 0; j < 8; j++) col[j] = hi[j];
  col[7] |= (unsigned long long)top << 32;
}

// z = a m (nine limbs).
__device__ __forceinline__ void small_mul(uint32_t (&z)[9], const uint32_t (&a)[8], uint32_t m) {
  uint32_t o[8];
  asm("mul.lo.u32 %0, %8, %12; mul.hi.u32 %1, %8, %12; mul.lo.u32 %2, %9, %12; mul.hi.u32 %3, %9, %12;\n\t"
      "mul.lo.u32 %4, %10, %12; mul.hi.u32 %5, %10, %12; mul.lo.u32 %6, %11, %12; mul.hi.u32 %7, %11, %12;"
      : "=&r"(z[0]), "=&r"(z[1]), "=&r"(z[2]), "=&r"(z[3]), "=&r"(z[4]), "=&r"(z[5]), "=&r"(z[6]), "=&r"(z[7])
      : "r"(a[0]), "r"(a[2]), "r"(a[4]), "r"(a[6]), "r"(m));
  asm("mul.lo.u32 %0, %8, %12; mul.hi.u32 %1, %8, %12; mul.lo.u32 %2, %9, %12; mul.hi.u32 %3, %9, %12;\n\t"
      "mul.lo.u32 %4, %10, %12; mul.hi.u32 %5, %10, %12; mul.lo.u32 %6, %11, %12; mul.hi.u32 %7, %11, %12;"
      : "=&r"(o[0]), "=&r"(o[1]), "=&r"(o[2]), "=&r"(o[3]), "=&r"(o[4]), "=&r"(o[5]), "=&r"(o[6]), "=&r"(o[7])
      : "r"(a[1]), "r"(a[3]), "r"(a[5]), "r"(a[7]), "r"(m));
  asm("add.cc.u32 %0, %0, %8; addc.cc.u32 %1, %1, %9; addc.cc.u32 %2, %2, %10; addc.cc.u32 %3, %3, %11;\n\t"
      "addc.cc.u32 %4, %4, %12; addc.cc.u32 %5, %5, %13; addc.cc.u32 %6, %6, %14; addc.u32 %7, %15, 0;"
      : "+&r"(z[1]), "+&r"(z[2]), "+&r"(z[3]), "+&r"(z[4]), "+&r"(z[5]), "+&r"(z[6]), "+&r"(z[7]), "=&r"(z[8])
      : "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]));
}

// t mod r for t < 2^273: Barrett with a 32-bit quotient estimate.  With x =
// floor(t / 2^241) and M = floor(2^273 / r), q = floor(x M / 2^32) satisfies
// t / r - 2.0001 < q <= t / r: the remainder is below 2.0001 r < 2^256.
__device__ __forceinline__ Fr small_reduce(const uint32_t (&t)[9]) {
  uint32_t p[9];
  const uint32_t x = (t[8] << 15) | (t[7] >> 17);
  const uint32_t q = __umulhi(x, 289441u);
  const uint32_t r[8] = {r_limb(0), r_limb(1), r_limb(2), r_limb(3), r_limb(4), r_limb(5), r_limb(6), r_limb(7)};
  small_mul(p, r, q);
  Fr out;
  const uint32_t lo[8] = {t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7]};
  const uint32_t ql[8] = {p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7]};
  (void)sub8(out.v, lo, ql);  // the ninth limbs cancel
  cond_sub_r(out.v, 0);
  cond_sub_r(out.v, 0);
  return out;
}

// a m mod r for m < 2^18 (a reduced): an eighth of a Montgomery product's
// multiply-adds.
__device__ __forceinline__ Fr small_mul_mod(const Fr& a, uint32_t m) {
  uint32_t t[9];
  small_mul(t, a.v, m);
  return small_reduce(t);
}

// t += z (nine limbs).
__device__ __forceinline__ void add9(uint32_t (&t)[9], const uint32_t (&z)[9]) {
  asm("add.cc.u32 %0, %0, %9; addc.cc.u32 %1, %1, %10; addc.cc.u32 %2, %2, %11; addc.cc.u32 %3, %3, %12;\n\t"
      "addc.cc.u32 %4, %4, %13; addc.cc.u32 %5, %5, %14; addc.cc.u32 %6, %6, %15; addc.cc.u32 %7, %7, %16;\n\t"
      "addc.u32 %8, %8, %17;"
      : "+&r"(t[0]), "+&r"(t[1]), "+&r"(t[2]), "+&r"(t[3]), "+&r"(t[4]), "+&r"(t[5]), "+&r"(t[6]), "+&r"(t[7]),
        "+&r"(t[8])
      : "r"(z[0]), "r"(z[1]), "r"(z[2]), "r"(z[3]), "r"(z[4]), "r"(z[5]), "r"(z[6]), "r"(z[7]), "r"(z[8]));
}

// w += a z for a nine-limb z (the caller keeps the sum below 2^544).
__device__ __forceinline__ void wide_mac9(uint32_t (&w)[17], const Fr& a, const uint32_t (&z)[9]) {
  uint32_t y[9];
  Fr zl;
#pragma unroll
  for (int i = 0; i < 8; i++) zl.v[i] = z[i];
  wide_mac(w, a, zl);
  small_mul(y, a.v, z[8]);
  asm("add.cc.u32 %0, %0, %9; addc.cc.u32 %1, %1, %10; addc.cc.u32 %2, %2, %11; addc.cc.u32 %3, %3, %12;\n\t"
      "addc.cc.u32 %4, %4, %13; addc.cc.u32 %5, %5, %14; addc.cc.u32 %6, %6, %15; addc.cc.u32 %7, %7, %16;\n\t"
      "addc.u32 %8, %8, %17;"
      : "+&r"(w[8]), "+&r"(w[9]), "+&r"(w[10]), "+&r"(w[11]), "+&r"(w[12]), "+&r"(w[13]), "+&r"(w[14]), "+&r"(w[15]),
        "+&r"(w[16])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(y[8]));
}

// w += a (b m) for m < 2^16: up to 2^17 terms of at most 2^526.
__device__ __forceinline__ void wide_mac_small(uint32_t (&w)[17], const Fr& a, const Fr& b, uint32_t m) {
  uint32_t z[9];
  small_mul(z, b.v, m);
  wide_mac9(w, a, z);
}

// s += a for a nine-limb sum of reduced elements.
__device__ __forceinline__ void sum9_add(uint32_t (&s)[9], const Fr& a) {
  asm("add.cc.u32 %0, %0, %9; addc.cc.u32 %1, %1, %10; addc.cc.u32 %2, %2, %11; addc.cc.u32 %3, %3, %12;\n\t"
      "addc.cc.u32 %4, %4, %13; addc.cc.u32 %5, %5, %14; addc.cc.u32 %6, %6, %15; addc.cc.u32 %7, %7, %16;\n\t"
      "addc.u32 %8, %8, 0;"
      : "+&r"(s[0]), "+&r"(s[1]), "+&r"(s[2]), "+&r"(s[3]), "+&r"(s[4]), "+&r"(s[5]), "+&r"(s[6]), "+&r"(s[7]),
        "+&r"(s[8])
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]), "r"(a.v[7]));
}
__device__ __forceinline__ void sum9_columns(const uint32_t (&s)[9], unsigned long long (&col)[8]) {
#pragma unroll
  for (int j = 0; j < 8; j++) col[j] = s[j];
  col[7] |= (unsigned long long)s[8] << 32;
}
#endif

// t - r if t >= r else t  (t < 2^256 given as 8 limbs plus an overflow limb hi).
VL_HD void cond_sub_r(uint32_t (&t)[8], uint32_t hi) {
  uint32_t d[8];
#if defined(__CUDA_ARCH__)
  const uint32_t r[8] = {r_limb(0), r_limb(1), r_limb(2), r_limb(3), r_limb(4), r_limb(5), r_limb(6), r_limb(7)};
  const uint32_t borrow = sub8(d, t, r);
#else
  uint64_t borrow = 0;
  for (int i = 0; i < 8; i++) {
    uint64_t x = (uint64_t)t[i] - r_limb(i) - borrow;
    d[i] = (uint32_t)x;
    borrow = (x >> 63) & 1;
  }
#endif
  // t >= r iff no borrow out of the 256-bit subtraction, or hi is set.
  bool take = (hi != 0) || (borrow == 0);
#pragma unroll
  for (int i = 0; i < 8; i++) t[i] = take ? d[i] : t[i];
}

VL_HD bool lt_r(const Fr& a) {
  uint64_t borrow = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    uint64_t x = (uint64_t)a.v[i] - r_limb(i) - borrow;
    borrow = (x >> 63) & 1;
  }
  return borrow != 0;
}

VL_HD Fr fr_add(const Fr& a, const Fr& b) {
  Fr s;
#if defined(__CUDA_ARCH__)
  add8(s.v, a.v, b.v);  // below 2r < 2^256: no carry out
  cond_sub_r(s.v, 0);
#else
  uint64_t c = 0;
  for (int i = 0; i < 8; i++) {
    c += (uint64_t)a.v[i] + b.v[i];
    s.v[i] = (uint32_t)c;
    c >>= 32;
  }
  cond_sub_r(s.v, (uint32_t)c);
#endif
  return s;
}

VL_HD Fr fr_sub(const Fr& a, const Fr& b) {
  Fr d;
#if defined(__CUDA_ARCH__)
  // Add r back when the subtraction wrapped.
  const uint32_t w = sub8(d.v, a.v, b.v);
  const uint32_t rw[8] = {r_limb(0) & w, r_limb(1) & w, r_limb(2) & w, r_limb(3) & w,
                          r_limb(4) & w, r_limb(5) & w, r_limb(6) & w, r_limb(7) & w};
  add8(d.v, d.v, rw);
#else
  uint64_t borrow = 0;
  for (int i = 0; i < 8; i++) {
    uint64_t x = (uint64_t)a.v[i] - b.v[i] - borrow;
    d.v[i] = (uint32_t)x;
    borrow = (x >> 63) & 1;
  }
  // Add r back when the subtraction wrapped.
  uint32_t mask = borrow ? 0xffffffffu : 0u;
  uint64_t c = 0;
  for (int i = 0; i < 8; i++) {
    c += (uint64_t)d.v[i] + (r_limb(i) & mask);
    d.v[i] = (uint32_t)c;
    c >>= 32;
  }
#endif
  return d;
}

VL_HD Fr fr_neg(const Fr& a) { return fr_sub(fr_zero(), a); }
VL_HD Fr fr_dbl(const Fr& a) { return fr_add(a, a); }

// Montgomery product a.b.R^-1 mod r (row by row, one reduction row after each
// row of products).  Inputs a < 2^256, b < r; the output is reduced (< r).
VL_HD Fr mont_mul(const Fr& a, const Fr& b) {
#if defined(__CUDA_ARCH__)
  // The rows run over a's limbs: a row adds b a_i < r 2^32 and m r < r 2^32 to
  // a value below 2r, which fits the nine words for any a < 2^256.
  uint32_t e[8], o[8];
  mul_row0(e, o, b.v, a.v[0]);
  redc_row(e, o);
#pragma unroll
  for (int i = 1; i < 8; i++) {
    mul_row(e, o, b.v, a.v[i]);
    redc_row(e, o);
  }
  Fr out = join_rows(e, o);  // below 2r: a b / 2^256 < r, m r / 2^256 < r
  cond_sub_r(out.v, 0);
  return out;
#else
  uint32_t t[10];
  for (int j = 0; j < 10; j++) t[j] = 0;
  for (int i = 0; i < 8; i++) {
    uint64_t c = 0;
    for (int j = 0; j < 8; j++) {
      c += (uint64_t)a.v[j] * b.v[i] + t[j];
      t[j] = (uint32_t)c;
      c >>= 32;
    }
    c += t[8];
    t[8] = (uint32_t)c;
    t[9] = (uint32_t)(c >> 32);
    uint32_t m = t[0] * NPRIME;
    c = ((uint64_t)m * r_limb(0) + t[0]) >> 32;
    for (int j = 1; j < 8; j++) {
      c += (uint64_t)m * r_limb(j) + t[j];
      t[j - 1] = (uint32_t)c;
      c >>= 32;
    }
    c += t[8];
    t[7] = (uint32_t)c;
    t[8] = t[9] + (uint32_t)(c >> 32);
  }
  Fr out;
  for (int j = 0; j < 8; j++) out.v[j] = t[j];
  cond_sub_r(out.v, t[8]);
  return out;
#endif
}

VL_HD Fr to_mont(const Fr& a) { return mont_mul(a, fr_r2()); }
VL_HD Fr from_mont(const Fr& a) {
#if defined(__CUDA_ARCH__)
  Fr x = redc_low(a.v);  // the product by 1: only the reduction rows
  cond_sub_r(x.v, 0);
  return x;
#else
  return mont_mul(a, fr_small(1));
#endif
}

#if defined(__CUDACC__)
// The ten limbs of V = sum_l acc[l] . 2^(32 l), one carry chain over the words
// of the columns.
__device__ __forceinline__ void column_limbs(const uint64_t (&acc)[8], uint32_t (&t)[10]) {
  uint32_t w[16];
#pragma unroll
  for (int l = 0; l < 8; l++) {
    w[2 * l] = (uint32_t)acc[l];
    w[2 * l + 1] = (uint32_t)(acc[l] >> 32);
  }
  t[0] = w[0];
  asm("add.cc.u32 %0, %9, %10; addc.cc.u32 %1, %11, %12; addc.cc.u32 %2, %13, %14; addc.cc.u32 %3, %15, %16;\n\t"
      "addc.cc.u32 %4, %17, %18; addc.cc.u32 %5, %19, %20; addc.cc.u32 %6, %21, %22; addc.cc.u32 %7, %23, 0;\n\t"
      "addc.u32 %8, 0, 0;"
      : "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]), "=&r"(t[6]), "=&r"(t[7]), "=&r"(t[8]),
        "=&r"(t[9])
      : "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(w[8]), "r"(w[9]), "r"(w[10]),
        "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]));
}
#endif

// Montgomery reduction of a wide value V = sum_l acc[l] . 2^(32 l) given as
// eight unsigned 64-bit column sums: returns V . R^-1 mod r (reduced).
// V < 2^289, so the REDC result is below 2r before the final subtraction.
VL_HD Fr redc_columns(const uint64_t acc[8]) {
#if defined(__CUDA_ARCH__)
  uint32_t v[10], t[8], top[8];
  const uint64_t c[8] = {acc[0], acc[1], acc[2], acc[3], acc[4], acc[5], acc[6], acc[7]};
  column_limbs(c, v);
#pragma unroll
  for (int j = 0; j < 8; j++) {
    t[j] = v[j];
    top[j] = j < 2 ? v[8 + j] : 0u;
  }
  // V / 2^256 = (low 256 bits) / 2^256 (Montgomery, at most r) + the top limbs (below 2^33)
  Fr out = redc_low(t);
  add8(out.v, out.v, top);
  cond_sub_r(out.v, 0);
  return out;
#else
  uint32_t t[18];
  uint64_t carry = 0;
  for (int l = 0; l < 8; l++) {
    uint64_t s = (acc[l] & 0xffffffffull) + carry;
    t[l] = (uint32_t)s;
    carry = (acc[l] >> 32) + (s >> 32);
  }
  t[8] = (uint32_t)carry;
  t[9] = (uint32_t)(carry >> 32);
  for (int j = 10; j < 18; j++) t[j] = 0;
  for (int i = 0; i < 8; i++) {
    uint32_t m = t[i] * NPRIME;
    uint64_t c = 0;
    for (int j = 0; j < 8; j++) {
      c += (uint64_t)m * r_limb(j) + t[i + j];
      t[i + j] = (uint32_t)c;
      c >>= 32;
    }
    for (int j = i + 8; j < 18; j++) {
      c += t[j];
      t[j] = (uint32_t)c;
      c >>= 32;
    }
  }
  Fr out;
  for (int j = 0; j < 8; j++) out.v[j] = t[8 + j];
  cond_sub_r(out.v, t[16]);
  return out;
#endif
}

// Reduce a 512-bit little-endian value (lo + hi.2^256) mod r; canonical out.
VL_HD Fr reduce_512(const Fr& lo, const Fr& hi) {
  // hi.2^256 = hi.R = mont_mul(hi, R^2) (valid for unreduced hi < 2^256).
  Fr h = mont_mul(hi, fr_r2());
  Fr l = lo;
  cond_sub_r(l.v, 0);
  cond_sub_r(l.v, 0);  // 2^256 < 3r: two subtractions reduce any 256-bit value
  return fr_add(l, h);
}

// Inverse of a canonical nonzero a (canonical result; 0 for 0), by the binary
// GCD with batched updates of T. Pornin, "Optimized Binary GCD for Modular
// Inversion" (IACR ePrint 2020/972): x, y start at a, r with x = a u, y = a v
// (mod r).  A batch runs 31 steps on 64-bit approximations of x and y (their low
// 31 and top 33 bits), collecting the steps as a 2 x 2 matrix with entries of at
// most 2^31, then applies the matrix once to (x, y), dividing by 2^31 exactly,
// and to (u, v), dividing by 2^31 mod r (r = 1 mod 2^31: the multiple of r to
// add is -t mod 2^31).  17 batches (2 . 255 - 1 <= 17 . 31) leave y = 1, v = 1/a.
// One thread needs about 12 us on the GPU, against 110 us for a plain binary
// Euclid on eight limbs, which moves every limb in every step.
VL_HD int bit_length(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return 32 - __clz((int)x);
#else
  int n = 0;
  for (; x; x >>= 1) n++;
  return n;
#endif
}
VL_HD uint64_t inv_approx(const uint32_t (&x)[8], int n) {  // n >= 64: bits of max(x, y)
  const int sft = n - 33, i = sft >> 5, b = sft & 31;
  const uint64_t lo = (uint64_t)x[i] | ((uint64_t)x[i + 1] << 32);  // i <= 6
  const uint64_t hi = i + 2 < 8 ? x[i + 2] : 0u;
  const uint64_t top = ((lo >> b) | (b ? hi << (64 - b) : 0)) & 0x1ffffffffull;
  return (top << 31) | (x[0] & 0x7fffffffu);
}
// w = f x + g y as nine limbs (two's complement; |f| + |g| <= 2^31).
VL_HD void inv_combine(const uint32_t (&x)[8], int64_t f, const uint32_t (&y)[8], int64_t g, uint32_t (&w)[9]) {
  int64_t c = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    c += (int64_t)x[i] * f + (int64_t)y[i] * g;
    w[i] = (uint32_t)c;
    c >>= 32;
  }
  w[8] = (uint32_t)c;
}
// out = |w / 2^31| for w a multiple of 2^31; true if w was negative.
VL_HD bool inv_shift_abs(const uint32_t (&w)[9], uint32_t (&out)[8]) {
  const bool neg = w[8] >> 31;
  uint64_t c = neg ? 1 : 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const uint32_t t = (w[i] >> 31) | (w[i + 1] << 1);
    c += neg ? (uint32_t)~t : t;
    out[i] = (uint32_t)c;
    c >>= 32;
  }
  return neg;
}
// w / 2^31 mod r for |w| <= 2^31 r.
VL_HD void inv_shift_mod(uint32_t (&w)[9], Fr& out) {
  const uint32_t k = (0u - w[0]) & 0x7fffffffu;  // w + k r = 0 mod 2^31
  uint64_t c = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    c += (uint64_t)k * r_limb(i) + w[i];
    w[i] = (uint32_t)c;
    c >>= 32;
  }
  w[8] += (uint32_t)c;  // in (-2^31 r, 2^32 r): after the shift in (-r, 2 r)
  const bool neg = w[8] >> 31;
#pragma unroll
  for (int i = 0; i < 8; i++) out.v[i] = (w[i] >> 31) | (w[i + 1] << 1);
  if (neg) {
    uint64_t d = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
      d += (uint64_t)out.v[i] + r_limb(i);
      out.v[i] = (uint32_t)d;
      d >>= 32;
    }
  } else {
    cond_sub_r(out.v, 0);
  }
}
VL_HD Fr fr_inv_canonical(const Fr& a) {
  uint32_t x[8], y[8];
  Fr u = fr_small(1), v = fr_zero();
  for (int i = 0; i < 8; i++) {
    x[i] = a.v[i];
    y[i] = r_limb(i);
  }
  for (int batch = 0; batch < 17; batch++) {
    int n = 64;  // bits of max(x, y), at least 64
#pragma unroll
    for (int i = 2; i < 8; i++) {
      const uint32_t t = x[i] | y[i];
      if (t) n = 32 * i + bit_length(t);
    }
    uint64_t xa = inv_approx(x, n), ya = inv_approx(y, n);
    int64_t f0 = 1, g0 = 0, f1 = 0, g1 = 1;
    for (int j = 0; j < 31; j++) {
      const bool odd = xa & 1, swap = odd && xa < ya;
      const uint64_t xs = swap ? ya : xa, ys = swap ? xa : ya;
      const int64_t fa = swap ? f1 : f0, fb = swap ? f0 : f1, ga = swap ? g1 : g0, gb = swap ? g0 : g1;
      xa = (xs - (odd ? ys : 0)) >> 1;
      ya = ys;
      f0 = fa - (odd ? fb : 0);
      g0 = ga - (odd ? gb : 0);
      f1 = 2 * fb;
      g1 = 2 * gb;
    }
    uint32_t w0[9], w1[9];
    inv_combine(x, f0, y, g0, w0);
    inv_combine(x, f1, y, g1, w1);
    if (inv_shift_abs(w0, x)) f0 = -f0, g0 = -g0;
    if (inv_shift_abs(w1, y)) f1 = -f1, g1 = -g1;
    inv_combine(u.v, f0, v.v, g0, w0);
    inv_combine(u.v, f1, v.v, g1, w1);
    inv_shift_mod(w0, u);
    inv_shift_mod(w1, v);
  }
  return v;  // for a = 0: y stays r and v stays 0
}
// Inverse in Montgomery form (x.R -> x^-1.R): from_mont, canonical inverse, to_mont.
VL_HD Fr fr_inv_mont(const Fr& a) { return to_mont(fr_inv_canonical(from_mont(a))); }

// Signed integer x (|x| < 2^63) as a canonical field element.
VL_HD Fr fr_from_i64(int64_t x) {
  uint64_t mag = x < 0 ? (uint64_t)(-(x + 1)) + 1u : (uint64_t)x;
  Fr a = fr_zero();
  a.v[0] = (uint32_t)mag;
  a.v[1] = (uint32_t)(mag >> 32);
  return x < 0 ? fr_neg(a) : a;
}

}  // namespace vl
