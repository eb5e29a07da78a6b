// zc_field.cuh -- arithmetic in the BLS12-381 scalar field r on sm_103a.
//
// Elements are 8 x 32-bit little-endian limbs (32 bytes).  The device
// multiplier is a CIOS Montgomery product (Koc, Acar, Kaliski 1996) whose
// 64-bit partial products are accumulated in place by carry chains of wide
// multiply-adds (see zc_mul_row); r's low limb is 1, so -r^{-1} mod 2^32 =
// 0xffffffff and the per-row quotient digit is just the negated low word.
// r < 2^255 keeps every intermediate of a row inside nine words.
//
// "Level" bookkeeping: a Montgomery product of values x (stored as x R^i)
// and y (stored as y R^j) returns x y R^(i+j-1).  Canonical storage is level
// 0, the usual Montgomery form level 1.  The provers keep tables at whatever
// level makes the gate need no conversions and fold the R powers into
// per-proof constants.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define ZC_HD __host__ __device__ __forceinline__
#define ZC_D __device__ __forceinline__
#else
#define ZC_HD inline
#define ZC_D inline
#endif

namespace zc {

struct fr {
  uint32_t v[8];
};

// r = 0x73eda753299d7d483339d80809a1d80553bda402fffe5bfeffffffff00000001
#define ZC_P0 0x00000001u
#define ZC_P1 0xffffffffu
#define ZC_P2 0xfffe5bfeu
#define ZC_P3 0x53bda402u
#define ZC_P4 0x09a1d805u
#define ZC_P5 0x3339d808u
#define ZC_P6 0x299d7d48u
#define ZC_P7 0x73eda753u

// limb i of r (i is a compile-time constant after unrolling)
ZC_HD uint32_t p_limb(int i) {
  switch (i) {
    case 0: return ZC_P0;
    case 1: return ZC_P1;
    case 2: return ZC_P2;
    case 3: return ZC_P3;
    case 4: return ZC_P4;
    case 5: return ZC_P5;
    case 6: return ZC_P6;
    default: return ZC_P7;
  }
}

ZC_HD fr fr_zero() {
  fr z;
  for (int i = 0; i < 8; i++) z.v[i] = 0;
  return z;
}

ZC_HD bool fr_is_zero(const fr& a) {
  uint32_t x = 0;
  for (int i = 0; i < 8; i++) x |= a.v[i];
  return x == 0;
}

ZC_HD bool fr_equal(const fr& a, const fr& b) {
  uint32_t x = 0;
  for (int i = 0; i < 8; i++) x |= a.v[i] ^ b.v[i];
  return x == 0;
}

// a < r as an integer (canonical check)
ZC_HD bool fr_is_canonical(const fr& a) {
  const uint32_t P[8] = {ZC_P0, ZC_P1, ZC_P2, ZC_P3, ZC_P4, ZC_P5, ZC_P6, ZC_P7};
  for (int i = 7; i >= 0; i--) {
    if (a.v[i] != P[i]) return a.v[i] < P[i];
  }
  return false;
}

// ---------------------------------------------------------------- generic --
// Portable versions (host verifier, set-up constants).  64-bit intermediates.

ZC_HD fr fr_add_g(const fr& a, const fr& b) {
  const uint32_t P[8] = {ZC_P0, ZC_P1, ZC_P2, ZC_P3, ZC_P4, ZC_P5, ZC_P6, ZC_P7};
  fr s, t;
  uint64_t c = 0;
  for (int i = 0; i < 8; i++) {
    c += (uint64_t)a.v[i] + b.v[i];
    s.v[i] = (uint32_t)c;
    c >>= 32;
  }
  int64_t br = 0;
  for (int i = 0; i < 8; i++) {
    int64_t d = (int64_t)s.v[i] - P[i] + br;
    t.v[i] = (uint32_t)d;
    br = d >> 32;  // 0 or -1
  }
  return (c == 0 && br < 0) ? s : t;
}

ZC_HD fr fr_sub_g(const fr& a, const fr& b) {
  const uint32_t P[8] = {ZC_P0, ZC_P1, ZC_P2, ZC_P3, ZC_P4, ZC_P5, ZC_P6, ZC_P7};
  fr s;
  int64_t br = 0;
  for (int i = 0; i < 8; i++) {
    int64_t d = (int64_t)a.v[i] - b.v[i] + br;
    s.v[i] = (uint32_t)d;
    br = d >> 32;
  }
  if (br < 0) {
    uint64_t c = 0;
    for (int i = 0; i < 8; i++) {
      c += (uint64_t)s.v[i] + P[i];
      s.v[i] = (uint32_t)c;
      c >>= 32;
    }
  }
  return s;
}

// Montgomery product a b 2^-256 mod r, inputs < r, output < r.
ZC_HD fr fr_mul_g(const fr& a, const fr& b) {
  const uint32_t P[8] = {ZC_P0, ZC_P1, ZC_P2, ZC_P3, ZC_P4, ZC_P5, ZC_P6, ZC_P7};
  uint32_t t[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
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
    uint32_t m = 0u - t[0];  // t0 * (-r^{-1}) mod 2^32, r0 = 1
    c = (uint64_t)m * P[0] + t[0];
    c >>= 32;
    for (int j = 1; j < 8; j++) {
      c += (uint64_t)m * P[j] + t[j];
      t[j - 1] = (uint32_t)c;
      c >>= 32;
    }
    c += t[8];
    t[7] = (uint32_t)c;
    t[8] = t[9] + (uint32_t)(c >> 32);
  }
  fr r;
  for (int i = 0; i < 8; i++) r.v[i] = t[i];
  if (t[8] != 0 || !fr_is_canonical(r)) {
    int64_t br = 0;
    for (int i = 0; i < 8; i++) {
      int64_t d = (int64_t)r.v[i] - P[i] + br;
      r.v[i] = (uint32_t)d;
      br = d >> 32;
    }
  }
  return r;
}

// ---- multiplication by a known constant
// y w mod r for a multiplier w whose quotient q = floor(2^256 w / r) is kept
// beside it (Shoup's method): qh = floor(y q / 2^256), y w - qh r, whose low
// 256 bits are all that is needed.  Only the word sums 6 and up of y q are
// formed (43 of 64 products): what is left out is below 6 2^224, so qh is
// short of y w / r by less than 1 + y / 2^256 + 6 / 2^32 and the result is
// below 2r for every y < 2r.  The low halves of y w and of qh r take 28 + 15
// wide products and 14 low ones (-r = 2^32 - 1 + 2^64 N, N = ~r / 2^64: the
// two lowest words of r need none); every carry chain of theirs ends at word
// 7, so they need no additions besides the chains.  86 wide and 14 low
// products against 112 wide: 372 cycles of the multiplier pipe a product
// against 448, and 35 other instructions against 90.  Measured (dependent
// products, 16 warps per SM, one GB300): 9.1e10 products/s, 9.3e10 with the
// constant in the kernel parameters, against 7.1e10 for fr_mul_inl in the
// same run.
struct frc {
  fr w, q;  // canonical w, floor(2^256 w / r)
};

// floor(2^256 w / r) from w R mod r: 2^256 w = q r + (w R mod r), so
// q = (w R mod r) (-r^-1) mod 2^256
ZC_HD fr fr_quot(const fr& w1) {
  const uint32_t ninv[8] = {0xffffffffu, 0xfffffffeu, 0xfffe5bfdu, 0x53ba5bffu,
                            0x0004ec06u, 0x181b2c17u, 0xd7bf2839u, 0x3d443ab0u};
  fr t = fr_zero();
  for (int i = 0; i < 8; i++) {
    uint64_t k = 0;
    for (int j = 0; i + j < 8; j++) {
      k += (uint64_t)w1.v[i] * ninv[j] + t.v[i + j];
      t.v[i + j] = (uint32_t)k;
      k >>= 32;
    }
  }
  return t;
}

// ---------------------------------------------------------------- device --
#if defined(__CUDACC__)

ZC_D fr fr_add(const fr& a, const fr& b) {
  fr s, t;
  uint32_t bw;
  asm("add.cc.u32 %0, %8, %16;\n\t"
      "addc.cc.u32 %1, %9, %17;\n\t"
      "addc.cc.u32 %2, %10, %18;\n\t"
      "addc.cc.u32 %3, %11, %19;\n\t"
      "addc.cc.u32 %4, %12, %20;\n\t"
      "addc.cc.u32 %5, %13, %21;\n\t"
      "addc.cc.u32 %6, %14, %22;\n\t"
      "addc.u32 %7, %15, %23;"
      : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]),
        "=r"(s.v[6]), "=r"(s.v[7])
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
        "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
        "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
  asm("sub.cc.u32 %0, %9, %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32 %8, 0, 0;"
      : "=r"(t.v[0]), "=r"(t.v[1]), "=r"(t.v[2]), "=r"(t.v[3]), "=r"(t.v[4]), "=r"(t.v[5]),
        "=r"(t.v[6]), "=r"(t.v[7]), "=r"(bw)
      : "r"(s.v[0]), "r"(s.v[1]), "r"(s.v[2]), "r"(s.v[3]), "r"(s.v[4]), "r"(s.v[5]),
        "r"(s.v[6]), "r"(s.v[7]), "n"(ZC_P0), "n"(ZC_P1), "n"(ZC_P2), "n"(ZC_P3), "n"(ZC_P4),
        "n"(ZC_P5), "n"(ZC_P6), "n"(ZC_P7));
  // bw == 0xffffffff: s < r, keep s
#pragma unroll
  for (int i = 0; i < 8; i++) s.v[i] = bw ? s.v[i] : t.v[i];
  return s;
}

// Lazily reduced sum and difference of canonical a, b: results in [0, 2r)
// (2r < 2^256) without the conditional correction.  Such a value may be the
// SECOND operand of fr_mul: its rows run over b's limbs with a < r, so every
// row stays below 2r + 1 and the product below 2r before its final
// subtraction, whatever b < 2^256 is.  fr_reduce1 brings it to [0, r).
ZC_D fr fr_add_lazy(const fr& a, const fr& b) {
  fr s;
  asm("add.cc.u32 %0, %8, %16;\n\t"
      "addc.cc.u32 %1, %9, %17;\n\t"
      "addc.cc.u32 %2, %10, %18;\n\t"
      "addc.cc.u32 %3, %11, %19;\n\t"
      "addc.cc.u32 %4, %12, %20;\n\t"
      "addc.cc.u32 %5, %13, %21;\n\t"
      "addc.cc.u32 %6, %14, %22;\n\t"
      "addc.u32 %7, %15, %23;"
      : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]),
        "=r"(s.v[6]), "=r"(s.v[7])
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
        "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
        "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
  return s;
}

// a - b + r mod 2^256, in (0, 2r) for canonical a, b
ZC_D fr fr_sub_lazy(const fr& a, const fr& b) {
  fr s;
  asm("sub.cc.u32 %0, %8, %16;\n\t"
      "subc.cc.u32 %1, %9, %17;\n\t"
      "subc.cc.u32 %2, %10, %18;\n\t"
      "subc.cc.u32 %3, %11, %19;\n\t"
      "subc.cc.u32 %4, %12, %20;\n\t"
      "subc.cc.u32 %5, %13, %21;\n\t"
      "subc.cc.u32 %6, %14, %22;\n\t"
      "subc.u32 %7, %15, %23;"
      : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]),
        "=r"(s.v[6]), "=r"(s.v[7])
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
        "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
        "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
  asm("add.cc.u32 %0, %0, %8;\n\t"
      "addc.cc.u32 %1, %1, %9;\n\t"
      "addc.cc.u32 %2, %2, %10;\n\t"
      "addc.cc.u32 %3, %3, %11;\n\t"
      "addc.cc.u32 %4, %4, %12;\n\t"
      "addc.cc.u32 %5, %5, %13;\n\t"
      "addc.cc.u32 %6, %6, %14;\n\t"
      "addc.u32 %7, %7, %15;"
      : "+r"(s.v[0]), "+r"(s.v[1]), "+r"(s.v[2]), "+r"(s.v[3]), "+r"(s.v[4]), "+r"(s.v[5]),
        "+r"(s.v[6]), "+r"(s.v[7])
      : "n"(ZC_P0), "n"(ZC_P1), "n"(ZC_P2), "n"(ZC_P3), "n"(ZC_P4), "n"(ZC_P5), "n"(ZC_P6),
        "n"(ZC_P7));
  return s;
}

// x - r when x >= r, for x < 2r
ZC_D fr fr_reduce1(const fr& x) {
  fr t;
  uint32_t bw;
  asm("sub.cc.u32 %0, %9, %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32 %8, 0, 0;"
      : "=r"(t.v[0]), "=r"(t.v[1]), "=r"(t.v[2]), "=r"(t.v[3]), "=r"(t.v[4]), "=r"(t.v[5]),
        "=r"(t.v[6]), "=r"(t.v[7]), "=r"(bw)
      : "r"(x.v[0]), "r"(x.v[1]), "r"(x.v[2]), "r"(x.v[3]), "r"(x.v[4]), "r"(x.v[5]),
        "r"(x.v[6]), "r"(x.v[7]), "n"(ZC_P0), "n"(ZC_P1), "n"(ZC_P2), "n"(ZC_P3), "n"(ZC_P4),
        "n"(ZC_P5), "n"(ZC_P6), "n"(ZC_P7));
  fr r;
#pragma unroll
  for (int i = 0; i < 8; i++) r.v[i] = bw ? x.v[i] : t.v[i];
  return r;
}

ZC_D fr fr_sub(const fr& a, const fr& b) {
  fr s;
  uint32_t bw;
  asm("sub.cc.u32 %0, %9, %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32 %8, 0, 0;"
      : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]),
        "=r"(s.v[6]), "=r"(s.v[7]), "=r"(bw)
      : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
        "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
        "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
  asm("add.cc.u32 %0, %0, %8;\n\t"
      "addc.cc.u32 %1, %1, %9;\n\t"
      "addc.cc.u32 %2, %2, %10;\n\t"
      "addc.cc.u32 %3, %3, %11;\n\t"
      "addc.cc.u32 %4, %4, %12;\n\t"
      "addc.cc.u32 %5, %5, %13;\n\t"
      "addc.cc.u32 %6, %6, %14;\n\t"
      "addc.u32 %7, %7, %15;"
      : "+r"(s.v[0]), "+r"(s.v[1]), "+r"(s.v[2]), "+r"(s.v[3]), "+r"(s.v[4]), "+r"(s.v[5]),
        "+r"(s.v[6]), "+r"(s.v[7])
      : "r"(bw & ZC_P0), "r"(bw & ZC_P1), "r"(bw & ZC_P2), "r"(bw & ZC_P3), "r"(bw & ZC_P4),
        "r"(bw & ZC_P5), "r"(bw & ZC_P6), "r"(bw & ZC_P7));
  return s;
}

// t - r when t >= r, for t < 2r given as words
ZC_D fr fr_reduce_final(uint32_t t0, uint32_t t1, uint32_t t2, uint32_t t3, uint32_t t4,
                        uint32_t t5, uint32_t t6, uint32_t t7) {
  fr s, r;
  uint32_t bw;
  asm("sub.cc.u32 %0, %9, %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32 %8, 0, 0;"
      : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]),
        "=r"(s.v[6]), "=r"(s.v[7]), "=r"(bw)
      : "r"(t0), "r"(t1), "r"(t2), "r"(t3), "r"(t4), "r"(t5), "r"(t6), "r"(t7), "n"(ZC_P0),
        "n"(ZC_P1), "n"(ZC_P2), "n"(ZC_P3), "n"(ZC_P4), "n"(ZC_P5), "n"(ZC_P6), "n"(ZC_P7));
  r.v[0] = bw ? t0 : s.v[0];
  r.v[1] = bw ? t1 : s.v[1];
  r.v[2] = bw ? t2 : s.v[2];
  r.v[3] = bw ? t3 : s.v[3];
  r.v[4] = bw ? t4 : s.v[4];
  r.v[5] = bw ? t5 : s.v[5];
  r.v[6] = bw ? t6 : s.v[6];
  r.v[7] = bw ? t7 : s.v[7];
  return r;
}

// Montgomery rows (CIOS) with the even/odd split of the partial products
// (Emmart, Luitjens, Weems, Woolley, "Optimizing Modular Multiplication for
// NVIDIA's Maxwell GPUs", ARITH 2016).  The accumulator is E + 2^32 O: a_j b
// is 64 bits wide, so the products with even j fill E's word pairs and those
// with odd j O's, and each half is one carry chain of mad.lo.cc / madc.hi.cc
// pairs that the integer multiplier accumulates in place (one wide
// multiply-add per product, the carry in a predicate): no separate additions.
// Dropping the zero low word after a reduction swaps the halves: the new E is
// O, the new O is E from word 2 on, and E's word 1 (X) enters the next row at
// word 0, its carry flowing into the O chain, which starts at word 1.
//
// The reduction adds m r, m = -t0 (r0 = 1).  r1 = 2^32 - 1 needs no product:
// m (2^32 - 1) = (m - [m != 0]) 2^32 + t0.
//
// Bound: a wide multiply-add holds the multiplier pipe four cycles per warp
// and SM quarter, so 64 + 48 products take 448 cycles: at most 9.0e10
// products/s at 2070 MHz.  Measured (chains of dependent products, 16 warps
// per SM, one GB300): 7.59e10 inlined, 85 % of that, against 5.08e10 for rows
// of plain 64-bit products joined by add-with-carry chains (426 instructions
// a product, the ALU pipe's additions the bound); with m r1 as a ninth wide
// product 6.4e10, with m r0 too 6.1e10.

// E[0..8], O[0..7] = a b (E[8] = 0)
ZC_D void zc_mul_first(const fr& a, uint32_t b, uint32_t (&E)[9], uint32_t (&O)[8]) {
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    asm("mul.lo.u32 %0, %2, %3;\n\tmul.hi.u32 %1, %2, %3;" : "=r"(E[j]), "=r"(E[j + 1]) : "r"(a.v[j]), "r"(b));
    asm("mul.lo.u32 %0, %2, %3;\n\tmul.hi.u32 %1, %2, %3;" : "=r"(O[j]), "=r"(O[j + 1]) : "r"(a.v[j + 1]), "r"(b));
  }
  E[8] = 0;
}

// E[0..7] + 2^32 O[0..6] + X + a b -> E[0..8], O[0..7]
ZC_D void zc_mul_row(const fr& a, uint32_t b, uint32_t X, uint32_t (&E)[9], uint32_t (&O)[8]) {
  asm("add.cc.u32 %0, %0, %17;\n\t"
      "madc.lo.cc.u32 %9, %19, %26, %9;\n\t"
      "madc.hi.cc.u32 %10, %19, %26, %10;\n\t"
      "madc.lo.cc.u32 %11, %21, %26, %11;\n\t"
      "madc.hi.cc.u32 %12, %21, %26, %12;\n\t"
      "madc.lo.cc.u32 %13, %23, %26, %13;\n\t"
      "madc.hi.cc.u32 %14, %23, %26, %14;\n\t"
      "madc.lo.cc.u32 %15, %25, %26, %15;\n\t"
      "madc.hi.u32 %16, %25, %26, 0;\n\t"
      "mad.lo.cc.u32 %0, %18, %26, %0;\n\t"
      "madc.hi.cc.u32 %1, %18, %26, %1;\n\t"
      "madc.lo.cc.u32 %2, %20, %26, %2;\n\t"
      "madc.hi.cc.u32 %3, %20, %26, %3;\n\t"
      "madc.lo.cc.u32 %4, %22, %26, %4;\n\t"
      "madc.hi.cc.u32 %5, %22, %26, %5;\n\t"
      "madc.lo.cc.u32 %6, %24, %26, %6;\n\t"
      "madc.hi.cc.u32 %7, %24, %26, %7;\n\t"
      "addc.u32 %8, 0, 0;"
      : "+r"(E[0]), "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "=r"(E[8]),
        "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "=r"(O[7])
      : "r"(X), "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]),
        "r"(a.v[7]), "r"(b));
}

// E + 2^32 O += m r, m = -E[0]; E[0] becomes 0
ZC_D void zc_mul_reduce(uint32_t (&E)[9], uint32_t (&O)[8]) {
  uint32_t m, h;
  asm("sub.cc.u32 %0, 0, %2;\n\tsubc.u32 %1, %0, 0;" : "=&r"(m), "=&r"(h) : "r"(E[0]));
  asm("add.cc.u32 %0, %0, %9;\n\t"
      "addc.cc.u32 %1, %1, %10;\n\t"
      "madc.lo.cc.u32 %2, %8, %11, %2;\n\t"
      "madc.hi.cc.u32 %3, %8, %11, %3;\n\t"
      "madc.lo.cc.u32 %4, %8, %12, %4;\n\t"
      "madc.hi.cc.u32 %5, %8, %12, %5;\n\t"
      "madc.lo.cc.u32 %6, %8, %13, %6;\n\t"
      "madc.hi.u32 %7, %8, %13, %7;"
      : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7])
      : "r"(m), "r"(E[0]), "r"(h), "n"(ZC_P3), "n"(ZC_P5), "n"(ZC_P7));
  asm("add.cc.u32 %0, %0, %9;\n\t"
      "addc.cc.u32 %1, %1, 0;\n\t"
      "madc.lo.cc.u32 %2, %9, %10, %2;\n\t"
      "madc.hi.cc.u32 %3, %9, %10, %3;\n\t"
      "madc.lo.cc.u32 %4, %9, %11, %4;\n\t"
      "madc.hi.cc.u32 %5, %9, %11, %5;\n\t"
      "madc.lo.cc.u32 %6, %9, %12, %6;\n\t"
      "madc.hi.cc.u32 %7, %9, %12, %7;\n\t"
      "addc.u32 %8, %8, 0;"
      : "+r"(E[0]), "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(E[8])
      : "r"(m), "n"(ZC_P2), "n"(ZC_P4), "n"(ZC_P6));
}

// a b R^-1 in [0, 2r) for a < r and any b < 2^256.  Between rows the
// accumulator is below 2r (b's digits come one a row), within one below
// 2^288: E needs nine words and O, at most the whole shifted by a word, eight.
ZC_D fr fr_mul_lazy_inl(const fr& a, const fr& b) {
  uint32_t E[9], O[8];
  zc_mul_first(a, b.v[0], E, O);
  zc_mul_reduce(E, O);
#pragma unroll
  for (int i = 1; i < 8; i++) {
    uint32_t nE[9], nO[8];
#pragma unroll
    for (int j = 0; j < 8; j++) nE[j] = O[j];
#pragma unroll
    for (int j = 0; j < 7; j++) nO[j] = E[j + 2];
    zc_mul_row(a, b.v[i], E[1], nE, nO);
    zc_mul_reduce(nE, nO);
#pragma unroll
    for (int j = 0; j < 9; j++) E[j] = nE[j];
#pragma unroll
    for (int j = 0; j < 8; j++) O[j] = nO[j];
  }
  fr t;
  asm("add.cc.u32 %0, %8, %16;\n\t"
      "addc.cc.u32 %1, %9, %17;\n\t"
      "addc.cc.u32 %2, %10, %18;\n\t"
      "addc.cc.u32 %3, %11, %19;\n\t"
      "addc.cc.u32 %4, %12, %20;\n\t"
      "addc.cc.u32 %5, %13, %21;\n\t"
      "addc.cc.u32 %6, %14, %22;\n\t"
      "addc.u32 %7, %15, %23;"
      : "=r"(t.v[0]), "=r"(t.v[1]), "=r"(t.v[2]), "=r"(t.v[3]), "=r"(t.v[4]), "=r"(t.v[5]), "=r"(t.v[6]),
        "=r"(t.v[7])
      : "r"(O[0]), "r"(O[1]), "r"(O[2]), "r"(O[3]), "r"(O[4]), "r"(O[5]), "r"(O[6]), "r"(O[7]), "r"(E[1]), "r"(E[2]),
        "r"(E[3]), "r"(E[4]), "r"(E[5]), "r"(E[6]), "r"(E[7]), "r"(E[8]));
  return t;
}

ZC_D fr fr_mul_inl(const fr& a, const fr& b) {
  const fr t = fr_mul_lazy_inl(a, b);
  return fr_reduce_final(t.v[0], t.v[1], t.v[2], t.v[3], t.v[4], t.v[5], t.v[6], t.v[7]);
}

// Product by a constant (see frc): y w mod r in [0, 2r), for y < 2r.
// c[0..2NP) += b (a0, a1, ...) as one carry chain of 64-bit products.  TAIL 0:
// the chain ends there (no carry out), 1: the carry is added to c[2NP], 2: the
// low word of al b (with the carry) is added to c[2NP].
template <int NP, int TAIL>
ZC_D void zc_chain(uint32_t* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b, uint32_t al = 0) {
  if constexpr (NP == 0) {
    if constexpr (TAIL == 2) asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(c[0]) : "r"(al), "r"(b));
  } else if constexpr (NP == 1) {
    if constexpr (TAIL == 0)
      asm("mad.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.u32 %1, %2, %3, %1;" : "+r"(c[0]), "+r"(c[1]) : "r"(a0), "r"(b));
    else if constexpr (TAIL == 1)
      asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\tmadc.hi.cc.u32 %1, %3, %4, %1;\n\taddc.u32 %2, %2, 0;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]) : "r"(a0), "r"(b));
    else
      asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\tmadc.hi.cc.u32 %1, %3, %4, %1;\n\tmadc.lo.u32 %2, %5, %4, %2;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]) : "r"(a0), "r"(b), "r"(al));
  } else if constexpr (NP == 2) {
#define ZC_C2 "mad.lo.cc.u32 %0, %5, %7, %0;\n\tmadc.hi.cc.u32 %1, %5, %7, %1;\n\tmadc.lo.cc.u32 %2, %6, %7, %2;\n\t"
    if constexpr (TAIL == 0)
      asm(ZC_C2 "madc.hi.u32 %3, %6, %7, %3;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(al) : "r"(a0), "r"(a1), "r"(b));
    else if constexpr (TAIL == 1)
      asm(ZC_C2 "madc.hi.cc.u32 %3, %6, %7, %3;\n\taddc.u32 %4, %4, 0;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]) : "r"(a0), "r"(a1), "r"(b));
    else
      asm(ZC_C2 "madc.hi.cc.u32 %3, %6, %7, %3;\n\tmadc.lo.u32 %4, %8, %7, %4;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]) : "r"(a0), "r"(a1), "r"(b), "r"(al));
  } else if constexpr (NP == 3) {
#define ZC_C3                                                                                                     \
  "mad.lo.cc.u32 %0, %7, %10, %0;\n\tmadc.hi.cc.u32 %1, %7, %10, %1;\n\tmadc.lo.cc.u32 %2, %8, %10, %2;\n\t"       \
  "madc.hi.cc.u32 %3, %8, %10, %3;\n\tmadc.lo.cc.u32 %4, %9, %10, %4;\n\t"
    if constexpr (TAIL == 0)
      asm(ZC_C3 "madc.hi.u32 %5, %9, %10, %5;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(al)
          : "r"(a0), "r"(a1), "r"(a2), "r"(b));
    else if constexpr (TAIL == 1)
      asm(ZC_C3 "madc.hi.cc.u32 %5, %9, %10, %5;\n\taddc.u32 %6, %6, 0;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6])
          : "r"(a0), "r"(a1), "r"(a2), "r"(b));
    else
      asm(ZC_C3 "madc.hi.cc.u32 %5, %9, %10, %5;\n\tmadc.lo.u32 %6, %11, %10, %6;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6])
          : "r"(a0), "r"(a1), "r"(a2), "r"(b), "r"(al));
  } else {
#define ZC_C4                                                                                                     \
  "mad.lo.cc.u32 %0, %9, %13, %0;\n\tmadc.hi.cc.u32 %1, %9, %13, %1;\n\tmadc.lo.cc.u32 %2, %10, %13, %2;\n\t"      \
  "madc.hi.cc.u32 %3, %10, %13, %3;\n\tmadc.lo.cc.u32 %4, %11, %13, %4;\n\tmadc.hi.cc.u32 %5, %11, %13, %5;\n\t"   \
  "madc.lo.cc.u32 %6, %12, %13, %6;\n\t"
    if constexpr (TAIL == 0)
      asm(ZC_C4 "madc.hi.u32 %7, %12, %13, %7;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6]), "+r"(c[7]), "+r"(al)
          : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b));
    else
      asm(ZC_C4 "madc.hi.cc.u32 %7, %12, %13, %7;\n\taddc.u32 %8, %8, 0;"
          : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6]), "+r"(c[7]), "+r"(c[8])
          : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b));
  }
}

ZC_D fr fr_mulc_lazy(const frc& W, const fr& y) {
  const uint32_t* p = W.q.v;
  uint32_t E[10] = {}, O[9] = {};  // words 6..15 (products of even word sums) and 7..15 (odd) of y q
  zc_chain<1, 0>(E, p[6], 0, 0, 0, y.v[0]);
  zc_chain<1, 0>(O, p[7], 0, 0, 0, y.v[0]);
  zc_chain<2, 0>(E, p[5], p[7], 0, 0, y.v[1]);
  zc_chain<1, 1>(O, p[6], 0, 0, 0, y.v[1]);
  zc_chain<2, 1>(E, p[4], p[6], 0, 0, y.v[2]);
  zc_chain<2, 0>(O, p[5], p[7], 0, 0, y.v[2]);
  zc_chain<3, 0>(E, p[3], p[5], p[7], 0, y.v[3]);
  zc_chain<2, 1>(O, p[4], p[6], 0, 0, y.v[3]);
  zc_chain<3, 1>(E, p[2], p[4], p[6], 0, y.v[4]);
  zc_chain<3, 0>(O, p[3], p[5], p[7], 0, y.v[4]);
  zc_chain<4, 0>(E, p[1], p[3], p[5], p[7], y.v[5]);
  zc_chain<3, 1>(O, p[2], p[4], p[6], 0, y.v[5]);
  zc_chain<4, 1>(E, p[0], p[2], p[4], p[6], y.v[6]);
  zc_chain<4, 0>(O, p[1], p[3], p[5], p[7], y.v[6]);
  zc_chain<4, 0>(E + 2, p[1], p[3], p[5], p[7], y.v[7]);
  zc_chain<4, 1>(O, p[0], p[2], p[4], p[6], y.v[7]);
  fr q;
  asm("add.cc.u32 %0, %9, %18;\n\t"
      "addc.cc.u32 %1, %10, %19;\n\t"
      "addc.cc.u32 %2, %11, %20;\n\t"
      "addc.cc.u32 %3, %12, %21;\n\t"
      "addc.cc.u32 %4, %13, %22;\n\t"
      "addc.cc.u32 %5, %14, %23;\n\t"
      "addc.cc.u32 %6, %15, %24;\n\t"
      "addc.cc.u32 %7, %16, %25;\n\t"
      "addc.u32 %8, %17, %26;"
      : "+r"(E[0]), "=r"(q.v[0]), "=r"(q.v[1]), "=r"(q.v[2]), "=r"(q.v[3]), "=r"(q.v[4]), "=r"(q.v[5]), "=r"(q.v[6]),
        "=r"(q.v[7])
      : "r"(E[1]), "r"(E[2]), "r"(E[3]), "r"(E[4]), "r"(E[5]), "r"(E[6]), "r"(E[7]), "r"(E[8]), "r"(E[9]), "r"(O[0]),
        "r"(O[1]), "r"(O[2]), "r"(O[3]), "r"(O[4]), "r"(O[5]), "r"(O[6]), "r"(O[7]), "r"(O[8]));
  // y w - q r mod 2^256, -r = -1 + 2^32 + 2^64 N: A = -q - 1 (words 0..7), B = q (words 1..7)
  constexpr uint32_t N0 = ~ZC_P2, N1 = ~ZC_P3, N2 = ~ZC_P4, N3 = ~ZC_P5, N4 = ~ZC_P6, N5 = ~ZC_P7;
  uint32_t A[8], B[8];
#pragma unroll
  for (int i = 0; i < 8; i++) A[i] = ~q.v[i];
#pragma unroll
  for (int i = 0; i < 7; i++) B[i] = q.v[i];
  const uint32_t* w = W.w.v;
  zc_chain<4, 0>(A, w[0], w[2], w[4], w[6], y.v[0]);
  zc_chain<3, 2>(B, w[1], w[3], w[5], 0, y.v[0], w[7]);
  zc_chain<3, 0>(A + 2, w[1], w[3], w[5], 0, y.v[1]);
  zc_chain<3, 2>(B, w[0], w[2], w[4], 0, y.v[1], w[6]);
  zc_chain<3, 0>(A + 2, w[0], w[2], w[4], 0, y.v[2]);
  zc_chain<2, 2>(B + 2, w[1], w[3], 0, 0, y.v[2], w[5]);
  zc_chain<2, 0>(A + 4, w[1], w[3], 0, 0, y.v[3]);
  zc_chain<2, 2>(B + 2, w[0], w[2], 0, 0, y.v[3], w[4]);
  zc_chain<2, 0>(A + 4, w[0], w[2], 0, 0, y.v[4]);
  zc_chain<1, 2>(B + 4, w[1], 0, 0, 0, y.v[4], w[3]);
  zc_chain<1, 0>(A + 6, w[1], 0, 0, 0, y.v[5]);
  zc_chain<1, 2>(B + 4, w[0], 0, 0, 0, y.v[5], w[2]);
  zc_chain<1, 0>(A + 6, w[0], 0, 0, 0, y.v[6]);
  zc_chain<0, 2>(B + 6, 0, 0, 0, 0, y.v[6], w[1]);
  zc_chain<0, 2>(B + 6, 0, 0, 0, 0, y.v[7], w[0]);
  // q N at word 2
  zc_chain<3, 0>(A + 2, N0, N2, N4, 0, q.v[0]);
  zc_chain<2, 2>(B + 2, N1, N3, 0, 0, q.v[0], N5);
  zc_chain<2, 0>(A + 4, N1, N3, 0, 0, q.v[1]);
  zc_chain<2, 2>(B + 2, N0, N2, 0, 0, q.v[1], N4);
  zc_chain<2, 0>(A + 4, N0, N2, 0, 0, q.v[2]);
  zc_chain<1, 2>(B + 4, N1, 0, 0, 0, q.v[2], N3);
  zc_chain<1, 0>(A + 6, N1, 0, 0, 0, q.v[3]);
  zc_chain<1, 2>(B + 4, N0, 0, 0, 0, q.v[3], N2);
  zc_chain<1, 0>(A + 6, N0, 0, 0, 0, q.v[4]);
  zc_chain<0, 2>(B + 6, 0, 0, 0, 0, q.v[4], N1);
  zc_chain<0, 2>(B + 6, 0, 0, 0, 0, q.v[5], N0);
  fr t;
  asm("add.cc.u32 %0, %8, 1;\n\t"
      "addc.cc.u32 %1, %9, %16;\n\t"
      "addc.cc.u32 %2, %10, %17;\n\t"
      "addc.cc.u32 %3, %11, %18;\n\t"
      "addc.cc.u32 %4, %12, %19;\n\t"
      "addc.cc.u32 %5, %13, %20;\n\t"
      "addc.cc.u32 %6, %14, %21;\n\t"
      "addc.u32 %7, %15, %22;"
      : "=r"(t.v[0]), "=r"(t.v[1]), "=r"(t.v[2]), "=r"(t.v[3]), "=r"(t.v[4]), "=r"(t.v[5]), "=r"(t.v[6]), "=r"(t.v[7])
      : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(B[0]), "r"(B[1]),
        "r"(B[2]), "r"(B[3]), "r"(B[4]), "r"(B[5]), "r"(B[6]));
  return t;
}

ZC_D fr fr_mulc(const frc& W, const fr& y) { return fr_reduce1(fr_mulc_lazy(W, y)); }

// Sums of products with one reduction: (a0 b0 + ... + a_{K-1} b_{K-1}) R^-1
// mod r, for inputs below r, K = 2 or 3.  Each row adds a_p b_p[i] for every
// p, then one reduction and the one-word shift.  Between rows the accumulator
// stays below (K+1) r < 2^257, before the shift below 2^289, so E takes ten
// words and O nine; at the end it is (sum a_p b_p + M r) / 2^256
// < r (K r / 2^256 + 1) < 2.36 r for K = 3: at most two subtractions of r
// give the canonical result.  Against K separate products and K - 1 additions
// this saves K - 1 reductions (48 of 112 wide products each).

// E[0..9] + 2^32 O[0..8] + X += a b
ZC_D void zc_acc_row(const fr& a, uint32_t b, uint32_t X, uint32_t (&E)[10], uint32_t (&O)[9]) {
  asm("add.cc.u32 %0, %0, %19;\n\t"
      "madc.lo.cc.u32 %10, %21, %28, %10;\n\t"
      "madc.hi.cc.u32 %11, %21, %28, %11;\n\t"
      "madc.lo.cc.u32 %12, %23, %28, %12;\n\t"
      "madc.hi.cc.u32 %13, %23, %28, %13;\n\t"
      "madc.lo.cc.u32 %14, %25, %28, %14;\n\t"
      "madc.hi.cc.u32 %15, %25, %28, %15;\n\t"
      "madc.lo.cc.u32 %16, %27, %28, %16;\n\t"
      "madc.hi.cc.u32 %17, %27, %28, %17;\n\t"
      "addc.u32 %18, %18, 0;\n\t"
      "mad.lo.cc.u32 %0, %20, %28, %0;\n\t"
      "madc.hi.cc.u32 %1, %20, %28, %1;\n\t"
      "madc.lo.cc.u32 %2, %22, %28, %2;\n\t"
      "madc.hi.cc.u32 %3, %22, %28, %3;\n\t"
      "madc.lo.cc.u32 %4, %24, %28, %4;\n\t"
      "madc.hi.cc.u32 %5, %24, %28, %5;\n\t"
      "madc.lo.cc.u32 %6, %26, %28, %6;\n\t"
      "madc.hi.cc.u32 %7, %26, %28, %7;\n\t"
      "addc.cc.u32 %8, %8, 0;\n\t"
      "addc.u32 %9, %9, 0;"
      : "+r"(E[0]), "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(E[8]),
        "+r"(E[9]), "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7]),
        "+r"(O[8])
      : "r"(X), "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]),
        "r"(a.v[7]), "r"(b));
}

// E + 2^32 O += m r, m = -E[0] (as zc_mul_reduce, on the wider accumulator)
ZC_D void zc_acc_reduce(uint32_t (&E)[10], uint32_t (&O)[9]) {
  uint32_t m, h;
  asm("sub.cc.u32 %0, 0, %2;\n\tsubc.u32 %1, %0, 0;" : "=&r"(m), "=&r"(h) : "r"(E[0]));
  asm("add.cc.u32 %0, %0, %10;\n\t"
      "addc.cc.u32 %1, %1, %11;\n\t"
      "madc.lo.cc.u32 %2, %9, %12, %2;\n\t"
      "madc.hi.cc.u32 %3, %9, %12, %3;\n\t"
      "madc.lo.cc.u32 %4, %9, %13, %4;\n\t"
      "madc.hi.cc.u32 %5, %9, %13, %5;\n\t"
      "madc.lo.cc.u32 %6, %9, %14, %6;\n\t"
      "madc.hi.cc.u32 %7, %9, %14, %7;\n\t"
      "addc.u32 %8, %8, 0;"
      : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7]), "+r"(O[8])
      : "r"(m), "r"(E[0]), "r"(h), "n"(ZC_P3), "n"(ZC_P5), "n"(ZC_P7));
  asm("add.cc.u32 %0, %0, %10;\n\t"
      "addc.cc.u32 %1, %1, 0;\n\t"
      "madc.lo.cc.u32 %2, %10, %11, %2;\n\t"
      "madc.hi.cc.u32 %3, %10, %11, %3;\n\t"
      "madc.lo.cc.u32 %4, %10, %12, %4;\n\t"
      "madc.hi.cc.u32 %5, %10, %12, %5;\n\t"
      "madc.lo.cc.u32 %6, %10, %13, %6;\n\t"
      "madc.hi.cc.u32 %7, %10, %13, %7;\n\t"
      "addc.cc.u32 %8, %8, 0;\n\t"
      "addc.u32 %9, %9, 0;"
      : "+r"(E[0]), "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(E[8]),
        "+r"(E[9])
      : "r"(m), "n"(ZC_P2), "n"(ZC_P4), "n"(ZC_P6));
}

// t (nine words, below 3r) minus r when it is at least r
ZC_D void zc_sub_r_if(uint32_t& t0, uint32_t& t1, uint32_t& t2, uint32_t& t3, uint32_t& t4, uint32_t& t5,
                      uint32_t& t6, uint32_t& t7, uint32_t& t8) {
  uint32_t s0, s1, s2, s3, s4, s5, s6, s7, s8, bw;
  asm("sub.cc.u32 %0, %10, %19;\n\t"
      "subc.cc.u32 %1, %11, %20;\n\t"
      "subc.cc.u32 %2, %12, %21;\n\t"
      "subc.cc.u32 %3, %13, %22;\n\t"
      "subc.cc.u32 %4, %14, %23;\n\t"
      "subc.cc.u32 %5, %15, %24;\n\t"
      "subc.cc.u32 %6, %16, %25;\n\t"
      "subc.cc.u32 %7, %17, %26;\n\t"
      "subc.cc.u32 %8, %18, 0;\n\t"
      "subc.u32 %9, 0, 0;"
      : "=r"(s0), "=r"(s1), "=r"(s2), "=r"(s3), "=r"(s4), "=r"(s5), "=r"(s6), "=r"(s7), "=r"(s8), "=r"(bw)
      : "r"(t0), "r"(t1), "r"(t2), "r"(t3), "r"(t4), "r"(t5), "r"(t6), "r"(t7), "r"(t8), "n"(ZC_P0),
        "n"(ZC_P1), "n"(ZC_P2), "n"(ZC_P3), "n"(ZC_P4), "n"(ZC_P5), "n"(ZC_P6), "n"(ZC_P7));
  // bw == 0xffffffff: t < r, keep it
  t0 = bw ? t0 : s0; t1 = bw ? t1 : s1; t2 = bw ? t2 : s2; t3 = bw ? t3 : s3; t4 = bw ? t4 : s4;
  t5 = bw ? t5 : s5; t6 = bw ? t6 : s6; t7 = bw ? t7 : s7; t8 = bw ? t8 : s8;
}

template <int K>
ZC_D fr fr_mul_sum_inl(const fr (&a)[K], const fr (&b)[K]) {
  uint32_t E[10] = {}, O[9] = {}, X = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
#pragma unroll
    for (int p = 0; p < K; p++) zc_acc_row(a[p], b[p].v[i], p == 0 ? X : 0u, E, O);
    zc_acc_reduce(E, O);
    uint32_t nE[10], nO[9];
#pragma unroll
    for (int j = 0; j < 9; j++) nE[j] = O[j];
    nE[9] = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) nO[j] = E[j + 2];
    nO[8] = 0;
    X = E[1];
#pragma unroll
    for (int j = 0; j < 10; j++) E[j] = nE[j];
#pragma unroll
    for (int j = 0; j < 9; j++) O[j] = nO[j];
  }
  uint32_t t0, t1, t2, t3, t4, t5, t6, t7, t8;
  asm("add.cc.u32 %0, %9, %18;\n\t"
      "addc.cc.u32 %1, %10, %19;\n\t"
      "addc.cc.u32 %2, %11, %20;\n\t"
      "addc.cc.u32 %3, %12, %21;\n\t"
      "addc.cc.u32 %4, %13, %22;\n\t"
      "addc.cc.u32 %5, %14, %23;\n\t"
      "addc.cc.u32 %6, %15, %24;\n\t"
      "addc.cc.u32 %7, %16, %25;\n\t"
      "addc.u32 %8, %17, %26;"
      : "=r"(t0), "=r"(t1), "=r"(t2), "=r"(t3), "=r"(t4), "=r"(t5), "=r"(t6), "=r"(t7), "=r"(t8)
      : "r"(E[0]), "r"(E[1]), "r"(E[2]), "r"(E[3]), "r"(E[4]), "r"(E[5]), "r"(E[6]), "r"(E[7]), "r"(E[8]), "r"(X),
        "r"(O[0]), "r"(O[1]), "r"(O[2]), "r"(O[3]), "r"(O[4]), "r"(O[5]), "r"(O[6]), "r"(O[7]));
  zc_sub_r_if(t0, t1, t2, t3, t4, t5, t6, t7, t8);
  if (K > 2) zc_sub_r_if(t0, t1, t2, t3, t4, t5, t6, t7, t8);
  fr x;
  x.v[0] = t0; x.v[1] = t1; x.v[2] = t2; x.v[3] = t3; x.v[4] = t4; x.v[5] = t5; x.v[6] = t6; x.v[7] = t7;
  return x;
}

// out-of-line copy shared by the kernels (see fr_mul_call)
static __device__ __noinline__ fr fr_mul_sum3_call(fr a0, fr b0, fr a1, fr b1, fr a2, fr b2) {
  const fr a[3] = {a0, a1, a2}, b[3] = {b0, b1, b2};
  return fr_mul_sum_inl<3>(a, b);
}
// (a0 b0 + a1 b1 + a2 b2) R^-1, canonical
ZC_D fr fr_mul_sum3(const fr& a0, const fr& b0, const fr& a1, const fr& b1, const fr& a2, const fr& b2) {
  return fr_mul_sum3_call(a0, b0, a1, b1, a2, b2);
}

// Kernels call one out-of-line copy of the multiplier so that their code fits
// the instruction cache (inlined at every call site, a round body of ~30
// products missed the cache on almost every instruction).
static __device__ __noinline__ fr fr_mul_call(fr a, fr b) { return fr_mul_inl(a, b); }
ZC_D fr fr_mul(const fr& a, const fr& b) { return fr_mul_call(a, b); }

// the constant c from its level-1 form c R mod r
ZC_D frc frc_of(const fr& c1) {
  frc c;
  fr one = fr_zero();
  one.v[0] = 1;
  c.w = fr_mul(one, c1);
  c.q = fr_quot(c1);
  return c;
}

#else
inline fr fr_add(const fr& a, const fr& b) { return fr_add_g(a, b); }
inline fr fr_sub(const fr& a, const fr& b) { return fr_sub_g(a, b); }
inline fr fr_mul(const fr& a, const fr& b) { return fr_mul_g(a, b); }
#endif

ZC_HD fr fr_from_u32(uint32_t x) {
  fr z = fr_zero();
  z.v[0] = x;
  return z;
}

}  // namespace zc
