// BN254 prime fields on 8 x 32-bit limbs in Montgomery form, and Fp2 = Fp[i]/(i^2 + 1).
//
// The Groth16 prover of zkVC (Sec. IV: libsnark's groth16 backend) works in the scalar
// field Fr (witness, QAP polynomials, NTT) and the base field Fp (curve coordinates).
// Both moduli are below 2^254, which the bounds below rely on.
//
// Multiplication is Montgomery's by operand scanning: for each limb b_i of the multiplier
// t += a b_i, then m = t_0 (-N^-1 mod 2^32) and t = (t + m N) / 2^32, with the terms split
// by parity over two accumulators (below).  Cost: 2 * 8 * 8 wide multiply-adds and 8 low
// products, counted as 4 * 8 * 8 + 8 = 264 IMADs per product.
#pragma once
#include <cstdint>

namespace zkvc {

// ------------------------------------------------------------------ compile-time bignum
struct U256c {
  uint32_t w[8];
};

constexpr U256c cx_dbl_mod(U256c x, U256c m) {
  U256c r{};
  uint32_t c = 0;
  for (int i = 0; i < 8; i++) {
    uint64_t v = ((uint64_t)x.w[i] << 1) | c;
    r.w[i] = (uint32_t)v;
    c = (uint32_t)(v >> 32);
  }
  bool ge = c != 0;
  if (!ge) {
    ge = true;
    for (int i = 7; i >= 0; i--) {
      if (r.w[i] != m.w[i]) {
        ge = r.w[i] > m.w[i];
        break;
      }
    }
  }
  if (ge) {
    uint64_t br = 0;
    for (int i = 0; i < 8; i++) {
      uint64_t v = (uint64_t)r.w[i] - m.w[i] - br;
      r.w[i] = (uint32_t)v;
      br = (v >> 63) & 1;
    }
  }
  return r;
}

constexpr U256c cx_pow2_mod(int k, U256c m) {
  U256c x{};
  x.w[0] = 1;
  for (int i = 0; i < k; i++) x = cx_dbl_mod(x, m);
  return x;
}

constexpr U256c cx_twice(U256c x) {  // 2x below 2^256
  U256c r{};
  for (int i = 0; i < 8; i++) r.w[i] = (x.w[i] << 1) | (i ? x.w[i - 1] >> 31 : 0u);
  return r;
}

constexpr uint32_t cx_neg_inv32(uint32_t m0) {
  uint32_t x = m0;  // Newton iteration for m0^-1 mod 2^32 (m0 odd)
  for (int i = 0; i < 5; i++) x = x * (2u - m0 * x);
  return 0u - x;
}

// ------------------------------------------------------------------ field parameters
// p and r of BN254 (alt_bn128), little-endian 32-bit limbs.
struct FpCfg {
  static constexpr U256c MOD = {{0xd87cfd47u, 0x3c208c16u, 0x6871ca8du, 0x97816a91u,
                                 0x8181585du, 0xb85045b6u, 0xe131a029u, 0x30644e72u}};
  static constexpr U256c MOD2 = cx_twice(MOD);
  static constexpr U256c R1 = cx_pow2_mod(256, MOD);
  static constexpr U256c R2 = cx_pow2_mod(512, MOD);
  static constexpr U256c R3 = cx_pow2_mod(768, MOD);
  static constexpr uint32_t INV = cx_neg_inv32(MOD.w[0]);
};

struct FrCfg {
  static constexpr U256c MOD = {{0xf0000001u, 0x43e1f593u, 0x79b97091u, 0x2833e848u,
                                 0x8181585du, 0xb85045b6u, 0xe131a029u, 0x30644e72u}};
  static constexpr U256c MOD2 = cx_twice(MOD);
  static constexpr U256c R1 = cx_pow2_mod(256, MOD);
  static constexpr U256c R2 = cx_pow2_mod(512, MOD);
  static constexpr U256c R3 = cx_pow2_mod(768, MOD);
  static constexpr uint32_t INV = cx_neg_inv32(MOD.w[0]);
};

#define ZKVC_LIMB_SWITCH(ARR, i)                                               \
  switch (i) {                                                                 \
    case 0: return ARR.w[0];                                                   \
    case 1: return ARR.w[1];                                                   \
    case 2: return ARR.w[2];                                                   \
    case 3: return ARR.w[3];                                                   \
    case 4: return ARR.w[4];                                                   \
    case 5: return ARR.w[5];                                                   \
    case 6: return ARR.w[6];                                                   \
    default: return ARR.w[7];                                                  \
  }

template <class C>
__host__ __device__ __forceinline__ constexpr uint32_t mod_limb(int i) { ZKVC_LIMB_SWITCH(C::MOD, i) }
template <class C>
__host__ __device__ __forceinline__ constexpr uint32_t mod2_limb(int i) { ZKVC_LIMB_SWITCH(C::MOD2, i) }
template <class C>
__host__ __device__ __forceinline__ constexpr uint32_t r1_limb(int i) { ZKVC_LIMB_SWITCH(C::R1, i) }
template <class C>
__host__ __device__ __forceinline__ constexpr uint32_t r2_limb(int i) { ZKVC_LIMB_SWITCH(C::R2, i) }
template <class C>
__host__ __device__ __forceinline__ constexpr uint32_t r3_limb(int i) { ZKVC_LIMB_SWITCH(C::R3, i) }

// ------------------------------------------------------------------ carry-chain rows
// t[0..8] += a[0..7] * b : low halves into t[0..7] (carry into t[8]), then high halves
// into t[1..8].  The caller guarantees that the 288-bit sum fits.
__device__ __forceinline__ void mac_row(uint32_t (&t)[9], const uint32_t (&a)[8], uint32_t b) {
  asm("mad.lo.cc.u32  %0, %9,  %17, %0;\n\t"
      "madc.lo.cc.u32 %1, %10, %17, %1;\n\t"
      "madc.lo.cc.u32 %2, %11, %17, %2;\n\t"
      "madc.lo.cc.u32 %3, %12, %17, %3;\n\t"
      "madc.lo.cc.u32 %4, %13, %17, %4;\n\t"
      "madc.lo.cc.u32 %5, %14, %17, %5;\n\t"
      "madc.lo.cc.u32 %6, %15, %17, %6;\n\t"
      "madc.lo.cc.u32 %7, %16, %17, %7;\n\t"
      "addc.u32       %8, %8, 0;\n\t"
      "mad.hi.cc.u32  %1, %9,  %17, %1;\n\t"
      "madc.hi.cc.u32 %2, %10, %17, %2;\n\t"
      "madc.hi.cc.u32 %3, %11, %17, %3;\n\t"
      "madc.hi.cc.u32 %4, %12, %17, %4;\n\t"
      "madc.hi.cc.u32 %5, %13, %17, %5;\n\t"
      "madc.hi.cc.u32 %6, %14, %17, %6;\n\t"
      "madc.hi.cc.u32 %7, %15, %17, %7;\n\t"
      "madc.hi.u32    %8, %16, %17, %8;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]),
        "+r"(t[7]), "+r"(t[8])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
        "r"(b));
}

// r = a + b over 8 limbs; returns the carry out.
__device__ __forceinline__ uint32_t add8(uint32_t (&r)[8], const uint32_t (&a)[8], const uint32_t (&b)[8]) {
  uint32_t c;
  asm("add.cc.u32  %0, %9,  %17;\n\t"
      "addc.cc.u32 %1, %10, %18;\n\t"
      "addc.cc.u32 %2, %11, %19;\n\t"
      "addc.cc.u32 %3, %12, %20;\n\t"
      "addc.cc.u32 %4, %13, %21;\n\t"
      "addc.cc.u32 %5, %14, %22;\n\t"
      "addc.cc.u32 %6, %15, %23;\n\t"
      "addc.cc.u32 %7, %16, %24;\n\t"
      "addc.u32    %8, 0, 0;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(c)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
        "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  return c;
}

// r = a - b over 8 limbs; returns 1 if it borrowed (a < b).
__device__ __forceinline__ uint32_t sub8(uint32_t (&r)[8], const uint32_t (&a)[8], const uint32_t (&b)[8]) {
  uint32_t br;
  asm("sub.cc.u32  %0, %9,  %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32    %8, 0, 0;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(br)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
        "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  return br & 1u;
}

// ------------------------------------------------------------------ prime field element
template <class C>
struct Field {
  uint32_t v[8];

  __device__ __forceinline__ static Field zero() {
    Field r;
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = 0;
    return r;
  }
  __device__ __forceinline__ static Field one() {  // R mod N (Montgomery form of 1)
    Field r;
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = r1_limb<C>(i);
    return r;
  }
  __device__ __forceinline__ static Field modulus() {
    Field r;
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = mod_limb<C>(i);
    return r;
  }
  __device__ __forceinline__ bool is_zero() const {
    uint32_t acc = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) acc |= v[i];
    return acc == 0;
  }
  __device__ __forceinline__ bool operator==(const Field& o) const {
    uint32_t acc = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) acc |= v[i] ^ o.v[i];
    return acc == 0;
  }
  __device__ __forceinline__ bool operator!=(const Field& o) const { return !(*this == o); }
};

template <class C>
__device__ __forceinline__ Field<C> f_add(const Field<C>& a, const Field<C>& b) {
  Field<C> s, d;
  add8(s.v, a.v, b.v);  // a + b < 2N < 2^255: no carry out
  const Field<C> m = Field<C>::modulus();
  uint32_t br = sub8(d.v, s.v, m.v);
  return br ? s : d;
}

template <class C>
__device__ __forceinline__ Field<C> f_sub(const Field<C>& a, const Field<C>& b) {
  Field<C> d, e;
  uint32_t br = sub8(d.v, a.v, b.v);
  const Field<C> m = Field<C>::modulus();
  add8(e.v, d.v, m.v);
  return br ? e : d;
}

template <class C>
__device__ __forceinline__ Field<C> f_neg(const Field<C>& a) {
  return f_sub(Field<C>::zero(), a);
}

template <class C>
__device__ __forceinline__ Field<C> f_dbl(const Field<C>& a) { return f_add(a, a); }

// Montgomery product a b R^-1 mod N, CIOS with carry-chain rows (reference form; the
// even/odd f_mul below is the one the kernels use).
template <class C>
__device__ __forceinline__ Field<C> f_mul_cios(const Field<C>& a, const Field<C>& b) {
  uint32_t t[9];
#pragma unroll
  for (int i = 0; i < 9; i++) t[i] = 0;
  uint32_t m[8];
#pragma unroll
  for (int i = 0; i < 8; i++) m[i] = mod_limb<C>(i);
#pragma unroll
  for (int i = 0; i < 8; i++) {
    mac_row(t, a.v, b.v[i]);
    uint32_t q = t[0] * C::INV;
    mac_row(t, m, q);  // t[0] becomes 0
#pragma unroll
    for (int j = 0; j < 8; j++) t[j] = t[j + 1];
    t[8] = 0;
  }
  Field<C> r, d;
#pragma unroll
  for (int i = 0; i < 8; i++) r.v[i] = t[i];
  uint32_t br = sub8(d.v, r.v, m);
  return br ? r : d;
}

// ------------------------------------------------------------------ even/odd products
// The kernels' products keep a number as two accumulators: e holds the limbs of the terms
// x_i y_j with i + j even and o those with i + j odd (o[k] weighs 2^(32 (k + 1))).  The
// terms x_s y, x_(s+2) y, x_(s+4) y, x_(s+6) y of one row then land on neighbouring aligned
// limb pairs of one accumulator, so a row is two carry chains of four 32 x 32 + 64 -> 64-bit
// multiply-adds each (mad.lo.cc / madc.hi.cc on a register pair) with the carry handed on
// inside the chain: one multiply-add instruction per term, against one multiply-add and one
// carry addition in product scanning.  The row-by-row form follows Koc, Acar and Kaliski's
// operand scanning (1996); two accumulators for terms that are and are not aligned are known
// from CUDA multiprecision work (Emmart, Luitjens, Weems and Woolley, "Optimizing modular
// multiplication for NVIDIA's Maxwell GPUs", 2016).
//
// What bounds it: the multiplier's 32 wide multiply-adds per SM and clock; a product has
// 128 of them and 8 low products, 132 clocks per warp and SM.  Measured on GB300 (2,070
// MHz, 32 warps per SM): 147 clocks = 68.4 G products/s (product scanning before: 159,
// 63.2 G); one warp alone 900 cycles per product (1,141); f_sqr 125 clocks, 80.6 G;
// f_mul2 217 clocks, 46.4 G (two products and an addition before: 323); Fp2 product 387
// clocks, 26.0 G (546); Fp2 square 301 (358).
#define ZKVC_CHAIN_3                                                          \
  "mad.lo.cc.u32  %0, %8,  %12, %0;\n\tmadc.hi.cc.u32 %1, %8,  %12, %1;\n\t"   \
  "madc.lo.cc.u32 %2, %9,  %12, %2;\n\tmadc.hi.cc.u32 %3, %9,  %12, %3;\n\t"   \
  "madc.lo.cc.u32 %4, %10, %12, %4;\n\tmadc.hi.cc.u32 %5, %10, %12, %5;\n\t"
#define ZKVC_CHAIN_4C                                                         \
  "mad.lo.cc.u32  %0, %9,  %13, %0;\n\tmadc.hi.cc.u32 %1, %9,  %13, %1;\n\t"   \
  "madc.lo.cc.u32 %2, %10, %13, %2;\n\tmadc.hi.cc.u32 %3, %10, %13, %3;\n\t"   \
  "madc.lo.cc.u32 %4, %11, %13, %4;\n\tmadc.hi.cc.u32 %5, %11, %13, %5;\n\t"   \
  "madc.lo.cc.u32 %6, %12, %13, %6;\n\tmadc.hi.cc.u32 %7, %12, %13, %7;\n\t"
#define ZKVC_CHAIN_X(x, s, y) "r"(x[s]), "r"(x[s + 2]), "r"(x[s + 4]), "r"(x[s + 6]), "r"(y)

namespace eo {
// t[0..7] += (x_s, x_(s+2), x_(s+4), x_(s+6)) y; the caller's bound leaves no carry out
__device__ __forceinline__ void chain(uint32_t* t, const uint32_t* x, int s, uint32_t y) {
  asm(ZKVC_CHAIN_3 "madc.lo.cc.u32 %6, %11, %12, %6;\n\tmadc.hi.u32 %7, %11, %12, %7;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7])
      : ZKVC_CHAIN_X(x, s, y));
}
// the same with t[7] fresh (zero before)
__device__ __forceinline__ void chain_f1(uint32_t* t, const uint32_t* x, int s, uint32_t y) {
  asm(ZKVC_CHAIN_3 "madc.lo.cc.u32 %6, %11, %12, %6;\n\tmadc.hi.u32 %7, %11, %12, 0;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "=r"(t[7])
      : ZKVC_CHAIN_X(x, s, y));
}
// t[6] and t[7] fresh
__device__ __forceinline__ void chain_f2(uint32_t* t, const uint32_t* x, int s, uint32_t y) {
  asm(ZKVC_CHAIN_3 "madc.lo.cc.u32 %6, %11, %12, 0;\n\tmadc.hi.u32 %7, %11, %12, 0;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "=r"(t[6]), "=r"(t[7])
      : ZKVC_CHAIN_X(x, s, y));
}
// the carry out is added to top
__device__ __forceinline__ void chain_c(uint32_t* t, uint32_t& top, const uint32_t* x, int s, uint32_t y) {
  asm(ZKVC_CHAIN_4C "addc.u32 %8, %8, 0;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]), "+r"(top)
      : ZKVC_CHAIN_X(x, s, y));
}
// the carry out becomes top
__device__ __forceinline__ void chain_cf(uint32_t* t, uint32_t& top, const uint32_t* x, int s, uint32_t y) {
  asm(ZKVC_CHAIN_4C "addc.u32 %8, 0, 0;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]), "=r"(top)
      : ZKVC_CHAIN_X(x, s, y));
}
// w += pend with its carry into t, then chain_f2
__device__ __forceinline__ void chain_p2(uint32_t& w, uint32_t pend, uint32_t* t, const uint32_t* x, int s,
                                         uint32_t y) {
  asm("add.cc.u32 %8, %8, %14;\n\t"
      "madc.lo.cc.u32 %0, %9,  %13, %0;\n\tmadc.hi.cc.u32 %1, %9,  %13, %1;\n\t"
      "madc.lo.cc.u32 %2, %10, %13, %2;\n\tmadc.hi.cc.u32 %3, %10, %13, %3;\n\t"
      "madc.lo.cc.u32 %4, %11, %13, %4;\n\tmadc.hi.cc.u32 %5, %11, %13, %5;\n\t"
      "madc.lo.cc.u32 %6, %12, %13, 0;\n\tmadc.hi.u32 %7, %12, %13, 0;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "=r"(t[6]), "=r"(t[7]), "+r"(w)
      : ZKVC_CHAIN_X(x, s, y), "r"(pend));
}
// t[0..7] = (x_s, x_(s+2), x_(s+4), x_(s+6)) y
__device__ __forceinline__ void mul4(uint32_t* t, const uint32_t* x, int s, uint32_t y) {
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const uint64_t p = (uint64_t)x[s + 2 * j] * y;
    t[2 * j] = (uint32_t)p;
    t[2 * j + 1] = (uint32_t)(p >> 32);
  }
}
// Short chains of a square's rows: N products x0 y, x1 y, .. into t[0 .. 2N - 1].  MODE 0:
// the carry out becomes t[2N]; 1: t[2N - 1] is fresh; 2: the last two limbs are fresh.
template <int N, int MODE>
__device__ __forceinline__ void chain_s(uint32_t* t, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t y) {
  if constexpr (N == 3 && MODE == 0)
    asm("mad.lo.cc.u32  %0, %7, %10, %0;\n\tmadc.hi.cc.u32 %1, %7, %10, %1;\n\t"
        "madc.lo.cc.u32 %2, %8, %10, %2;\n\tmadc.hi.cc.u32 %3, %8, %10, %3;\n\t"
        "madc.lo.cc.u32 %4, %9, %10, %4;\n\tmadc.hi.cc.u32 %5, %9, %10, %5;\n\taddc.u32 %6, 0, 0;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "=r"(t[6])
        : "r"(x0), "r"(x1), "r"(x2), "r"(y));
  else if constexpr (N == 3 && MODE == 1)
    asm("mad.lo.cc.u32  %0, %6, %9, %0;\n\tmadc.hi.cc.u32 %1, %6, %9, %1;\n\t"
        "madc.lo.cc.u32 %2, %7, %9, %2;\n\tmadc.hi.cc.u32 %3, %7, %9, %3;\n\t"
        "madc.lo.cc.u32 %4, %8, %9, %4;\n\tmadc.hi.u32 %5, %8, %9, 0;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "=r"(t[5])
        : "r"(x0), "r"(x1), "r"(x2), "r"(y));
  else if constexpr (N == 3)
    asm("mad.lo.cc.u32  %0, %6, %9, %0;\n\tmadc.hi.cc.u32 %1, %6, %9, %1;\n\t"
        "madc.lo.cc.u32 %2, %7, %9, %2;\n\tmadc.hi.cc.u32 %3, %7, %9, %3;\n\t"
        "madc.lo.cc.u32 %4, %8, %9, 0;\n\tmadc.hi.u32 %5, %8, %9, 0;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "=r"(t[4]), "=r"(t[5])
        : "r"(x0), "r"(x1), "r"(x2), "r"(y));
  else if constexpr (N == 2 && MODE == 0)
    asm("mad.lo.cc.u32  %0, %5, %7, %0;\n\tmadc.hi.cc.u32 %1, %5, %7, %1;\n\t"
        "madc.lo.cc.u32 %2, %6, %7, %2;\n\tmadc.hi.cc.u32 %3, %6, %7, %3;\n\taddc.u32 %4, 0, 0;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "=r"(t[4])
        : "r"(x0), "r"(x1), "r"(y));
  else if constexpr (N == 2)
    asm("mad.lo.cc.u32  %0, %4, %6, %0;\n\tmadc.hi.cc.u32 %1, %4, %6, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %6, %2;\n\tmadc.hi.u32 %3, %5, %6, 0;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "=r"(t[3])
        : "r"(x0), "r"(x1), "r"(y));
  else if constexpr (MODE == 0)
    asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\tmadc.hi.cc.u32 %1, %3, %4, %1;\n\taddc.u32 %2, 0, 0;"
        : "+r"(t[0]), "+r"(t[1]), "=r"(t[2])
        : "r"(x0), "r"(y));
  else
    asm("mad.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.u32 %1, %2, %3, 0;" : "+r"(t[0]), "=r"(t[1]) : "r"(x0), "r"(y));
}

// One reduction row: q = e_0 (-N^-1) mod 2^32 and (e, o) += q N, which clears e_0.
template <class C>
__device__ __forceinline__ void red_row(uint32_t* e, uint32_t* o) {
  uint32_t n[8];
#pragma unroll
  for (int i = 0; i < 8; i++) n[i] = mod_limb<C>(i);
  const uint32_t q = e[0] * C::INV;
  chain(o, n, 1, q);
  chain_c(e, o[7], n, 0, q);
}

// The division by 2^32 after a row: o becomes the even accumulator, e_2.. the odd one, and
// e_1 stays pending (added to the new e_0 by the next chain_p2 or by merge).
__device__ __forceinline__ void shift(uint32_t* e, uint32_t* o, uint32_t* pend) {
  *pend = e[1];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const uint32_t up = j < 6 ? e[j + 2] : 0u;
    e[j] = o[j];
    o[j] = up;
  }
}

// r = e + 2^32 o + pend over eight limbs, for the state after a shift (o_6 = o_7 = 0)
__device__ __forceinline__ void merge(uint32_t (&r)[8], const uint32_t* e, const uint32_t* o, uint32_t pend) {
  asm("add.cc.u32  %0, %8,  %16;\n\taddc.cc.u32 %1, %9,  %17;\n\taddc.cc.u32 %2, %10, %18;\n\t"
      "addc.cc.u32 %3, %11, %19;\n\taddc.cc.u32 %4, %12, %20;\n\taddc.cc.u32 %5, %13, %21;\n\t"
      "addc.cc.u32 %6, %14, %22;\n\taddc.u32 %7, %15, 0;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(e[0]), "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(pend), "r"(o[0]),
        "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]));
}

// the whole product a b: e[0..15], o[0..14]
__device__ __forceinline__ void mul_wide(uint32_t* e, uint32_t* o, const uint32_t* a, const uint32_t* b) {
  mul4(e, a, 0, b[0]);
  mul4(o, a, 1, b[0]);
#pragma unroll
  for (int i = 1; i < 8; i += 2) {
    if (i == 1)
      chain_f2(e + 2, a, 1, b[1]);
    else
      chain_f1(e + i + 1, a, 1, b[i]);
    chain_cf(o + i - 1, o[i + 7], a, 0, b[i]);
    if (i < 7) {
      chain_cf(e + i + 1, e[i + 9], a, 0, b[i + 1]);
      chain_f1(o + i + 1, a, 1, b[i + 1]);
    }
  }
}

// the whole square a^2 (a < 2^255): 28 products a_i a_j (i < j) against limbs of 2a, whose
// row i starts at limb i + 1 without the bit that comes up from a_i, then the 8 diagonals
__device__ __forceinline__ void sqr_wide(uint32_t* e, uint32_t* o, const uint32_t* a) {
  uint32_t d[8], s[8];
#pragma unroll
  for (int j = 1; j < 8; j++) {
    d[j] = __funnelshift_l(a[j - 1], a[j], 1);
    s[j] = a[j] << 1;
  }
  const uint32_t x[8] = {s[1], d[2], d[3], d[4], d[5], d[6], d[7], 0};
  mul4(o, x, 0, a[0]);
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const uint64_t p = (uint64_t)d[2 + 2 * j] * a[0];
    e[2 + 2 * j] = (uint32_t)p;
    e[3 + 2 * j] = (uint32_t)(p >> 32);
  }
  chain_s<3, 0>(o + 2, s[2], d[4], d[6], a[1]);
  chain_s<3, 2>(e + 4, d[3], d[5], d[7], a[1]);
  chain_s<3, 1>(o + 4, s[3], d[5], d[7], a[2]);
  chain_s<2, 0>(e + 6, d[4], d[6], 0, a[2]);
  chain_s<2, 0>(o + 6, s[4], d[6], 0, a[3]);
  chain_s<2, 1>(e + 8, d[5], d[7], 0, a[3]);
  chain_s<2, 1>(o + 8, s[5], d[7], 0, a[4]);
  chain_s<1, 0>(e + 10, d[6], 0, 0, a[4]);
  chain_s<1, 0>(o + 10, s[6], 0, 0, a[5]);
  chain_s<1, 1>(e + 12, d[7], 0, 0, a[5]);
  chain_s<1, 1>(o + 12, s[7], 0, 0, a[6]);
  o[14] = 0;
  asm("mul.lo.u32     %0,  %16, %16;\n\tmul.hi.u32     %1,  %16, %16;\n\t"
      "mad.lo.cc.u32  %2,  %17, %17, %2;\n\tmadc.hi.cc.u32 %3,  %17, %17, %3;\n\t"
      "madc.lo.cc.u32 %4,  %18, %18, %4;\n\tmadc.hi.cc.u32 %5,  %18, %18, %5;\n\t"
      "madc.lo.cc.u32 %6,  %19, %19, %6;\n\tmadc.hi.cc.u32 %7,  %19, %19, %7;\n\t"
      "madc.lo.cc.u32 %8,  %20, %20, %8;\n\tmadc.hi.cc.u32 %9,  %20, %20, %9;\n\t"
      "madc.lo.cc.u32 %10, %21, %21, %10;\n\tmadc.hi.cc.u32 %11, %21, %21, %11;\n\t"
      "madc.lo.cc.u32 %12, %22, %22, %12;\n\tmadc.hi.cc.u32 %13, %22, %22, %13;\n\t"
      "madc.lo.cc.u32 %14, %23, %23, 0;\n\tmadc.hi.u32 %15, %23, %23, 0;"
      : "=&r"(e[0]), "=&r"(e[1]), "+&r"(e[2]), "+&r"(e[3]), "+&r"(e[4]), "+&r"(e[5]), "+&r"(e[6]), "+&r"(e[7]),
        "+&r"(e[8]), "+&r"(e[9]), "+&r"(e[10]), "+&r"(e[11]), "+&r"(e[12]), "+&r"(e[13]), "=&r"(e[14]), "=&r"(e[15])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]));
}

// t = e + 2^32 o, 16 limbs
__device__ __forceinline__ void merge_wide(uint32_t* t, const uint32_t* e, const uint32_t* o) {
  uint32_t c;
  t[0] = e[0];
  asm("add.cc.u32  %0, %8,  %15;\n\taddc.cc.u32 %1, %9,  %16;\n\taddc.cc.u32 %2, %10, %17;\n\t"
      "addc.cc.u32 %3, %11, %18;\n\taddc.cc.u32 %4, %12, %19;\n\taddc.cc.u32 %5, %13, %20;\n\t"
      "addc.cc.u32 %6, %14, %21;\n\taddc.u32 %7, 0, 0;"
      : "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]), "=r"(t[7]), "=r"(c)
      : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(o[0]), "r"(o[1]), "r"(o[2]),
        "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]));
  asm("add.cc.u32  %8, %8,  0xffffffff;\n\taddc.cc.u32 %0, %9,  %17;\n\taddc.cc.u32 %1, %10, %18;\n\t"
      "addc.cc.u32 %2, %11, %19;\n\taddc.cc.u32 %3, %12, %20;\n\taddc.cc.u32 %4, %13, %21;\n\t"
      "addc.cc.u32 %5, %14, %22;\n\taddc.cc.u32 %6, %15, %23;\n\taddc.u32 %7, %16, %24;"
      : "=&r"(t[8]), "=&r"(t[9]), "=&r"(t[10]), "=&r"(t[11]), "=&r"(t[12]), "=&r"(t[13]), "=&r"(t[14]), "=&r"(t[15]),
        "+&r"(c)
      : "r"(e[8]), "r"(e[9]), "r"(e[10]), "r"(e[11]), "r"(e[12]), "r"(e[13]), "r"(e[14]), "r"(e[15]), "r"(o[7]),
        "r"(o[8]), "r"(o[9]), "r"(o[10]), "r"(o[11]), "r"(o[12]), "r"(o[13]), "r"(o[14]));
}

// x += y and x -= y over 16 limbs modulo 2^512; w_sub returns 1 if it borrowed
__device__ __forceinline__ void w_add(uint32_t* x, const uint32_t* y) {
  uint32_t lo[8], hi[8], a[8], b[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    a[i] = x[i];
    b[i] = y[i];
  }
  uint32_t c = add8(lo, a, b);
  asm("add.cc.u32  %8, %8,  0xffffffff;\n\taddc.cc.u32 %0, %9,  %17;\n\taddc.cc.u32 %1, %10, %18;\n\t"
      "addc.cc.u32 %2, %11, %19;\n\taddc.cc.u32 %3, %12, %20;\n\taddc.cc.u32 %4, %13, %21;\n\t"
      "addc.cc.u32 %5, %14, %22;\n\taddc.cc.u32 %6, %15, %23;\n\taddc.u32 %7, %16, %24;"
      : "=&r"(hi[0]), "=&r"(hi[1]), "=&r"(hi[2]), "=&r"(hi[3]), "=&r"(hi[4]), "=&r"(hi[5]), "=&r"(hi[6]),
        "=&r"(hi[7]), "+&r"(c)
      : "r"(x[8]), "r"(x[9]), "r"(x[10]), "r"(x[11]), "r"(x[12]), "r"(x[13]), "r"(x[14]), "r"(x[15]), "r"(y[8]),
        "r"(y[9]), "r"(y[10]), "r"(y[11]), "r"(y[12]), "r"(y[13]), "r"(y[14]), "r"(y[15]));
#pragma unroll
  for (int i = 0; i < 8; i++) {
    x[i] = lo[i];
    x[8 + i] = hi[i];
  }
}
__device__ __forceinline__ uint32_t w_sub(uint32_t* x, const uint32_t* y) {
  uint32_t lo[8], hi[8], a[8], b[8], c;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    a[i] = x[i];
    b[i] = y[i];
  }
  const uint32_t br = sub8(lo, a, b);
  asm("sub.cc.u32  %8, 0,   %25;\n\tsubc.cc.u32 %0, %9,  %17;\n\tsubc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\tsubc.cc.u32 %3, %12, %20;\n\tsubc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\tsubc.cc.u32 %6, %15, %23;\n\tsubc.cc.u32 %7, %16, %24;\n\tsubc.u32 %8, 0, 0;"
      : "=&r"(hi[0]), "=&r"(hi[1]), "=&r"(hi[2]), "=&r"(hi[3]), "=&r"(hi[4]), "=&r"(hi[5]), "=&r"(hi[6]),
        "=&r"(hi[7]), "=&r"(c)
      : "r"(x[8]), "r"(x[9]), "r"(x[10]), "r"(x[11]), "r"(x[12]), "r"(x[13]), "r"(x[14]), "r"(x[15]), "r"(y[8]),
        "r"(y[9]), "r"(y[10]), "r"(y[11]), "r"(y[12]), "r"(y[13]), "r"(y[14]), "r"(y[15]), "r"(br));
#pragma unroll
  for (int i = 0; i < 8; i++) {
    x[i] = lo[i];
    x[8 + i] = hi[i];
  }
  return c & 1u;
}
}  // namespace eo

// r < 2N brought below N
template <class C>
__device__ __forceinline__ Field<C> f_once(const Field<C>& r) {
  Field<C> d;
  const Field<C> m = Field<C>::modulus();
  const uint32_t br = sub8(d.v, r.v, m.v);
  return br ? r : d;
}

// Montgomery product a b R^-1 mod N, not brought below N.  For a <= 4N and any b < 2^256:
// after each row the state is below a + N <= 5N < 2^256 and before the division below
// 2^288, so nothing leaves limb 8; the result is below a b / R + N: below 2N for a < 4N and
// b < N, for a, b < 2N, and for a < N and any b.
template <class C>
__device__ __forceinline__ Field<C> f_mul_lazy(const Field<C>& a, const Field<C>& b) {
  uint32_t e[8], o[8], pend;
  eo::mul4(e, a.v, 0, b.v[0]);
  eo::mul4(o, a.v, 1, b.v[0]);
  eo::red_row<C>(e, o);
  eo::shift(e, o, &pend);
#pragma unroll
  for (int i = 1; i < 8; i++) {
    eo::chain_p2(e[0], pend, o, a.v, 1, b.v[i]);
    eo::chain_c(e, o[7], a.v, 0, b.v[i]);
    eo::red_row<C>(e, o);
    eo::shift(e, o, &pend);
  }
  Field<C> r;
  eo::merge(r.v, e, o, pend);
  return r;
}

// Products by a constant w known ahead (a transform's twiddles) with its quotient
// wq = floor(w 2^256 / N) beside it (Shoup's method, as in Harvey, "Faster arithmetic for
// number-theoretic transforms", 2014): q = floor(x wq / 2^256) is the quotient of x w / N or
// a little less, so x w - q N is found from its low 256 bits alone.  Neither product is
// needed whole: q from the columns 6 .. 14 of x wq (43 multiply-adds, short of the true
// quotient by less than x / 2^256 + 1 + 2^-29), and the columns 0 .. 7 of x w and of
// q (2^256 - N), summed in one pair of accumulators (28 and 8 low products each): 99
// multiply-adds and 16 low products against the Montgomery product's 128 and 8.
namespace eo {
// N products x0 y, x1 y, x2 y into t[0 .. 2N - 1], the carry out dropped; LOW: one more
// whose low half alone goes to t[2N]
template <int N, bool LOW>
__device__ __forceinline__ void chain_low(uint32_t* t, const uint32_t* x, uint32_t y) {
  if constexpr (N == 3 && LOW)
    asm("mad.lo.cc.u32  %0, %7, %11, %0;\n\tmadc.hi.cc.u32 %1, %7, %11, %1;\n\t"
        "madc.lo.cc.u32 %2, %8, %11, %2;\n\tmadc.hi.cc.u32 %3, %8, %11, %3;\n\t"
        "madc.lo.cc.u32 %4, %9, %11, %4;\n\tmadc.hi.cc.u32 %5, %9, %11, %5;\n\tmadc.lo.u32 %6, %10, %11, %6;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6])
        : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(y));
  else if constexpr (N == 2 && LOW)
    asm("mad.lo.cc.u32  %0, %5, %8, %0;\n\tmadc.hi.cc.u32 %1, %5, %8, %1;\n\t"
        "madc.lo.cc.u32 %2, %6, %8, %2;\n\tmadc.hi.cc.u32 %3, %6, %8, %3;\n\tmadc.lo.u32 %4, %7, %8, %4;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4])
        : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(y));
  else if constexpr (N == 1 && LOW)
    asm("mad.lo.cc.u32 %0, %3, %5, %0;\n\tmadc.hi.cc.u32 %1, %3, %5, %1;\n\tmadc.lo.u32 %2, %4, %5, %2;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2])
        : "r"(x[0]), "r"(x[2]), "r"(y));
  else if constexpr (LOW)
    t[0] += x[0] * y;
  else if constexpr (N == 4)
    chain(t, x, 0, y);
  else if constexpr (N == 3)
    asm("mad.lo.cc.u32  %0, %6, %9, %0;\n\tmadc.hi.cc.u32 %1, %6, %9, %1;\n\t"
        "madc.lo.cc.u32 %2, %7, %9, %2;\n\tmadc.hi.cc.u32 %3, %7, %9, %3;\n\t"
        "madc.lo.cc.u32 %4, %8, %9, %4;\n\tmadc.hi.u32 %5, %8, %9, %5;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5])
        : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(y));
  else if constexpr (N == 2)
    asm("mad.lo.cc.u32  %0, %4, %6, %0;\n\tmadc.hi.cc.u32 %1, %4, %6, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %6, %2;\n\tmadc.hi.u32 %3, %5, %6, %3;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3])
        : "r"(x[0]), "r"(x[2]), "r"(y));
  else
    asm("mad.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.u32 %1, %2, %3, %1;"
        : "+r"(t[0]), "+r"(t[1])
        : "r"(x[0]), "r"(y));
}
// rows I .. 7 of the low half of x y: e[0..7] + 2^32 o[0..6] += x y_I 2^(32 I) + .. mod 2^256
template <int I>
__device__ __forceinline__ void low_rows(uint32_t* e, uint32_t* o, const uint32_t* x, const uint32_t* y) {
  if constexpr (I < 8) {
    // even columns I + j <= 6 and odd ones I + j <= 7 (the last by its low half)
    if constexpr (I % 2 == 0) {
      chain_low<4 - I / 2, false>(e + I, x, y[I]);
      chain_low<3 - I / 2, true>(o + I, x + 1, y[I]);
    } else {
      if constexpr (I < 7) chain_low<3 - I / 2, false>(e + I + 1, x + 1, y[I]);
      chain_low<3 - I / 2, true>(o + I - 1, x, y[I]);
    }
    low_rows<I + 1>(e, o, x, y);
  }
}
}  // namespace eo

// x w mod N, not brought below N: below 2N for x < 4N (w < N in plain form, wq its quotient)
template <class C>
__device__ __forceinline__ Field<C> f_mul_const(const Field<C>& x, const Field<C>& w, const Field<C>& wq) {
  uint32_t e[10], o[9], q[8], n[8];
  const uint32_t* a = x.v;
  {  // columns 6 .. 14 of x wq: e[c - 6], e[c - 5] even c; o[c - 7], o[c - 6] odd c
    const uint64_t p6 = (uint64_t)a[6] * wq.v[0], p7 = (uint64_t)a[7] * wq.v[0];
    e[0] = (uint32_t)p6;
    e[1] = (uint32_t)(p6 >> 32);
    e[2] = 0;
    o[0] = (uint32_t)p7;
    o[1] = (uint32_t)(p7 >> 32);
    eo::chain_s<2, 1>(e, a[5], a[7], 0, wq.v[1]);
    eo::chain_s<1, 0>(o, a[6], 0, 0, wq.v[1]);
    eo::chain_s<2, 0>(e, a[4], a[6], 0, wq.v[2]);
    eo::chain_s<2, 1>(o, a[5], a[7], 0, wq.v[2]);
    eo::chain_s<3, 1>(e, a[3], a[5], a[7], wq.v[3]);
    eo::chain_s<2, 0>(o, a[4], a[6], 0, wq.v[3]);
    eo::chain_s<3, 0>(e, a[2], a[4], a[6], wq.v[4]);
    eo::chain_s<3, 1>(o, a[3], a[5], a[7], wq.v[4]);
    eo::chain_f1(e, a, 1, wq.v[5]);
    eo::chain_s<3, 0>(o, a[2], a[4], a[6], wq.v[5]);
    eo::chain_cf(e, e[8], a, 0, wq.v[6]);
    eo::chain_f1(o, a, 1, wq.v[6]);
    eo::chain_f1(e + 2, a, 1, wq.v[7]);
    eo::chain_cf(o, o[8], a, 0, wq.v[7]);
    asm("{\n\t.reg .u32 c;\n\tadd.cc.u32 c, %8, %17;\n\t"
        "addc.cc.u32 %0, %9,  %18;\n\taddc.cc.u32 %1, %10, %19;\n\taddc.cc.u32 %2, %11, %20;\n\t"
        "addc.cc.u32 %3, %12, %21;\n\taddc.cc.u32 %4, %13, %22;\n\taddc.cc.u32 %5, %14, %23;\n\t"
        "addc.cc.u32 %6, %15, %24;\n\taddc.u32 %7, %16, %25;\n\t}"
        : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7])
        : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(e[8]), "r"(e[9]), "r"(o[0]),
          "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]), "r"(o[8]));
  }
#pragma unroll
  for (int i = 0; i < 8; i++) n[i] = i == 0 ? 0u - mod_limb<C>(0) : ~mod_limb<C>(i);  // 2^256 - N (N is odd)
  eo::mul4(e, a, 0, w.v[0]);
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const uint64_t p = (uint64_t)a[1 + 2 * j] * w.v[0];
    o[2 * j] = (uint32_t)p;
    o[2 * j + 1] = (uint32_t)(p >> 32);
  }
  o[6] = a[7] * w.v[0];
  eo::low_rows<1>(e, o, a, w.v);
  eo::low_rows<0>(e, o, n, q);
  Field<C> r;
  r.v[0] = e[0];
  asm("add.cc.u32  %0, %7,  %14;\n\taddc.cc.u32 %1, %8,  %15;\n\taddc.cc.u32 %2, %9, %16;\n\t"
      "addc.cc.u32 %3, %10, %17;\n\taddc.cc.u32 %4, %11, %18;\n\taddc.cc.u32 %5, %12, %19;\n\t"
      "addc.u32 %6, %13, %20;"
      : "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]), "=r"(r.v[7])
      : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(o[0]), "r"(o[1]), "r"(o[2]),
        "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]));
  return r;
}

// the product below N, for operands whose lazy product is below 2N.  (Values that may exceed
// N come second: f_to_mont reduces an arbitrary 256-bit value.)
template <class C>
__device__ __forceinline__ Field<C> f_mul(const Field<C>& a, const Field<C>& b) {
  return f_once(f_mul_lazy(a, b));
}

// Lazy butterfly arithmetic: x < 4N brought below 2N; a + b below 2N and a - b + 2N below 4N
// for a, b < 2N
template <class C>
__device__ __forceinline__ Field<C> f_red2(const Field<C>& x) {
  Field<C> m, d;
#pragma unroll
  for (int i = 0; i < 8; i++) m.v[i] = mod2_limb<C>(i);
  const uint32_t br = sub8(d.v, x.v, m.v);
  return br ? x : d;
}
template <class C>
__device__ __forceinline__ Field<C> f_add_raw(const Field<C>& a, const Field<C>& b) {
  Field<C> s;
  add8(s.v, a.v, b.v);
  return s;
}
template <class C>
__device__ __forceinline__ Field<C> f_add2(const Field<C>& a, const Field<C>& b) { return f_red2(f_add_raw(a, b)); }
template <class C>
__device__ __forceinline__ Field<C> f_sub2(const Field<C>& a, const Field<C>& b) {
  Field<C> m, s, d;
#pragma unroll
  for (int i = 0; i < 8; i++) m.v[i] = mod2_limb<C>(i);
  add8(s.v, a.v, m.v);
  sub8(d.v, s.v, b.v);
  return d;
}

// (a b + c d) R^-1 mod N with one reduction, for operands up to N: the state stays below
// a + c + N <= 3N < 2^256, the result below 2N^2 / R + N < 2N.
template <class C>
__device__ __forceinline__ Field<C> f_mul2(const Field<C>& a, const Field<C>& b, const Field<C>& c,
                                           const Field<C>& d) {
  uint32_t e[8], o[8], pend;
  eo::mul4(e, a.v, 0, b.v[0]);
  eo::mul4(o, a.v, 1, b.v[0]);
  eo::chain(o, c.v, 1, d.v[0]);
  eo::chain_c(e, o[7], c.v, 0, d.v[0]);
  eo::red_row<C>(e, o);
  eo::shift(e, o, &pend);
#pragma unroll
  for (int i = 1; i < 8; i++) {
    eo::chain_p2(e[0], pend, o, a.v, 1, b.v[i]);
    eo::chain_c(e, o[7], a.v, 0, b.v[i]);
    eo::chain(o, c.v, 1, d.v[i]);
    eo::chain_c(e, o[7], c.v, 0, d.v[i]);
    eo::red_row<C>(e, o);
    eo::shift(e, o, &pend);
  }
  Field<C> r;
  eo::merge(r.v, e, o, pend);
  return f_once(r);
}

// t R^-1 mod N for a 16-limb t < N R given as low limbs e[0..7] + 2^32 o[0..7] (o[7] = 0)
// and its top half: the low half reduces to at most N + 1, the sum to less than 2N.
template <class C>
__device__ __forceinline__ Field<C> f_redc(uint32_t* e, uint32_t* o, const uint32_t (&top)[8]) {
  uint32_t n[8], pend;
#pragma unroll
  for (int i = 0; i < 8; i++) n[i] = mod_limb<C>(i);
  eo::red_row<C>(e, o);
  eo::shift(e, o, &pend);
#pragma unroll
  for (int i = 1; i < 8; i++) {
    const uint32_t q = (e[0] + pend) * C::INV;
    eo::chain_p2(e[0], pend, o, n, 1, q);
    eo::chain_c(e, o[7], n, 0, q);
    eo::shift(e, o, &pend);
  }
  Field<C> r;
  uint32_t lo[8];
  eo::merge(lo, e, o, pend);
  add8(r.v, lo, top);
  return f_once(r);
}

// the same for t[0..15]
template <class C>
__device__ __forceinline__ Field<C> f_redc_wide(const uint32_t* t) {
  uint32_t e[8], o[8], top[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    e[i] = t[i];
    o[i] = 0;
    top[i] = t[8 + i];
  }
  return f_redc<C>(e, o, top);
}

// a^2 R^-1 mod N for a <= N: 36 products and a reduction instead of 64
template <class C>
__device__ __forceinline__ Field<C> f_sqr(const Field<C>& a) {
  uint32_t E[16], O[15], e[8], o[8], x[8], y[8], top[8];
  eo::sqr_wide(E, O, a.v);
#pragma unroll
  for (int i = 0; i < 8; i++) {
    e[i] = E[i];
    o[i] = i < 7 ? O[i] : 0u;
    x[i] = E[8 + i];
    y[i] = O[7 + i];
  }
  add8(top, x, y);
  return f_redc<C>(e, o, top);
}

// Out-of-line Montgomery product with 64-bit accumulation: CIOS rows written with
// 32 x 32 + 64-bit multiply-adds in plain C (reference form: 12.6 T IMAD-equivalents/s in
// zkvc_imad_rate form 6, against 18.1 T/s for product scanning and 19 T/s for f_mulc below).
template <class C>
__device__ __noinline__ Field<C> f_mulc_cios(Field<C> a, Field<C> b) {
  uint32_t t[10];
#pragma unroll
  for (int i = 0; i < 10; i++) t[i] = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    uint64_t c = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      uint64_t s = (uint64_t)a.v[j] * b.v[i] + t[j] + c;  // < 2^64
      t[j] = (uint32_t)s;
      c = s >> 32;
    }
    uint64_t s8 = (uint64_t)t[8] + c;
    t[8] = (uint32_t)s8;
    t[9] = (uint32_t)(s8 >> 32);
    uint32_t q = t[0] * C::INV;
    c = ((uint64_t)q * mod_limb<C>(0) + t[0]) >> 32;  // low word cancels
#pragma unroll
    for (int j = 1; j < 8; j++) {
      uint64_t s = (uint64_t)q * mod_limb<C>(j) + t[j] + c;
      t[j - 1] = (uint32_t)s;
      c = s >> 32;
    }
    uint64_t s7 = (uint64_t)t[8] + c;
    t[7] = (uint32_t)s7;
    t[8] = t[9] + (uint32_t)(s7 >> 32);
    t[9] = 0;
  }
  Field<C> r, d;
  uint32_t m[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    r.v[i] = t[i];
    m[i] = mod_limb<C>(i);
  }
  uint32_t br = sub8(d.v, r.v, m);  // result < 2N < 2^255, so t[8] = 0 here
  return br ? r : d;
}

// Out-of-line products for the point formulas: called, not inlined, so that the large
// formulas keep one copy of each (fully inlined point formulas stall on instruction fetch).
template <class C>
__device__ __noinline__ Field<C> f_mulc(Field<C> a, Field<C> b) {
  return f_mul(a, b);
}
template <class C>
__device__ __noinline__ Field<C> f_sqrc(Field<C> a) {
  return f_sqr(a);
}
template <class C>
__device__ __noinline__ Field<C> f_mul2c(Field<C> a, Field<C> b, Field<C> c, Field<C> d) {
  return f_mul2(a, b, c, d);
}

// t < 64 N (nine limbs) mod N: the quotient from the top bits, at most one short (both
// moduli begin with the same bits: N / 2^240 lies in (12388, 12389))
template <class C>
__device__ __forceinline__ Field<C> f_mod9(const uint32_t (&t)[9]) {
  static_assert(C::MOD.w[7] >> 16 == 12388, "the quotient estimate's divisor");
  const uint32_t h = (t[7] >> 16) | (t[8] << 16);  // t / 2^240 < 2^20
  const uint32_t q = __umulhi(h, 346675u);         // 2^32 / 12389
  uint32_t p[8];
  Field<C> r, x;
  uint64_t c = 0;
#pragma unroll
  for (int i = 0; i < 8; i++) {
    c += (uint64_t)q * mod_limb<C>(i);
    p[i] = (uint32_t)c;
    c >>= 32;
    x.v[i] = t[i];
  }
  sub8(r.v, x.v, p);  // below 2N: the ninth limbs cancel
  return f_once(r);
}

// a R mod N for any a < 2^256 (the second operand of f_mul may exceed N)
template <class C>
__device__ __forceinline__ Field<C> f_to_mont(const Field<C>& a) {
  Field<C> r2;
#pragma unroll
  for (int i = 0; i < 8; i++) r2.v[i] = r2_limb<C>(i);
  return f_mul(r2, a);
}

template <class C>
__device__ __forceinline__ Field<C> f_from_mont(const Field<C>& a) {
  Field<C> one_raw = Field<C>::zero();
  one_raw.v[0] = 1;
  return f_mul(a, one_raw);
}

// Canonical value from a small signed integer (|v| < 2^31), already in Montgomery form.
template <class C>
__device__ __forceinline__ Field<C> f_from_int(int32_t v) {
  Field<C> x = Field<C>::zero();
  uint32_t mag = v < 0 ? (uint32_t)(-(int64_t)v) : (uint32_t)v;
  x.v[0] = mag;
  x = f_to_mont(x);
  return v < 0 ? f_neg(x) : x;
}

// a^e for an exponent given as 8 limbs (plain square-and-multiply, MSB first).
template <class C>
__device__ __forceinline__ Field<C> f_pow(const Field<C>& a, const uint32_t (&e)[8]) {
  Field<C> r = Field<C>::one();
  for (int i = 7; i >= 0; i--) {
    for (int bit = 31; bit >= 0; bit--) {
      r = f_sqr(r);
      if ((e[i] >> bit) & 1u) r = f_mul(r, a);
    }
  }
  return r;
}

// Inverse of a Montgomery-form element (a R -> a^-1 R); 0 maps to 0.  Not constant-time.
//
// Binary division (Stehle and Zimmermann, "A binary recursive gcd algorithm", 2004) on
// (f, g) = (N, a R), f odd: halve g until it is odd, counting the halvings j past those the
// division before has brought for free; then (f, g) <- (g, f + q g) with the odd q of least
// magnitude that makes the sum divisible by 2^(j + 1) (|q| < 2^j).  All of it is decided by
// low bits, so 30 halvings at a time run on the low words alone and give a matrix
//   2^30 (f, g)' = [[fa, fb], [ga, gb]] (f, g),  row sums of magnitudes at most 2^30
// (as in the jumps of Bernstein and Yang, "Fast constant-time gcd computation and modular
// inversion", 2019), which then updates the whole numbers.  f and g stay in [-N, N] and end
// as +-1 and 0; d and e stay in [0, 3N/2] with d a R = f c and e a R = g c modulo N for one
// c, which a batch divides by 4: the pair is multiplied by the matrix and divided by 2^32, a
// limb, as one row of a Montgomery product does it, where f and g are divided by 2^30.
// Remainders grow by (1 + sqrt 17) / 4 per division at the most, so 2 * 254 /
// (2 - log2((1 + sqrt 17) / 2)) = 790 halvings reach |g| = 1 (about 540 on average) and one
// more division 0: 28 batches, 18 on average.
//
// What bounds it: the latency of one thread, in equal parts in the divisions and in the
// updates' wide products, and the first fetch of its code: a proof runs it a few times, each
// in another kernel.  So the two rows' updates are a loop.  Measured: one thread 32.2 k cycles,
// a warp of 32 inversions 42.0 k, 1.83 G inversions/s on the whole GPU, the chain-mode proof of
// [49,320]x[320,512] 700 us; with the rows written out 30.0 k, 39.8 k, 1.99 G and 707 us
// (divsteps on signed limbs, the form before: 30.5 k, 39.4 k, 1.70 G and 700 us).
namespace inv {
constexpr int BATCH = 30;         // halvings per matrix
constexpr int QUOTIENT_BITS = 5;  // bits of a quotient found at once

struct Rows {
  int32_t fa, fb, ga, gb;
};

// A batch on the low words of f and g.  due: halvings since the last division less its j, so
// the next division's j once positive; returned for the next batch.
__device__ __forceinline__ int batch(int due, uint32_t f, uint32_t g, Rows& m) {
  int32_t fa = 1, fb = 0, ga = 0, gb = 1;
  uint32_t left = BATCH;
  for (;;) {
    const uint32_t z = min((uint32_t)__ffs((int)g) - 1u, left);  // g = 0: what is left
    g >>= z;
    fa <<= z;
    fb <<= z;
    left -= z;
    due += (int)z;
    if (left == 0) break;
    if (due > 0) {  // g takes f's place
      const uint32_t t = f;
      f = g;
      g = t;
      const int32_t ta = fa, tb = fb;
      fa = ga;
      fb = gb;
      ga = ta;
      gb = tb;
      due = -due;
    }
    // g + w f clears bits of g: w = -g / f modulo 2^bits, of least magnitude where these
    // complete the quotient ((3 f) xor 2 is 1 / f modulo 32)
    const uint32_t want = (uint32_t)(1 - due), bits = min(min(want, left), (uint32_t)QUOTIENT_BITS);
    const uint32_t w0 = (0u - g * ((3u * f) ^ 2u)) << (32u - bits);
    const int32_t w = bits == want ? (int32_t)w0 >> (32u - bits) : (int32_t)(w0 >> (32u - bits));
    g += f * (uint32_t)w;
    ga += fa * w;
    gb += fb * w;
  }
  // either row may change its sign, and with it that of f and d or of g and e
  m = {abs(fa), fa < 0 ? -fb : fb, abs(ga), ga < 0 ? -gb : gb};
  return due;
}

// r = (a x + b y) / 2^30 (exact), x and y in two's complement, a >= 0: a and |b| times x and
// y or its complement, and what the complement and the unsigned reading of a negative number
// leave out: 1 for the one, 2^256 for the other
__device__ __forceinline__ void combine(uint32_t (&r)[8], const uint32_t (&x)[8], uint32_t a, const uint32_t (&y)[8],
                                        int32_t b) {
  const uint32_t s = (uint32_t)(b >> 31), m = ((uint32_t)b ^ s) - s;
  uint64_t e[4], o[4];
#pragma unroll
  for (int j = 0; j < 4; j++) {  // a + |b| <= 2^30: each below 2^62
    e[j] = (uint64_t)x[2 * j] * a + (uint64_t)(y[2 * j] ^ s) * m;
    o[j] = (uint64_t)x[2 * j + 1] * a + (uint64_t)(y[2 * j + 1] ^ s) * m;
  }
  e[0] += m & s;
  const uint32_t high = (a & (uint32_t)((int32_t)x[7] >> 31)) + (m & ((uint32_t)((int32_t)y[7] >> 31) ^ s));
  uint32_t t[9];
  t[0] = (uint32_t)e[0];
  asm("add.cc.u32  %0, %8,  %15;\n\taddc.cc.u32 %1, %9,  %16;\n\taddc.cc.u32 %2, %10, %17;\n\t"
      "addc.cc.u32 %3, %11, %18;\n\taddc.cc.u32 %4, %12, %19;\n\taddc.cc.u32 %5, %13, %20;\n\t"
      "addc.cc.u32 %6, %14, %21;\n\taddc.u32 %7, %22, %23;"
      : "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]), "=&r"(t[6]), "=&r"(t[7]), "=&r"(t[8])
      : "r"((uint32_t)(e[0] >> 32)), "r"((uint32_t)e[1]), "r"((uint32_t)(e[1] >> 32)), "r"((uint32_t)e[2]),
        "r"((uint32_t)(e[2] >> 32)), "r"((uint32_t)e[3]), "r"((uint32_t)(e[3] >> 32)), "r"((uint32_t)o[0]),
        "r"((uint32_t)(o[0] >> 32)), "r"((uint32_t)o[1]), "r"((uint32_t)(o[1] >> 32)), "r"((uint32_t)o[2]),
        "r"((uint32_t)(o[2] >> 32)), "r"((uint32_t)o[3]), "r"((uint32_t)(o[3] >> 32)), "r"(0u - high));
#pragma unroll
  for (int i = 0; i < 8; i++) r[i] = __funnelshift_r(t[i], t[i + 1], BATCH);
}

// (a x + b y) / 2^32 modulo N, ny = 2N - y: for x and y up to 3N / 2 below 2N 2^30 / 2^32 + N
template <class C>
__device__ __forceinline__ Field<C> combine_mod(const Field<C>& x, uint32_t a, const Field<C>& y, const Field<C>& ny,
                                                int32_t b) {
  const uint32_t m = (uint32_t)abs(b);
  uint32_t e[8], o[8];
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const uint64_t p = (uint64_t)x.v[j] * a + (uint64_t)(b < 0 ? ny.v[j] : y.v[j]) * m;
    (j & 1 ? o : e)[j & ~1] = (uint32_t)p;
    (j & 1 ? o : e)[j | 1] = (uint32_t)(p >> 32);
  }
  eo::red_row<C>(e, o);
  Field<C> r;
  asm("add.cc.u32  %0, %8,  %15;\n\taddc.cc.u32 %1, %9,  %16;\n\taddc.cc.u32 %2, %10, %17;\n\t"
      "addc.cc.u32 %3, %11, %18;\n\taddc.cc.u32 %4, %12, %19;\n\taddc.cc.u32 %5, %13, %20;\n\t"
      "addc.cc.u32 %6, %14, %21;\n\taddc.u32 %7, %22, 0;"
      : "=&r"(r.v[0]), "=&r"(r.v[1]), "=&r"(r.v[2]), "=&r"(r.v[3]), "=&r"(r.v[4]), "=&r"(r.v[5]), "=&r"(r.v[6]),
        "=&r"(r.v[7])
      : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(o[0]), "r"(o[1]), "r"(o[2]),
        "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]));
  return r;
}
}  // namespace inv

template <class C>
__device__ __noinline__ Field<C> f_inv(const Field<C>& a) {
  if (a.is_zero()) return Field<C>::zero();
  Field<C> f = Field<C>::modulus(), g = a, d = Field<C>::zero(), e;
#pragma unroll
  for (int i = 0; i < 8; i++) e.v[i] = r3_limb<C>(i);
  int due = 0, n = 1;
  for (; n < 31; n++) {
    inv::Rows m;
    due = inv::batch(due, f.v[0], g.v[0], m);
    Field<C> m2, ne;
#pragma unroll
    for (int i = 0; i < 8; i++) m2.v[i] = mod2_limb<C>(i);
    sub8(ne.v, m2.v, e.v);
    const Field<C> f0 = f, g0 = g, d0 = d, e0 = e;
#pragma unroll 1
    for (int row = 0; row < 2; row++) {  // f's row, then g's
      f = g;
      d = e;
      inv::combine(g.v, f0.v, (uint32_t)m.fa, g0.v, m.fb);
      e = inv::combine_mod(d0, (uint32_t)m.fa, e0, ne, m.fb);
      m.fa = m.ga;
      m.fb = m.gb;
    }
    if (g.is_zero()) break;
  }
  // d = +-(R^3 / 4^n) / (a R): times 4^n / R
  const uint64_t c = uint64_t(1) << (2 * n);
  Field<C> back = Field<C>::zero();
  back.v[0] = (uint32_t)c;
  back.v[1] = (uint32_t)(c >> 32);
  const Field<C> r = f_mul(d, back);
  return f.v[7] >> 31 ? f_neg(r) : r;
}

using Fp = Field<FpCfg>;
using Fr = Field<FrCfg>;

// ------------------------------------------------------------------ Fp2 = Fp[i]/(i^2+1)
struct Fp2 {
  Fp c0, c1;
  __device__ __forceinline__ static Fp2 zero() { return {Fp::zero(), Fp::zero()}; }
  __device__ __forceinline__ static Fp2 one() { return {Fp::one(), Fp::zero()}; }
  __device__ __forceinline__ bool is_zero() const { return c0.is_zero() && c1.is_zero(); }
  __device__ __forceinline__ bool operator==(const Fp2& o) const { return c0 == o.c0 && c1 == o.c1; }
  __device__ __forceinline__ bool operator!=(const Fp2& o) const { return !(*this == o); }
};

__device__ __forceinline__ Fp2 f_add(const Fp2& a, const Fp2& b) { return {f_add(a.c0, b.c0), f_add(a.c1, b.c1)}; }
__device__ __forceinline__ Fp2 f_sub(const Fp2& a, const Fp2& b) { return {f_sub(a.c0, b.c0), f_sub(a.c1, b.c1)}; }
__device__ __forceinline__ Fp2 f_neg(const Fp2& a) { return {f_neg(a.c0), f_neg(a.c1)}; }
__device__ __forceinline__ Fp2 f_dbl(const Fp2& a) { return {f_dbl(a.c0), f_dbl(a.c1)}; }

// Products of Fp2 with lazy reduction: (a0 + a1 i)(b0 + b1 i) takes the three whole products
// a0 b0, a1 b1 and (a0 + a1)(b0 + b1) (Karatsuba; the sums stay unreduced, below 2^255),
// adds and subtracts them at full width and reduces the two coefficients once each: 3 x 64
// + 2 x 72 multiply-adds instead of 3 x 136 (Aranha, Karabina, Longa, Gebotys and Lopez,
// "Faster explicit formulas for computing pairings over ordinary curves", 2011).  Operands
// up to N.  Out of line: G2 formulas call them about ten times each.
namespace eo {
// re = Re(a b), im = Im(a b) at full width: im < 2 N^2; re modulo 2^512, returning 1 if
// negative
__device__ __forceinline__ uint32_t mul2_wide(uint32_t* re, uint32_t* im, const Fp2& a, const Fp2& b) {
  uint32_t t1[16], e[16], o[15], sa[8], sb[8];
  mul_wide(e, o, a.c0.v, b.c0.v);
  merge_wide(re, e, o);
  mul_wide(e, o, a.c1.v, b.c1.v);
  merge_wide(t1, e, o);
  add8(sa, a.c0.v, a.c1.v);
  add8(sb, b.c0.v, b.c1.v);
  mul_wide(e, o, sa, sb);
  merge_wide(im, e, o);
  w_sub(im, re);
  w_sub(im, t1);
  return w_sub(re, t1);
}
// t += N R if neg
__device__ __forceinline__ void fix_neg(uint32_t* t, uint32_t neg) {
  uint32_t h[8], m[8], x[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    m[i] = mod_limb<FpCfg>(i) & (0u - neg);
    x[i] = t[8 + i];
  }
  add8(h, x, m);
#pragma unroll
  for (int i = 0; i < 8; i++) t[8 + i] = h[i];
}
}  // namespace eo

static __device__ __noinline__ Fp2 f_mul(Fp2 a, Fp2 b) {
  uint32_t re[16], im[16];
  const uint32_t neg = eo::mul2_wide(re, im, a, b);
  eo::fix_neg(re, neg);
  return {f_redc_wide<FpCfg>(re), f_redc_wide<FpCfg>(im)};
}

// a b + c d: |Re| < 2 N^2 < N R and Im < 4 N^2 < N R, so one reduction each still holds
static __device__ __noinline__ Fp2 f_mul2(Fp2 a, Fp2 b, Fp2 c, Fp2 d) {
  uint32_t re[16], im[16], r2[16], i2[16];
  eo::mul2_wide(re, im, a, b);
  eo::mul2_wide(r2, i2, c, d);
  eo::w_add(im, i2);
  eo::w_add(re, r2);
  eo::fix_neg(re, re[15] >> 31);
  return {f_redc_wide<FpCfg>(re), f_redc_wide<FpCfg>(im)};
}

// (a0 + a1 i)^2 = (a0 + a1)(a0 - a1) + 2 a0 a1 i, the factors unreduced (below 2N)
static __device__ __noinline__ Fp2 f_sqr(Fp2 a) {
  Fp s, d, t, u;
  const Fp m = Fp::modulus();
  add8(s.v, a.c0.v, a.c1.v);
  sub8(u.v, m.v, a.c1.v);
  add8(d.v, a.c0.v, u.v);
  add8(t.v, a.c0.v, a.c0.v);
  return {f_mulc(s, d), f_mulc(t, a.c1)};
}

__device__ __forceinline__ Fp2 f_inv(const Fp2& a) {
  Fp n = f_add(f_sqr(a.c0), f_sqr(a.c1));
  Fp ni = f_inv(n);
  return {f_mul(a.c0, ni), f_neg(f_mul(a.c1, ni))};
}

__device__ __forceinline__ Fp2 f_to_mont(const Fp2& a) { return {f_to_mont(a.c0), f_to_mont(a.c1)}; }
__device__ __forceinline__ Fp2 f_from_mont(const Fp2& a) { return {f_from_mont(a.c0), f_from_mont(a.c1)}; }

// ------------------------------------------------------------------ memory helpers
template <class F>
__device__ __forceinline__ F ld_field(const F* p) {
  static_assert(sizeof(F) % 16 == 0, "16-byte vector loads");
  F r;
  uint32_t* d = reinterpret_cast<uint32_t*>(&r);
  const uint4* s = reinterpret_cast<const uint4*>(p);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(F) / 16); i++) {
    uint4 q = s[i];
    d[4 * i] = q.x;
    d[4 * i + 1] = q.y;
    d[4 * i + 2] = q.z;
    d[4 * i + 3] = q.w;
  }
  return r;
}

template <class F>
__device__ __forceinline__ void st_field(F* p, const F& x) {
  uint4* d = reinterpret_cast<uint4*>(p);
  const uint32_t* s = reinterpret_cast<const uint32_t*>(&x);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(F) / 16); i++) d[i] = make_uint4(s[4 * i], s[4 * i + 1], s[4 * i + 2], s[4 * i + 3]);
}

}  // namespace zkvc
