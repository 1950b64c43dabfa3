// Optimal ate pairing over BN254 on the GPU, for Groth16 verification (zkVC Sec. II:
// Verify checks e(A, B) = e(alpha, beta) e(IC(x), gamma) e(C, delta)), by one block per
// pairing or proof.
//
// Tower: Fp6 = Fp2[v]/(v^3 - xi), Fp12 = Fp6[w]/(w^2 - v), xi = 9 + i, so w^6 = xi and an
// element is sum_m c_m w^m (c_m in Fp2, m = 2j + k for the coefficient j of v in part k).
// G2 lives on the D-type twist y^2 = x^3 + b', b' = 3/xi; psi(x, y) = (x w^2, y w^3) maps it
// into E(Fp12).
//
// What bounds it: latency.  A pairing is about 450 products of Fp12 one after another, and
// a verifier's queue is a few dozen proofs, so a thread per pairing leaves the GPU idle.
// Here the 36 Fp2 products of an Fp12 product run side by side: three warps, 12 results
// (6 coefficients x 2 parts) of six lanes, each lane one coefficient product's real or
// imaginary part as a sum of two Fp products with one reduction (f_mul2).  A fourth warp
// runs the point arithmetic of the Miller loop a step ahead, one lane per part of a
// product.  Measured for 32 proofs (128 Miller loops, 32 final exponentiations): Miller
// loops 16.5 -> 0.32 ms, final exponentiations 18.6 -> 0.33, the subgroup test (a 254-bit
// multiplication per proof before) 6.2 -> 0.
//
// Miller loop f_(6u+2, Q)(P) over the signed digits of 6u + 2 (66 digits, 22 nonzero), T in
// homogeneous projective coordinates (Aranha, Karabina, Longa, Gebotys and Lopez, "Faster
// explicit formulas for computing pairings over ordinary curves", 2011).  The tangent / chord
// through T (and Q) evaluated at P is l = yP - lambda xP w + (lambda xR - yR) w^3 for a point
// R on the line; each line is used scaled by a factor in Fp2 (2 Y Z for doublings, X - xQ Z
// for additions), which the final exponentiation removes, as it does the vertical lines that
// negative digits leave out.  Two closing additions with pi(Q) and -pi^2(Q) (Frobenius on
// the twist) complete the optimal ate loop; 6u + 2 > 0 for this curve, so no final conjugation.
//
// Final exponentiation f^((p^12 - 1)/r): the easy part f^((p^6 - 1)(p^2 + 1)) with one
// inversion and a Frobenius, then the hard part (p^4 - p^2 + 1)/r = p^3 + l2 p^2 + l1 p + l0
// with l2 = 6u^2 + 1, l1 = -36u^3 - 18u^2 - 12u + 1, l0 = -36u^3 - 30u^2 - 18u - 2 (an
// identity in u checked by the tests), through three exponentiations by u; in the
// cyclotomic subgroup an inverse is a conjugation.  The result is exactly the pairing
// value, not a power of it.
#pragma once
#include "fp2_rounds.cuh"

namespace zkvc {

static constexpr uint64_t BN_U = 4965661367192848881ull;  // the curve parameter u

__device__ __forceinline__ Fp2 f2_conj(const Fp2& a) { return {a.c0, f_neg(a.c1)}; }

// an element of Fp12: c[2 m + part] the real or imaginary part of the coefficient of w^m
struct alignas(16) E12 {
  Fp c[12];
};

// Frobenius constants gam[k][m] = xi^(m (p^k - 1) / 6) for k = 1, 2, 3 and m < 6 (index
// k-1), and the twist's b' and 3 b'
struct FrobTab {
  Fp2 g[3][6];
  Fp2 b, b3;
};

// signed digits (non-adjacent form) of a positive number, least significant first
struct Naf {
  int8_t d[72];
  int n;
};
constexpr Naf naf_digits(uint64_t lo, bool bit64) {
  Naf r{};
  // the number as lo + 2^64 bit64: halve, taking out +-1 where odd
  uint64_t x = lo;
  uint64_t top = bit64 ? 1 : 0;
  while (x || top) {
    int8_t z = 0;
    if (x & 1) {
      z = (x & 3) == 3 ? -1 : 1;
      if (z == 1) {
        x -= 1;
      } else {
        x += 1;
        if (x == 0) top += 1;
      }
    }
    r.d[r.n++] = z;
    x = (x >> 1) | (top << 63);
    top >>= 1;
  }
  return r;
}
// 6u + 2 has 65 bits: the low 64 wrap, bit 64 is set
__device__ constexpr Naf ATE_NAF = naf_digits(6ull * BN_U + 2ull, true);
__device__ constexpr Naf U_NAF = naf_digits(BN_U, false);

// ------------------------------------------------------------------ Fp12 on three warps
constexpr int PAIR_F = 96;   // threads of the Fp12 arithmetic
constexpr int PAIR_BT = 128;  // and a warp of point arithmetic in the Miller loop

__device__ __forceinline__ void f12_bar() { asm volatile("bar.sync 1, 96;" ::: "memory"); }

// t += x over nine limbs
__device__ __forceinline__ void add9(uint32_t (&t)[9], const uint32_t (&x)[9]) {
  asm("add.cc.u32  %0, %0, %9;\n\taddc.cc.u32 %1, %1, %10;\n\taddc.cc.u32 %2, %2, %11;\n\t"
      "addc.cc.u32 %3, %3, %12;\n\taddc.cc.u32 %4, %4, %13;\n\taddc.cc.u32 %5, %5, %14;\n\t"
      "addc.cc.u32 %6, %6, %15;\n\taddc.cc.u32 %7, %7, %16;\n\taddc.u32 %8, %8, %17;"
      : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]), "+r"(t[8])
      : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]), "r"(x[8]));
}

// dst = a b on threads 0 .. 95 (dst may be a or b).  Lane 6 g + i of warp w (g < 4, i < 6)
// computes part g & 1 of a_i b_(m-i), m = 2 w + (g >> 1), b's index modulo 6; the terms that
// wrap (i > m) carry w^6 = xi: xi (x + y i) = (9 x - y) + (x + 9 y) i.  The six lanes' values
// (each below 10 N) are summed unreduced.
static __device__ __noinline__ void f12_mul(E12* dst, const E12* a, const E12* b) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = lane < 24 ? lane / 6 : 3, i = lane < 24 ? lane % 6 : 5;
  const int m = 2 * w + (g >> 1), part = g & 1;
  const bool wrap = i > m;
  const int j = wrap ? m - i + 6 : m - i;
  const Fp a0 = ld_field(&a->c[2 * i]), a1 = ld_field(&a->c[2 * i + 1]);
  const Fp b0 = ld_field(&b->c[2 * j + part]), b1 = ld_field(&b->c[2 * j + 1 - part]);
  // part 0: a0 b.re + (N - a1) b.im; part 1: a0 b.im + a1 b.re
  Fp n1 = f_comp(a1);
#pragma unroll
  for (int l = 0; l < 8; l++) n1.v[l] = part ? a1.v[l] : n1.v[l];
  const Fp v = f_mul2(a0, b0, n1, b1);
  // the other part of the same product
  Fp o;
  const int mate = part ? lane - 6 : lane + 6;
#pragma unroll
  for (int l = 0; l < 8; l++) o.v[l] = __shfl_sync(0xffffffffu, v.v[l], mate & 31);
  uint32_t t[9];
  {
    // wrapped: 9 v + (part ? o : N - o)
    const Fp co = f_comp(o);
    const uint32_t k = wrap ? 9u : 1u;
    uint64_t c = 0;
#pragma unroll
    for (int l = 0; l < 8; l++) {
      c += (uint64_t)k * v.v[l] + (wrap ? (part ? o.v[l] : co.v[l]) : 0u);
      t[l] = (uint32_t)c;
      c >>= 32;
    }
    t[8] = (uint32_t)c;
  }
  uint32_t x[9], y[9];
#pragma unroll
  for (int l = 0; l < 9; l++) x[l] = __shfl_sync(0xffffffffu, t[l], (lane + 3) & 31);
  add9(t, x);  // i < 3: terms i and i + 3
#pragma unroll
  for (int l = 0; l < 9; l++) {
    x[l] = __shfl_sync(0xffffffffu, t[l], (lane + 1) & 31);
    y[l] = __shfl_sync(0xffffffffu, t[l], (lane + 2) & 31);
  }
  add9(x, y);
  add9(t, x);
  const Fp r = f_mod9<FpCfg>(t);
  f12_bar();  // every operand has been read
  if (lane < 24 && i == 0) st_field(&dst->c[2 * m + part], r);
  f12_bar();
}

__device__ __forceinline__ void f12_set_one(E12* dst) {  // threads 0 .. 11 of the caller
  if (threadIdx.x < 12) st_field(&dst->c[threadIdx.x], threadIdx.x == 0 ? Fp::one() : Fp::zero());
}
__device__ __forceinline__ void f12_copy(E12* dst, const E12* a) {
  if (threadIdx.x < 12) st_field(&dst->c[threadIdx.x], ld_field(&a->c[threadIdx.x]));
  f12_bar();
}
// a -> conj(a): the odd powers of w change sign (f^(p^6))
__device__ __forceinline__ void f12_conj(E12* dst, const E12* a) {
  if (threadIdx.x < 12) {
    const Fp x = ld_field(&a->c[threadIdx.x]);
    st_field(&dst->c[threadIdx.x], (threadIdx.x >> 1) & 1 ? f_neg(x) : x);
  }
  f12_bar();
}
// f^(p^k): c_m -> c_m^(p^k) gam[k][m] with c^(p^k) = conj(c) for odd k
static __device__ __noinline__ void f12_frob(E12* dst, const E12* a, const FrobTab* T, int k) {
  const int t = threadIdx.x;
  Fp r = Fp::zero();
  if (t < 12) {
    const int m = t >> 1, part = t & 1;
    const Fp x = ld_field(&a->c[2 * m]);
    Fp y = ld_field(&a->c[2 * m + 1]);
    if (k & 1) y = f_neg(y);
    const Fp2 g = ld_field(&T->g[k - 1][m]);
    r = part ? f_mul2(x, g.c1, y, g.c0) : f_mul2(x, g.c0, f_comp(y), g.c1);
  }
  f12_bar();
  if (t < 12) st_field(&dst->c[t], r);
  f12_bar();
}

// ------------------------------------------------------------------ final exponentiation
// r = a^u for a in the cyclotomic subgroup (conj(a) = a^-1 in ac)
static __device__ __noinline__ void f12_pow_u(E12* r, const E12* a, E12* ac) {
  f12_conj(ac, a);
  f12_copy(r, a);
  for (int i = U_NAF.n - 2; i >= 0; i--) {
    f12_mul(r, r, r);
    const int d = U_NAF.d[i];
    if (d) f12_mul(r, r, d > 0 ? a : ac);
  }
}

// f <- f^((p^12 - 1)/r) on threads 0 .. 95; s: scratch
struct alignas(16) FinalScratch {
  E12 t, a, b, c, x, y, z;
};
static __device__ __noinline__ void final_exp(E12* f, FinalScratch* s, const FrobTab* T) {
  // f^-1 = conj(f) g^(p^2) g^(p^4) / n, g = f conj(f) in Fp6 and n = g g^(p^2) g^(p^4) in Fp2
  f12_conj(&s->x, f);
  f12_mul(&s->y, f, &s->x);
  f12_frob(&s->a, &s->y, T, 2);
  f12_frob(&s->b, &s->a, T, 2);
  f12_mul(&s->a, &s->a, &s->b);
  f12_mul(&s->z, &s->y, &s->a);
  if (threadIdx.x == 0) {
    const Fp2 n{ld_field(&s->z.c[0]), ld_field(&s->z.c[1])}, ni = f_inv(n);
    for (int i = 0; i < 12; i++) st_field(&s->z.c[i], i == 0 ? ni.c0 : i == 1 ? ni.c1 : Fp::zero());
  }
  f12_bar();
  f12_mul(&s->a, &s->a, &s->z);
  f12_mul(&s->a, &s->a, &s->x);
  // easy part: t = f^(p^6 - 1) = conj(f) / f, then ^(p^2 + 1)
  f12_mul(&s->x, &s->x, &s->a);
  f12_frob(&s->y, &s->x, T, 2);
  f12_mul(&s->t, &s->x, &s->y);
  // hard part: a = t^u, b = t^(u^2), c = t^(u^3)
  f12_pow_u(&s->a, &s->t, &s->x);
  f12_pow_u(&s->b, &s->a, &s->x);
  f12_pow_u(&s->c, &s->b, &s->x);
  E12 *x = &s->x, *y = &s->y, *z = &s->z, *a = &s->a, *b = &s->b, *c = &s->c, *t = &s->t;
  // c <- c^36
  f12_mul(x, c, c);
  f12_mul(x, x, x);
  f12_mul(x, x, x);
  f12_mul(c, x, c);  // c^9
  f12_mul(c, c, c);
  f12_mul(c, c, c);
  // b: y = b^6, b <- b^18
  f12_mul(x, b, b);
  f12_mul(x, x, b);
  f12_mul(y, x, x);     // b^6
  f12_mul(z, y, y);     // b^12
  f12_mul(b, z, y);     // b^18
  f12_mul(z, b, z);     // b^30
  f12_mul(y, y, t);     // t^l2 = b^6 t
  f12_frob(f, y, T, 2);
  f12_mul(z, z, c);     // c^36 b^30
  f12_mul(b, b, c);     // c^36 b^18
  // a: x = a^12, a <- a^18
  f12_mul(x, a, a);
  f12_mul(a, x, a);     // a^3
  f12_mul(a, a, a);     // a^6
  f12_mul(x, a, a);     // a^12
  f12_mul(a, x, a);     // a^18
  f12_mul(b, b, x);     // c^36 b^18 a^12
  f12_conj(b, b);
  f12_mul(b, b, t);     // t^l1
  f12_frob(b, b, T, 1);
  f12_mul(z, z, a);
  f12_mul(x, t, t);
  f12_mul(z, z, x);     // c^36 b^30 a^18 t^2
  f12_conj(z, z);       // t^l0
  f12_frob(t, t, T, 3);
  f12_mul(f, f, t);
  f12_mul(f, f, b);
  f12_mul(f, f, z);
}

// ------------------------------------------------------------------ Miller loop
// The point warp's variables (fp2_rounds.cuh)
enum MillerVar : uint8_t {
  MV_X, MV_Y, MV_Z, MV_QX, MV_QY, MV_XN, MV_YP, MV_B3,  // T, the point added, (-xP, 0), (yP, 0), 3 b'
  MV_0, MV_1, MV_2, MV_3, MV_4, MV_5, MV_6, MV_7, MV_8, MV_9, MV_L0, MV_L1, MV_L3, MV_COUNT
};
// Doubling: B = Y^2, E = 3 b' Z^2, F = 3 E; X3 = 2 X Y (B - F), Y3 = (B + F)^2 - 12 E^2,
// Z3 = 8 B Y Z (four times the usual coordinates); l0 = 2 Y Z yP, l1 = -3 X^2 xP, l3 = B - E.
static __device__ const RoundOp MILLER_DBL[][ROUND_OPS] = {
    {{MV_0, MV_X, MV_Y, OP_MUL}, {MV_1, MV_Y, MV_Y, OP_MUL}, {MV_2, MV_Z, MV_Z, OP_MUL}, {MV_3, MV_Y, MV_Z, OP_MUL},
     {MV_4, MV_X, MV_X, OP_MUL}},
    {{MV_0, MV_0, MV_0, OP_ADD}, {MV_5, MV_1, MV_1, OP_ADD}, {MV_3, MV_3, MV_3, OP_ADD}, {MV_6, MV_4, MV_4, OP_ADD}},
    {{MV_4, MV_6, MV_4, OP_ADD}, {MV_7, MV_3, MV_3, OP_ADD}},
    {{MV_2, MV_B3, MV_2, OP_MUL}, {MV_L0, MV_3, MV_YP, OP_MUL}, {MV_L1, MV_4, MV_XN, OP_MUL}},
    {{MV_6, MV_2, MV_2, OP_ADD}, {MV_L3, MV_1, MV_2, OP_SUB}},
    {{MV_8, MV_6, MV_2, OP_ADD}},
    {{MV_2, MV_1, MV_8, OP_ADD}, {MV_1, MV_1, MV_8, OP_SUB}, {MV_8, MV_8, MV_8, OP_ADD}},
    {{MV_X, MV_0, MV_1, OP_MUL}, {MV_2, MV_2, MV_2, OP_MUL}, {MV_6, MV_6, MV_8, OP_MUL}, {MV_Z, MV_5, MV_7, OP_MUL}},
    {{MV_Y, MV_2, MV_6, OP_SUB}},
};
// Addition of Q: th = Y - yQ Z, la = X - xQ Z, C = th^2, D = la^2, E = la D, F = Z C,
// G = X D, H = E + F - 2 G; X3 = la H, Y3 = th (G - H) - E Y, Z3 = Z E; l0 = la yP,
// l1 = -th xP, l3 = th xQ - la yQ.
static __device__ const RoundOp MILLER_ADD[][ROUND_OPS] = {
    {{MV_0, MV_QY, MV_Z, OP_MUL}, {MV_1, MV_QX, MV_Z, OP_MUL}},
    {{MV_0, MV_Y, MV_0, OP_SUB}, {MV_1, MV_X, MV_1, OP_SUB}},
    {{MV_2, MV_0, MV_0, OP_MUL}, {MV_3, MV_1, MV_1, OP_MUL}, {MV_4, MV_0, MV_QX, OP_MUL}, {MV_5, MV_1, MV_QY, OP_MUL},
     {MV_L0, MV_1, MV_YP, OP_MUL}},
    {{MV_L3, MV_4, MV_5, OP_SUB}},
    {{MV_4, MV_1, MV_3, OP_MUL}, {MV_5, MV_Z, MV_2, OP_MUL}, {MV_6, MV_X, MV_3, OP_MUL}, {MV_L1, MV_0, MV_XN, OP_MUL}},
    {{MV_7, MV_4, MV_5, OP_ADD}, {MV_8, MV_6, MV_6, OP_ADD}},
    {{MV_7, MV_7, MV_8, OP_SUB}},
    {{MV_8, MV_6, MV_7, OP_SUB}},
    {{MV_X, MV_1, MV_7, OP_MUL}, {MV_2, MV_0, MV_8, OP_MUL}, {MV_3, MV_4, MV_Y, OP_MUL}, {MV_Z, MV_Z, MV_4, OP_MUL}},
    {{MV_Y, MV_2, MV_3, OP_SUB}},
};

struct alignas(16) MillerShared {
  E12 f, line[2];
  Fp2 V[MV_COUNT];
  Fp2 Q[2], nQy;   // Q, -yQ
  Fp2 Q1[2], Q2[2];  // pi(Q), -pi^2(Q)
};

// steps of the loop: for each digit below the top a doubling (0), then +-Q (1, 2) where the
// digit is not zero, then pi(Q) (3) and -pi^2(Q) (4)
struct AteSteps {
  uint8_t k[96];
  int n;
};
constexpr AteSteps ate_steps() {
  AteSteps s{};
  const Naf d = naf_digits(6ull * BN_U + 2ull, true);
  for (int i = d.n - 2; i >= 0; i--) {
    s.k[s.n++] = 0;
    if (d.d[i]) s.k[s.n++] = d.d[i] > 0 ? 1 : 2;
  }
  s.k[s.n++] = 3;
  s.k[s.n++] = 4;
  return s;
}
__device__ constexpr AteSteps ATE_STEPS = ate_steps();

// f_(6u+2, Q)(P) with the two closing additions into sh->f, by a block of PAIR_BT threads; P,
// Q affine (Montgomery), one at infinity: one.  Returns (to every thread of the fourth warp)
// whether [6u + 2]Q + pi(Q) - pi^2(Q) = -pi^3(Q): as pi satisfies X^2 - t X + p on the twist
// and the norm of X^3 - X^2 + X + 6u + 2 modulo that polynomial is r times a number prime to
// the twist's order (checked by the tests), the equation holds exactly for the points of
// order r.  (An addition that meets T = +-Q or O, which no point of order r does, leaves
// Z = 0 for good, and the test fails.)
__device__ __forceinline__ bool miller_loop(MillerShared* sh, const G1A& P, const G2A& Q, const FrobTab* T) {
  const int t = threadIdx.x, warp = t >> 5;
  Fp2* const V = sh->V;
  f12_set_one(&sh->f);
  if (t < 24) st_field(&sh->line[t / 12].c[t % 12], Fp::zero());
  if (P.is_inf() || Q.is_inf()) {
    __syncthreads();
    return true;
  }
  if (t == 96) {
    V[MV_X] = Q.x;
    V[MV_Y] = Q.y;
    V[MV_Z] = Fp2::one();
    V[MV_XN] = {f_neg(P.x), Fp::zero()};
    V[MV_YP] = {P.y, Fp::zero()};
    V[MV_B3] = T->b3;
    sh->Q[0] = Q.x;
    sh->Q[1] = Q.y;
    sh->nQy = f_neg(Q.y);
    // pi(Q) = (conj(x) xi^((p-1)/3), conj(y) xi^((p-1)/2)), pi^2(Q) = (x xi^((p^2-1)/3), y xi^((p^2-1)/2))
    sh->Q1[0] = f_mul(f2_conj(Q.x), T->g[0][2]);
    sh->Q1[1] = f_mul(f2_conj(Q.y), T->g[0][3]);
    sh->Q2[0] = f_mul(Q.x, T->g[1][2]);
    sh->Q2[1] = f_neg(f_mul(Q.y, T->g[1][3]));
  }
  __syncthreads();
  const int n = ATE_STEPS.n;
  for (int s = 0; s <= n; s++) {
    if (warp == 3) {  // the point warp, one step ahead
      if (s < n) {
        const int k = ATE_STEPS.k[s], lane = t & 31;
        if (k) {
          if (lane < 4) {
            const Fp2* const q = k == 3 ? sh->Q1 : k == 4 ? sh->Q2 : sh->Q;
            const Fp2* const y = k == 2 ? &sh->nQy : q + 1;
            const Fp* const src = lane < 2 ? &q->c0 : &y->c0;
            st_field(&V[lane < 2 ? MV_QX : MV_QY].c0 + (lane & 1), ld_field(src + (lane & 1)));
          }
          __syncwarp();
          for (const auto& r : MILLER_ADD) fp2_round(V, r);
        } else {
          for (const auto& r : MILLER_DBL) fp2_round(V, r);
        }
        E12* const L = &sh->line[s & 1];
        if (lane < 6) {  // l0, l1 w, l3 w^3
          const int c = lane >> 1, part = lane & 1;
          st_field(&L->c[(c == 2 ? 6 : 2 * c) + part], ld_field(&V[MV_L0 + c].c0 + part));
        }
      }
    } else if (s > 0) {
      if (s > 1 && ATE_STEPS.k[s - 1] == 0) f12_mul(&sh->f, &sh->f, &sh->f);
      f12_mul(&sh->f, &sh->f, &sh->line[(s - 1) & 1]);
    }
    __syncthreads();
  }
  if (warp != 3) return true;
  // T = -pi^3(Q) = (conj(x) xi^((p^3-1)/3), -conj(y) xi^((p^3-1)/2))?
  if ((t & 31) == 0) {
    V[MV_0] = f_mul(f_mul(f2_conj(Q.x), T->g[2][2]), V[MV_Z]);
    V[MV_1] = f_neg(f_mul(f_mul(f2_conj(Q.y), T->g[2][3]), V[MV_Z]));
  }
  __syncwarp();
  return V[MV_0] == V[MV_X] && V[MV_1] == V[MV_Y] && !V[MV_Z].is_zero();
}

}  // namespace zkvc
