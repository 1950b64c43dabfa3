// Fp2 programs on one warp: variables in shared memory, operations in rounds.
//
// A chain of G2 point operations is bound by the latency of its products, and one thread's
// Fp2 product takes about 2,250 cycles.  Here two lanes share a product, the real part on
// one and the imaginary part on the other, each a sum of two Fp products with a single
// reduction (f_mul2, 1,305 cycles), and up to sixteen independent products run side by side.
// A program is a list of rounds; a round is up to ROUND_OPS operations of one kind, all of
// which read their operands before any stores its result.  A round costs about 1,450 cycles
// for products and 170 for sums.
#pragma once
#include "curve.cuh"

namespace zkvc {

enum : uint8_t { OP_NONE, OP_MUL, OP_ADD, OP_SUB };
struct RoundOp {
  uint8_t dst, a, b, op;
};
constexpr int ROUND_OPS = 5;
using Round = RoundOp[ROUND_OPS];

// one round on the calling warp (every lane calls): lane 2 s + part computes part `part` of
// operation s; rounds are uniform in kind
__device__ __forceinline__ void fp2_round(Fp2* V, const RoundOp* ops) {
  const int lane = threadIdx.x & 31, s = lane >> 1, part = lane & 1;
  const RoundOp o = ops[s < ROUND_OPS ? s : 0];
  const bool mul = ops[0].op == OP_MUL;
  const Fp* const A = &V[o.a].c0;
  const Fp* const B = &V[o.b].c0;
  Fp r;
  if (mul) {
    const Fp a0 = ld_field(A), a1 = ld_field(A + 1), b0 = ld_field(B + part), b1 = ld_field(B + 1 - part);
    Fp n1 = f_comp(a1);
#pragma unroll
    for (int l = 0; l < 8; l++) n1.v[l] = part ? a1.v[l] : n1.v[l];
    r = f_mul2(a0, b0, n1, b1);
  } else {
    const Fp x = ld_field(A + part), y = ld_field(B + part);
    const Fp add = f_add(x, y), sub = f_sub(x, y);
#pragma unroll
    for (int l = 0; l < 8; l++) r.v[l] = o.op == OP_ADD ? add.v[l] : sub.v[l];
  }
  __syncwarp();
  if (s < ROUND_OPS && o.op != OP_NONE) st_field(&V[o.dst].c0 + part, r);
  __syncwarp();
}

// ------------------------------------------------------------------ G2 doublings
// variables of a G2 point in XYZZ coordinates and its doubling's temporaries
enum G2Var : uint8_t { GV_X, GV_Y, GV_ZZ, GV_ZZZ, GV_0, GV_1, GV_2, GV_3, GV_4, GV_5, GV_COUNT };

// dbl-2008-s-1 with U = 2Y, V = U^2, M = X 3X, W = U V, 2S = 2X V, 3S = 3X V: X3 = M^2 - 2S,
// Y3 = M (3S - M^2) - W Y, ZZ3 = V ZZ, ZZZ3 = W ZZZ.  Infinity (ZZ = 0) stays infinity; no
// point has Y = 0 (the curve's order is odd).
static __device__ const RoundOp G2_DBL[][ROUND_OPS] = {
    {{GV_0, GV_Y, GV_Y, OP_ADD}, {GV_1, GV_X, GV_X, OP_ADD}},
    {{GV_2, GV_1, GV_X, OP_ADD}},
    {{GV_3, GV_0, GV_0, OP_MUL}, {GV_4, GV_X, GV_2, OP_MUL}},
    {{GV_0, GV_0, GV_3, OP_MUL}, {GV_5, GV_4, GV_4, OP_MUL}, {GV_1, GV_1, GV_3, OP_MUL}, {GV_2, GV_2, GV_3, OP_MUL},
     {GV_ZZ, GV_3, GV_ZZ, OP_MUL}},
    {{GV_X, GV_5, GV_1, OP_SUB}, {GV_2, GV_2, GV_5, OP_SUB}},
    {{GV_1, GV_4, GV_2, OP_MUL}, {GV_2, GV_0, GV_Y, OP_MUL}, {GV_ZZZ, GV_0, GV_ZZZ, OP_MUL}},
    {{GV_Y, GV_1, GV_2, OP_SUB}},
};

// V's point <- 2^n times it, on the calling warp (about 5,000 cycles per doubling; a quad of
// lanes takes about 10,000).  Infinity stays what it is: a sum of small scalars has nothing
// in its upper windows, and Horner's doublings of nothing were two thirds of its time (16
// points with the scalar 1: 566 us with them)
__device__ __forceinline__ void g2_doublings(Fp2* V, uint32_t n) {
  if (V[GV_ZZ].is_zero()) return;
  for (uint32_t i = 0; i < n; i++)
    for (const auto& r : G2_DBL) fp2_round(V, r);
}

}  // namespace zkvc
