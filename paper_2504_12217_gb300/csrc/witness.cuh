// Device bodies of the witness, CRPC and proof-encoding steps, shared by the one-proof
// prover and the batched prover (each kernel there maps its blocks to these bodies).
//
// CRPC (zkVC Sec. III-A): with z drawn at setup, the matmul Y = X W is proven through
// the n row constraints a_k b_k = c_k, where a_k = sum_i z^(ib) x_ik and
// b_k = sum_j z^j w_kj, and Y(z) = sum_(i,j) z^(ib + j) y_ij.  PSQ (Sec. III-B) chains
// the products through prefix sums S_k = S_(k-1) + c_k, closing S_(n-2) + c_(n-1) = Y(z).
#pragma once
#include "curve.cuh"

namespace zkvc {

// Sums of small integers times field elements stay whole numbers until the end: a 320-bit
// two's complement accumulator takes z |x| (8 multiply-adds) added or subtracted, the block's
// accumulators are summed as they are, and one reduction per row follows.  (2^254 x 2^31 x
// 2^32 terms stay below 2^318.)  What bounds it: the reads of the z powers from L2, shared by
// the ROWS rows of a block.  Measured for the 64-proof batch: a_k and b_k 179 us, Y(z)
// 52 (1,143 and 235 with two Montgomery products per entry and a tree of field additions);
// one [197,768] x [768,3072] proof 27 and 12 (94 and 38).
struct Wide {
  uint32_t v[10];
};
__device__ __forceinline__ Wide wide_zero() {
  Wide w;
#pragma unroll
  for (int i = 0; i < 10; i++) w.v[i] = 0;
  return w;
}
// w += (x ^ m) + (m & 1), m = 0 or all ones: w + x or w - x
__device__ __forceinline__ void wide_add(Wide& w, const uint32_t (&x)[10], uint32_t m) {
  asm("{\n\t.reg .u32 c;\n\tadd.cc.u32 c, %20, 0xffffffff;\n\t"
      "addc.cc.u32 %0, %0, %10;\n\taddc.cc.u32 %1, %1, %11;\n\taddc.cc.u32 %2, %2, %12;\n\t"
      "addc.cc.u32 %3, %3, %13;\n\taddc.cc.u32 %4, %4, %14;\n\taddc.cc.u32 %5, %5, %15;\n\t"
      "addc.cc.u32 %6, %6, %16;\n\taddc.cc.u32 %7, %7, %17;\n\taddc.cc.u32 %8, %8, %18;\n\taddc.u32 %9, %9, %19;\n\t}"
      : "+r"(w.v[0]), "+r"(w.v[1]), "+r"(w.v[2]), "+r"(w.v[3]), "+r"(w.v[4]), "+r"(w.v[5]), "+r"(w.v[6]), "+r"(w.v[7]),
        "+r"(w.v[8]), "+r"(w.v[9])
      : "r"(x[0] ^ m), "r"(x[1] ^ m), "r"(x[2] ^ m), "r"(x[3] ^ m), "r"(x[4] ^ m), "r"(x[5] ^ m), "r"(x[6] ^ m),
        "r"(x[7] ^ m), "r"(x[8] ^ m), "r"(x[9] ^ m), "r"(m & 1u));
}
// w += z x
__device__ __forceinline__ void wide_mac(Wide& w, const Fr& z, int32_t x) {
  const uint32_t mag = x < 0 ? 0u - (uint32_t)x : (uint32_t)x;
  uint32_t e[8], o[8], t[10];
  eo::mul4(e, z.v, 0, mag);
  eo::mul4(o, z.v, 1, mag);
  t[0] = e[0];
  asm("add.cc.u32  %0, %8,  %15;\n\taddc.cc.u32 %1, %9,  %16;\n\taddc.cc.u32 %2, %10, %17;\n\t"
      "addc.cc.u32 %3, %11, %18;\n\taddc.cc.u32 %4, %12, %19;\n\taddc.cc.u32 %5, %13, %20;\n\t"
      "addc.cc.u32 %6, %14, %21;\n\taddc.u32 %7, %22, 0;"
      : "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]), "=&r"(t[6]), "=&r"(t[7]), "=&r"(t[8])
      : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(o[0]), "r"(o[1]), "r"(o[2]),
        "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]));
  t[9] = 0;
  wide_add(w, t, x < 0 ? 0xffffffffu : 0u);
}
__device__ __forceinline__ Wide wide_shfl_down(const Wide& w, int d) {
  Wide r;
#pragma unroll
  for (int i = 0; i < 10; i++) r.v[i] = __shfl_down_sync(0xffffffffu, w.v[i], d);
  return r;
}
// w mod N (w a whole number in two's complement; Montgomery forms stay what they are)
__device__ __forceinline__ Fr wide_mod(const Wide& w) {
  const bool neg = (w.v[9] >> 31) != 0;
  Wide a = wide_zero();
  wide_add(a, w.v, neg ? 0xffffffffu : 0u);
  const uint32_t lo[9] = {a.v[0], a.v[1], a.v[2], a.v[3], a.v[4], a.v[5], a.v[6], a.v[7], 0};
  Fr hi = Fr::zero();  // the words above 2^256 = R: hi R
  hi.v[0] = a.v[8];
  hi.v[1] = a.v[9];
  const Fr r = f_add(f_mod9<FrCfg>(lo), f_to_mont(hi));
  return neg ? f_neg(r) : r;
}

constexpr int CRPC_ROWS = 4;  // rows of W per block: one load of a z power serves them all

// Sums of CRPC_ROWS accumulators over a block of 256 threads, the row r's in lane r of warp
// 0 (others: zero); sh: 8 x CRPC_ROWS accumulators.
template <int ROWS>
__device__ __forceinline__ Wide block_sums(Wide (&w)[ROWS], Wide* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int r = 0; r < ROWS; r++) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) wide_add(w[r], wide_shfl_down(w[r], d).v, 0);
    if (lane == 0) sh[wid * ROWS + r] = w[r];
  }
  __syncthreads();
  Wide s = wide_zero();
  if (wid == 0 && lane < ROWS)
    for (int i = 0; i < 8; i++) wide_add(s, sh[i * ROWS + lane].v, 0);
  __syncthreads();
  return s;
}

// Block body for the rows k0 .. k0 + CRPC_ROWS - 1 below n: a_k and b_k (256 threads).
__device__ __forceinline__ void crpc_ab_rows(const int8_t* __restrict__ X, const int8_t* __restrict__ W,
                                             const Fr* __restrict__ zA, const Fr* __restrict__ zB, int a, int n, int b,
                                             int k0, Fr* ak, Fr* bk, Wide* sh) {
  Wide s[CRPC_ROWS];
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < CRPC_ROWS; r++) s[r] = wide_zero();
  for (int i = threadIdx.x; i < a; i += blockDim.x) {
    const Fr z = ld_field(zA + i);
#pragma unroll
    for (int r = 0; r < CRPC_ROWS; r++) wide_mac(s[r], z, k0 + r < n ? X[size_t(i) * n + k0 + r] : 0);
  }
  Wide t = block_sums(s, sh);
  if (threadIdx.x < CRPC_ROWS && k0 + lane < n) st_field(ak + k0 + lane, wide_mod(t));
#pragma unroll
  for (int r = 0; r < CRPC_ROWS; r++) s[r] = wide_zero();
  for (int j = threadIdx.x; j < b; j += blockDim.x) {
    const Fr z = ld_field(zB + j);
#pragma unroll
    for (int r = 0; r < CRPC_ROWS; r++) wide_mac(s[r], z, k0 + r < n ? W[size_t(k0 + r) * b + j] : 0);
  }
  t = block_sums(s, sh);
  if (threadIdx.x < CRPC_ROWS && k0 + lane < n) st_field(bk + k0 + lane, wide_mod(t));
}

// Block body for row i < a of Y: z^(ib) sum_j z^j y_ij (256 threads).
__device__ __forceinline__ void crpc_y_row(const int32_t* __restrict__ Y, const Fr* __restrict__ zA,
                                           const Fr* __restrict__ zB, int b, int i, Fr* part, Wide* sh) {
  Wide s[1] = {wide_zero()};
  for (int j = threadIdx.x; j < b; j += blockDim.x) wide_mac(s[0], ld_field(zB + j), Y[size_t(i) * b + j]);
  const Wide t = block_sums(s, sh);
  if (threadIdx.x == 0) st_field(part + i, f_mul(wide_mod(t), ld_field(zA + i)));
}

// Block body (1024 threads, sh of 1024 entries): c_k = a_k b_k, the prefix sums
// S_k = c_0 + ... + c_k for k <= n - 2, the closing check against Y(z) (flag bit 1), and
// the first n domain evaluations A_ev = a, B_ev = b, C_ev = c.
// Fr value of lane src (shuffle of the eight words); every lane of the warp calls it
__device__ __forceinline__ Fr fr_shfl_up(const Fr& x, int d) {
  Fr r;
#pragma unroll
  for (int i = 0; i < 8; i++) r.v[i] = __shfl_up_sync(0xffffffffu, x.v[i], d);
  return r;
}
__device__ __forceinline__ Fr fr_shfl_down(const Fr& x, int d) {
  Fr r;
#pragma unroll
  for (int i = 0; i < 8; i++) r.v[i] = __shfl_down_sync(0xffffffffu, x.v[i], d);
  return r;
}

// Inclusive scan of Fr sums over a warp (five shuffle rounds); every lane calls it.
__device__ __forceinline__ Fr warp_scan_fr(Fr v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const Fr u = fr_shfl_up(v, d);
    if (lane >= d) v = f_add(v, u);
  }
  return v;
}

__device__ __forceinline__ void psq_chain(const Fr* __restrict__ ak, const Fr* __restrict__ bk,
                                          const Fr* __restrict__ ypart, int a, int n, Fr* S, Fr* Aev, Fr* Bev, Fr* Cev,
                                          int* flags, Fr* sh) {
  const int T = blockDim.x;
  const int per = (n + T - 1) / T;
  const int k0 = threadIdx.x * per;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Fr local = Fr::zero();
  for (int k = k0; k < k0 + per && k < n; k++) {
    Fr a_ = ld_field(ak + k), b_ = ld_field(bk + k);
    Fr c = f_mul(a_, b_);
    st_field(Aev + k, a_);
    st_field(Bev + k, b_);
    st_field(Cev + k, c);
    local = f_add(local, c);
  }
  // inclusive scan of the per-thread sums: within each warp by shuffles, then over the
  // warps' totals by warp 0
  const Fr incl = warp_scan_fr(local);
  if (lane == 31) st_field(sh + wid, incl);
  __syncthreads();
  if (wid == 0) {
    Fr t = lane < T / 32 ? ld_field(sh + lane) : Fr::zero();
    t = warp_scan_fr(t);
    st_field(sh + 32 + lane, t);  // inclusive totals of warps 0 .. lane
  }
  __syncthreads();
  Fr run = f_sub(incl, local);  // this thread's exclusive prefix within its warp
  if (wid) run = f_add(run, ld_field(sh + 32 + wid - 1));
  for (int k = k0; k < k0 + per && k < n; k++) {
    run = f_add(run, ld_field(Cev + k));  // c_k as this thread stored it above
    if (k < n - 1) st_field(S + k, run);
  }
  // closing check against Y(z) = sum_i ypart_i (warp 1: strided sums, then a shuffle tree)
  if (wid == (T > 32 ? 1 : 0)) {
    Fr yz = Fr::zero();
    for (int i = lane; i < a; i += 32) yz = f_add(yz, ld_field(ypart + i));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) yz = f_add(yz, fr_shfl_down(yz, d));
    if (lane == 0) {
      const Fr total = ld_field(sh + 32 + (T / 32) - 1);  // S_(n-2) + c_(n-1)
      if (total != yz) atomicOr(flags, 1);
    }
  }
}

// Domain row k >= n: A_ev[n + v] = w_v for v = 0 .. l (one, X, Y), zeros elsewhere
// (the input-consistency rows).
__device__ __forceinline__ void domain_rest_row(const int8_t* __restrict__ X, const int32_t* __restrict__ Y, int n,
                                                uint32_t an, uint32_t l, size_t k, Fr* Aev, Fr* Bev, Fr* Cev) {
  size_t v = k - n;
  Fr w = Fr::zero();
  if (v == 0)
    w = Fr::one();
  else if (v <= an)
    w = f_from_int<FrCfg>(X[v - 1]);
  else if (v <= l)
    w = f_from_int<FrCfg>(Y[v - 1 - an]);
  st_field(Aev + k, w);
  st_field(Bev + k, Fr::zero());
  st_field(Cev + k, Fr::zero());
}

__device__ __forceinline__ bool canonical_fr(const Fr& x) {
  for (int i = 7; i >= 0; i--) {
    uint32_t m = mod_limb<FrCfg>(i);
    if (x.v[i] != m) return x.v[i] < m;
  }
  return false;
}

__device__ __forceinline__ void write_canon(uint8_t* out, const Fp& x) {
  Fp c = f_from_mont(x);
  for (int i = 0; i < 8; i++) {
    out[4 * i] = (uint8_t)c.v[i];
    out[4 * i + 1] = (uint8_t)(c.v[i] >> 8);
    out[4 * i + 2] = (uint8_t)(c.v[i] >> 16);
    out[4 * i + 3] = (uint8_t)(c.v[i] >> 24);
  }
}

__device__ __forceinline__ G1A g1_affine_with(const G1J& p, const Fp& inv_zz_zzz) {
  if (p.is_inf()) return G1A::inf();
  return {f_mul(p.X, f_mul(inv_zz_zzz, p.ZZZ)), f_mul(p.Y, f_mul(inv_zz_zzz, p.ZZ))};
}

// Canonical affine encoding of one G1 point (64 bytes: x, y; infinity as zeros); one thread.
__device__ __forceinline__ void encode_g1(const G1J& P, uint8_t* out) {
  const Fp inv = P.is_inf() ? Fp::one() : f_inv(f_mul(P.ZZ, P.ZZZ));
  const G1A q = g1_affine_with(P, inv);
  write_canon(out, q.x);
  write_canon(out + 32, q.y);
}

// Canonical encodings of A (bytes 0..63) and C (192..255) with one shared inversion
// (Montgomery's trick); one thread.
__device__ __forceinline__ void encode_a_c(const G1J& A, const G1J& C, uint8_t* proof) {
  Fp za = A.is_inf() ? Fp::one() : f_mul(A.ZZ, A.ZZZ);
  Fp zc = C.is_inf() ? Fp::one() : f_mul(C.ZZ, C.ZZZ);
  Fp inv = f_inv(f_mul(za, zc));
  G1A a = g1_affine_with(A, f_mul(inv, zc));
  G1A c = g1_affine_with(C, f_mul(inv, za));
  write_canon(proof + 0, a.x);
  write_canon(proof + 32, a.y);
  write_canon(proof + 192, c.x);
  write_canon(proof + 224, c.y);
}

// Canonical encoding of B (bytes 64..191: x.c0, x.c1, y.c0, y.c1); one thread.
__device__ __forceinline__ void encode_b(const G2J& B, uint8_t* proof) {
  G2A q = p_to_affine(B);
  write_canon(proof + 64, q.x.c0);
  write_canon(proof + 96, q.x.c1);
  write_canon(proof + 128, q.y.c0);
  write_canon(proof + 160, q.y.c1);
}

}  // namespace zkvc
