// Radix-2 NTT over Fr for the QAP quotient h(x) (zkVC Sec. II: the R1CS is encoded as a
// QAP by interpolation over the domain H = <omega_N>; the prover divides A B - C by
// t(x) = x^N - 1 through evaluations on the coset gH).
//
// GB300 design: every pass takes k <= 10 consecutive radix-2 stages of one group of 2^k
// elements, staged through shared memory as two planes of 16-byte halves.  A block holds
// G groups whose global indices differ in the low bits, so each global load or store of
// the block touches G consecutive elements (G * 32 contiguous bytes).  N = 2^16 takes
// two passes (two HBM round trips), N = 2^24 three.  Decimation in frequency maps
// natural order to bit-reversed order and decimation in time maps it back, so the prove
// path (INTT -> coset NTT -> pointwise -> coset INTT) never runs a bit-reversal pass:
// the coset shift g^i and 1/N are applied at the bit-reversed store of the inverse
// transforms.  The transform is linear and its twiddles are in plain form, so data in
// either form (Montgomery or not) goes through unconverted.
//
// Each stage reads its twiddles omega^(j 2^s) from a table of its own, so neighbouring
// butterflies read neighbouring entries at every stage (out of one table of N/2, the entries
// of a later stage lie in a line each), and a second table holds their quotients
// floor(omega^e 2^256 / r) (f_mul_const).  The inverse transforms read the same tables:
// omega^-e = -omega^(N/2 - e), the sign taken by exchanging the operands of the butterfly's
// difference.  2^22 coset inverse: Montgomery twiddles from one table 950 us, quotients from
// one table 977, Montgomery twiddles by stages 928, quotients by stages 875; 2^24: 3,769 us
// with Montgomery twiddles by stages, 3,493 with quotients.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "ntt.h"

namespace zkvc {

// first entry of the twiddle table of decimation-in-frequency stage s (2^(L - 1 - s) + 1
// entries omega^(j 2^s), in whole 128-byte lines); s = L: all of them
__host__ __device__ __forceinline__ size_t tw_offset(uint32_t L, uint32_t s) {
  return (size_t(1) << L) - (size_t(1) << (L - s)) + 4 * s;
}
// After them, at 2^t + j: the coset forms g^(2^s) omega^(j 2^s), s = L - 1 - t, of the DIT
// stages t = 1 .. COSET_STAGES - 1; quotients this many entries further on
constexpr uint32_t COSET_STAGES = 4;  // no transform of two passes has a shorter last pass
__host__ __device__ __forceinline__ size_t tw_total(uint32_t L) { return tw_offset(L, L) + (1u << COSET_STAGES); }

struct ScaleTabs {
  const Fr* coset;
  const Fr* g_lo;
  const Fr* gi_lo;
  const Fr* g_hi;
  const Fr* g_hi_n;
  const Fr* gi_hi_n;
  const Fr* consts;
};

__device__ __forceinline__ uint32_t brev_bits(uint32_t x, uint32_t logN) {
  return logN ? (__brev(x) >> (32 - logN)) : 0u;
}

__device__ __forceinline__ Fr scale_factor(const ScaleTabs& t, int mode, uint32_t i) {
  switch (mode) {
    case SC_G: return f_mul(ld_field(t.g_lo + (i & 1023u)), ld_field(t.g_hi + (i >> 10)));
    case SC_NG: return f_mul(ld_field(t.g_lo + (i & 1023u)), ld_field(t.g_hi_n + (i >> 10)));
    case SC_NGI: return f_mul(ld_field(t.gi_lo + (i & 1023u)), ld_field(t.gi_hi_n + (i >> 10)));
    case SC_N: return ld_field(t.consts + 0);
    default: return Fr::one();
  }
}

__device__ __forceinline__ Fr f_pow_u32(Fr base, uint32_t e) {
  Fr r = Fr::one();
  while (e) {
    if (e & 1u) r = f_mul(r, base);
    base = f_sqr(base);
    e >>= 1;
  }
  return r;
}

// consts: [0] N^-1 [1] 1/(g^N - 1) [2] omega [3] omega^-1 [4] g [5] g^-1 [6] g^1024
//         [7] g^-1024 [8] one
__global__ void k_domain_consts(Fr* consts, uint32_t logN) {
  // omega_(2^28) = g^((r - 1) / 2^28), g = 5 (a quadratic non-residue of Fr)
  uint32_t e[8];
  {
    uint32_t m[8];
#pragma unroll
    for (int i = 0; i < 8; i++) m[i] = mod_limb<FrCfg>(i);
    m[0] -= 1;  // r - 1 (r is odd, no borrow)
#pragma unroll
    for (int i = 0; i < 8; i++) e[i] = (m[i] >> 28) | (i < 7 ? (m[i + 1] << 4) : 0u);
  }
  Fr g = f_from_int<FrCfg>(5);
  Fr w = f_pow(g, e);
  for (uint32_t i = logN; i < 28; i++) w = f_sqr(w);
  Fr gN = g;
  for (uint32_t i = 0; i < logN; i++) gN = f_sqr(gN);
  Fr nm = f_from_int<FrCfg>((int32_t)(1u << logN));
  Fr gi = f_inv(g);
  consts[0] = f_inv(nm);
  consts[1] = f_inv(f_sub(gN, Fr::one()));
  consts[2] = w;
  consts[3] = f_inv(w);
  consts[4] = g;
  consts[5] = gi;
  consts[6] = f_pow_u32(g, 1024);
  consts[7] = f_pow_u32(gi, 1024);
  consts[8] = Fr::one();
}

// out[e] = mult * base^e for e < count; each thread fills a run of 16.
__global__ void k_fill_pows(Fr* out, size_t count, const Fr* base_p, const Fr* mult_p) {
  size_t e0 = (size_t(blockIdx.x) * blockDim.x + threadIdx.x) * 16;
  if (e0 >= count) return;
  Fr base = *base_p;
  Fr x = f_mul(*mult_p, f_pow_u32(base, (uint32_t)e0));
  for (size_t e = e0; e < e0 + 16 && e < count; e++) {
    st_field(out + e, x);
    x = f_mul(x, base);
  }
}

// From the Montgomery forms m = w 2^256 mod r of the twiddles in out[0 .. total): the plain w
// there and out[total + e] = floor(w 2^256 / r) = (w 2^256 - m) / r, which is -m / r mod 2^256
// (limb by limb, as in a reduction).
__global__ void k_fill_twiddles(Fr* out, size_t total) {
  const size_t e = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const Fr m = ld_field(out + e);
  st_field(out + e, f_from_mont(m));
  uint32_t t[8];
  Fr q;
#pragma unroll
  for (int i = 0; i < 8; i++) t[i] = m.v[i];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    q.v[i] = t[i] * FrCfg::INV;
    uint64_t c = 0;
#pragma unroll
    for (int j = 0; i + j < 8; j++) {
      c += (uint64_t)q.v[i] * mod_limb<FrCfg>(j) + t[i + j];
      t[i + j] = (uint32_t)c;
      c >>= 32;
    }
  }
  st_field(out + total + e, q);
}

// the tables of the stages s >= 1 (every 2^s-th entry of stage 0's) and the coset forms
__global__ void k_fill_stages(Fr* out, uint32_t L, ScaleTabs tabs) {
  const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;  // 2^(L - 1 - s) + j, j < 2^(L - 1 - s); 0: the last entries
  if (e >= 1u << (L - 1)) return;
  if (e == 0) {
    for (uint32_t s = 1; s < L; s++) st_field(out + tw_offset(L, s) + (1u << (L - 1 - s)), ld_field(out + (1u << (L - 1))));
    for (uint32_t k = 0; k < 1u << COSET_STAGES; k++) {
      const uint32_t t = k < 2 ? 0u : 31 - __clz(k);
      st_field(out + tw_offset(L, L) + k,
               t && t < L ? f_mul(scale_factor(tabs, SC_G, 1u << (L - 1 - t)), ld_field(out + (size_t(k - (1u << t)) << (L - 1 - t))))
                          : Fr::zero());
    }
    return;
  }
  const uint32_t lg = 31 - __clz(e), s = L - 1 - lg, j = e - (1u << lg);
  if (s >= 1) st_field(out + tw_offset(L, s) + j, ld_field(out + (size_t(j) << s)));
}

// The factors left of N^-1 g^i when the DIT's first COSET_STAGES stages run in coset form:
// for position p (natural index i = bit-reversed p) N^-1 g^(i mod N / 16), times g^(N/2) for
// odd p (stage 0's coset factor, so that stage keeps no product); entry 2 (p / 16) + p mod 2.
__global__ void k_fill_coset(Fr* out, uint32_t L, ScaleTabs tabs) {
  const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x, lb = L - COSET_STAGES;
  if (e >= 2u << lb) return;
  const Fr c = scale_factor(tabs, SC_NG, brev_bits(e >> 1, lb));
  st_field(out + e, (e & 1u) ? f_mul(c, scale_factor(tabs, SC_G, 1u << (L - 1))) : c);
}

static int fill_pows(Fr* out, size_t count, const Fr* base, const Fr* mult, cudaStream_t st) {
  size_t runs = (count + 15) / 16;
  unsigned blocks = (unsigned)((runs + 127) / 128);
  k_fill_pows<<<blocks, 128, 0, st>>>(out, count, base, mult); ZK_COUNT_LAUNCH();
  ZK_CUDA(cudaGetLastError());
  return ZKVC_OK;
}

static ScaleTabs tabs_of(const NttDomain* d) {
  return {d->coset, d->g_lo, d->gi_lo, d->g_hi, d->g_hi_n, d->gi_hi_n, d->consts};
}

static std::mutex g_dom_mu;
static std::map<std::pair<int, uint32_t>, NttDomain*> g_domains;

int ntt_domain(uint32_t logN, const NttDomain** out) {
  ZK_CHECK(logN >= 1 && logN <= 28, ZKVC_EINVAL, "ntt: log N = %u outside [1, 28]", logN);
  int dev = 0;
  ZK_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_dom_mu);
  auto it = g_domains.find({dev, logN});
  if (it != g_domains.end()) {
    *out = it->second;
    return ZKVC_OK;
  }
  NttDomain* d = new NttDomain();
  d->logN = logN;
  d->N = size_t(1) << logN;
  size_t half = d->N / 2;
  size_t hi = d->N >= 1024 ? d->N / 1024 : 1;
  cudaStream_t st;
  ZK_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
  ZK_CUDA(cudaMalloc(&d->consts, 16 * sizeof(Fr)));
  const size_t total = tw_total(logN), ncoset = logN > COSET_STAGES ? size_t(2) << (logN - COSET_STAGES) : 0;
  ZK_CUDA(cudaMalloc(&d->tw, 2 * total * sizeof(Fr)));
  if (ncoset) ZK_CUDA(cudaMalloc(&d->coset, 2 * ncoset * sizeof(Fr)));
  ZK_CUDA(cudaMalloc(&d->g_lo, 1024 * sizeof(Fr)));
  ZK_CUDA(cudaMalloc(&d->gi_lo, 1024 * sizeof(Fr)));
  ZK_CUDA(cudaMalloc(&d->g_hi, hi * sizeof(Fr)));
  ZK_CUDA(cudaMalloc(&d->g_hi_n, hi * sizeof(Fr)));
  ZK_CUDA(cudaMalloc(&d->gi_hi_n, hi * sizeof(Fr)));
  k_domain_consts<<<1, 1, 0, st>>>(d->consts, logN); ZK_COUNT_LAUNCH();
  ZK_CUDA(cudaGetLastError());
  const Fr* c = d->consts;
  ZK_TRY(fill_pows(d->tw, half + 1, c + 2, c + 8, st));
  ZK_TRY(fill_pows(d->g_lo, 1024, c + 4, c + 8, st));
  ZK_TRY(fill_pows(d->gi_lo, 1024, c + 5, c + 8, st));
  ZK_TRY(fill_pows(d->g_hi, hi, c + 6, c + 8, st));
  ZK_TRY(fill_pows(d->g_hi_n, hi, c + 6, c + 0, st));
  ZK_TRY(fill_pows(d->gi_hi_n, hi, c + 7, c + 0, st));
  const ScaleTabs tabs = tabs_of(d);
  k_fill_stages<<<(unsigned)((half + 255) / 256), 256, 0, st>>>(d->tw, logN, tabs); ZK_COUNT_LAUNCH();
  k_fill_twiddles<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(d->tw, total); ZK_COUNT_LAUNCH();
  if (ncoset) {
    k_fill_coset<<<(unsigned)((ncoset + 255) / 256), 256, 0, st>>>(d->coset, logN, tabs); ZK_COUNT_LAUNCH();
    k_fill_twiddles<<<(unsigned)((ncoset + 255) / 256), 256, 0, st>>>(d->coset, ncoset); ZK_COUNT_LAUNCH();
  }
  ZK_CUDA(cudaGetLastError());
  ZK_CUDA(cudaStreamSynchronize(st));
  ZK_CUDA(cudaStreamDestroy(st));
  g_domains[{dev, logN}] = d;
  *out = d;
  return ZKVC_OK;
}

// One pass: k consecutive radix-2 stages from stage s0, over G = 2^logG groups of 2^k
// elements per block (E = G 2^k elements, staged in shared memory as two planes of 16-byte
// halves: an element is two vector accesses, and neighbouring elements are conflict-free).
struct PassGeo {
  uint32_t L, s0, k, logG;
};

// global index of the block's e-th staged element (N <= 2^28)
template <bool DIT>
__device__ __forceinline__ uint32_t pass_index(const PassGeo& g, uint32_t gid0, uint32_t e) {
  const uint32_t gg = e & ((1u << g.logG) - 1u), j = e >> g.logG;
  const uint32_t gid = gid0 + gg;
  const uint32_t sbits = DIT ? g.s0 : (g.L - g.s0 - g.k);
  const uint32_t lo = gid & ((1u << sbits) - 1u), hi = gid >> sbits;
  const uint32_t base = DIT ? ((hi << (g.s0 + g.k)) | lo) : ((hi << (g.L - g.s0)) | lo);
  return base + (j << sbits);
}

__device__ __forceinline__ Fr sm_get(const uint4* sm, uint32_t E, uint32_t e) {
  const uint4 a = sm[e], b = sm[E + e];
  return {{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
__device__ __forceinline__ void sm_put(uint4* sm, uint32_t E, uint32_t e, const Fr& x) {
  sm[e] = make_uint4(x.v[0], x.v[1], x.v[2], x.v[3]);
  sm[E + e] = make_uint4(x.v[4], x.v[5], x.v[6], x.v[7]);
}

// What bounds a pass on a large grid: the products, at 0.8 of the multiplier's rate where
// the twiddles stay in L1 (the passes after the first).  Measured at 2^22, passes of 8 + 7 +
// 7 stages: 285 + 228 + 217 us (306 + 257 + 226 with Montgomery products by twiddles from
// one table; 378 + 296 + 293 with eight scalar shared-memory accesses per element, full
// reductions and 64-bit indices before that); the first reads its twiddles from memory, as
// many bytes as the data.
//
// Values stay lazily reduced between loads and stores: below 2N in a decimation-in-frequency
// pass, below 4N in a decimation-in-time pass, so a butterfly's product needs no
// conditional subtraction and its sums one at most.  raw: the input is any 256-bit value.
template <bool DIT>
__device__ __forceinline__ void pass_load(const Fr* arr, const PassGeo& g, uint32_t gid0, uint4* sm, int load_scale,
                                          int raw, const ScaleTabs& tabs) {
  const uint32_t E = 1u << (g.logG + g.k);
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x) {
    const uint32_t idx = pass_index<DIT>(g, gid0, e);
    Fr x = ld_field(arr + idx);
    if (load_scale) {  // (the product reduces a raw value too)
      x = f_mul_lazy(scale_factor(tabs, load_scale, idx), x);
    } else if (raw) {
      const uint32_t t[9] = {x.v[0], x.v[1], x.v[2], x.v[3], x.v[4], x.v[5], x.v[6], x.v[7], 0};
      x = f_mod9<FrCfg>(t);
    }
    sm_put(sm, E, e, x);
  }
}

// last: the transform's last pass, whose values go out below N
template <bool DIT>
__device__ __forceinline__ void pass_store(Fr* arr, const PassGeo& g, uint32_t gid0, const uint4* sm, int store_scale,
                                           bool last, const ScaleTabs& tabs) {
  const uint32_t E = 1u << (g.logG + g.k);
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x) {
    const uint32_t idx = pass_index<DIT>(g, gid0, e);
    Fr x = sm_get(sm, E, e);
    if (store_scale) {
      x = f_mul(scale_factor(tabs, store_scale, brev_bits(idx, g.L)), x);
    } else if (last) {
      if (DIT) x = f_red2(x);
      x = f_once(x);
    }
    st_field(arr + idx, x);
  }
}

// The pass's k stages on NPOLY staged arrays (2 E vectors apart).  Radix 2 (R4 false):
// one stage per shared-memory round trip, one butterfly per element pair.  R4: two stages
// at a time: a radix-4 unit reads four elements, runs their four butterflies of stages t
// and t + 1 in registers (two independent products per stage) and writes them back, so a
// pair of stages costs one round trip and one barrier instead of two; an odd last stage
// runs as radix 2.  Barriers between rounds (the first one orders the loads before it).
//   DIF, stage t of half h (block 2h), then h/2: a unit is j0 = blk 2h + off (off < h/2)
//     and j0 + h/2, j0 + h, j0 + 3h/2; twiddles w_t(off), w_t(off + h/2), w_(t+1)(off).
//   DIT, stage t of half h (block 2h), then 2h: a unit is j0 = blk 4h + off (off < h) and
//     j0 + h, j0 + 2h, j0 + 3h; twiddles w_t(off), w_(t+1)(off), w_(t+1)(off + h).
// w_t(q) is entry (q << sbits) + lo of the table of DIF stage s = s0 + t, in DIT entry
// (q << s0) + lo of that of stage L - 1 - s, lo the group's low index bits; INV (DIF only): minus
// the entry as far from the table's end, so the difference is taken the other way round.  The
// transform's stage of half 1 over neighbouring elements (DIF s = L - 1, DIT s = 0) has
// w = 1 throughout and takes no product.
template <bool DIT, int NPOLY, bool R4, bool INV, bool COSET = false>
__device__ __forceinline__ void pass_stages(uint4* sm, const PassGeo& g, uint32_t gid0, const Fr* tw) {
  const uint32_t G = 1u << g.logG, E = G << g.k, L = g.L, logG = g.logG;
  const uint32_t sbits = DIT ? g.s0 : (L - g.s0 - g.k);
  const uint32_t smask = (1u << sbits) - 1u;
  static_assert(!(DIT && INV), "the forward transforms alone run by decimation in time");
  // the table of stage s and its entry for a butterfly
  auto stage_tab = [&](uint32_t s) -> const Fr* {
    if (COSET && s > 0 && s < COSET_STAGES) return tw + tw_offset(L, L) + (1u << s);
    const uint32_t sd = DIT ? L - 1 - s : s;
    return tw + tw_offset(L, sd) + (INV ? 1u << (L - 1 - sd) : 0u);
  };
  const size_t total = tw_total(L);
  auto entry = [&](const Fr* tab, uint32_t q, uint32_t lo) -> const Fr* {
    const uint32_t p = DIT ? (q << g.s0) + lo : (q << sbits) + lo;
    return INV ? tab - p : tab + p;
  };
  auto mul_tw = [&](const Fr& x, const Fr* tab, uint32_t q, uint32_t lo) -> Fr {
    const Fr* w = entry(tab, q, lo);
    return f_mul_const(x, ld_field(w), ld_field(w + total));
  };
  auto diff = [&](const Fr& x, const Fr& y) -> Fr { return INV ? f_sub2(y, x) : f_sub2(x, y); };
  __syncthreads();
  uint32_t t = 0;
  const uint32_t nq = E >> 2;
  for (; R4 && t + 1 < g.k; t += 2) {
    const uint32_t s = g.s0 + t;
    const Fr *tab0 = stage_tab(s), *tab1 = stage_tab(s + 1);
    for (uint32_t ua = threadIdx.x; ua < nq * (uint32_t)NPOLY; ua += blockDim.x) {
      const uint32_t poly = NPOLY == 1 ? 0u : ua / nq, u = ua - poly * nq;
      uint4* smp = sm + size_t(poly) * 2 * E;
      const uint32_t gg = u & (G - 1), q = u >> logG;
      const uint32_t lo = (gid0 + gg) & smask;
      if (DIT) {
        const uint32_t lh = t, h = 1u << lh;  // stage t: half h; stage t + 1: half 2h
        const uint32_t off = q & (h - 1), j0 = ((q >> lh) << (lh + 2)) + off;
        const uint32_t p0 = (j0 << logG) + gg, p1 = ((j0 + h) << logG) + gg, p2 = ((j0 + 2 * h) << logG) + gg,
                       p3 = ((j0 + 3 * h) << logG) + gg;
        Fr x1 = sm_get(smp, E, p1), x3 = sm_get(smp, E, p3);
        if (s == 0) {
          x1 = f_red2(x1);
          x3 = f_red2(x3);
        } else {
          x1 = mul_tw(x1, tab0, off, lo);
          x3 = mul_tw(x3, tab0, off, lo);
        }
        const Fr x0 = f_red2(sm_get(smp, E, p0)), x2 = f_red2(sm_get(smp, E, p2));
        const Fr vc = mul_tw(f_add_raw(x2, x3), tab1, off, lo);
        const Fr a = f_red2(f_add_raw(x0, x1));
        sm_put(smp, E, p0, f_add_raw(a, vc));
        sm_put(smp, E, p2, f_sub2(a, vc));
        const Fr vd = mul_tw(f_sub2(x2, x3), tab1, off + h, lo);
        const Fr b = f_red2(f_sub2(x0, x1));
        sm_put(smp, E, p1, f_add_raw(b, vd));
        sm_put(smp, E, p3, f_sub2(b, vd));
      } else {
        const uint32_t lh = g.k - 1 - t, h = 1u << lh, hq = h >> 1;  // stage t: half h; t + 1: h/2
        const uint32_t off = q & (hq - 1), j0 = ((q >> (lh - 1)) << (lh + 1)) + off;
        const uint32_t p0 = (j0 << logG) + gg, p1 = ((j0 + hq) << logG) + gg, p2 = ((j0 + h) << logG) + gg,
                       p3 = ((j0 + h + hq) << logG) + gg;
        Fr a, b, c, d;
        {
          const Fr x0 = sm_get(smp, E, p0), x2 = sm_get(smp, E, p2);
          a = f_add2(x0, x2);
          b = mul_tw(diff(x0, x2), tab0, off, lo);
        }
        {
          const Fr x1 = sm_get(smp, E, p1), x3 = sm_get(smp, E, p3);
          c = f_add2(x1, x3);
          d = mul_tw(diff(x1, x3), tab0, off + hq, lo);
        }
        sm_put(smp, E, p0, f_add2(a, c));
        sm_put(smp, E, p2, f_add2(b, d));
        if (s + 1 == L - 1) {
          a = f_red2(f_sub2(a, c));
          b = f_red2(f_sub2(b, d));
        } else {
          a = mul_tw(diff(a, c), tab1, off, lo);
          b = mul_tw(diff(b, d), tab1, off, lo);
        }
        sm_put(smp, E, p1, a);
        sm_put(smp, E, p3, b);
      }
    }
    __syncthreads();
  }
  for (; t < g.k; t++) {  // radix 2: every stage, or the last of an odd count
    const uint32_t s = g.s0 + t, nbf = E >> 1;
    const Fr* tab = stage_tab(s);
    const uint32_t logh = DIT ? t : (g.k - 1 - t), h = 1u << logh;
    const bool unit = DIT ? s == 0 : s == L - 1;
    auto place = [&](uint32_t bf, uint32_t& pu, uint32_t& pv, uint32_t& qh, uint32_t& lo) {
      const uint32_t gg = bf & (G - 1), q = bf >> logG;
      qh = q & (h - 1);
      const uint32_t ju = ((q >> logh) << (logh + 1)) + qh;
      pu = (ju << logG) + gg;
      pv = ((ju + h) << logG) + gg;
      lo = (gid0 + gg) & smask;
    };
    auto butterfly = [&](uint4* smp, uint32_t pu, uint32_t pv, auto&& mul) {
      const Fr v = sm_get(smp, E, pv);
      if (DIT) {
        const Fr y = unit ? f_red2(v) : mul(v), x = f_red2(sm_get(smp, E, pu));
        sm_put(smp, E, pu, f_add_raw(x, y));
        sm_put(smp, E, pv, f_sub2(x, y));
      } else {
        const Fr u = sm_get(smp, E, pu);
        sm_put(smp, E, pu, f_add2(u, v));
        sm_put(smp, E, pv, unit ? f_red2(f_sub2(u, v)) : mul(diff(u, v)));
      }
    };
    if (NPOLY > 1 && !R4) {
      // a thread takes a butterfly's place in each array, for one read of its twiddle
      // (quotient turns of a 64-proof batch: 4,976 us with the arrays side by side, 4,716 so)
      for (uint32_t bf = threadIdx.x; bf < nbf; bf += blockDim.x) {
        uint32_t pu, pv, qh, lo;
        place(bf, pu, pv, qh, lo);
        const Fr* w = entry(tab, qh, lo);
        const Fr w0 = ld_field(w), w1 = ld_field(w + total);
#pragma unroll 1
        for (uint32_t p = 0; p < NPOLY; p++)
          butterfly(sm + size_t(p) * 2 * E, pu, pv, [&](const Fr& x) { return f_mul_const(x, w0, w1); });
      }
    } else {
      for (uint32_t bfa = threadIdx.x; bfa < nbf * (uint32_t)NPOLY; bfa += blockDim.x) {
        const uint32_t poly = NPOLY == 1 ? 0u : bfa / nbf;
        uint32_t pu, pv, qh, lo;
        place(bfa - poly * nbf, pu, pv, qh, lo);
        butterfly(sm + size_t(poly) * 2 * E, pu, pv, [&](const Fr& x) { return mul_tw(x, tab, qh, lo); });
      }
    }
    __syncthreads();
  }
}

// Resident blocks the registers are cut to: radix 2 at 64 registers (32 warps per SM, the
// large grids), radix 4 at 128 (the small ones, which have fewer blocks than that).
template <bool R4>
constexpr int pass_min_blocks() { return R4 ? 2 : 4; }

// One pass of k stages over G groups per block; see the file comment.
template <bool DIT, bool R4, bool INV>
__global__ void __launch_bounds__(256, pass_min_blocks<R4>())
    k_ntt_pass(Fr* data, size_t bstride, const Fr* __restrict__ tw, uint32_t logN, uint32_t s0, uint32_t k,
               uint32_t logG, int load_scale, int store_scale, int raw, ScaleTabs tabs) {
  extern __shared__ uint4 sm[];
  const PassGeo g{logN, s0, k, logG};
  Fr* arr = data + size_t(blockIdx.y) * bstride;
  const uint32_t gid0 = blockIdx.x << logG;
  pass_load<DIT>(arr, g, gid0, sm, load_scale, raw, tabs);
  pass_stages<DIT, 1, R4, INV>(sm, g, gid0, tw);
  pass_store<DIT>(arr, g, gid0, sm, store_scale, s0 + k == logN, tabs);
}

// The turn of an inverse DIF transform into a forward DIT transform, in one pass: the
// DIF's last pass (its k stages end at stage L - 1, groups of 2^k consecutive elements),
// the inverse's scaling by N^-1 and the coset's powers g^i, and the DIT's first pass over the
// same groups.  Saves a global round trip and a launch.  Most of g^i goes into the twiddles of
// the DIT's first stages (k_fill_coset), which leaves one product by a constant per element
// out of a table of N / 8 (two Montgomery products before: the turns of a 64-proof batch took
// 5,756 us, 5,172 so).
template <bool R4>
__global__ void __launch_bounds__(256, pass_min_blocks<R4>())
    k_ntt_turn(Fr* data, size_t bstride, const Fr* __restrict__ tw, uint32_t L, uint32_t k,
               uint32_t logG, ScaleTabs tabs) {
  extern __shared__ uint4 sm[];
  const PassGeo gdif{L, L - k, k, logG}, gdit{L, 0, k, logG};
  Fr* arr = data + size_t(blockIdx.y) * bstride;
  const uint32_t gid0 = blockIdx.x << logG;
  const uint32_t E = 1u << (logG + k), ncoset = 2u << (L - COSET_STAGES);
  pass_load<false>(arr, gdif, gid0, sm, SC_NONE, 0, tabs);
  pass_stages<false, 1, R4, true>(sm, gdif, gid0, tw);
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x) {
    const uint32_t idx = pass_index<false>(gdif, gid0, e);
    const Fr* c = tabs.coset + 2 * (idx / (1u << COSET_STAGES)) + (idx & 1u);
    sm_put(sm, E, e, f_mul_const(sm_get(sm, E, e), ld_field(c), ld_field(c + ncoset)));
  }
  pass_stages<true, 1, R4, false, true>(sm, gdit, gid0, tw);
  pass_store<true>(arr, gdit, gid0, sm, SC_NONE, false, tabs);
}

// The quotient turn, one instance per blockIdx.y (arrays A_i, B_i, C_i, H_i of N
// elements at i, m + i, 2m + i, 3m + i): the last DIT pass of A, B and C (strided groups),
// h_ev = (A B - C) / (g^N - 1) on the staged elements, and the first DIF pass of the
// inverse transform of h over the same groups; only H is written.  Its three staged arrays
// leave two blocks per SM: 512 threads of radix 2 on large grids, up to 768 (the three
// forward passes side by side) of radix 4 on small ones.
template <bool R4>
__global__ void __launch_bounds__(R4 ? 768 : 512, R4 ? 1 : 2)
    k_ntt_quotient_turn(Fr* ev, uint32_t m, size_t N, const Fr* __restrict__ tw, uint32_t L, uint32_t k,
                        uint32_t logG, ScaleTabs tabs) {
  extern __shared__ uint4 sm[];
  const PassGeo gdit{L, L - k, k, logG}, gdif{L, 0, k, logG};
  const uint32_t gid0 = blockIdx.x << logG;
  const uint32_t E = 1u << (logG + k);
  const size_t i = blockIdx.y;
  for (int p = 0; p < 3; p++)
    pass_load<true>(ev + (size_t(p) * m + i) * N, gdit, gid0, sm + size_t(p) * 2 * E, SC_NONE, 0, tabs);
  pass_stages<true, 3, R4, false>(sm, gdit, gid0, tw);
  const Fr zinv = ld_field(tabs.consts + 1);
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x) {
    const Fr a = f_red2(sm_get(sm, E, e)), b = f_red2(sm_get(sm + 2 * E, E, e)), c = f_red2(sm_get(sm + 4 * E, E, e));
    sm_put(sm, E, e, f_mul_lazy(f_sub2(f_mul_lazy(a, b), c), zinv));
  }
  pass_stages<false, 1, R4, true>(sm, gdif, gid0, tw);
  pass_store<false>(ev + (size_t(3) * m + i) * N, gdif, gid0, sm, SC_NONE, false, tabs);
}

int ntt_init() {
  static OncePerDevice once;
  constexpr size_t one = 64 << 10, three = 192 << 10;
  return smem_limits(once, {{(const void*)k_ntt_pass<true, false, false>, one},
                            {(const void*)k_ntt_pass<true, true, false>, one},
                            {(const void*)k_ntt_pass<false, false, false>, one},
                            {(const void*)k_ntt_pass<false, true, false>, one},
                            {(const void*)k_ntt_pass<false, false, true>, one},
                            {(const void*)k_ntt_pass<false, true, true>, one},
                            {(const void*)k_ntt_turn<false>, one},
                            {(const void*)k_ntt_turn<true>, one},
                            {(const void*)k_ntt_quotient_turn<false>, three},
                            {(const void*)k_ntt_quotient_turn<true>, three}});
}

// Stage split of an N = 2^L transform into passes of at most min(elog, 10) stages, the
// first passes one stage longer.
static std::vector<uint32_t> pass_split(uint32_t L, int elog) {
  const uint32_t kmax = (uint32_t)elog < 10 ? (uint32_t)elog : 10;
  const uint32_t P = (L + kmax - 1) / kmax;
  const uint32_t kb = L / P, rem = L % P;
  std::vector<uint32_t> ks(P);
  for (uint32_t p = 0; p < P; p++) ks[p] = kb + (p < rem ? 1 : 0);
  return ks;
}

// groups per block (log2) and the block shape of a pass of k stages
struct PassShape {
  uint32_t logG, E, threads;
  dim3 grid;
};
static PassShape pass_shape(uint32_t L, uint32_t k, int elog, int batch) {
  PassShape sh;
  const uint32_t groups_log = L - k;
  sh.logG = (uint32_t)elog - k;
  if (sh.logG > groups_log) sh.logG = groups_log;
  sh.E = 1u << (sh.logG + k);
  sh.threads = sh.E / 2 < 256 ? sh.E / 2 : 256;
  sh.grid = dim3((unsigned)(size_t(1) << (groups_log - sh.logG)), (unsigned)batch);
  return sh;
}

// Radix 4 for grids below four blocks per SM (latency-bound: fewer, longer-lived threads
// with two independent products per stage finish sooner), radix 2 above (throughput:
// twice the resident warps).
static bool radix4(dim3 grid) { return uint64_t(grid.x) * grid.y < 4ull * (uint64_t)device_sm_count(); }

static int launch_pass(bool dit, Fr* data, int batch, size_t bstride, const NttDomain* d, bool inverse, uint32_t s0,
                       uint32_t k, int elog, int ls, int ss, int tm, cudaStream_t st) {
  const uint32_t L = d->logN;
  const PassShape sh = pass_shape(L, k, elog, batch);
  const bool r4 = radix4(sh.grid);
  auto* f = dit ? (r4 ? k_ntt_pass<true, true, false> : k_ntt_pass<true, false, false>)
          : inverse ? (r4 ? k_ntt_pass<false, true, true> : k_ntt_pass<false, false, true>)
                    : (r4 ? k_ntt_pass<false, true, false> : k_ntt_pass<false, false, false>);
  f<<<sh.grid, sh.threads, size_t(sh.E) * 32, st>>>(data, bstride, d->tw, L, s0, k, sh.logG, ls, ss, tm, tabs_of(d));
  ZK_COUNT_LAUNCH();
  ZK_CUDA(cudaGetLastError());
  return ZKVC_OK;
}

static int run_passes(bool dit, Fr* data, int batch, size_t bstride, const NttDomain* d, bool inverse,
                      int load_scale, int store_scale, bool raw, int elog, cudaStream_t st) {
  ZK_CHECK(elog >= 8 && elog <= 11, ZKVC_EINVAL, "ntt: 2^%d elements per block outside [2^8, 2^11]", elog);
  ZK_CHECK(batch >= 1 && batch <= 65535, ZKVC_EINVAL, "ntt: batch of %d arrays", batch);
  ZK_TRY(ntt_init());
  const std::vector<uint32_t> ks = pass_split(d->logN, elog);
  const uint32_t P = (uint32_t)ks.size();
  uint32_t s0 = 0;
  for (uint32_t p = 0; p < P; p++) {
    const bool first = p == 0, last = p + 1 == P;
    ZK_TRY(launch_pass(dit, data, batch, bstride, d, inverse, s0, ks[p], elog, first ? load_scale : 0,
                       last ? store_scale : 0, (first && raw) ? 1 : 0, st));
    s0 += ks[p];
  }
  return ZKVC_OK;
}

int ntt_quotient_chain(Fr* ev, int m, size_t N, const NttDomain* d, cudaStream_t st, int elog) {
  ZK_CHECK(elog >= 8 && elog <= 11, ZKVC_EINVAL, "ntt: 2^%d elements per block outside [2^8, 2^11]", elog);
  ZK_CHECK(m >= 1 && 3 * m <= 65535, ZKVC_EINVAL, "ntt: %d instances", m);
  ZK_CHECK(N == d->N, ZKVC_EINVAL, "ntt: array stride %zu is not N", N);
  ZK_TRY(ntt_init());
  const uint32_t L = d->logN;
  const std::vector<uint32_t> ks = pass_split(L, elog);
  const uint32_t P = (uint32_t)ks.size();
  Fr* H = ev + size_t(3) * m * N;
  if (P < 2 || L < 2) {  // one pass: no turn to fuse
    ZK_TRY(run_passes(false, ev, 3 * m, N, d, true, SC_NONE, SC_NG, false, elog, st));
    ZK_TRY(run_passes(true, ev, 3 * m, N, d, false, SC_NONE, SC_NONE, false, elog, st));
    ZK_TRY(ntt_quotient(ev, ev + size_t(m) * N, ev + size_t(2) * m * N, H, d, st, size_t(m) * N));
    return run_passes(false, H, m, N, d, true, SC_NONE, SC_NGI, false, elog, st);
  }
  const ScaleTabs tabs = tabs_of(d);
  // inverse DIF transforms of A, B, C up to their last pass
  uint32_t s0 = 0;
  for (uint32_t p = 0; p + 1 < P; p++) {
    ZK_TRY(launch_pass(false, ev, 3 * m, N, d, true, s0, ks[p], elog, 0, 0, 0, st));
    s0 += ks[p];
  }
  // turn: the inverse's last pass, x N^-1 g^i, the forward DIT's first pass
  {
    const uint32_t k = ks[P - 1];
    const PassShape sh = pass_shape(L, k, elog, 3 * m);
    if (radix4(sh.grid))
      k_ntt_turn<true><<<sh.grid, sh.threads, size_t(sh.E) * 32, st>>>(ev, N, d->tw, L, k, sh.logG, tabs);
    else
      k_ntt_turn<false><<<sh.grid, sh.threads, size_t(sh.E) * 32, st>>>(ev, N, d->tw, L, k, sh.logG, tabs);
    ZK_COUNT_LAUNCH();
    ZK_CUDA(cudaGetLastError());
  }
  // the forward DIT's middle passes: the mirror of the DIF split (its pass q covers the
  // groups of the DIF's pass P - 1 - q)
  uint32_t s0d = ks[P - 1];
  for (uint32_t q = 1; q + 1 < P; q++) {
    ZK_TRY(launch_pass(true, ev, 3 * m, N, d, false, s0d, ks[P - 1 - q], elog, 0, 0, 0, st));
    s0d += ks[P - 1 - q];
  }
  // quotient turn: the forward's last pass of A, B, C, the quotient, the first inverse
  // DIF pass of h
  {
    const uint32_t k = ks[0];
    const PassShape sh = pass_shape(L, k, elog, m);
    // three times the threads where the grid is too small to fill the GPU (latency-bound)
    const uint64_t blocks = uint64_t(sh.grid.x) * sh.grid.y;
    const uint32_t threads = blocks < 2 * uint64_t(device_sm_count()) ? std::min<uint32_t>(3 * sh.threads, 768)
                             : radix4(sh.grid)                         ? sh.threads
                                                                       : std::min<uint32_t>(2 * sh.threads, 512);
    if (radix4(sh.grid))
      k_ntt_quotient_turn<true><<<sh.grid, threads, size_t(3) * sh.E * 32, st>>>(ev, (uint32_t)m, N, d->tw, L, k, sh.logG, tabs);
    else
      k_ntt_quotient_turn<false><<<sh.grid, threads, size_t(3) * sh.E * 32, st>>>(ev, (uint32_t)m, N, d->tw, L, k, sh.logG, tabs);
    ZK_COUNT_LAUNCH();
    ZK_CUDA(cudaGetLastError());
  }
  // the rest of h's inverse DIF transform, x N^-1 g^-i at the last store
  s0 = ks[0];
  for (uint32_t p = 1; p < P; p++) {
    ZK_TRY(launch_pass(false, H, m, N, d, true, s0, ks[p], elog, 0, p + 1 == P ? SC_NGI : 0, 0, st));
    s0 += ks[p];
  }
  return ZKVC_OK;
}

int ntt_dif(Fr* data, int batch, size_t bstride, const NttDomain* d, bool inverse, int load_scale,
            int store_scale, bool raw, cudaStream_t st, int elog) {
  return run_passes(false, data, batch, bstride, d, inverse, load_scale, store_scale, raw, elog, st);
}

// The element at bit-reversed position q, natural index p, on its way out: times the factor
// of p, below N (x: below 4N).
__device__ __forceinline__ Fr bitrev_value(const Fr& x, int scale, uint32_t p, const ScaleTabs& tabs) {
  return scale ? f_mul(scale_factor(tabs, scale, p), x) : f_once(f_red2(x));
}

__global__ void k_bitrev_small(Fr* a, uint32_t logN, int scale, ScaleTabs tabs) {
  const uint32_t N = 1u << logN, p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  const uint32_t q = brev_bits(p, logN);
  if (p > q) return;
  const Fr x = ld_field(a + p), y = ld_field(a + q);
  st_field(a + p, bitrev_value(y, scale, p, tabs));
  if (p != q) st_field(a + q, bitrev_value(x, scale, q, tabs));
}

// Bit reversal of N >= 256 elements in tiles: index (hi, mid, lo) with four bits in hi and
// lo goes to (lo^r, mid^r, hi^r), so the 16 x 16 elements of one mid trade places with those
// of mid^r, transposed and reversed, through shared memory; both sides move in runs of 512
// bytes and every thread has work (one thread per index, half of them past the diagonal,
// took 350 us at 2^22 with a scale, 131 now).
constexpr int BR_ROW = 17;  // padded: a column's 16-byte halves fall in different banks
__global__ void __launch_bounds__(256) k_bitrev_tiles(Fr* a, uint32_t logN, int scale, ScaleTabs tabs) {
  __shared__ uint4 sm[2][2 * 16 * BR_ROW];
  const uint32_t mid = blockIdx.x, mrev = logN == 8 ? 0u : brev_bits(mid, logN - 8);
  if (mid > mrev) return;
  const uint32_t hi = threadIdx.x >> 4, lo = threadIdx.x & 15, E = 16 * BR_ROW;
  const uint32_t p = (hi << (logN - 4)) | (mid << 4) | lo, q = (hi << (logN - 4)) | (mrev << 4) | lo;
  sm_put(sm[0], E, hi * BR_ROW + lo, ld_field(a + p));
  sm_put(sm[1], E, hi * BR_ROW + lo, ld_field(a + q));
  __syncthreads();
  const uint32_t e = (__brev(lo) >> 28) * BR_ROW + (__brev(hi) >> 28);
  st_field(a + q, bitrev_value(sm_get(sm[0], E, e), scale, q, tabs));
  if (mid != mrev) st_field(a + p, bitrev_value(sm_get(sm[1], E, e), scale, p, tabs));
}

int ntt_bitrev(Fr* data, const NttDomain* d, int scale, cudaStream_t st) {
  if (d->logN >= 8)
    k_bitrev_tiles<<<1u << (d->logN - 8), 256, 0, st>>>(data, d->logN, scale, tabs_of(d));
  else
    k_bitrev_small<<<1, 128, 0, st>>>(data, d->logN, scale, tabs_of(d));
  ZK_COUNT_LAUNCH();
  ZK_CUDA(cudaGetLastError());
  return ZKVC_OK;
}

__global__ void k_quotient(const Fr* __restrict__ A, const Fr* __restrict__ B, const Fr* __restrict__ C, Fr* H,
                           size_t N, const Fr* consts) {
  size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= N) return;
  Fr zinv = ld_field(consts + 1);
  Fr v = f_sub(f_mul(ld_field(A + i), ld_field(B + i)), ld_field(C + i));
  st_field(H + i, f_mul(v, zinv));
}

int ntt_quotient(const Fr* A, const Fr* B, const Fr* C, Fr* H, const NttDomain* d, cudaStream_t st, size_t count) {
  size_t n = count ? count : d->N;
  unsigned blocks = (unsigned)((n + 255) / 256);
  k_quotient<<<blocks, 256, 0, st>>>(A, B, C, H, n, d->consts); ZK_COUNT_LAUNCH();
  ZK_CUDA(cudaGetLastError());
  return ZKVC_OK;
}

}  // namespace zkvc
