// tc.cuh -- building blocks of the tensor-core (tcgen05) kernels whose
// operands are cut into exact fixed-point bf16 slices: mbarrier waits with a
// time limit, bulk copies, MMA issue, shared-memory descriptors and the
// slicing arithmetic.
#pragma once
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "df64.cuh"

namespace tw {

// ------------------------------------------------------------ addresses
__device__ __forceinline__ uint32_t tc_su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// byte offset of the 16-byte chunk q (0..3) of row r in a K-major tile of 32
// bf16 per row with the 64-byte swizzle (chunk index XOR bits 1-2 of the row)
__host__ __device__ __forceinline__ uint32_t tc_swz64(int r, int q) {
  return (uint32_t)r * 64u + ((uint32_t)(q ^ ((r >> 1) & 3)) << 4);
}
// shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512
// bytes apart; bits 46-48 = 0b001 (descriptor version), bits 61-63 = 4 (64B)
__device__ __forceinline__ uint64_t tc_sdesc64(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}
// instruction descriptor, kind::f16: D F32, A and B BF16, both K-major
__host__ __device__ __forceinline__ uint32_t tc_idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ------------------------------------------------------------ mbarriers
__device__ __forceinline__ void tc_mbar_init(uint32_t bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mbar_arrive_tx(uint32_t bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool tc_mbar_try(uint32_t bar, unsigned parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.b32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long tc_time() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr unsigned long long TC_WAIT_NS = 4000000000ull;   // bound of every wait (4 s)
// true once the phase of this parity has completed; false after TC_WAIT_NS or
// (fail != nullptr) once another role of the CTA has failed
__device__ __forceinline__ bool tc_mbar_wait(uint32_t bar, unsigned parity, volatile int *fail) {
  unsigned long long t0 = 0;
  for (unsigned it = 1;; ++it) {
    if (tc_mbar_try(bar, parity)) return true;
    if ((it & 255u) == 0) {
      if (fail && *fail) return false;
      const unsigned long long t = tc_time();
      if (t0 == 0) t0 = t;
      else if (t - t0 > TC_WAIT_NS) return false;
    }
  }
}

// ------------------------------------------------------ copies and MMAs
__device__ __forceinline__ void tc_bulk_g2s(uint32_t dst, const void *src, unsigned bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// D (TMEM) (+)= A (TMEM) B (shared memory): bf16 operands, FP32 accumulators
__device__ __forceinline__ void tc_mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\t"
               "setp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
               ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// one lane of a converged warp.  MMAs and commits are issued by a warp whose 32
// lanes run the issuing loop together, one elected lane doing the work of each
// unrolled group: 15 cycles per 128 x 16 x 16 MMA; issued inside a branch taken by lane 0 alone
// they took 45 (operands moved to uniform registers one MMA at a time)
__device__ __forceinline__ bool tc_elect() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0;
}
// TMEM stores: 4 consecutive columns of the warp's 32 lanes
__device__ __forceinline__ void tc_st4(uint32_t addr, const uint32_t *v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
               ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
// 8 consecutive columns
__device__ __forceinline__ void tc_st8(uint32_t addr, uint4 a, uint4 b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"r"(addr), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_ld4(uint32_t *v, uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr));
}
__device__ __forceinline__ void tc_ld2(uint32_t *v, uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(addr));
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------ slicing
// 2^e as a float, e in [-126, 127]
__device__ __forceinline__ float tc_pow2f(int e) { return __int_as_float((e + 127) << 23); }
// bf16 bits of two floats of at most 8 significant bits (exact): upper halves
__device__ __forceinline__ uint32_t tc_pack_bf16(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
// smallest e in [-100, 127] with |hi + lo| < 2^e for every float pair whose
// |hi| <= mx (the low half may lift the sum past mx by one unit in the last
// place); the upper clamp keeps e in 8 bits and costs one bit of headroom
__device__ __forceinline__ int tc_exp_above(float mx) {
  mx *= 1.0f + 1.0f / 1048576.0f;
  if (!(mx > 0.f)) return -100;
  const int e = (int)((__float_as_uint(mx) >> 23) & 0xffu) - 126;
  return e < -100 ? -100 : (e > 127 ? 127 : e);
}

// Seven 8-bit slices of a float pair scaled to |hi + lo| < 2^7: step s rounds
// what is left to a multiple of 2^-8s (adding and subtracting 1.5 2^(23-8s)),
//   hi + lo = s0 + s1 + ... + s6 + r,  |s_p| <= 2^(7-8p) (s2: 129/128 of it), |r| <= 2^-49,
// every s_p an integer of at most 8 significant bits times 2^-8p: exact in
// bf16.  The first two steps act on hi alone (exact); what is left of it is
// then joined with lo (TwoSum, its error added back before slice 4).
// Two pairs at a time in packed f32x2 instructions: each lane rounds like the
// scalar one, in half the issue slots, which is what the slicing warps of a
// product kernel compete for.
struct Slicer7 {
  f2 r, e;
  __device__ __forceinline__ void init(float hi0, float lo0, float hi1, float lo1, f2 scale) {
    r = mul2(f2_make(hi0, hi1), scale);
    e = mul2(f2_make(lo0, lo1), scale);
  }
  // slice S of both pairs as two bf16 (the first in the low half); S = 0 .. 6 in order
  template <int S> __device__ __forceinline__ uint32_t next() {
    if (S == 2) {
      const f2 s = add2(r, e), bb = sub2(s, r);
      e = add2(sub2(r, sub2(s, bb)), sub2(e, bb));
      r = s;
    }
    if (S == 4) r = add2(r, e);
    constexpr float m = 1.5f * (float)(1 << 23) / (float)(1ull << (8 * S));
    const f2 M = f2_make(m, m), s = sub2(add2(r, M), M);
    r = sub2(r, s);
    const float2 v = f2_split(s);
    return tc_pack_bf16(v.x, v.y);
  }
};

// f(integral_constant<int, S>) for S = 0..6, in order
template <class F> __device__ __forceinline__ void for_slices7(F &f) {
  f(std::integral_constant<int, 0>{});
  f(std::integral_constant<int, 1>{});
  f(std::integral_constant<int, 2>{});
  f(std::integral_constant<int, 3>{});
  f(std::integral_constant<int, 4>{});
  f(std::integral_constant<int, 5>{});
  f(std::integral_constant<int, 6>{});
}

// ------------------------------------------- products of seven slices
constexpr int TC_NSL = 7;                // slices per operand
constexpr int TC_NACC = 6;               // accumulators: levels 0..4, and 5..6
constexpr int TC_NPAIR = 28;             // slice pairs of levels 0..6
// level of slice pair p = 0..27 (levels in order, pair (i, L - i) of level L)
__host__ __device__ constexpr int tc_pair_level(int p) {
  int l = 0, first = 0;
  while (p >= first + l + 1) { first += l + 1; ++l; }
  return l;
}
// the MMA of slice pair PR: operand addresses are compile-time selections of
// the precomputed ones, so the issuing thread spends a few instructions on it
// (computing the pair's descriptors in the loop cost about 50 cycles an MMA)
template <bool FIRST, int PR>
__device__ __forceinline__ void tc_issue_pair(const uint32_t *d, uint32_t a, const uint64_t *b, uint32_t idesc) {
  constexpr int L = tc_pair_level(PR), si = PR - L * (L + 1) / 2, sj = L - si;
  constexpr int ac = L < 5 ? L : 5;
  // the first MMA of a chunk into each accumulator overwrites it
  tc_mma_ts(d[ac], a + 8u * si, b[sj], idesc, FIRST && si == 0 && L < 6 ? 0u : 1u);
}
template <bool FIRST, int P0, int... PR>
__device__ __forceinline__ void tc_issue_pairs(std::integer_sequence<int, PR...>, const uint32_t *d, uint32_t a,
                                            const uint64_t *b, uint32_t idesc) {
  (tc_issue_pair<FIRST, P0 + PR>(d, a, b, idesc), ...);
}
// half H of a stage's pairs (14 each)
template <int H>
__device__ __forceinline__ void tc_issue_half(bool first, const uint32_t *d, uint32_t a, const uint64_t *b,
                                           uint32_t idesc) {
  if (first)
    tc_issue_pairs<true, H * TC_NPAIR / 2>(std::make_integer_sequence<int, TC_NPAIR / 2>{}, d, a, b, idesc);
  else
    tc_issue_pairs<false, H * TC_NPAIR / 2>(std::make_integer_sequence<int, TC_NPAIR / 2>{}, d, a, b, idesc);
}

// D0 + .. + D4 + D56 as a float pair.  D_L is a multiple of 2^-8L of at most
// (L+1) 204 2^(14-8L): a running sum below 2^22 leaves a TwoSum error of at
// most 2^-3, and adding that to D2 (below 2^7.4, multiples of 2^-16), then to
// D3 (below 0.8, multiples of 2^-24), is exact in 24 bits; from D4 on the
// rounding is that of the pair's low half.
// Two values at a time (packed f32x2).
__device__ __forceinline__ void tc_two_sum2(f2 a, f2 b, f2 &s, f2 &e) {
  s = add2(a, b);
  const f2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}
__device__ __forceinline__ void tc_join_levels(const f2 *d, f2 &hi, f2 &lo) {
  f2 s, e;
  tc_two_sum2(d[0], d[1], s, e);
  tc_two_sum2(s, add2(e, d[2]), s, e);
  tc_two_sum2(s, add2(e, d[3]), s, e);
  e = add2(e, add2(d[4], d[5]));
  hi = add2(s, e);
  lo = sub2(e, sub2(hi, s));
}

// ------------------------------------------- guards of the sliced products
// A sum of n products of sliced operands is off by about sqrt(n) 2^-56 T (rms),
// T the product of the two exponents' powers: the dropped levels and residues
// are uniform over 2^-56 of the largest entries, however small the entries that
// meet.  Double-float rounds such a sum at about 2^-47 of S, the sum of the
// products' magnitudes.  A guard computes S (bf16 magnitudes rounded down, FP32
// sums: a lower bound to a few percent) and has every sum with
//   sqrt(n) 2^-56 T > 2^-47 S
// formed again in double-float, so that no sum loses digits to the slices.  S = 0: every
// product is zero, in slices as well.  A NaN or infinite S is taken again too.
__device__ __forceinline__ bool tc_guard_fails(float S, float sqrt_n_T) {
  return S != 0.f && !(512.f * S >= sqrt_n_T && S < __int_as_float(0x7f800000));
}
// C (16 x 8) += A (16 x 16) B (16 x 8), one warp, fragments in registers.  With
// g = lane / 4, c = lane % 4 the 16 k are dealt out alike on both sides (a sum
// does not mind): a[0], a[2] are row g, k 4c .. 4c+3, a[1], a[3] row g + 8; b[0],
// b[1] column g, k 4c .. 4c+3; d[0], d[1] are (g, 2c), (g, 2c+1), d[2], d[3] row g + 8.
// (Magnitudes take a hundredth of the slices' arithmetic: mma.sync from
// registers, with nothing staged, keeps up with HBM.)
__device__ __forceinline__ void tc_mma_mag(float *d, const uint32_t *a, const uint32_t *b) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// sum over the warp's lanes, the same bits in every lane (dd_add commutes)
__device__ __forceinline__ dd tc_warp_sum(dd a) {
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    dd o;
    o.hi = __shfl_xor_sync(0xffffffffu, a.hi, m);
    o.lo = __shfl_xor_sync(0xffffffffu, a.lo, m);
    a = dd_add(a, o);
  }
  return a;
}

}  // namespace tw
