// gemm_fwd_sl64.cu -- the FP64-class batched forward product on the
// 5th-generation tensor cores, both operands cut into seven exact bf16 slices.
//
// Per frequency w the forward map is the complex product
//   Y^(w) = F^(w) X^(w)            (Nr x Nm) (Nm x B)
// (Sec. "FFT-based Hessian matvecs"), a contraction over the grid.  Written
// over reals, with K' = 2 Nm and the entries of one grid point adjacent:
//   a row of F^:            (Fr, Fi)
//   two rows of X^ per RHS: (Xr, -Xi) -> Yr,   (Xi, Xr) -> Yi.
// Either operand can take the 128 MMA rows (TMEM): F^ (FM: 128 rows of F^
// against 2 x 32 columns) or X^ (XM: 64 right-hand sides x 2 against up to 64
// rows of F^), whichever needs less MMA time for the reserved batch: few
// forecast points leave the 128 rows of FM mostly empty.
//
// Accuracy.  Every row of F^ and of X^ has one power-of-two exponent per
// frequency and range of 4128 grid points (k_row_scan; F^: once per load; X^: one
// pass per call); slices, levels and exact accumulation as in gemm_sl64.cu.  The
// level sums are exact over chunks of 96 grid points (K' = 192); the chunks of a
// range are added in double-float in shared memory, the
// ranges in a fixed order by k_fwd_join.  The SIMT product rounds its running sum
// after every one of the 2 Nm terms.  A field that is large where a row of F^ is small
// leaves fewer digits to their sum than double-float does; such sums are found from
// their magnitudes, bounded from below per 32 grid points for every frequency
// (k_fwd_check) and formed in full for those that this leaves open (k_fwd_mag), and
// taken again in double-float (k_fwd_join).
//
// What bounds it.  The SIMT form (gemm.cu) spends about 60 FP32 operations on
// an entry and right-hand side.  Here 28 MMAs of 128 x N x 16 serve 8 grid
// points; cutting the slices (about 32 FP32 operations a real, once per
// operand row and tile) takes about as long, on its own warps.  Measured (401
// frequencies, 50,000 grid points): 20 rows and 64 right-hand sides (XM) 54.4 ->
// 17.7 ms, of which 3.3 ms are the exponents' pass over X^; 100 rows and 32
// (FM) 147 -> 18.9 ms.
//
// Kernel: persistent, one CTA per SM over (frequency, range, row tiles), the
// tiles of one range fastest (its operands are then read from L2).  Warps
// 0-15: two groups that copy rows of the M operand (cp.async, 128 bytes a row
// and stage), slice them and fill alternate TMEM stages; 16-19: the same for
// the N operand into swizzled shared memory; 20-27 drain the accumulators; 28
// issues the MMAs.  Every wait is bounded: on expiry the kernel records
// TW_ERR_TIMEOUT, drains its copies and MMAs, frees TMEM and returns.
#include <algorithm>

#include "../../include/tw.h"
#include "kernels.h"
#include "tc.cuh"

namespace tw {

namespace {

constexpr int TM = 128;                  // MMA M
constexpr int SK = 8;                    // grid points per stage (K' = 16)
constexpr int CH_STAGES = 12;            // stages per exact chunk (96 grid points)
constexpr int RANGE = 43 * CH_STAGES * SK;   // 4128 grid points per work item
constexpr int NSL = TC_NSL, NACC = TC_NACC;
constexpr int A_COLS = NSL * 8;          // TMEM columns of a stage
constexpr int NGRP = 256, NPROD = 2 * NGRP, NNB = 128, NEPI = 256;
constexpr int NTHR = NPROD + NNB + NEPI + 32;
constexpr int MAXA = 4, SBH = 4;         // M stages (at most), N stages
constexpr int RAW_ROW = SK * 16 + 16;    // a row's 8 entries, padded (bank conflicts)
constexpr int RAWN_D = 3;                // raw slots of the N operand

__device__ __forceinline__ void note(int *err, volatile int *fail, int info) {
  if (!*fail && atomicCAS(err, 0, TW_ERR_TIMEOUT) == 0) err[1] = info;
  *fail = 1;
}

// One pass over rows of Nm complex entries, row y of frequency x = blockIdx.x from
// A + x * ws + y * rs, range z = blockIdx.z of it: its exponent e[(x nrange + z) es +
// y], and for the guard one bf16 value (rounded down) per block of 32 entries, blk[(x
// es + y) nbp + i]: the least |Re| + |Im| of the block (LOW: the operator) or their
// sum (the data)
template <bool LOW>
__global__ void __launch_bounds__(256)
k_row_scan(const float4 *__restrict__ A, long ws, long rs, int Nm, int8_t *__restrict__ e, int es,
           uint16_t *__restrict__ blk, int nbp, int *__restrict__ open) {
  __shared__ float red[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = blockIdx.z;
  const int kb = rg * RANGE, kend = min(Nm, kb + RANGE);
  if (!LOW && blockIdx.y == 0 && rg == 0 && threadIdx.x == 0) open[blockIdx.x] = 0;    // for k_fwd_check
  const float4 *p = A + (long)blockIdx.x * ws + (long)blockIdx.y * rs;
  uint16_t *out = blk + ((size_t)blockIdx.x * es + blockIdx.y) * nbp;
  float mx = 0.f;
  for (int k0 = kb + 128 * warp; k0 < kend; k0 += 1024) {
    float s[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + 32 * j + lane;
      s[j] = LOW ? __int_as_float(0x7f800000) : 0.f;
      if (k < kend) {
        const float4 v = __ldg(p + k);
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.z)));
        s[j] = fabsf(v.x) + fabsf(v.z);
      }
    }
    // four values a lane over 32 lanes: block j ends in the lanes whose bits 4 and 3 are j's bits 0 and 1
    auto join = [](float a, float b) { return LOW ? fminf(a, b) : a + b; };
    auto halve = [&](float lo, float hi, int m) {
      const float keep = lane & m ? hi : lo;
      return join(keep, __shfl_xor_sync(0xffffffffu, lane & m ? lo : hi, m));
    };
    float r = halve(halve(s[0], s[1], 16), halve(s[2], s[3], 16), 8);
#pragma unroll
    for (int m = 4; m >= 1; m >>= 1) r = join(r, __shfl_xor_sync(0xffffffffu, r, m));
    const int i = k0 / 32 + (lane >> 4) + 2 * ((lane >> 3) & 1);
    if ((lane & 7) == 0 && 32 * i < kend) out[i] = (uint16_t)(__float_as_uint(r) >> 16);
  }
  if (kend == Nm)
    for (int i = (Nm + 31) / 32 + threadIdx.x; i < nbp; i += 256) out[i] = 0;
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
  if (lane == 0) red[warp] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) mx = fmaxf(mx, red[i]);
    e[((size_t)blockIdx.x * gridDim.z + rg) * es + blockIdx.y] = (int8_t)tc_exp_above(mx);
  }
}

// ------------------------------------------------------ the guard (tc.cuh)
// sqrt(n) T of a row and a column: root of the sum of n T^2 over the ranges, n = 2
// entries a point; er, eb: their exponents in range 0, strides sr, sb
__device__ __forceinline__ float guard_scale(int Nm, int nrange, const int8_t *er, int sr, const int8_t *eb, int sb) {
  int top = -1000;
  for (int g = 0; g < nrange; ++g) top = max(top, (int)er[(size_t)g * sr] + (int)eb[(size_t)g * sb]);
  float t = 0.f;
  for (int g = 0; g < nrange; ++g)
    t += scalbnf(2.f * (float)min(RANGE, Nm - g * RANGE), 2 * ((int)er[(size_t)g * sr] + (int)eb[(size_t)g * sb] - top));
  return scalbnf(sqrtf(t), top);
}

// open[w] = 1 if the blocks' bound sum_i low F^ x (sum of |X^|) leaves some sum of
// this frequency unsettled.  A CTA takes 16 rows and 64 columns, its warps the
// blocks in turn
__global__ void __launch_bounds__(256)
k_fwd_check(const int8_t *__restrict__ ef, const uint16_t *__restrict__ low, const int8_t *__restrict__ ex,
            const uint16_t *__restrict__ xsum, int nbp, int nrange, int Nr, int Nm, int B, int *__restrict__ open,
            unsigned long long *__restrict__ Sq) {
  __shared__ float sS[8][16][65], sM[8][64];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int w = blockIdx.y, col0 = blockIdx.z * 64, r0 = blockIdx.x * 16, nf = min(8, (B - col0 + 7) / 8);
  const uint16_t *la = low + ((size_t)w * Nr + min(r0 + g, Nr - 1)) * nbp + 4 * c;
  const uint16_t *lb = low + ((size_t)w * Nr + min(r0 + g + 8, Nr - 1)) * nbp + 4 * c;
  float S[8][4] = {}, M[8][4] = {};
  for (int s = 16 * warp; s < nbp; s += 128) {
    const uint2 p = __ldg(reinterpret_cast<const uint2 *>(la + s)), q = __ldg(reinterpret_cast<const uint2 *>(lb + s));
    const uint32_t a[4] = {p.x, q.x, p.y, q.y}, one[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
#pragma unroll
    for (int f = 0; f < 8; ++f)
      if (f < nf) {
        const int b = min(col0 + 8 * f + g, B - 1);
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(xsum + ((size_t)w * B + b) * nbp + 4 * c + s));
        const uint32_t bb[2] = {v.x, v.y};
        tc_mma_mag(S[f], a, bb);
        tc_mma_mag(M[f], one, bb);                         // zero: an empty column
      }
  }
#pragma unroll
  for (int f = 0; f < 8; ++f)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sS[warp][g + 8 * (i >> 1)][8 * f + 2 * c + (i & 1)] = S[f][i];
      if (g == 0 && i < 2) sM[warp][8 * f + 2 * c + i] = M[f][i];
    }
  __syncthreads();
  for (int t = threadIdx.x; t < 1024; t += 256) {
    const int rl = t >> 6, bl = t & 63, r = r0 + rl, b = col0 + bl;
    if (r >= Nr || b >= B) continue;
    Sq[((size_t)w * Nr + r) * B + b] = 0;                  // k_fwd_mag's sum
    float v = 0.f, m = 0.f;
    for (int k = 0; k < 8; ++k) { v += sS[k][rl][bl]; m += sM[k][bl]; }
    if (m != 0.f && (v == 0.f || tc_guard_fails(v, guard_scale(Nm, nrange, ef + (size_t)w * nrange * Nr + r, Nr,
                                                               ex + (size_t)w * nrange * B + b, B))))
      open[w] = 1;
  }
}

// Sq[w][r][b] += sum_k |F^[r][k]| |X^[b][k]| over SUB grid points, of the open
// frequencies: 32 rows and 32 columns a CTA, whose warps take 16 points in turn,
// straight from both operands.  The pieces are added as integers, in units of
// 2^-24 sqrt(n) T, so that their order does not matter (a sum that fails is below
// 2^15); bit 63: not finite.  Bound by the operands' second reading, and for a few open
// frequencies by a CTA's own latency, hence the short pieces (whole ranges: 70 us).
constexpr int SUB = 688;                 // 43 steps of 16
constexpr unsigned long long S_BAD = 1ull << 63;
__global__ void __launch_bounds__(256, 2)
k_fwd_mag(const float4 *__restrict__ F, const float4 *__restrict__ X, long xs, const int8_t *__restrict__ ef,
          const int8_t *__restrict__ ex, const int *__restrict__ open, int nrt, int nbt, int nrange, int Nr, int Nm,
          int B, unsigned long long *__restrict__ Sq) {
  const int w = blockIdx.y;
  if (!open[w]) return;
  __shared__ float sh[8][32][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int r0 = blockIdx.x % nrt * 32, b0 = blockIdx.x / nrt % nbt * 32, kb = blockIdx.x / (nrt * nbt) * SUB;
  const int kend = min(Nm, kb + SUB);
  float d[2][4][4] = {};
  for (int k = kb + 16 * warp + c; k - c < kend; k += 128) {
    // four entries' magnitudes, zero past the range (a lane's k are c, c + 4, .. on
    // both sides: a load instruction takes 64 bytes in a row)
    auto quad = [&](const float4 *row, uint32_t *o) {
      float m[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = __ldg(row + min(k + 4 * j, kend - 1));
        m[j] = k + 4 * j < kend ? fabsf(v.x) + fabsf(v.z) : 0.f;
      }
      o[0] = tc_pack_bf16(m[0], m[1]);
      o[1] = tc_pack_bf16(m[2], m[3]);
    };
    uint32_t bq[4][2];
#pragma unroll
    for (int f = 0; f < 4; ++f) quad(X + (long)min(b0 + 8 * f + g, B - 1) * xs + (long)w * Nm, bq[f]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t lo[2], hi[2];
      quad(F + ((long)w * Nr + min(r0 + 16 * h + g, Nr - 1)) * Nm, lo);
      quad(F + ((long)w * Nr + min(r0 + 16 * h + g + 8, Nr - 1)) * Nm, hi);
      const uint32_t a[4] = {lo[0], hi[0], lo[1], hi[1]};
#pragma unroll
      for (int f = 0; f < 4; ++f) tc_mma_mag(d[h][f], a, bq[f]);
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int i = 0; i < 4; ++i) sh[warp][16 * h + g + 8 * (i >> 1)][8 * f + 2 * c + (i & 1)] = d[h][f][i];
  __syncthreads();
  for (int t = threadIdx.x; t < 1024; t += 256) {
    const int r = t >> 5, b = t & 31;
    if (r0 + r >= Nr || b0 + b >= B) continue;
    float S = 0.f;
    for (int v = 0; v < 8; ++v) S += sh[v][r][b];
    unsigned long long *o = Sq + ((size_t)w * Nr + r0 + r) * B + b0 + b;
    if (!(S < __int_as_float(0x7f800000))) {
      atomicOr(o, S_BAD);
    } else if (S > 0.f) {
      const float gs = guard_scale(Nm, nrange, ef + (size_t)w * nrange * Nr + r0 + r, Nr,
                                   ex + (size_t)w * nrange * B + b0 + b, B);
      // at least one unit: a sum that is not zero stays so; at most 2^40 a piece
      const float u = fminf(S / gs * 16777216.f, 1.0995116e12f);
      atomicAdd(o, u >= 1.f ? (unsigned long long)u : 1ull);
    }
  }
}

// Yo[b][w][r]: the ranges' partial sums in order; then the sums of open frequencies
// that fail the guard again in double-float, by all of the CTA's threads.  (A CTA's
// outputs are gridDim.x apart: those of one frequency, which fail together, go to
// different CTAs.)
__global__ void __launch_bounds__(256)
k_fwd_join(const cdd *__restrict__ part, const cdd *__restrict__ F, const cdd *__restrict__ X, long xs,
           const int *__restrict__ open, const unsigned long long *__restrict__ Sq, cdd *__restrict__ Yo,
           long y_bstride, int nrange, int Nf, int Nr, int Nm, int B) {
  __shared__ int list[256], count;
  __shared__ cdd sh[8];
  const int lane = threadIdx.x & 31;
  const long i = blockIdx.x + (long)gridDim.x * threadIdx.x;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  if (i < (long)B * Nf * Nr) {
    const int r = (int)(i % Nr), w = (int)(i / Nr % Nf), b = (int)(i / Nr / Nf);
    const cdd *p = part + (size_t)(i / Nr) * nrange * Nr + r;
    cdd acc = cdd_zero();
    for (int c = 0; c < nrange; ++c) acc = cdd_add(acc, ld_cdd(p + (size_t)c * Nr));
    st_cdd(Yo + (size_t)b * y_bstride + (size_t)w * Nr + r, acc);
    if (open[w]) {
      const unsigned long long S = Sq[((size_t)w * Nr + r) * B + b];
      if ((S & S_BAD) || (S != 0 && S < (1ull << 15)))     // as tc_guard_fails: 512 S < sqrt(n) T
        list[atomicAdd(&count, 1)] = threadIdx.x;
    }
  }
  __syncthreads();
  for (int it = 0; it < count; ++it) {
    const long q = blockIdx.x + (long)gridDim.x * list[it];
    const int r = (int)(q % Nr), w = (int)(q / Nr % Nf), b = (int)(q / Nr / Nf);
    const cdd *f = F + ((size_t)w * Nr + r) * Nm, *x = X + (long)b * xs + (size_t)w * Nm;
    cdd a[4] = {cdd_zero(), cdd_zero(), cdd_zero(), cdd_zero()};      // four chains in flight
    for (int k = threadIdx.x; k < Nm; k += 1024)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + 256 * u < Nm) a[u] = cdd_add(a[u], cdd_mul(ld_cdd(f + k + 256 * u), ld_cdd(x + k + 256 * u)));
    cdd y = cdd_add(cdd_add(a[0], a[1]), cdd_add(a[2], a[3]));
    y.re = tc_warp_sum(y.re);
    y.im = tc_warp_sum(y.im);
    __syncthreads();                     // the sum before is read
    if (lane == 0) sh[threadIdx.x >> 5] = y;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int v = 1; v < 8; ++v) y = cdd_add(y, sh[v]);
      st_cdd(Yo + (size_t)b * y_bstride + (size_t)w * Nr + r, y);
    }
  }
}

template <int N, bool XM>
struct Cfg {
  static constexpr int nbuf = 2 * NACC * N + 2 * A_COLS <= 512 ? 2 : 1;
  static constexpr int left = (512 - nbuf * NACC * N) / A_COLS;
  static constexpr int SA = left < MAXA ? left : MAXA;
  static constexpr int MROWS = XM ? 64 : 128;      // raw rows of the M operand per tile
  static constexpr int NROWS = XM ? N : N / 2;     // of the N operand
  static constexpr uint32_t b_slice = (uint32_t)N * 64u, b_atom = NSL * b_slice;   // two stages
  static constexpr uint32_t rawm = MROWS * RAW_ROW, rawn = NROWS * RAW_ROW;        // one slot
  static constexpr uint32_t acc = N * TM * 8;
  static constexpr size_t smem = 1024 + SBH / 2 * b_atom + 4 * rawm + RAWN_D * rawn + acc;
  static_assert(SA >= 2 && smem <= 227 * 1024, "stages");
};

// rows of X^ and F^: X^[b][w][k] (stride xs per right-hand side), F^[w][r][k]
template <int N, bool XM>
__global__ void __launch_bounds__(NTHR, 1)
k_gemm_fwd_sl64(const float4 *__restrict__ F, const int8_t *__restrict__ ef, const float4 *__restrict__ X, long xs,
                const int8_t *__restrict__ ex, float2 *__restrict__ part, int nrange, int Nf, int Nr, int Nm,
                int B, int nmt, int nnt, int *err) {
  typedef Cfg<N, XM> C;
  constexpr int SA = C::SA, nbuf = C::nbuf;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * MAXA + 2 * SBH + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int T = nmt * nnt * nrange * Nf;
  const int my_items = (int)blockIdx.x < T ? (T - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const uint32_t sB0 = (tc_su32(smem_raw) + 1023u) & ~1023u;
  uint8_t *gB0 = smem_raw + (sB0 - tc_su32(smem_raw));
  uint8_t *gRawM = gB0 + SBH / 2 * C::b_atom, *gRawN = gRawM + 4 * C::rawm;
  float2 *sAcc = reinterpret_cast<float2 *>(gRawN + RAWN_D * C::rawn);      // [N][128]
  const uint32_t bar0 = tc_su32(&bars[0]);
  auto fullA = [&](int st) { return bar0 + 8u * st; };
  auto emptyA = [&](int st) { return bar0 + 8u * (MAXA + st); };
  auto fullB = [&](int st) { return bar0 + 8u * (2 * MAXA + st); };
  auto emptyB = [&](int st) { return bar0 + 8u * (2 * MAXA + SBH + st); };
  auto tfull = [&](int bf) { return bar0 + 8u * (2 * MAXA + 2 * SBH + bf); };
  auto tempty = [&](int bf) { return bar0 + 8u * (2 * MAXA + 2 * SBH + 2 + bf); };
  const uint32_t drain = bar0 + 8u * (2 * MAXA + 2 * SBH + 4);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(tc_su32(&tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    fail = 0;
    for (int st = 0; st < SA; ++st) {
      tc_mbar_init(fullA(st), NGRP);
      tc_mbar_init(emptyA(st), 1);
    }
    for (int st = 0; st < SBH; ++st) {
      tc_mbar_init(fullB(st), NNB);
      tc_mbar_init(emptyB(st), 1);
    }
    for (int bf = 0; bf < 2; ++bf) {
      tc_mbar_init(tfull(bf), 1);
      tc_mbar_init(tempty(bf), NEPI);
    }
    tc_mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  constexpr uint32_t tmem = 0;           // all 512 columns are allocated
  constexpr uint32_t tmemA = tmem + (uint32_t)(nbuf * NACC * N);
  volatile int *vfail = &fail;
  struct Item { int w, rg, mt, nt, k0, nst; };   // nst: stages, even
  auto item_of = [&](int i) {
    Item it;
    int t = (int)blockIdx.x + i * (int)gridDim.x;
    it.nt = t % nnt; t /= nnt;
    it.mt = t % nmt; t /= nmt;
    it.rg = t % nrange;
    it.w = t / nrange;
    it.k0 = it.rg * RANGE;
    it.nst = (min(Nm - it.k0, RANGE) + 2 * SK - 1) / (2 * SK) * 2;
    return it;
  };
  // first entry of raw row q of an operand's tile t, nullptr past the rows
  auto x_row = [&](int w, int b) { return b < B ? X + (long)b * xs + (long)w * Nm : nullptr; };
  auto f_row = [&](int w, int r) { return r < Nr ? F + ((long)w * Nr + r) * Nm : nullptr; };
  auto m_row = [&](const Item &it, int q) { return XM ? x_row(it.w, it.mt * 64 + q) : f_row(it.w, it.mt * 128 + q); };
  auto n_row = [&](const Item &it, int q) {
    return XM ? f_row(it.w, it.nt * N + q) : x_row(it.w, it.nt * (N / 2) + q);
  };
  auto x_exp = [&](const Item &it, int b) { return (int)ex[((size_t)it.w * nrange + it.rg) * B + b]; };
  auto f_exp = [&](const Item &it, int r) { return (int)ef[((size_t)it.w * nrange + it.rg) * Nr + r]; };
  auto m_exp = [&](const Item &it, int q) {
    const int i = XM ? it.mt * 64 + q : it.mt * 128 + q;
    return XM ? (i < B ? x_exp(it, i) : 0) : (i < Nr ? f_exp(it, i) : 0);
  };
  auto n_exp = [&](const Item &it, int q) {
    const int i = XM ? it.nt * N + q : it.nt * (N / 2) + q;
    return XM ? (i < Nr ? f_exp(it, i) : 0) : (i < B ? x_exp(it, i) : 0);
  };
  auto copy16 = [&](uint32_t dst, const float4 *row, int k, int kend) {
    const bool in = row != nullptr && k < kend;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 ::"r"(dst), "l"(in ? row + k : F), "r"(in ? 16 : 0) : "memory");
  };

  if (warp < NPROD / 32) {
    // ---------------- M operand: slices into TMEM.  Group g fills the stages
    // of its parity; 8 threads copy a row's 8 grid points, thread = MMA row r,
    // points 4h .. 4h+3 cuts them
    const int tg = tid & (NGRP - 1), r = tg & (TM - 1), h = tg >> 7, g = tid / NGRP;
    constexpr int NCP = C::MROWS * 8 / NGRP;
    const uint8_t *rawp = gRawM + g * 2 * C::rawm;
    const uint32_t raw0 = tc_su32(rawp);
    int ii = 0, is = g, islot = 0;
    Item cp = item_of(0);
    const float4 *rows[NCP];
    auto set_rows = [&]() {
#pragma unroll
      for (int u = 0; u < NCP; ++u) rows[u] = m_row(cp, (u * NGRP + tg) >> 3);
    };
    if (my_items > 0) set_rows();
    auto load = [&]() {
      if (ii < my_items) {
        const int k = cp.k0 + is * SK + (tg & 7);
#pragma unroll
        for (int u = 0; u < NCP; ++u)
          copy16(raw0 + (uint32_t)(islot * C::rawm + ((u * NGRP + tg) >> 3) * RAW_ROW + (tg & 7) * 16), rows[u], k, Nm);
        is += 2;
        if (is >= cp.nst) {
          is = g;
          if (++ii < my_items) { cp = item_of(ii); set_rows(); }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      islot ^= 1;
    };
    load();
    int slot = 0, st = g, use = 0;
    bool ok = true;
    const uint32_t lane_base = tmemA + ((uint32_t)(32 * (warp & 3)) << 16) + 4u * h;
    const uint32_t flip = XM && !(r & 1) ? 0x80000000u : 0u;
    for (int i = 0; i < my_items && ok; ++i) {
      const Item it = item_of(i);
      const float sc1 = tc_pow2f(7 - m_exp(it, XM ? r >> 1 : r));
      const f2 sc = f2_make(sc1, sc1);
      for (int s = g; s < it.nst; s += 2) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // the group's copies of this slot are in, and every thread has read the other one
        asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(NGRP) : "memory");
        load();
        Slicer7 sl[4];
        const float4 *p = reinterpret_cast<const float4 *>(rawp + slot * C::rawm + (XM ? r >> 1 : r) * RAW_ROW + h * 64);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 v = p[u];
          sl[u].init(v.x, v.y, v.z, v.w, sc);
        }
        slot ^= 1;
        if (use > 0) {
          const bool got = tc_mbar_wait(emptyA(st), (unsigned)((use - 1) & 1), vfail);
          if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) note(err, vfail, 61);
            ok = false;
          }
        }
        if (ok) {      // after a failure the group's barriers still have to be met
          tc_fence_after();
          const uint32_t at = lane_base + (uint32_t)(st * A_COLS);
          auto put = [&](auto S) {
            uint32_t wd[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const uint32_t w = sl[u].template next<S.value>();
              // XM: (Xr, -Xi) in even rows, (Xi, Xr) in odd ones
              wd[u] = XM && (r & 1) ? __byte_perm(w, 0, 0x1032) : w ^ flip;
            }
            tc_st4(at + 8u * S.value, wd);
          };
          for_slices7(put);
          tc_wait_st();
          tc_fence_before();
          tc_mbar_arrive(fullA(st));
        }
        st += 2;
        while (st >= SA) { st -= SA; ++use; }
      }
      int all;         // leave together: a warp that failed must not strand the others at the barrier
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
                   "barrier.cta.red.and.pred q, %2, %3, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                   : "=r"(all) : "r"((int)ok), "r"(1 + g), "r"(NGRP) : "memory");
      ok = all != 0;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // own copies drained before exit
  } else if (warp < (NPROD + NNB) / 32) {
    // ---------------- N operand: slices into shared memory (K-major, 64-byte
    // swizzle; a stage is half of a 32-wide atom).  Task = (row, 4 grid points)
    const int tg = tid - NPROD;
    constexpr int NCP = (C::NROWS * 8 + NNB - 1) / NNB, NTASK = C::NROWS * 2;
    static_assert(NTASK <= NNB, "one task a thread");
    const uint32_t raw0 = tc_su32(gRawN);
    int ii = 0, is = 0, islot = 0;
    Item cp = item_of(0);
    const float4 *rows[NCP];
    auto set_rows = [&]() {
#pragma unroll
      for (int u = 0; u < NCP; ++u) {
        const int q = (u * NNB + tg) >> 3;
        rows[u] = q < C::NROWS ? n_row(cp, q) : nullptr;
      }
    };
    if (my_items > 0) set_rows();
    auto load = [&]() {
      if (ii < my_items) {
        const int k = cp.k0 + is * SK + (tg & 7);
#pragma unroll
        for (int u = 0; u < NCP; ++u) {
          const int q = (u * NNB + tg) >> 3;
          if (q < C::NROWS)
            copy16(raw0 + (uint32_t)(islot * C::rawn + q * RAW_ROW + (tg & 7) * 16), rows[u], k, Nm);
        }
        if (++is >= cp.nst) {
          is = 0;
          if (++ii < my_items) { cp = item_of(ii); set_rows(); }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (++islot == RAWN_D) islot = 0;
    };
#pragma unroll
    for (int d = 0; d < RAWN_D - 1; ++d) load();
    const int q = tg >> 1, hh = tg & 1;                // row and 4-point half of this thread's task
    int slot = 0, st = 0, use = 0;
    bool ok = true;
    for (int i = 0; i < my_items && ok; ++i) {
      const Item it = item_of(i);
      const float sc1 = tg < NTASK ? tc_pow2f(7 - n_exp(it, q)) : 0.f;
      const f2 sc = f2_make(sc1, sc1);
      for (int s = 0; s < it.nst; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(RAWN_D - 2) : "memory");
        asm volatile("bar.sync 3, %0;" ::"r"(NNB) : "memory");
        load();
        if (use > 0) {
          const bool got = tc_mbar_wait(emptyB(st), (unsigned)((use - 1) & 1), vfail);
          if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) note(err, vfail, 62);
            ok = false;
          }
        }
        if (ok && tg < NTASK) {
          Slicer7 sl[4];
          const float4 *p = reinterpret_cast<const float4 *>(gRawN + slot * C::rawn + q * RAW_ROW + hh * 64);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 v = p[u];
            sl[u].init(v.x, v.y, v.z, v.w, sc);
          }
          uint8_t *atom = gB0 + (st >> 1) * C::b_atom;
          const int qc = 2 * (st & 1) + hh;
          auto put = [&](auto S) {
            uint32_t wd[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) wd[u] = sl[u].template next<S.value>();
            uint8_t *sl_at = atom + S.value * C::b_slice;
            if (XM) {
              *reinterpret_cast<uint4 *>(sl_at + tc_swz64(q, qc)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
            } else {
              // row q: (Xr, -Xi), row N/2 + q: (Xi, Xr)
              *reinterpret_cast<uint4 *>(sl_at + tc_swz64(q, qc)) =
                  make_uint4(wd[0] ^ 0x80000000u, wd[1] ^ 0x80000000u, wd[2] ^ 0x80000000u, wd[3] ^ 0x80000000u);
              *reinterpret_cast<uint4 *>(sl_at + tc_swz64(N / 2 + q, qc)) =
                  make_uint4(__byte_perm(wd[0], 0, 0x1032), __byte_perm(wd[1], 0, 0x1032),
                             __byte_perm(wd[2], 0, 0x1032), __byte_perm(wd[3], 0, 0x1032));
            }
          };
          for_slices7(put);
        }
        if (ok) {
          // generic-proxy writes -> visible to the tensor cores (async proxy)
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          tc_mbar_arrive(fullB(st));
        }
        if (++slot == RAWN_D) slot = 0;
        if (++st == SBH) { st = 0; ++use; }
      }
      int all;
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
                   "barrier.cta.red.and.pred q, 3, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                   : "=r"(all) : "r"((int)ok), "r"(NNB) : "memory");
      ok = all != 0;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp < (NPROD + NNB + NEPI) / 32) {
    // ---------------- epilogue (two warps a TMEM lane quarter, each half of the columns)
    const int lg = warp & 3, half = (warp - (NPROD + NNB) / 32) >> 2;
    const int r = 32 * lg + lane;
    constexpr int CW = N / 2;
    bool ok = true;
    int bf = 0, use = 0;
    float2 *acc = sAcc + half * CW * TM + r;
    for (int i = 0; i < my_items && ok; ++i) {
      const Item it = item_of(i);
      const int nch = (it.nst + CH_STAGES - 1) / CH_STAGES;
      for (int c = 0; c < nch; ++c) {
        const bool got = tc_mbar_wait(tfull(bf), (unsigned)(use & 1), vfail);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) note(err, vfail, 63);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t trow = tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)(bf * NACC * N + half * CW);
#pragma unroll 1
        for (int c0 = 0; c0 < CW; c0 += 4) {
          uint32_t d[NACC][4];
#pragma unroll
          for (int L = 0; L < NACC; ++L) tc_ld4(d[L], trow + (uint32_t)(L * N + c0));
          tc_wait_ld();
          if (c0 + 4 >= CW) {
            // the buffer is read: the MMAs of a later chunk may overwrite it
            tc_fence_before();
            tc_mbar_arrive(tempty(bf));
          }
#pragma unroll
          for (int j = 0; j < 4; j += 2) {             // two columns at once
            f2 v[NACC], xh, xl;
#pragma unroll
            for (int L = 0; L < NACC; ++L) v[L] = f2_make(__uint_as_float(d[L][j]), __uint_as_float(d[L][j + 1]));
            tc_join_levels(v, xh, xl);
            float2 *ac = acc + (c0 + j) * TM;
            if (c > 0) {
              const float2 o = ac[0], o2 = ac[TM];
              f2 h = f2_make(o.x, o2.x), l = f2_make(o.y, o2.y);
              dd_add2(h, l, xh, xl);
              xh = h;
              xl = l;
            }
            const float2 h = f2_split(xh), l = f2_split(xl);
            ac[0] = make_float2(h.x, l.x);
            ac[TM] = make_float2(h.y, l.y);
          }
        }
        if (++bf == nbuf) { bf = 0; ++use; }
      }
      if (!ok) break;
      // scaled partial sums of the range: part[b][w][range][r], real and imaginary halves apart
      const float sa = tc_pow2f(m_exp(it, XM ? r >> 1 : r) - 7);
#pragma unroll 1
      for (int c0 = 0; c0 < CW; ++c0) {
        const int n = half * CW + c0;
        const int b = XM ? it.mt * 64 + (r >> 1) : it.nt * (N / 2) + c0;
        const int rr = XM ? it.nt * N + n : it.mt * 128 + r;
        const int im = XM ? r & 1 : half;
        if (b >= B || rr >= Nr) continue;
        const float sb = tc_pow2f(n_exp(it, XM ? n : c0) - 7);
        const float2 v = acc[c0 * TM];
        part[2 * ((((size_t)b * Nf + it.w) * nrange + it.rg) * Nr + rr) + im] =
            make_float2(v.x * sa * sb, v.y * sa * sb);
      }
    }
  } else {
    // ---------------- MMA issuer (the warp's lanes run together, one is elected to issue)
    const uint32_t idesc = tc_idesc_bf16(TM, N);
    auto wait = [&](uint32_t bar, int parity) {
      return __all_sync(0xffffffffu, tc_mbar_wait(bar, (unsigned)(parity & 1), vfail));
    };
    bool ok = true;
    int sa = 0, usea = 0, sb = 0, useb = 0, bf = 0, used = 0;
    for (int i = 0; i < my_items && ok; ++i) {
      const Item it = item_of(i);
      for (int c0 = 0; c0 < it.nst && ok; c0 += CH_STAGES) {
        if (used > 0 && !wait(tempty(bf), used - 1)) { ok = false; break; }
        tc_fence_after();
        uint32_t dc[NACC];
#pragma unroll
        for (int L = 0; L < NACC; ++L) dc[L] = tmem + (uint32_t)((bf * NACC + L) * N);
        const int ns = min(CH_STAGES, it.nst - c0);
        if (!wait(fullB(sb), useb) || !wait(fullA(sa), usea)) { ok = false; break; }
        // the next stage is waited for between the halves of this one's MMAs
        for (int s = 0; s < ns; ++s) {
          tc_fence_after();
          const uint32_t aT = tmemA + (uint32_t)(sa * A_COLS);
          const uint64_t bd0 = tc_sdesc64(sB0 + (uint32_t)(sb >> 1) * C::b_atom + 32u * (sb & 1));
          uint64_t bd[NSL];
#pragma unroll
          for (int j = 0; j < NSL; ++j) bd[j] = bd0 + (uint64_t)(j * (C::b_slice >> 4));
          const bool last = s == ns - 1;
          if (tc_elect()) tc_issue_half<0>(s == 0, dc, aT, bd, idesc);
          __syncwarp();
          const uint32_t eA = emptyA(sa), eB = emptyB(sb);
          if (++sa == SA) { sa = 0; ++usea; }
          if (++sb == SBH) { sb = 0; ++useb; }
          if (!last && (!wait(fullB(sb), useb) || !wait(fullA(sa), usea))) ok = false;
          if (tc_elect()) {
            tc_issue_half<1>(s == 0, dc, aT, bd, idesc);
            tc_commit(eA);
            tc_commit(eB);
            if (last) tc_commit(tfull(bf));
          }
          __syncwarp();
          if (!ok) break;
        }
        if (++bf == nbuf) { bf = 0; ++used; }
      }
    }
    if (!ok && lane == 0) note(err, vfail, 64);
    // every issued MMA complete before TMEM is released
    if (tc_elect()) tc_commit(drain);
    tc_mbar_wait(drain, 0, nullptr);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(512u) : "memory");
}

// columns per tile for `rows` of the N operand, each taking `per` columns
int cols_for(int rows, int per) {
  const int most = 64 / per, nt = (rows + most - 1) / most;
  return ((rows + nt - 1) / nt * per + 15) / 16 * 16;
}
// relative MMA time of a stage: tiles x columns (an MMA of 16 columns takes as long as one of 32)
long stage_cost(int mtiles, int ntiles, int N) { return (long)mtiles * ntiles * std::max(N, 32); }

}  // namespace

// ------------------------------------------------------------------ host side
int gemm_fwd_sl64_nrange(int Nm) { return (Nm + RANGE - 1) / RANGE; }

static int fwd_nbp(int Nm) { return ((Nm + 31) / 32 + 15) / 16 * 16; }
static size_t up16(size_t n) { return (n + 15) / 16 * 16; }
// a map's tables: row exponents, then (16-byte aligned) the guard's block minima
size_t fwd_exp64_bytes(int Nf, int Nr, int Nm) {
  return up16((size_t)Nf * gemm_fwd_sl64_nrange(Nm) * Nr) + (size_t)Nf * Nr * fwd_nbp(Nm) * sizeof(uint16_t);
}
static const uint16_t *fwd_low(const int8_t *ef, int Nf, int Nr, int Nm) {
  return reinterpret_cast<const uint16_t *>(ef + up16((size_t)Nf * gemm_fwd_sl64_nrange(Nm) * Nr));
}
cudaError_t launch_fwd_exp64(const void *F, int8_t *ef, int Nf, int Nr, int Nm, int row0, int nrows,
                             cudaStream_t s) {
  if (nrows <= 0) return cudaSuccess;
  const int nbp = fwd_nbp(Nm);
  k_row_scan<true><<<dim3(Nf, nrows, gemm_fwd_sl64_nrange(Nm)), 256, 0, s>>>(reinterpret_cast<const float4 *>(F) + (size_t)row0 * Nm,
                                                   (long)Nr * Nm, Nm, Nm, ef + row0, Nr,
                                                   const_cast<uint16_t *>(fwd_low(ef, Nf, Nr, Nm)) + (size_t)row0 * nbp, nbp,
                                                   nullptr);
  count_launches(1);
  return cudaGetLastError();
}

// per call: open frequencies, exponents and block sums of X^, magnitude sums
size_t gemm_fwd_sl64_ws_bytes(int Nf, int Nr, int Nm, int B) {
  const size_t nr = gemm_fwd_sl64_nrange(Nm);
  return up16((size_t)Nf * sizeof(int)) + up16(Nf * nr * B) + (size_t)Nf * B * fwd_nbp(Nm) * sizeof(uint16_t) +
         (size_t)Nf * Nr * B * sizeof(unsigned long long);
}

// Yo[b][w][r] for b < B; ef: launch_fwd_exp64; ws: gemm_fwd_sl64_ws_bytes(B).
// bmax (the reserved batch) fixes which operand takes the MMA rows, so that a
// column's rounding does not depend on its batch
cudaError_t launch_gemm_fwd_sl64(const void *F, const int8_t *ef, const cdd *X, long x_bstride, void *ws,
                                 size_t ws_bytes, cdd *part, cdd *Yo, long y_bstride, int Nf, int Nr, int Nm, int B,
                                 int bmax, int *err, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  if (gemm_fwd_sl64_ws_bytes(Nf, Nr, Nm, B) > ws_bytes) return cudaErrorInvalidValue;
  const float4 *Xp = reinterpret_cast<const float4 *>(X), *Fp = reinterpret_cast<const float4 *>(F);
  const int nbp = fwd_nbp(Nm), nr = gemm_fwd_sl64_nrange(Nm);
  uint8_t *wp = reinterpret_cast<uint8_t *>(ws);
  int *open = reinterpret_cast<int *>(wp);
  int8_t *ex = reinterpret_cast<int8_t *>(wp += up16((size_t)Nf * sizeof(int)));
  uint16_t *xsum = reinterpret_cast<uint16_t *>(wp += up16((size_t)Nf * nr * B));
  unsigned long long *Sq = reinterpret_cast<unsigned long long *>(wp + (size_t)Nf * B * nbp * sizeof(uint16_t));
  k_row_scan<false><<<dim3(Nf, B, nr), 256, 0, s>>>(Xp, Nm, x_bstride, Nm, ex, B, xsum, nbp, open);
  k_fwd_check<<<dim3((Nr + 15) / 16, Nf, (B + 63) / 64), 256, 0, s>>>(ef, fwd_low(ef, Nf, Nr, Nm), ex, xsum, nbp, nr, Nr,
                                                                     Nm, B, open, Sq);
  count_launches(2);
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  auto plan = [&](bool xm, int b, int &nmt, int &nnt) {
    const int N = xm ? cols_for(Nr, 1) : cols_for(b, 2);
    nmt = xm ? (b + 63) / 64 : (Nr + 127) / 128;
    nnt = xm ? (Nr + N - 1) / N : (b + N / 2 - 1) / (N / 2);
    return N;
  };
  int m0, n0, m1, n1;
  const int Nx = plan(true, bmax, m0, n0), Nfm = plan(false, bmax, m1, n1);
  const bool xm = stage_cost(m0, n0, Nx) < stage_cost(m1, n1, Nfm);
  int nmt, nnt;
  const int N = plan(xm, B, nmt, nnt);
  const long T = (long)nmt * nnt * nr * Nf;
  const unsigned grid = (unsigned)std::max<long>(1, std::min<long>(T, nsm));
  auto run = [&](auto NC, auto XC) {
    constexpr int NN = NC.value;
    constexpr bool XM = XC.value;
    constexpr size_t sm = Cfg<NN, XM>::smem;
    cudaFuncSetAttribute(k_gemm_fwd_sl64<NN, XM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_gemm_fwd_sl64<NN, XM><<<grid, NTHR, sm, s>>>(Fp, ef, Xp, x_bstride, ex, reinterpret_cast<float2 *>(part), nr,
                                                   Nf, Nr, Nm, B, nmt, nnt, err);
  };
  auto pick = [&](auto XC) {
    switch (N) {
      case 16: run(std::integral_constant<int, 16>{}, XC); break;
      case 32: run(std::integral_constant<int, 32>{}, XC); break;
      case 48: run(std::integral_constant<int, 48>{}, XC); break;
      default: run(std::integral_constant<int, 64>{}, XC); break;
    }
  };
  if (xm) pick(std::true_type{});
  else pick(std::false_type{});
  const int nrt = (Nr + 31) / 32, nbt = (B + 31) / 32;
  k_fwd_mag<<<dim3(nrt * nbt * ((Nm + SUB - 1) / SUB), Nf), 256, 0, s>>>(Fp, Xp, x_bstride, ef, ex, open, nrt, nbt, nr,
                                                                        Nr, Nm, B, Sq);
  k_fwd_join<<<(unsigned)(((long)B * Nf * Nr + 255) / 256), 256, 0, s>>>(part, reinterpret_cast<const cdd *>(F), X,
                                                                        x_bstride, open, Sq, Yo, y_bstride, nr, Nf,
                                                                        Nr, Nm, B);
  count_launches(3);
  return cudaGetLastError();
}

}  // namespace tw
