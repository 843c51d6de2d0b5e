// gemm_sl.cu -- the reduced-precision adjoint product on the 5th-generation
// tensor cores, with both operands cut into exact fixed-point bf16 slices.
//
// Per frequency w the adjoint of a Toeplitz map is a complex product
//   X^(w) = F^(w)^H Y^(w)          (Nm x Nr) (Nr x B)
// (Sec. "FFT-based Hessian matvecs": the circulant embedding makes the map
// block diagonal in frequency).  With F^ = Ar + i Ai and Y = Yr + i Yi,
//   Xr = Ar^T Yr + Ai^T Yi,   Xi = Ar^T Yi - Ai^T Yr,
// one real product D = A' B'^T with K' = 2 Nr:
//   A'[m][2s] = Ar[s][m],  A'[m][2s+1] = Ai[s][m]                 (M: grid points)
//   B'[b][2s] = Yr[s][b],  B'[b][2s+1] = Yi[s][b]      -> D[m][b]      = Xr
//   B'[P+b][2s] = Yi[s][b], B'[P+b][2s+1] = -Yr[s][b]  -> D[m][P+b]    = Xi
// (P right-hand sides per tile, N = 2P columns).
//
// Accuracy.  F^T y cancels strongly (y = K^-1 d is large against m), so the
// sum has to be formed well below FP32 rounding of its terms, or the
// posterior mean and, through F_q's own cancellation, the forecast lose
// digits.  The tensor cores multiply bf16 exactly, but accumulate in FP32,
// which rounds at the running sum.  So each row m of A' (over all K') and
// each column of B' is scaled by a power of two to (-1, 1) and written in
// fixed point as four 8-bit integer slices (round to nearest at each step):
//   v = 2^(e-7) (s0 + s1/2^8 + s2/2^16 + s3/2^24),  |s_i| <= 128,
// (31 bits for the operator, an exact representation of every complex64 or
// bf16 hi+lo entry within 2^8 of its row maximum; the data side is cut from
// its double-float spectrum).  Every slice is an integer of at most 8
// significant bits, exact in bf16, so the products s_i t_j are integers of
// at most 2^14 and their sum over K' <= 1024 terms stays below 2^24: the
// leading level (s0 t0) accumulates EXACTLY in an FP32 accumulator D0, and
// the cancellation happens in exact arithmetic.  With slices pre-scaled by
// 2^-8i and 2^-8j, level 1 (s0 t1 + s1 t0, multiples of 2^-8 below 2^16 for
// K' <= 512) is exact in its own accumulator D1 as well.  Levels 2 and 3 go
// to D2, 2^-16 below the leading level; levels >= 4 are dropped (2^-32 of a
// term).  The separate exact D1 matters: the tensor cores truncate when they
// accumulate in FP32, and a truncated level-1 sum leaves a biased, spatially
// smooth error that the prior filter amplifies (measured: 13x the posterior
// mean's error of round-to-nearest); in D2 that bias is 2^8 smaller.  The
// result is
//   X = 2^(ea + eb - 14) ((D0 + D1) + D2),
// within a few units of 2^-30 of the terms: the error left is the rounding
// of the stored operator itself.  Ten MMAs per 16-wide k step.
//
// Kernel: persistent, one CTA per SM over (right-hand-side tile, 128 grid
// points, frequency), right-hand-side tile fastest.  Warps 0-7 and 8-15 stream
// the operator (complex64 or bf16 hi+lo, cp.async), slice it with its row's
// exponent and store alternate 16-wide A' stages to TMEM, from where the MMAs
// read them; warps 16-23 drain the accumulators; warp 24 issues the MMAs (one
// elected lane); warp 25 copies the B' slices (prepared once per call by
// k_bsl_build, cp.async.bulk).  TMEM: D0, D1, D2 of N columns, twice when that
// leaves two A' stages (N <= 72), the rest A' stages of 4 x 8 columns (N <=
// 144).  With A' in shared memory an MMA of N <= 32 took 40 cycles (A's 4 KB at
// 128 bytes a clock) against 16, eight producer warps were what bounded the
// small batches, and one warp a TMEM quarter the large ones' drain: 64
// right-hand sides of the 100-sensor case 10.0 -> 8.0 ms, 16 of the 200-sensor
// serving case 3.29 -> 3.10 ms.  Every
// wait is bounded: on expiry the kernel records TW_ERR_TIMEOUT, lets its
// copies and MMAs drain (bounded), frees TMEM and returns.
#include <stdint.h>

#include <algorithm>
#include <utility>

#include "../../include/tw.h"
#include "kernels.h"
#include "tc.cuh"

namespace tw {

namespace {

constexpr int TM = 128;                  // MMA M: grid points per tile
constexpr int KA = 32;                   // K' per B' atom: 16 rows (sensors) x (re, im)
constexpr int NSL = 4;                   // slices per operand
constexpr int A_COLS = NSL * 8;          // TMEM columns of a 16-wide A' stage
constexpr int NGRP = 256, NPROD = 2 * NGRP, NEPI = 256;
constexpr int NTHR = NPROD + NEPI + 64;
constexpr int MAXA = 4, SB = 4;          // A' stages (at most), B' stages
constexpr int RAW_D = 3;                 // operator atoms in shared memory (raw ring)
constexpr int RAW_SLOT = NPROD * 4 * 8;  // 16 KB: 16 rows x 128 grid points
constexpr int EXP_MIN = -100, EXP_MAX = 120;
constexpr int SL_PMAX = 72;              // right-hand sides per tile: 3 x 2P columns leave two A' stages

// round to the nearest integer (ties to even), |v| < 2^22
__device__ __forceinline__ float rnd_int(float v) {
  return __fsub_rn(__fadd_rn(v, 12582912.0f), 12582912.0f);
}
// smallest e with |v| < 2^e for the largest |v| = mx >= 0, clamped
__device__ __forceinline__ int exp_above(float mx) {
  if (!(mx > 0.f)) return EXP_MIN;
  const int E = (int)((__float_as_uint(mx) >> 23) & 0xffu);
  const int e = E - 126;
  return e < EXP_MIN ? EXP_MIN : (e > EXP_MAX ? EXP_MAX : e);
}

__device__ __forceinline__ float bf16lo(unsigned w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(unsigned w) { return __uint_as_float(w & 0xffff0000u); }

// operator entry (exact FP32 values) of the complex64 or bf16 hi+lo storage
template <int FMT> __device__ __forceinline__ float2 ld_entry(const void *A, size_t i);
template <> __device__ __forceinline__ float2 ld_entry<FMT_C64>(const void *A, size_t i) {
  return __ldcs(reinterpret_cast<const float2 *>(A) + i);
}
template <> __device__ __forceinline__ float2 ld_entry<FMT_BF16X2>(const void *A, size_t i) {
  const uint2 v = __ldcs(reinterpret_cast<const uint2 *>(A) + i);
  return make_float2(bf16lo(v.x) + bf16hi(v.x), bf16lo(v.y) + bf16hi(v.y));
}

// ------------------------------------------------------ row exponents
// ea[w][m] = smallest e with |Re|, |Im| of F^(w)[s][m] < 2^e for every row s
template <int FMT>
__global__ void k_row_exp(const void *__restrict__ A, int8_t *__restrict__ ea, int Nf, int Nr, int Nm) {
  const long total = (long)Nf * Nm;
  for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long)gridDim.x * blockDim.x) {
    const long w = idx / Nm, m = idx % Nm;
    float mx = 0.f;
    for (int s = 0; s < Nr; ++s) {
      const float2 v = ld_entry<FMT>(A, ((size_t)w * Nr + s) * Nm + m);
      mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    ea[idx] = (int8_t)exp_above(mx);
  }
}

// ------------------------------------------------------ B' slices
// tiles [w][nt][atom][slice][2P rows][32 bf16] (64-byte swizzle), eb[w][nt*P + b]
__global__ void __launch_bounds__(256)
k_bsl_build(const cdd *__restrict__ Y, long y_bstride, int Nr, int B, int P, int natoms,
            uint8_t *__restrict__ tiles, int *__restrict__ eb, int ntiles) {
  __shared__ int e_sh[SL_PMAX];
  const int w = blockIdx.x, nt = blockIdx.y;
  const int N = 2 * P;
  for (int bl = threadIdx.x; bl < P; bl += blockDim.x) {
    const int b = nt * P + bl;
    float mx = 0.f;
    if (b < B) {
      const cdd *y = Y + (size_t)b * y_bstride + (size_t)w * Nr;
      for (int s = 0; s < Nr; ++s) {
        const cdd v = ld_cdd(y + s);
        mx = fmaxf(mx, fmaxf(fabsf(v.re.hi), fabsf(v.im.hi)));
      }
    }
    // the low halves may lift |y| past the high half's bound by one unit in
    // the last place: bound the sum instead
    const int e = exp_above(mx * (1.0f + 1.0f / 1048576.0f));
    e_sh[bl] = e;
    eb[(size_t)w * ntiles * P + b] = e;
  }
  __syncthreads();
  const size_t slice_bytes = (size_t)N * 64;
  uint8_t *base = tiles + ((size_t)w * ntiles + nt) * natoms * NSL * slice_bytes;
  const int tasks = natoms * N * 4;
  for (int t = threadIdx.x; t < tasks; t += blockDim.x) {
    const int a = t / (N * 4), rem = t % (N * 4);
    const int n = rem >> 2, q = rem & 3;
    const int part = n >= P, bl = n - part * P, b = nt * P + bl;
    const float sc = tc_pow2f(7 - e_sh[bl]);
    uint32_t wd[NSL][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int s = 16 * a + 4 * q + u;
      cdd y = cdd_zero();
      if (b < B && s < Nr) y = ld_cdd(Y + (size_t)b * y_bstride + (size_t)w * Nr + s);
      // the two reals of this row: (yr, yi) for the real-part column, (yi, -yr) for the imaginary
      dd v[2];
      v[0] = part ? y.im : y.re;
      v[1] = part ? dd_neg(y.re) : y.im;
      float sl[2][NSL];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float hi = v[c].hi * sc, lo = v[c].lo * sc;   // exact: power-of-two scaling
#pragma unroll
        for (int i = 0; i < NSL; ++i) {
          const float si = rnd_int(hi);
          sl[c][i] = si * tc_pow2f(-8 * i);
          if (i + 1 < NSL) {
            float r, e;
            two_sum(__fsub_rn(hi, si), lo, r, e);      // hi - si is exact
            hi = r * 256.f;
            lo = e * 256.f;
          }
        }
      }
#pragma unroll
      for (int i = 0; i < NSL; ++i) wd[i][u] = tc_pack_bf16(sl[0][i], sl[1][i]);
    }
    uint8_t *at = base + (size_t)a * NSL * slice_bytes;
#pragma unroll
    for (int i = 0; i < NSL; ++i)
      *reinterpret_cast<uint4 *>(at + i * slice_bytes + tc_swz64(n, q)) =
          make_uint4(wd[i][0], wd[i][1], wd[i][2], wd[i][3]);
  }
}

// ------------------------------------------------------------------ the product
// pair p = 0..9 of slices (i, j), level L = i + j: p = 0 is level 0 (into
// D0), p = 1, 2 level 1 (into D1), p = 3..9 levels 2 and 3 (into D2)
template <int PR>
__device__ __forceinline__ void issue_pair(bool first, const uint32_t *d, uint32_t a, const uint64_t *b,
                                           uint32_t idesc) {
  constexpr int L = tc_pair_level(PR), si = PR - L * (L + 1) / 2, sj = L - si, ac = L < 2 ? L : 2;
  // the first MMA of a tile into each accumulator (pairs 0, 1, 3) overwrites it
  tc_mma_ts(d[ac], a + 8u * si, b[sj], idesc, first && si == 0 && L < 3 ? 0u : 1u);
}
template <int P0, int... PR>
__device__ __forceinline__ void issue_pairs(std::integer_sequence<int, PR...>, bool first, const uint32_t *d,
                                            uint32_t a, const uint64_t *b, uint32_t idesc) {
  (issue_pair<P0 + PR>(first, d, a, b, idesc), ...);
}

// the exact FP32 value of an operator entry held as 8 raw bytes
template <int FMT> __device__ __forceinline__ float2 decode_entry(uint2 v);
template <> __device__ __forceinline__ float2 decode_entry<FMT_C64>(uint2 v) {
  return make_float2(__uint_as_float(v.x), __uint_as_float(v.y));
}
template <> __device__ __forceinline__ float2 decode_entry<FMT_BF16X2>(uint2 v) {
  return make_float2(bf16lo(v.x) + bf16hi(v.x), bf16lo(v.y) + bf16hi(v.y));
}

__device__ __forceinline__ void note(int *err, volatile int *fail, int info) {
  if (!*fail && atomicCAS(err, 0, TW_ERR_TIMEOUT) == 0) err[1] = info;
  *fail = 1;
}

template <int FMT>
__global__ void __launch_bounds__(NTHR, 1)
k_gemm_adj_sl(const uint2 *__restrict__ A, const int8_t *__restrict__ ea, const uint8_t *__restrict__ Bt,
              const int *__restrict__ eb, cf *__restrict__ X, long x_bstride, int B, int P, int ntiles,
              int Nr, int Nm, int Nf, int natoms, int SA, int nbuf, int *err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * MAXA + 2 * SB + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int N = 2 * P;
  const int nmt = (Nm + TM - 1) / TM;
  const int T = nmt * Nf * ntiles;
  const int my_tiles = (int)blockIdx.x < T ? (T - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const uint32_t b_slice = (uint32_t)N * 64u, b_stage = NSL * b_slice;
  const uint32_t sB0 = (tc_su32(smem_raw) + 1023u) & ~1023u, sRaw = sB0 + (uint32_t)SB * b_stage;
  const uint32_t bar0 = tc_su32(&bars[0]);
  auto fullA = [&](int st) { return bar0 + 8u * st; };
  auto emptyA = [&](int st) { return bar0 + 8u * (MAXA + st); };
  auto fullB = [&](int st) { return bar0 + 8u * (2 * MAXA + st); };
  auto emptyB = [&](int st) { return bar0 + 8u * (2 * MAXA + SB + st); };
  auto tfull = [&](int bf) { return bar0 + 8u * (2 * MAXA + 2 * SB + bf); };
  auto tempty = [&](int bf) { return bar0 + 8u * (2 * MAXA + 2 * SB + 2 + bf); };
  const uint32_t drain = bar0 + 8u * (2 * MAXA + 2 * SB + 4);
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
    for (int st = 0; st < SB; ++st) {
      tc_mbar_init(fullB(st), 1);
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
  const uint32_t tmemA = tmem + (uint32_t)(nbuf * 3 * N);
  volatile int *vfail = &fail;
  auto tile_of = [&](int i, int &mt, int &w, int &nt) {
    const int t = (int)blockIdx.x + i * (int)gridDim.x;
    nt = t % ntiles;
    const int q = t / ntiles;
    mt = q % nmt;
    w = q / nmt;
  };

  if (warp < NPROD / 32) {
    // ---------------- producers: A' slices into TMEM.  Group g (8 warps) fills
    // every atom's stage g; thread = grid point r, rows 4h .. 4h+3 of the
    // stage's 8; its loads run RAW_D - 1 atoms ahead
    const int r = tid & (TM - 1), h = (tid >> 7) & 1, g = tid / NGRP;
    int ii = 0, ia = 0, islot = 0;
    const uint2 *ip = A;
    bool ivalid = false;
    auto set_issue_tile = [&]() {
      ivalid = false;
      if (ii >= my_tiles) return;
      int mt, w, nt;
      tile_of(ii, mt, w, nt);
      const int m = mt * TM + r;
      ivalid = m < Nm;
      ip = A + ((size_t)w * Nr + 8 * g + 4 * h) * Nm + (ivalid ? m : 0);
    };
    // raw ring: slot, entry u, producer thread (each thread reads only what it copied)
    const uint32_t raw0 = sRaw + 8u * tid;
    const uint8_t *rawp = smem_raw + (raw0 - tc_su32(smem_raw));
    auto load = [&]() {
      if (ii < my_tiles) {
        const int s0 = 16 * ia + 8 * g + 4 * h;
        const uint2 *p = ip + (size_t)(16 * ia) * Nm;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = ivalid && s0 + u < Nr;
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;"
                       ::"r"(raw0 + (uint32_t)(islot * RAW_SLOT + u * NPROD * 8)),
                         "l"(in ? p + (size_t)u * Nm : A), "r"(in ? 8 : 0) : "memory");
        }
        if (++ia == natoms) { ia = 0; ++ii; set_issue_tile(); }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (++islot == RAW_D) islot = 0;
    };
    auto row_scale_exp = [&](int i) {
      if (i >= my_tiles) return EXP_MIN;
      int mt, w, nt;
      tile_of(i, mt, w, nt);
      const int m = mt * TM + r;
      return m < Nm ? (int)ea[(size_t)w * Nm + m] : EXP_MIN;
    };
    set_issue_tile();
#pragma unroll
    for (int d = 0; d < RAW_D - 1; ++d) load();
    int slot = 0;
    int e_next = row_scale_exp(0);
    bool ok = true;
    const uint32_t lane_base = tmemA + ((uint32_t)(32 * (warp & 3)) << 16) + 4u * h;
    // the stages of the groups alternate; an atom whose second half holds no
    // rows (the last, for some Nr) has one
    const bool odd = 16 * (natoms - 1) + 8 >= Nr;
    int st = g, use = 0;
    auto step = [&](int n) {
      st += n;
      while (st >= SA) { st -= SA; ++use; }
    };
    for (int i = 0; i < my_tiles && ok; ++i) {
      const float sc1 = tc_pow2f(7 - e_next);
      const f2 sc = f2_make(sc1, sc1);
      e_next = row_scale_exp(i + 1);
      for (int a = 0; a < natoms; ++a) {
        asm volatile("cp.async.wait_group %0;" ::"n"(RAW_D - 2) : "memory");
        f2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 e = decode_entry<FMT>(
              *reinterpret_cast<const uint2 *>(rawp + slot * RAW_SLOT + u * NPROD * 8));
          v[u] = mul2(f2_make(e.x, e.y), sc);
        }
        if (++slot == RAW_D) slot = 0;
        load();
        const bool last_half = odd && a == natoms - 1;      // this atom has the first stage only
        if (use > 0) {
          const bool got = tc_mbar_wait(emptyA(st), (unsigned)((use - 1) & 1), vfail);
          if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) note(err, vfail, 21);
            ok = false;
            break;
          }
        }
        // (group 1 waits for the stage that it leaves to the next tile as well: a
        // jump of three stages could meet its next stage a whole phase early)
        if (last_half && g == 1) { step(1); continue; }
        tc_fence_after();
        // slice i = v rounded to the grid 2^-8i (v - slices so far, exact):
        // (x + 1.5 2^(23-8i)) - 1.5 2^(23-8i) rounds x to a multiple of 2^-8i
        const uint32_t at = lane_base + (uint32_t)(st * A_COLS);
#pragma unroll
        for (int il = 0; il < NSL; ++il) {
          const float m = tc_pow2f(23 - 8 * il) * 1.5f;
          const f2 M = f2_make(m, m);
          uint32_t wd[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const f2 s = sub2(add2(v[u], M), M);
            const float2 sv = f2_split(s);
            wd[u] = tc_pack_bf16(sv.x, sv.y);
            if (il + 1 < NSL) v[u] = sub2(v[u], s);
          }
          tc_st4(at + 8u * il, wd);
        }
        tc_wait_st();
        tc_fence_before();
        tc_mbar_arrive(fullA(st));
        step(last_half ? 1 : 2);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // own copies drained before exit
  } else if (warp < (NPROD + NEPI) / 32) {
    // ---------------- epilogue: (D0 + D1) + D2 from TMEM, scaled, complex64 out
    // (two warps a TMEM lane quarter, each half of the columns)
    const int lg = warp & 3, half = (warp - NPROD / 32) >> 2;
    const int r = 32 * lg + lane;
    const int CW = P / 2;
    bool ok = true;
    int bf = 0, use = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int mt, w, nt;
      tile_of(i, mt, w, nt);
      const int m = mt * TM + r;
      const float sa = tc_pow2f((m < Nm ? (int)ea[(size_t)w * Nm + m] : EXP_MIN) - 7);
      const int b0 = nt * P + half * CW;
      const int *ebw = eb + (size_t)w * ntiles * P + b0;
      cf *xp = X + (size_t)b0 * x_bstride + (size_t)w * Nm + m;
      const bool got = tc_mbar_wait(tfull(bf), (unsigned)(use & 1), vfail);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0) note(err, vfail, 22);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t trow = tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)(bf * 3 * N + half * CW);
#pragma unroll 1
      for (int c0 = 0; c0 < CW; c0 += 4) {
        uint32_t dr[3][4], di[3][4];
#pragma unroll
        for (int L = 0; L < 3; ++L) {
          tc_ld4(dr[L], trow + (uint32_t)(L * N + c0));
          tc_ld4(di[L], trow + (uint32_t)(L * N + P + c0));
        }
        tc_wait_ld();
        if (c0 + 4 >= CW) {
          // the buffer is read: the MMAs of a later tile may overwrite it
          tc_fence_before();
          tc_mbar_arrive(tempty(bf));
        }
        if (m < Nm) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (b0 + c0 + j >= B) continue;
            const float sb = tc_pow2f(ebw[c0 + j] - 7);
            const float re = __fadd_rn(__fadd_rn(__uint_as_float(dr[0][j]), __uint_as_float(dr[1][j])),
                                       __uint_as_float(dr[2][j])) * sa * sb;
            const float im = __fadd_rn(__fadd_rn(__uint_as_float(di[0][j]), __uint_as_float(di[1][j])),
                                       __uint_as_float(di[2][j])) * sa * sb;
            xp[(size_t)(c0 + j) * x_bstride] = cf_make(re, im);
          }
        }
      }
      if (++bf == nbuf) { bf = 0; ++use; }
    }
  } else if (warp == (NPROD + NEPI) / 32) {
    // ---------------- MMA issuer (the warp's lanes run together, one is elected to issue)
    const uint32_t idesc = tc_idesc_bf16(TM, N);
    auto wait = [&](uint32_t bar, int parity) {
      return __all_sync(0xffffffffu, tc_mbar_wait(bar, (unsigned)(parity & 1), vfail)) != 0;
    };
    bool ok = true;
    int sa = 0, usea = 0, sb = 0, useb = 0, bf = 0, used = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      // the epilogue has read this buffer's previous tile
      if (used > 0 && !wait(tempty(bf), used - 1)) { ok = false; break; }
      tc_fence_after();
      uint32_t dc[3];
#pragma unroll
      for (int L = 0; L < 3; ++L) dc[L] = tmem + (uint32_t)((bf * 3 + L) * N);
      if (!wait(fullB(sb), useb) || !wait(fullA(sa), usea)) { ok = false; break; }
      // stages of 8 rows; an atom's B' serves two.  The next stage is waited
      // for between the halves of this one's MMAs
      for (int s = 0; s < Nr; s += 8) {
        const int ks = (s >> 3) & 1;
        tc_fence_after();
        const uint32_t aT = tmemA + (uint32_t)(sa * A_COLS);
        const uint64_t bd0 = tc_sdesc64(sB0 + (uint32_t)sb * b_stage + 32u * ks);
        uint64_t bd[NSL];
#pragma unroll
        for (int j = 0; j < NSL; ++j) bd[j] = bd0 + (uint64_t)(j * (b_slice >> 4));
        const bool last = s + 8 >= Nr, b_done = ks == 1 || last;
        if (tc_elect()) issue_pairs<0>(std::make_integer_sequence<int, 5>{}, s == 0, dc, aT, bd, idesc);
        __syncwarp();
        const uint32_t eA = emptyA(sa), eB = emptyB(sb);
        if (++sa == SA) { sa = 0; ++usea; }
        if (b_done && ++sb == SB) { sb = 0; ++useb; }
        if (!last && ((b_done && !wait(fullB(sb), useb)) || !wait(fullA(sa), usea))) ok = false;
        if (tc_elect()) {
          issue_pairs<5>(std::make_integer_sequence<int, 5>{}, s == 0, dc, aT, bd, idesc);
          tc_commit(eA);
          if (b_done) tc_commit(eB);
          if (last) tc_commit(tfull(bf));
        }
        __syncwarp();
        if (!ok) break;
      }
      if (++bf == nbuf) { bf = 0; ++used; }
    }
    if (!ok && lane == 0) note(err, vfail, 23);
    // every issued MMA complete before TMEM is released
    if (tc_elect()) tc_commit(drain);
    tc_mbar_wait(drain, 0, nullptr);
  } else if (lane == 0) {
    // ---------------- B' slices: one bulk copy per atom
    int st = 0, use = 0, issued = 0;
    bool ok = true;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int mt, w, nt;
      tile_of(i, mt, w, nt);
      const uint8_t *Bw = Bt + ((size_t)w * ntiles + nt) * natoms * b_stage;
      for (int a = 0; a < natoms; ++a) {
        if (use > 0 && !tc_mbar_wait(emptyB(st), (unsigned)((use - 1) & 1), vfail)) { ok = false; break; }
        tc_mbar_arrive_tx(fullB(st), b_stage);
        tc_bulk_g2s(sB0 + (uint32_t)st * b_stage, Bw + (size_t)a * b_stage, b_stage, fullB(st));
        ++issued;
        if (++st == SB) { st = 0; ++use; }
      }
    }
    if (!ok) note(err, vfail, 24);
    // copies already issued must land before the CTA's shared memory goes
    for (int a = (issued > SB ? issued - SB : 0); a < issued; ++a)
      tc_mbar_wait(fullB(a % SB), (unsigned)((a / SB) & 1), nullptr);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(512u) : "memory");
}

}  // namespace

// ------------------------------------------------------------------ host side
int sl_natoms(int Nr) { return (Nr + KA / 2 - 1) / (KA / 2); }

size_t sl_ws_bytes(int Nf, int Nr, int bcols) {
  const int bc = (bcols + 7) / 8 * 8;
  return (size_t)Nf * sl_natoms(Nr) * NSL * 2 * (size_t)bc * 64;
}
size_t sl_eb_bytes(int Nf, int bcols) { return (size_t)Nf * ((bcols + 7) / 8 * 8) * sizeof(int); }

int sl_pick_tile(int B) {
  // right-hand sides per tile: one tile up to 72 (N = 144 columns, three
  // accumulators in 432 TMEM columns), else the fewest tiles of a multiple of 8
  const int P8 = (B + 7) / 8 * 8;
  if (P8 <= SL_PMAX) return P8;
  const int nt = (P8 + SL_PMAX - 1) / SL_PMAX;
  return ((P8 + nt - 1) / nt + 7) / 8 * 8;
}

cudaError_t launch_row_exp(const void *A, int fmt, int8_t *ea, int Nf, int Nr, int Nm, cudaStream_t s) {
  const long total = (long)Nf * Nm;
  long blocks = (total + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (fmt == FMT_C64)
    k_row_exp<FMT_C64><<<(unsigned)blocks, 256, 0, s>>>(A, ea, Nf, Nr, Nm);
  else if (fmt == FMT_BF16X2)
    k_row_exp<FMT_BF16X2><<<(unsigned)blocks, 256, 0, s>>>(A, ea, Nf, Nr, Nm);
  else
    return cudaErrorInvalidValue;
  count_launches(1);
  return cudaGetLastError();
}

// X[b][w][k] = sum_s conj(A[w][s][k]) Y[b][w][s] for b < B; P right-hand
// sides per tile (0: pick); ws: B' tiles of >= sl_ws_bytes(Nf, Nr, ntiles P)
cudaError_t launch_gemm_adj_sl(const void *A, int fmt, const int8_t *ea, const cdd *Y, long y_bstride,
                               cf *X, long x_bstride, int Nf, int Nr, int Nm, int B, int P,
                               void *ws, size_t ws_bytes, int *eb, size_t eb_bytes, int *err,
                               cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  if (Nr > 512 || (fmt != FMT_C64 && fmt != FMT_BF16X2)) return cudaErrorInvalidValue;
  if (P <= 0) P = sl_pick_tile(B);
  if (P % 8 != 0 || P > 80) return cudaErrorInvalidValue;
  P = P > SL_PMAX ? SL_PMAX : P;
  const int ntiles = (B + P - 1) / P, natoms = sl_natoms(Nr), N = 2 * P;
  if (sl_ws_bytes(Nf, Nr, ntiles * P) > ws_bytes || (size_t)Nf * ntiles * P * sizeof(int) > eb_bytes)
    return cudaErrorInvalidValue;
  k_bsl_build<<<dim3(Nf, ntiles), 256, 0, s>>>(Y, y_bstride, Nr, B, P, natoms,
                                               reinterpret_cast<uint8_t *>(ws), eb, ntiles);
  count_launches(1);
  // TMEM: three accumulators of N columns, twice if that leaves two A' stages,
  // the rest A' stages
  const int nbuf = 6 * N + 2 * A_COLS <= 512 ? 2 : 1;
  const int SA = std::min(MAXA, (512 - nbuf * 3 * N) / A_COLS);
  const size_t sm = 1024 + (size_t)RAW_D * RAW_SLOT + (size_t)SB * NSL * N * 64;
  // persistent: one CTA per SM (the registers allow no second one)
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const long tiles = (long)((Nm + TM - 1) / TM) * Nf * ntiles;
  const unsigned grid = (unsigned)(tiles < nsm ? tiles : (nsm > 0 ? nsm : 1));
  auto run = [&](auto *k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k<<<grid, NTHR, sm, s>>>(reinterpret_cast<const uint2 *>(A), ea, reinterpret_cast<const uint8_t *>(ws), eb, X,
                             x_bstride, B, P, ntiles, Nr, Nm, Nf, natoms, SA, nbuf, err);
  };
  if (fmt == FMT_C64) run(k_gemm_adj_sl<FMT_C64>);
  else run(k_gemm_adj_sl<FMT_BF16X2>);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace tw
