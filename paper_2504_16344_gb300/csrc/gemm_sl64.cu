// gemm_sl64.cu -- the FP64-class batched adjoint product on the 5th-generation
// tensor cores, with both operands cut into seven exact bf16 slices.
//
// Per frequency w the adjoint of a Toeplitz map is the complex product
//   X^(w) = F^(w)^H Y^(w)          (Nm x Nr) (Nr x B)
// (Sec. "FFT-based Hessian matvecs"), laid out as one real product
// D = A' B'^T with K' = 2 Nr exactly as in gemm_sl.cu:
//   A'[m][2s], A'[m][2s+1] = Re, Im F^[s][m]
//   B'[b] = (Yr, Yi) -> Xr,   B'[P + b] = (Yi, -Yr) -> Xi.
//
// Accuracy.  A row of A' (a grid point, over all Nr rows of F^) and a column
// of B' each get a power-of-two exponent, and every float pair is cut into
// seven 8-bit slices (tc.cuh: 56 bits below the row maximum; the pair holds 48
// of its own).  Slice products of levels L = i + j <= 6 are formed (28 MMAs
// per 16-wide k step, the dropped ones below 2^-54 of the row maxima).  The tensor
// cores accumulate in FP32 and truncate, so levels 0..4 have a TMEM
// accumulator each, in which every sum is exact: a level is a multiple of
// 2^-8L and at most (L+1) K' 2^14 2^-8L (one slice may reach 129: + 0.4%),
// below 2^24 units for K' <= 204.  Levels 5 and 6 share a sixth accumulator,
// 2^-40 below the terms, where truncation does no harm.  More than 102 rows
// are summed in chunks of 96 (K' = 192), added to X^ in double-float.  An entry
// 2^-p of its row's largest keeps 56 - p bits, so a sum whose large entries meet
// small ones would come out with fewer digits than in double-float, which rounds its
// running sum at 2^-48 after every one of the 2 Nr terms: those sums are found from
// their magnitudes and formed in double-float (k_adj_check, k_adj_guard).
//
// What bounds it.  The SIMT double-float product (gemm.cu) spends about 60
// FP32 operations per operator entry and right-hand side and is bound by the
// FP32 pipe; the 28 MMAs cost 28 x 4 bf16 multiply-adds there.  With both MMA
// operands in shared memory a 128 x 64 x 16 MMA would read 6 KB in the 32
// cycles its arithmetic takes (192 of the 128 bytes a clock that shared
// memory gives); so the A' slices, which are made in registers anyway, are
// stored to TMEM (tcgen05.st) and only B' is read from shared memory (64 bytes a
// clock).  TMEM holds the six accumulators of N = 2P <= 64 columns (384) and
// two to four 16-wide A' stages of 7 x 8 columns; for P <= 16 the accumulators
// are double-buffered as well.
// Measured (64 right-hand sides, 100 rows, 50,000 grid points, 401 frequencies):
// 25.1 ms (28.2 ms with scalar instead of packed slicing), against 246 ms for the SIMT product and 4.8 ms to read the operator;
// a stage takes 1,900 cycles where its MMAs need 900 (the accumulators are
// single-buffered at N = 64, so the MMAs of a tile wait for the drain of the
// one before).  Issuing the MMAs from one lane's branch instead of an elected
// lane of a converged warp: 43 ms.
//
// Kernel: persistent, one CTA per SM over (right-hand-side tile, 128 grid
// points, frequency), right-hand-side tile fastest: the CTAs running together
// read the same operator rows (from L2 for all but the first) and the same
// frequency's B' slices.  Warps 0-7 and 8-15 load the operator (two stages
// ahead), slice it and fill alternate A' stages; warps 16-23 drain the
// accumulators; warp 24 issues the MMAs; warp 25 copies B' slices
// (cp.async.bulk).  Every wait is bounded: on expiry the kernel records
// TW_ERR_TIMEOUT, lets its copies and MMAs drain (bounded), frees TMEM and
// returns.
#include <algorithm>

#include "../../include/tw.h"
#include "kernels.h"
#include "tc.cuh"

namespace tw {

namespace {

constexpr int TM = 128;                  // MMA M: grid points per tile
constexpr int KA = 32;                   // K' per B' atom: 16 rows x (re, im)
constexpr int NSL = TC_NSL, NACC = TC_NACC;
constexpr int EXACT_ROWS = 102;          // rows whose level sums stay exact
constexpr int CHUNK_ATOMS = 6;           // atoms per chunk beyond that (96 rows)
constexpr int A_COLS = NSL * 8;          // TMEM columns of a 16-wide A' stage
constexpr int NGRP = 256;                // producer threads of one group (8 warps)
constexpr int NPROD = 2 * NGRP, NEPI = 256;
constexpr int NTHR = NPROD + NEPI + 64;
constexpr int MAXA = 4, SB = 4;          // A' stages (at most), B' stages
constexpr int RAW_D = 3;                 // operator atoms in shared memory (raw ring)
constexpr int RAW_SLOT = NPROD * 4 * 16; // 32 KB: 16 rows x 128 grid points
constexpr int PMAX = 32;                 // right-hand sides per tile: 6 x 2P <= 384 TMEM columns

__device__ __forceinline__ void note(int *err, volatile int *fail, int info) {
  if (!*fail && atomicCAS(err, 0, TW_ERR_TIMEOUT) == 0) err[1] = info;
  *fail = 1;
}

// ea[w][m] = exponent of grid point m over the Nr rows of F^(w)
__global__ void k_row_exp64(const float4 *__restrict__ A, int8_t *__restrict__ ea, int Nf, int Nr, int Nm) {
  const long total = (long)Nf * Nm;
  for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long)gridDim.x * blockDim.x) {
    const float4 *p = A + (idx / Nm) * Nr * Nm + idx % Nm;
    float mx = 0.f;
    for (int s = 0; s < Nr; ++s) {
      const float4 v = __ldcs(p + (size_t)s * Nm);
      mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.z)));
    }
    ea[idx] = (int8_t)tc_exp_above(mx);
  }
}

// B' slices: tiles [w][nt][atom][slice][2P rows][32 bf16] (64-byte swizzle),
// column exponents eb[w][nt P + b], magnitudes mag[w][nt P + b][nrp] (bf16)
__global__ void __launch_bounds__(256)
k_bsl64_build(const cdd *__restrict__ Y, long y_bstride, int Nr, int B, int P, int natoms,
              uint8_t *__restrict__ tiles, int *__restrict__ eb, uint16_t *__restrict__ mag, int nrp, int *__restrict__ todo,
              int ntiles) {
  __shared__ int e_sh[PMAX];
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) todo[0] = 0;
  const int w = blockIdx.x, nt = blockIdx.y, N = 2 * P;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int bl = warp; bl < P; bl += 8) {
    const int b = nt * P + bl;
    float mx = 0.f;
    if (b < B)
      for (int s = lane; s < Nr; s += 32) {
        const cdd v = ld_cdd(Y + (size_t)b * y_bstride + (size_t)w * Nr + s);
        mx = fmaxf(mx, fmaxf(fabsf(v.re.hi), fabsf(v.im.hi)));
      }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
    if (lane == 0) {
      e_sh[bl] = tc_exp_above(mx);
      eb[(size_t)w * ntiles * P + b] = e_sh[bl];
    }
  }
  __syncthreads();
  // |Re| + |Im| below 2, for the guard
  for (int t = threadIdx.x; t < P * nrp; t += blockDim.x) {
    const int bl = t / nrp, s = t % nrp, b = nt * P + bl;
    float v = 0.f;
    if (b < B && s < Nr) {
      const cdd y = ld_cdd(Y + (size_t)b * y_bstride + (size_t)w * Nr + s);
      v = (fabsf(y.re.hi) + fabsf(y.im.hi)) * tc_pow2f(-e_sh[bl]);
    }
    mag[((size_t)w * ntiles * P + b) * nrp + s] = (uint16_t)(__float_as_uint(v) >> 16);
  }
  const size_t slice_bytes = (size_t)N * 64;
  uint8_t *base = tiles + ((size_t)w * ntiles + nt) * natoms * NSL * slice_bytes;
  for (int t = threadIdx.x; t < natoms * N * 4; t += blockDim.x) {
    const int a = t / (N * 4), n = (t >> 2) % N, q = t & 3;
    const int part = n >= P, bl = n - part * P, b = nt * P + bl;
    const float sc1 = tc_pow2f(7 - e_sh[bl]);
    const f2 sc = f2_make(sc1, sc1);
    Slicer7 sl[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int s = 16 * a + 4 * q + u;
      cdd y = cdd_zero();
      if (b < B && s < Nr) y = ld_cdd(Y + (size_t)b * y_bstride + (size_t)w * Nr + s);
      // the two reals of this row: (yr, yi) for the real-part column, (yi, -yr) for the imaginary
      const dd v0 = part ? y.im : y.re, v1 = part ? dd_neg(y.re) : y.im;
      sl[u].init(v0.hi, v0.lo, v1.hi, v1.lo, sc);
    }
    uint8_t *at = base + (size_t)a * NSL * slice_bytes + tc_swz64(n, q);
    auto put = [&](auto S) {
      uint32_t wd[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) wd[u] = sl[u].template next<S.value>();
      *reinterpret_cast<uint4 *>(at + S.value * slice_bytes) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
    };
    for_slices7(put);
  }
}

template <int P>
struct Cfg {
  static constexpr int N = 2 * P;
  // the accumulators twice if that leaves two A' stages, the rest A' stages
  static constexpr int nbuf = 2 * NACC * N + 2 * A_COLS <= 512 ? 2 : 1;
  static constexpr int left = (512 - nbuf * NACC * N) / A_COLS;
  static constexpr int SA = left < MAXA ? left : MAXA;
  static constexpr uint32_t b_slice = (uint32_t)N * 64u, b_stage = NSL * b_slice;
  // raw ring 96 KB, B' stages 112 KB at N = 64; never so little that a second
  // CTA (whose TMEM allocation would wait for this one's) fits beside it
  static constexpr size_t smem = 1024 + (size_t)RAW_D * RAW_SLOT + SB * b_stage;
  static_assert(SA >= 2 && smem > 114 * 1024 && smem <= 227 * 1024, "stages");
};

template <int P>
__global__ void __launch_bounds__(NTHR, 1)
k_gemm_adj_sl64(const float4 *__restrict__ A, const int8_t *__restrict__ ea, const uint8_t *__restrict__ Bt,
                const int *__restrict__ eb, cdd *__restrict__ X, long x_bstride, int B, int ntiles,
                int Nr, int Nm, int Nf, int natoms, int chunk, int *err) {
  constexpr int N = Cfg<P>::N, SA = Cfg<P>::SA, nbuf = Cfg<P>::nbuf;
  constexpr uint32_t b_slice = Cfg<P>::b_slice, b_stage = Cfg<P>::b_stage;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * MAXA + 2 * SB + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int nmt = (Nm + TM - 1) / TM;
  const int T = nmt * Nf * ntiles;
  const int my_tiles = (int)blockIdx.x < T ? (T - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int nchunk = (natoms + chunk - 1) / chunk;
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
  // all 512 columns are allocated, so the allocation starts at column 0; the
  // constant lets the MMA warp form its operands without register moves
  constexpr uint32_t tmem = 0;
  constexpr uint32_t tmemA = tmem + (uint32_t)(nbuf * NACC * N);
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
    // stage's 8; its loads run one atom (two stages) ahead
    const int r = tid & (TM - 1), h = (tid >> 7) & 1, g = tid / NGRP;
    int ii = 0, ia = 0;
    const float4 *ip = A;
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
    int islot = 0;
    const uint32_t raw0 = sRaw + 16u * tid;
    const uint8_t *rawp = smem_raw + (raw0 - tc_su32(smem_raw));
    auto load = [&]() {
      if (ii < my_tiles) {
        const int s0 = 16 * ia + 8 * g + 4 * h;
        const float4 *p = ip + (size_t)(16 * ia) * Nm;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = ivalid && s0 + u < Nr;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                       ::"r"(raw0 + (uint32_t)(islot * RAW_SLOT + u * NPROD * 16)),
                         "l"(in ? p + (size_t)u * Nm : A), "r"(in ? 16 : 0) : "memory");
        }
        if (++ia == natoms) { ia = 0; ++ii; set_issue_tile(); }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (++islot == RAW_D) islot = 0;
    };
    auto row_scale_exp = [&](int i) {
      if (i >= my_tiles) return 0;
      int mt, w, nt;
      tile_of(i, mt, w, nt);
      const int m = mt * TM + r;
      return m < Nm ? (int)ea[(size_t)w * Nm + m] : 0;
    };
    set_issue_tile();
#pragma unroll
    for (int d = 0; d < RAW_D - 1; ++d) load();
    int slot = 0;
    int e_next = row_scale_exp(0);
    bool ok = true;
    const uint32_t lane_base = tmemA + ((uint32_t)(32 * (warp & 3)) << 16) + 4u * h;
    // stage and its use count: the stages of the groups alternate, an atom
    // whose second half holds no rows (the last, for some Nr) has one
    const bool odd = 16 * (natoms - 1) + 8 >= Nr;
    int st = g, use = 0;
    if (st >= SA) { st -= SA; ++use; }
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
        Slicer7 sl[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 v = *reinterpret_cast<const float4 *>(rawp + slot * RAW_SLOT + u * NPROD * 16);
          sl[u].init(v.x, v.y, v.z, v.w, sc);
        }
        if (++slot == RAW_D) slot = 0;
        load();
        const bool last_half = odd && a == natoms - 1;      // this atom has the first stage only
        if (use > 0) {
          const bool got = tc_mbar_wait(emptyA(st), (unsigned)((use - 1) & 1), vfail);
          if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) note(err, vfail, 41);
            ok = false;
            break;
          }
        }
        // (group 1 waits for the stage that it leaves to the next tile as well: a
        // jump of three stages could meet its next stage a whole phase early)
        if (last_half && g == 1) { step(1); continue; }
        tc_fence_after();
        const uint32_t at = lane_base + (uint32_t)(st * A_COLS);
        auto put = [&](auto S) {
          uint32_t wd[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) wd[u] = sl[u].template next<S.value>();
          tc_st4(at + 8u * S.value, wd);
        };
        for_slices7(put);
        tc_wait_st();
        tc_fence_before();
        tc_mbar_arrive(fullA(st));
        step(last_half ? 1 : 2);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // own copies drained before exit
  } else if (warp < (NPROD + NEPI) / 32) {
    // ---------------- epilogue: level sums joined, scaled, stored as float pairs
    // (two warps a TMEM lane quarter, each half of the columns)
    const int lg = warp & 3, half = (warp - NPROD / 32) >> 2;
    const int r = 32 * lg + lane;
    constexpr int CW = P / 2;                       // right-hand sides of this warp
    bool ok = true;
    int bf = 0, use = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int mt, w, nt;
      tile_of(i, mt, w, nt);
      const int m = mt * TM + r;
      const float sa = tc_pow2f((m < Nm ? (int)ea[(size_t)w * Nm + m] : 0) - 7);
      const int b0 = nt * P + half * CW;
      const int *ebw = eb + (size_t)w * ntiles * P + b0;
      cdd *xp = X + (size_t)b0 * x_bstride + (size_t)w * Nm + m;
      for (int c = 0; c < nchunk; ++c) {
        const bool got = tc_mbar_wait(tfull(bf), (unsigned)(use & 1), vfail);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) note(err, vfail, 42);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t trow = tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)(bf * NACC * N + half * CW);
#pragma unroll 1
        for (int c0 = 0; c0 < CW; c0 += 2) {
          uint32_t dr[NACC][2], di[NACC][2];
#pragma unroll
          for (int L = 0; L < NACC; ++L) {
            tc_ld2(dr[L], trow + (uint32_t)(L * N + c0));
            tc_ld2(di[L], trow + (uint32_t)(L * N + P + c0));
          }
          tc_wait_ld();
          if (c0 + 2 >= CW) {
            // the buffer is read: the MMAs of a later chunk may overwrite it
            tc_fence_before();
            tc_mbar_arrive(tempty(bf));
          }
          f2 v[NACC], rh, rl, ih, il;                // both columns at once
#pragma unroll
          for (int L = 0; L < NACC; ++L) v[L] = f2_make(__uint_as_float(dr[L][0]), __uint_as_float(dr[L][1]));
          tc_join_levels(v, rh, rl);
#pragma unroll
          for (int L = 0; L < NACC; ++L) v[L] = f2_make(__uint_as_float(di[L][0]), __uint_as_float(di[L][1]));
          tc_join_levels(v, ih, il);
          const float2 arh = f2_split(rh), arl = f2_split(rl), aih = f2_split(ih), ail = f2_split(il);
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (m >= Nm || b0 + c0 + j >= B) continue;
            const float sb = tc_pow2f(ebw[c0 + j] - 7);
            cdd x;
            x.re = dd_make_raw(j ? arh.y : arh.x, j ? arl.y : arl.x);
            x.im = dd_make_raw(j ? aih.y : aih.x, j ? ail.y : ail.x);
            x = cdd_scale2(cdd_scale2(x, sa), sb);
            cdd *xo = xp + (size_t)(c0 + j) * x_bstride;
            if (c > 0) x = cdd_add(ld_cdd(xo), x);     // this thread stored the earlier chunks
            st_cdd(xo, x);
          }
        }
        if (++bf == nbuf) { bf = 0; ++use; }
      }
    }
  } else if (warp == (NPROD + NEPI) / 32) {
    // ---------------- MMA issuer (the warp's lanes run together, one is elected to issue)
    const uint32_t idesc = tc_idesc_bf16(TM, N);
    auto wait = [&](uint32_t bar, int parity) {
      return __all_sync(0xffffffffu, tc_mbar_wait(bar, (unsigned)(parity & 1), vfail));
    };
    bool ok = true;
    int sa = 0, usea = 0, sb = 0, useb = 0, bf = 0, used = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      for (int c = 0; c < nchunk && ok; ++c) {
        // the epilogue has read this buffer's previous chunk
        if (used > 0 && !wait(tempty(bf), used - 1)) { ok = false; break; }
        tc_fence_after();
        uint32_t dc[NACC];
#pragma unroll
        for (int L = 0; L < NACC; ++L) dc[L] = tmem + (uint32_t)((bf * NACC + L) * N);
        const int s0 = c * chunk * 16, s1 = min(Nr, s0 + chunk * 16);
        // stages of 8 rows; an atom's B' serves two.  The next stage is waited
        // for between the halves of this one's MMAs, so that the tensor cores
        // have work queued meanwhile
        if (!wait(fullB(sb), useb) || !wait(fullA(sa), usea)) { ok = false; break; }
        for (int s = s0; s < s1; s += 8) {
          const int ks = (s >> 3) & 1;
          tc_fence_after();
          const uint32_t aT = tmemA + (uint32_t)(sa * A_COLS);
          const uint64_t bd0 = tc_sdesc64(sB0 + (uint32_t)sb * b_stage + 32u * ks);
          uint64_t bd[NSL];
#pragma unroll
          for (int j = 0; j < NSL; ++j) bd[j] = bd0 + (uint64_t)(j * (b_slice >> 4));
          const bool last = s + 8 >= s1, b_done = ks == 1 || last;
          if (tc_elect()) tc_issue_half<0>(s == s0, dc, aT, bd, idesc);
          __syncwarp();
          const uint32_t eA = emptyA(sa), eB = emptyB(sb);
          if (++sa == SA) { sa = 0; ++usea; }
          if (b_done && ++sb == SB) { sb = 0; ++useb; }
          if (!last && ((b_done && !wait(fullB(sb), useb)) || !wait(fullA(sa), usea))) ok = false;
          if (tc_elect()) {
            tc_issue_half<1>(s == s0, dc, aT, bd, idesc);
            tc_commit(eA);
            if (b_done) tc_commit(eB);
            if (last) tc_commit(tfull(bf));
          }
          __syncwarp();
          if (!ok) break;
        }
        if (++bf == nbuf) { bf = 0; ++used; }
      }
    }
    if (!ok && lane == 0) note(err, vfail, 43);
    // every issued MMA complete before TMEM is released
    if (tc_elect()) tc_commit(drain);
    tc_mbar_wait(drain, 0, nullptr);
  } else {
    if (lane == 0) {
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
      if (!ok) note(err, vfail, 44);
      // copies already issued must land before the CTA's shared memory goes
      for (int a = (issued > SB ? issued - SB : 0); a < issued; ++a)
        tc_mbar_wait(fullB(a % SB), (unsigned)((a / SB) & 1), nullptr);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(512u) : "memory");
}

// ------------------------------------------------------ the guard (tc.cuh)
// low[w][tile][s]: the least |F^[s][m]| of a tile's 128 grid points, in units of
// the point's exponent (bf16, rounded down; rows past Nr zero).  Points that no
// sensor sees (no entry of 2^-100) are left out: their sums are zero
__global__ void __launch_bounds__(TM)
k_adj_low(const float4 *__restrict__ A, const int8_t *__restrict__ ea, uint16_t *__restrict__ low, int nrp, int Nr,
          int Nm) {
  __shared__ unsigned sh[2][TM / 32];
  const int w = blockIdx.y, m = blockIdx.x * TM + threadIdx.x;
  const int e = m < Nm ? (int)ea[(size_t)w * Nm + m] : -100;
  const float4 *p = A + (size_t)w * Nr * Nm + min(m, Nm - 1);
  uint16_t *out = low + ((size_t)w * gridDim.x + blockIdx.x) * nrp;
  for (int s = 0; s < nrp; ++s) {
    unsigned v = 0x7f800000u;
    if (s >= Nr) v = 0;
    else if (e > -100) {
      const float4 a = __ldcs(p + (size_t)s * Nm);
      v = __float_as_uint((fabsf(a.x) + fabsf(a.z)) * tc_pow2f(-e));
    }
    v = __reduce_min_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) sh[s & 1][threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      v = min(min(sh[s & 1][0], sh[s & 1][1]), min(sh[s & 1][2], sh[s & 1][3]));
      out[s] = (uint16_t)(min(v, 0x3f800000u) >> 16);      // (a tile without such points: any value)
    }
  }
}

// The tiles of 128 grid points and up to 64 columns (a piece of 64 of the ncols)
// with a sum whose bound over the whole tile, sum_s low |Y|, does not settle it:
// todo[1 ..], todo[0] of them (zeroed by k_bsl64_build).  A warp takes 16 tiles
__global__ void __launch_bounds__(128)
k_adj_check(const uint16_t *__restrict__ low, const uint16_t *__restrict__ mag, int nrp, int Nr, int ntl, int B,
            int ncols, int *__restrict__ todo) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int w = blockIdx.y, col0 = blockIdx.z * 64, t0 = (blockIdx.x * 4 + warp) * 16;
  if (t0 >= ntl) return;
  const int nf = min(8, (ncols - col0) / 8);
  const uint16_t *lo = low + (size_t)w * ntl * nrp + 4 * c;
  const uint16_t *mw = mag + ((size_t)w * ncols + col0 + g) * nrp + 4 * c;
  const size_t ra = (size_t)min(t0 + g, ntl - 1) * nrp, rb = (size_t)min(t0 + g + 8, ntl - 1) * nrp;
  float S[8][4] = {}, M[8][4] = {};
  for (int s = 0; s < nrp; s += 16) {
    const uint2 p = __ldg(reinterpret_cast<const uint2 *>(lo + ra + s)), q = __ldg(reinterpret_cast<const uint2 *>(lo + rb + s));
    const uint32_t a[4] = {p.x, q.x, p.y, q.y}, one[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
#pragma unroll
    for (int f = 0; f < 8; ++f)
      if (f < nf) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(mw + (size_t)(8 * f) * nrp + s));
        const uint32_t b[2] = {v.x, v.y};
        tc_mma_mag(S[f], a, b);
        tc_mma_mag(M[f], one, b);                          // zero: an empty column
      }
  }
  const float thr = sqrtf(2.f * (float)Nr);
  bool open[2] = {false, false};
#pragma unroll
  for (int f = 0; f < 8; ++f)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (col0 + 8 * f + 2 * c + (i & 1) < B && M[f][i] != 0.f && !(512.f * S[f][i] >= thr)) open[i >> 1] = true;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const unsigned any = __ballot_sync(0xffffffffu, open[h]);
    if (c == 0 && ((any >> lane) & 15u) && t0 + g + 8 * h < ntl)
      todo[1 + atomicAdd(todo, 1)] = (w * ntl + t0 + g + 8 * h) * (int)gridDim.z + (int)blockIdx.z;
  }
}

// S[m][b] = sum_s |F^[s][m]| |Y[s][b]| of those tiles, from the operator; sums that
// fail are formed in double-float and stored over the sliced ones.  A warp takes 16
// points.  Bound by the operator's second reading where every tile is on the list:
// 5.4 ms at 5.7 TB/s for 32 GB (64 right-hand sides of 100 sensors on 50,000
// points), beside the product's 25; with G^ there, smooth in space, few are, and
// both guard kernels take 0.7 ms.  Complex magnitudes: Re and Im of a sum share their
// bound, as in the complex double-float product.
__global__ void __launch_bounds__(256, 2)
k_adj_guard(const float4 *__restrict__ A, const int8_t *__restrict__ ea, const uint16_t *__restrict__ mag, int nrp,
            const cdd *__restrict__ Y, long y_bstride, cdd *__restrict__ X, long x_bstride, int Nr, int Nm, int B,
            int ncols, int ntl, int ngrp, const int *__restrict__ todo) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const float thr = sqrtf(2.f * (float)Nr);                // T = 1: both sides are scaled
  const int ntodo = todo[0];
  for (int it = blockIdx.x; it < ntodo; it += gridDim.x) {
    const int item = todo[1 + it], col0 = item % ngrp * 64, w = item / ngrp / ntl;
    const int m0 = item / ngrp % ntl * TM + 16 * warp;
    if (m0 >= Nm) continue;
    const int nf = min(8, (ncols - col0) / 8);               // fragments of 8 columns
    const int ma = min(m0 + g, Nm - 1), mb = min(m0 + g + 8, Nm - 1);
    const float sa = tc_pow2f(-(int)ea[(size_t)w * Nm + ma]), sb = tc_pow2f(-(int)ea[(size_t)w * Nm + mb]);
    const float4 *Aw = A + (size_t)w * Nr * Nm;
    const uint16_t *Mw = mag + ((size_t)w * ncols + col0 + g) * nrp + 4 * c;
    float4 v[2][4];
    auto load = [&](int s0) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int s = min(s0 + 4 * c + j, Nr - 1);           // past the rows: the data's magnitude is zero
        v[0][j] = __ldcs(Aw + (size_t)s * Nm + ma);
        v[1][j] = __ldcs(Aw + (size_t)s * Nm + mb);
      }
    };
    float d[8][4] = {};
    load(0);
    for (int s0 = 0; s0 < Nr; s0 += 16) {
      float r[2][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        r[0][j] = (fabsf(v[0][j].x) + fabsf(v[0][j].z)) * sa;
        r[1][j] = (fabsf(v[1][j].x) + fabsf(v[1][j].z)) * sb;
      }
      if (s0 + 16 < Nr) load(s0 + 16);
      const uint32_t a[4] = {tc_pack_bf16(r[0][0], r[0][1]), tc_pack_bf16(r[1][0], r[1][1]),
                             tc_pack_bf16(r[0][2], r[0][3]), tc_pack_bf16(r[1][2], r[1][3])};
#pragma unroll
      for (int f = 0; f < 8; ++f)
        if (f < nf) {
          const uint2 q = __ldg(reinterpret_cast<const uint2 *>(Mw + (size_t)(8 * f) * nrp + s0));
          const uint32_t b[2] = {q.x, q.y};
          tc_mma_mag(d[f], a, b);
        }
    }
    unsigned bad = 0;
#pragma unroll
    for (int f = 0; f < 8; ++f)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (m0 + g + 8 * (i >> 1) < Nm && col0 + 8 * f + 2 * c + (i & 1) < B && tc_guard_fails(d[f][i], thr))
          bad |= 1u << (4 * f + i);
    for (unsigned any = __reduce_or_sync(0xffffffffu, bad); any; any &= any - 1) {
      const int e = __ffs(any) - 1, f = e >> 2, i = e & 3;
      for (unsigned who = __ballot_sync(0xffffffffu, (bad >> e) & 1); who; who &= who - 1) {
        const int l = __ffs(who) - 1;
        const int m = m0 + (l >> 2) + 8 * (i >> 1), b = col0 + 8 * f + 2 * (l & 3) + (i & 1);
        const cdd *Yb = Y + (size_t)b * y_bstride + (size_t)w * Nr;
        cdd x = cdd_zero();
        for (int s = lane; s < Nr; s += 32)
          x = cdd_add(x, cdd_mul(cdd_conj(ld_cdd(reinterpret_cast<const cdd *>(Aw + (size_t)s * Nm + m))), ld_cdd(Yb + s)));
        x.re = tc_warp_sum(x.re);
        x.im = tc_warp_sum(x.im);
        if (lane == 0) st_cdd(X + (size_t)b * x_bstride + (size_t)w * Nm + m, x);
      }
    }
  }
}

int sl64_natoms(int Nr) { return (Nr + KA / 2 - 1) / (KA / 2); }
int sl64_nrp(int Nr) { return (Nr + 15) / 16 * 16; }
// right-hand sides per tile: the fewest tiles of at most PMAX, a multiple of 8
int sl64_tile(int B) {
  const int nt = (B + PMAX - 1) / PMAX;
  return ((B + nt - 1) / nt + 7) / 8 * 8;
}

}  // namespace

// ------------------------------------------------------------------ host side
// workspace for any batch of at most bcols right-hand sides: tiles hold fewer
// than 8 unused columns each, and there are at most ceil(bcols / PMAX) of them
static int sl64_cols(int bcols) { return bcols + 8 * ((bcols + PMAX - 1) / PMAX); }
size_t sl64_ws_bytes(int Nf, int Nr, int Nm, int bcols) {
  // slices, then the magnitudes, then the guard's list of tiles
  return (size_t)Nf * sl64_cols(bcols) * ((size_t)sl64_natoms(Nr) * NSL * 2 * 64 + (size_t)sl64_nrp(Nr) * 2) +
         sizeof(int) * (1 + (size_t)Nf * ((Nm + TM - 1) / TM) * ((sl64_cols(bcols) + 63) / 64));
}
size_t sl64_eb_bytes(int Nf, int bcols) { return (size_t)Nf * sl64_cols(bcols) * sizeof(int); }

// the operator's tables: row exponents, then (16-byte aligned) the guard's magnitudes
static const uint16_t *sl64_low(const int8_t *ea, int Nf, int Nm) {
  return reinterpret_cast<const uint16_t *>(ea + ((size_t)Nf * Nm + 15) / 16 * 16);
}
size_t row_exp64_bytes(int Nf, int Nr, int Nm) {
  return ((size_t)Nf * Nm + 15) / 16 * 16 + (size_t)Nf * ((Nm + TM - 1) / TM) * sl64_nrp(Nr) * sizeof(uint16_t);
}
cudaError_t launch_row_exp64(const void *A, int8_t *ea, int Nf, int Nr, int Nm, cudaStream_t s) {
  const long total = (long)Nf * Nm;
  const long blocks = std::min<long>((total + 255) / 256, 152 * 32);
  k_row_exp64<<<(unsigned)blocks, 256, 0, s>>>(reinterpret_cast<const float4 *>(A), ea, Nf, Nr, Nm);
  k_adj_low<<<dim3((Nm + TM - 1) / TM, Nf), TM, 0, s>>>(reinterpret_cast<const float4 *>(A), ea,
                                                        const_cast<uint16_t *>(sl64_low(ea, Nf, Nm)), sl64_nrp(Nr),
                                                        Nr, Nm);
  count_launches(2);
  return cudaGetLastError();
}

// X[b][w][k] = sum_s conj(A[w][s][k]) Y[b][w][s] for b < B
cudaError_t launch_gemm_adj_sl64(const void *A, const int8_t *ea, const cdd *Y, long y_bstride, cdd *X,
                                 long x_bstride, int Nf, int Nr, int Nm, int B, void *ws, size_t ws_bytes,
                                 int *eb, size_t eb_bytes, int *err, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  const int P = sl64_tile(B), N = 2 * P, ntiles = (B + P - 1) / P, natoms = sl64_natoms(Nr);
  const size_t b_stage = (size_t)NSL * N * 64, sl_bytes = (size_t)Nf * ntiles * natoms * b_stage;
  const int nrp = sl64_nrp(Nr), ncols = ntiles * P;
  const int ntl = (Nm + TM - 1) / TM, ngrp = (ncols + 63) / 64;
  const size_t mag_bytes = (size_t)Nf * ncols * nrp * 2;
  if (sl_bytes + mag_bytes + sizeof(int) * (1 + (size_t)Nf * ntl * ngrp) > ws_bytes || (size_t)Nf * ntiles * P * sizeof(int) > eb_bytes)
    return cudaErrorInvalidValue;
  uint16_t *mag = reinterpret_cast<uint16_t *>(reinterpret_cast<uint8_t *>(ws) + sl_bytes);
  int *todo = reinterpret_cast<int *>(reinterpret_cast<uint8_t *>(ws) + sl_bytes + mag_bytes);
  k_bsl64_build<<<dim3(Nf, ntiles), 256, 0, s>>>(Y, y_bstride, Nr, B, P, natoms,
                                                 reinterpret_cast<uint8_t *>(ws), eb, mag, nrp, todo,
                                                 ntiles);
  count_launches(1);
  const int chunk = Nr <= EXACT_ROWS ? natoms : CHUNK_ATOMS;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const long tiles = (long)((Nm + TM - 1) / TM) * Nf * ntiles;
  const unsigned grid = (unsigned)std::max<long>(1, std::min<long>(tiles, nsm));
  auto run = [&](auto PC) {
    constexpr int PP = PC.value;
    cudaFuncSetAttribute(k_gemm_adj_sl64<PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<PP>::smem);
    k_gemm_adj_sl64<PP><<<grid, NTHR, Cfg<PP>::smem, s>>>(reinterpret_cast<const float4 *>(A), ea,
                                                          reinterpret_cast<const uint8_t *>(ws), eb, X, x_bstride,
                                                          B, ntiles, Nr, Nm, Nf, natoms, chunk, err);
  };
  switch (P) {
    case 8: run(std::integral_constant<int, 8>{}); break;
    case 16: run(std::integral_constant<int, 16>{}); break;
    case 24: run(std::integral_constant<int, 24>{}); break;
    default: run(std::integral_constant<int, 32>{}); break;
  }
  k_adj_check<<<dim3((ntl + 63) / 64, Nf, ngrp), 128, 0, s>>>(sl64_low(ea, Nf, Nm), mag, nrp, Nr, ntl, B, ncols, todo);
  k_adj_guard<<<(unsigned)std::max<long>(1, std::min<long>((long)Nf * ntl * ngrp, 2L * nsm)), 256, 0, s>>>(
      reinterpret_cast<const float4 *>(A), ea, mag, nrp, Y, y_bstride, X, x_bstride, Nr, Nm, B, ncols, ntl, ngrp, todo);
  count_launches(3);
  return cudaGetLastError();
}

}  // namespace tw
