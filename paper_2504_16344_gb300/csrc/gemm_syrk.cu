// gemm_syrk.cu -- K's block products P = G G^T on the 5th-generation tensor
// cores, with G cut into exact fixed-point bf16 slices.
//
// Phase 2 forms K = sigma^2 I + F Gamma_pr F^T (Sec. "Real-time Bayesian
// inference and prediction framework"); with G = Phi C^{1/2} the block
// products are P = G G^T, a symmetric rank-Nm product over the grid, followed
// by prefix sums along the block diagonals (dense.cu).  K is factored in FP64
// and its conditioning amplifies rounding in these long sums, so P is needed
// to FP64 level.
//
// Slices.  Row i of G gets a power-of-two exponent e_i with |G_ik| < 2^e_i for
// every k, and each entry is written in fixed point as seven 8-bit integer
// slices (round to nearest at each step):
//   G_ik = 2^(e_i - 7) (s0 + s1 / 2^8 + ... + s6 / 2^48),  |s_p| <= 128,
// 55 bits below the row maximum (the double-float G has 48 bits of its own).
// Slice p is stored pre-scaled, s_p 2^-8p, exact in bf16.  The product of
// slices p and q is a multiple of 2^-8(p+q) of magnitude <= 2^14 2^-8(p+q);
// level L = p + q collects the L + 1 pairs of that scale, and pairs with
// L <= 6 are formed (28 MMAs per 16-wide k step; the dropped levels are
// below 2^-56 of a term).
//
// Exact accumulation.  The tensor cores accumulate in FP32 and truncate.  A
// level's sum over a chunk of 128 k is a multiple of 2^-8L below
// (L+1) 128 2^14 2^-8L <= 5 2^21 2^-8L for L <= 4, an integer count below
// 2^24: levels 0 .. 4 each accumulate EXACTLY in their own TMEM accumulator.
// Levels 5 and 6 share a sixth (2^-40 below a term, where the truncation of
// its ~100 accumulation steps stays near 2^-56 of the terms).  After each
// chunk the epilogue reads the six accumulators, scales each D_L by 2^8L to
// an integer D_L' and forms the exact
//   X = ((((D0' 2^8 + D1') 2^8 + D2') 2^8 + D3') 2^8 + D4') = (D0 + .. + D4) 2^32,
// adds it to an int64 total (exact) and D56 to an FP32 total.  At the end of
// a panel of k the tile adds 2^(e_i + e_j - 14) (T 2^-32 + F) to K in FP64:
// one rounding per panel.
//
// Kernel: persistent, one CTA per SM, over a host-ordered list of (128-row,
// 64-column) tiles of the lower triangle (groups of 8 row tiles, column tile
// outer, so the CTAs running together share their slice tiles in L2).  One
// thread issues the bulk copies of a k atom's slices (A: 7 x 128 rows, B: 7 x
// 64 rows of the same sliced panel) into a 2-stage ring; four warps move A's
// slices on to TMEM; one warp issues the MMAs (six accumulators of 64
// columns); eight warps drain them, half a row each.  Every wait is bounded:
// on expiry the kernel records TW_ERR_TIMEOUT, lets its copies and MMAs drain
// (bounded), frees TMEM and returns.
//
// Why this tile.  With both operands in shared memory an MMA of 128 x 32 x 16
// takes 45 cycles (A's 4 KB at 128 bytes a clock, issued from one lane's
// branch), three times its arithmetic, and each A slice is read again for
// every one of its up to seven pairs.  From TMEM a 128 x 64 x 16 MMA takes 32
// cycles, its arithmetic; shared memory then carries one read of A by the
// moving warps and B's 2 KB per MMA.  64 columns also halve the L2 reads of A.
// The sums keep their bits: chunks, panels and the order within an
// accumulator are what they were.  K of 10,000 rows from 12,500 grid points:
// 67 -> 37 ms.
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "../../include/tw.h"
#include "dense_api.h"
#include "kernels.h"
#include "tc.cuh"

namespace tw {

namespace {

constexpr int SK_TM = 128;                   // MMA M: rows of a tile
constexpr int SK_TN = 64;                    // MMA N: columns of a tile
constexpr int SK_KA = 32;                    // k per atom (two 16-wide MMA steps)
constexpr int SK_NSL = TC_NSL;               // slices per entry
constexpr int SK_NACC = TC_NACC;             // accumulators: levels 0 .. 4, and 5..6
constexpr int SK_CHUNK = 4;                  // atoms per exact chunk (128 k)
constexpr int SK_A_SLICE = SK_TM * SK_KA * 2;     // 8 KB
constexpr int SK_B_SLICE = SK_TN * SK_KA * 2;     // 4 KB
constexpr int SK_A_STAGE = SK_NSL * SK_A_SLICE;   // 56 KB
constexpr int SK_B_STAGE = SK_NSL * SK_B_SLICE;   // 28 KB
constexpr int SK_STAGE = SK_A_STAGE + SK_B_STAGE; // 84 KB
constexpr int SK_S = 2;                      // ring stages
constexpr int SK_SA = 2;                     // A stages in TMEM (16 k each)
constexpr int SK_A_COLS = SK_NSL * 8;        // TMEM columns of one
constexpr int SK_NMOV = 128, SK_NEPI = 256;  // moving and epilogue threads
constexpr int SK_NTHR = SK_NMOV + SK_NEPI + 64;
static_assert(SK_NACC * SK_TN + SK_SA * SK_A_COLS <= 512, "TMEM columns");
constexpr int SK_EXP_MIN = -100, SK_EXP_MAX = 120;

// round to the nearest integer (ties to even), |v| < 2^22
__device__ __forceinline__ float rnd_int(float v) {
  return __fsub_rn(__fadd_rn(v, 12582912.0f), 12582912.0f);
}
__device__ __forceinline__ int exp_above(float mx) {
  if (!(mx > 0.f)) return SK_EXP_MIN;
  const int e = (int)((__float_as_uint(mx) >> 23) & 0xffu) - 126;
  return e < SK_EXP_MIN ? SK_EXP_MIN : (e > SK_EXP_MAX ? SK_EXP_MAX : e);
}

// ------------------------------------------------------ row exponents
// eg[i] = smallest e with |G_ik| < 2^e for all k (rows >= n: the minimum)
__global__ void __launch_bounds__(256)
k_syrk_row_exp(const dd *__restrict__ G, long ldg, int n, int kdim, int *__restrict__ eg, int nrows) {
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (warp >= nrows) return;
  float mx = 0.f;
  if (warp < n) {
    const dd *row = G + (size_t)warp * ldg;
    for (int k = lane; k < kdim; k += 32) mx = fmaxf(mx, fabsf(row[k].hi));
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
  // the low half may lift |G| past the high half's bound by one unit in the
  // last place: bound the sum instead
  if (lane == 0) eg[warp] = warp < n ? exp_above(mx * (1.0f + 1.0f / 1048576.0f)) : SK_EXP_MIN;
}

// ------------------------------------------------------ slices of a k panel
// tiles[T][a][s][128 rows][32 bf16] (64-byte swizzle): rows 128 T .. +127 of
// G, columns k0 + 32 a .. +31 of the panel, slice s.  A 64-row column tile
// J is rows 64 (J mod 2) .. +63 of tile J / 2: 4 KB contiguous per slice.
__global__ void __launch_bounds__(256)
k_syrk_slice(const dd *__restrict__ G, long ldg, int n, int kdim, int k0, const int *__restrict__ eg,
             uint8_t *__restrict__ tiles, int natoms) {
  const int a = blockIdx.x, T = blockIdx.y;
  const int r = threadIdx.x & (SK_TM - 1), h = threadIdx.x >> 7;
  const int i = T * SK_TM + r;
  const int kb = k0 + SK_KA * a + 16 * h;
  const float sc = tc_pow2f(7 - eg[i]);
  float hi[16], lo[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    dd v = dd_zero();
    if (i < n && kb + u < kdim) v = G[(size_t)i * ldg + kb + u];
    hi[u] = v.hi * sc;   // exact: power-of-two scaling
    lo[u] = v.lo * sc;
  }
  uint8_t *base = tiles + ((size_t)T * natoms + a) * SK_NSL * SK_A_SLICE;
#pragma unroll
  for (int s = 0; s < SK_NSL; ++s) {
    uint32_t wd[8];
#pragma unroll
    for (int u2 = 0; u2 < 8; ++u2) {
      float sl[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int u = 2 * u2 + c;
        const float si = rnd_int(hi[u]);
        sl[c] = si * tc_pow2f(-8 * s);
        if (s + 1 < SK_NSL) {
          float rr, ee;
          two_sum(__fsub_rn(hi[u], si), lo[u], rr, ee);   // hi - si is exact
          hi[u] = rr * 256.f;
          lo[u] = ee * 256.f;
        }
      }
      wd[u2] = tc_pack_bf16(sl[0], sl[1]);
    }
    uint8_t *tile = base + (size_t)s * SK_A_SLICE;
    *reinterpret_cast<uint4 *>(tile + tc_swz64(r, 2 * h)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
    *reinterpret_cast<uint4 *>(tile + tc_swz64(r, 2 * h + 1)) = make_uint4(wd[4], wd[5], wd[6], wd[7]);
  }
}

// ------------------------------------------ FP64 panels (the Cholesky's updates)
// eg[i] = smallest e with |A_ik| < 2^e over the kdim columns of row i
__global__ void __launch_bounds__(256)
k_syrk_row_exp_d(const double *__restrict__ A, long ld, int n, int kdim, int *__restrict__ eg, int nrows) {
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (warp >= nrows) return;
  double mx = 0.0;
  if (warp < n)
    for (int k = lane; k < kdim; k += 32) mx = fmax(mx, fabs(A[(size_t)warp * ld + k]));
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, m));
  if (lane == 0) {
    int e = SK_EXP_MIN;
    if (warp < n && mx > 0.0) {
      frexp(mx, &e);                    // mx = f 2^e, f in [1/2, 1): mx < 2^e
      e = e < SK_EXP_MIN ? SK_EXP_MIN : (e > SK_EXP_MAX ? SK_EXP_MAX : e);
    }
    eg[warp] = e;
  }
}

// slices of an FP64 panel in the layout of k_syrk_slice: seven 8-bit slices
// hold the 53-bit significand of every entry within 2^2 of its row maximum
// exactly (steps in FP64: scaling by a power of two, rint, and (x - s) 256
// are exact)
__global__ void __launch_bounds__(256)
k_syrk_slice_d(const double *__restrict__ A, long ld, int n, int kdim, const int *__restrict__ eg,
               uint8_t *__restrict__ tiles, int natoms) {
  const int a = blockIdx.x, T = blockIdx.y;
  const int r = threadIdx.x & (SK_TM - 1), h = threadIdx.x >> 7;
  const int i = T * SK_TM + r;
  const int kb = SK_KA * a + 16 * h;
  const int e = eg[i];
  double x[16];
#pragma unroll
  for (int u = 0; u < 16; ++u)
    x[u] = (i < n && kb + u < kdim) ? ldexp(A[(size_t)i * ld + kb + u], 7 - e) : 0.0;
  uint8_t *base = tiles + ((size_t)T * natoms + a) * SK_NSL * SK_A_SLICE;
#pragma unroll
  for (int s = 0; s < SK_NSL; ++s) {
    uint32_t wd[8];
#pragma unroll
    for (int u2 = 0; u2 < 8; ++u2) {
      float sl[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int u = 2 * u2 + c;
        const double si = rint(x[u]);
        sl[c] = (float)si * tc_pow2f(-8 * s);
        x[u] = (x[u] - si) * 256.0;
      }
      wd[u2] = tc_pack_bf16(sl[0], sl[1]);
    }
    uint8_t *tile = base + (size_t)s * SK_A_SLICE;
    *reinterpret_cast<uint4 *>(tile + tc_swz64(r, 2 * h)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
    *reinterpret_cast<uint4 *>(tile + tc_swz64(r, 2 * h + 1)) = make_uint4(wd[4], wd[5], wd[6], wd[7]);
  }
}

// ------------------------------------------------------------------ the product
// tile number t: from the list tl, or (tl == nullptr) in row-major order over
// the lower triangle of 128-row tiles, row tile I holding column tiles
// 0 .. 2I+1.  A column tile at or past nc is empty (the last row tile of a
// size that is not a multiple of 128); every role skips it alike.
__device__ __forceinline__ bool tile_at(const int2 *__restrict__ tl, int t, int nc, int2 &out) {
  if (tl) { out = tl[t]; return true; }
  int I = (int)((sqrt(1.0 + 4.0 * (double)t) - 1.0) * 0.5);
  while ((I + 1) * (I + 2) <= t) ++I;
  while (I > 0 && I * (I + 1) > t) --I;
  out = make_int2(I, t - I * (I + 1));
  return out.y < nc;
}

__device__ __forceinline__ void note(int *err, volatile int *fail, int info) {
  if (!*fail && atomicCAS(err, 0, TW_ERR_TIMEOUT) == 0) err[1] = info;
  *fail = 1;
}

// K[i][j] = / += / -= P_ij (mode 0 / 1 / 2) over this panel for the tiles (row
// tile I of 128, column tile J of 64), entries of the lower 64-block triangle
// below n_pad only (n_pad a multiple of 64).
// Warp roles: 0-3 move A's slices to TMEM, 4-11 the epilogue (TMEM lane
// quarter = warp mod 4), 12 the bulk-copy issuer, 13 the MMA issuer.
__global__ void __launch_bounds__(SK_NTHR, 1)
k_syrk_sl(const uint8_t *__restrict__ Sl, const int *__restrict__ eg, const int2 *__restrict__ tl,
          int ntl, int natoms, double *__restrict__ K, long ldk, int n_pad, int mode, int *err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * SK_S + 2 * SK_SA + 3];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int my_tiles = (int)blockIdx.x < ntl ? (ntl - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int nchunk = (natoms + SK_CHUNK - 1) / SK_CHUNK;
  const int nc = (n_pad + SK_TN - 1) / SK_TN;
  const uint32_t sbase = (tc_su32(smem_raw) + 1023u) & ~1023u;
  const uint8_t *gbase = smem_raw + (sbase - tc_su32(smem_raw));
  const uint32_t bar0 = tc_su32(&bars[0]);
  auto full = [&](int st) { return bar0 + 8u * st; };
  auto empty = [&](int st) { return bar0 + 8u * (SK_S + st); };
  auto fullA = [&](int st) { return bar0 + 8u * (2 * SK_S + st); };
  auto emptyA = [&](int st) { return bar0 + 8u * (2 * SK_S + SK_SA + st); };
  const uint32_t tfull = bar0 + 8u * (2 * SK_S + 2 * SK_SA), tempty = tfull + 8u, drain = tfull + 16u;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(tc_su32(&tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    fail = 0;
    for (int st = 0; st < SK_S; ++st) {
      tc_mbar_init(full(st), 1);
      tc_mbar_init(empty(st), 1 + SK_NMOV / 32);     // the MMAs and each moving warp
    }
    for (int st = 0; st < SK_SA; ++st) {
      tc_mbar_init(fullA(st), SK_NMOV);
      tc_mbar_init(emptyA(st), 1);
    }
    tc_mbar_init(tfull, 1);
    tc_mbar_init(tempty, SK_NEPI);
    tc_mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  constexpr uint32_t tmem = 0;           // all 512 columns are allocated
  constexpr uint32_t tmemA = tmem + SK_NACC * SK_TN;
  volatile int *vfail = &fail;
  auto wait = [&](uint32_t bar, int parity) {      // by a whole warp
    return __all_sync(0xffffffffu, tc_mbar_wait(bar, (unsigned)(parity & 1), vfail)) != 0;
  };

  if (warp < SK_NMOV / 32) {
    // ---------------- A's slices from shared memory to TMEM: thread = row
    const uint32_t lane_base = tmemA + ((uint32_t)(32 * warp) << 16);
    int st = 0, use = 0, sa = 0, usea = 0;
    bool ok = true;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int2 t;
      if (!tile_at(tl, (int)blockIdx.x + i * (int)gridDim.x, nc, t)) continue;
      for (int a = 0; a < natoms && ok; ++a) {
        if (!wait(full(st), use)) { ok = false; break; }
        const uint8_t *src = gbase + (size_t)st * SK_STAGE;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          uint4 v[SK_NSL][2];
#pragma unroll
          for (int s = 0; s < SK_NSL; ++s)
#pragma unroll
            for (int q = 0; q < 2; ++q)
              v[s][q] = *reinterpret_cast<const uint4 *>(src + s * SK_A_SLICE + tc_swz64(tid, 2 * ks + q));
          if (ok && usea > 0 && !wait(emptyA(sa), usea - 1)) ok = false;
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int s = 0; s < SK_NSL; ++s)
            tc_st8(lane_base + (uint32_t)(sa * SK_A_COLS + 8 * s), v[s][0], v[s][1]);
          tc_wait_st();
          tc_fence_before();
          tc_mbar_arrive(fullA(sa));
          if (++sa == SK_SA) { sa = 0; ++usea; }
        }
        __syncwarp();
        if (lane == 0) tc_mbar_arrive(empty(st));
        if (++st == SK_S) { st = 0; ++use; }
      }
    }
    if (!ok && lane == 0) note(err, vfail, 34);
  } else if (warp < (SK_NMOV + SK_NEPI) / 32) {
    // ---------------- epilogue: exact level sums into int64, added to K at the end
    constexpr int CW = SK_TN / 2;
    const int lg = warp & 3, half = (warp - SK_NMOV / 32) >> 2;
    const int r = 32 * lg + lane;
    int use = 0;
    bool ok = true;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int2 t;
      if (!tile_at(tl, (int)blockIdx.x + i * (int)gridDim.x, nc, t)) continue;
      long long T[CW];
      float F[CW];
#pragma unroll
      for (int j = 0; j < CW; ++j) { T[j] = 0; F[j] = 0.f; }
      for (int c = 0; c < nchunk; ++c, ++use) {
        if (!wait(tfull, use)) { ok = false; break; }
        tc_fence_after();
        const uint32_t trow = tmem + ((uint32_t)(32 * lg) << 16) + (uint32_t)(half * CW);
#pragma unroll
        for (int c0 = 0; c0 < CW; c0 += 2) {
          uint32_t d[SK_NACC][2];
#pragma unroll
          for (int ac = 0; ac < SK_NACC; ++ac) tc_ld2(d[ac], trow + (uint32_t)(ac * SK_TN + c0));
          tc_wait_ld();
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            long long x = __float2int_rn(__uint_as_float(d[0][j]));
#pragma unroll
            for (int L = 1; L < 5; ++L)
              x = x * 256 + __float2int_rn(__uint_as_float(d[L][j]) * tc_pow2f(8 * L));
            T[c0 + j] += x;
            F[c0 + j] += __uint_as_float(d[5][j]);
          }
        }
        // the accumulators are read: the next chunk's MMAs may overwrite them
        tc_fence_before();
        tc_mbar_arrive(tempty);
      }
      if (!ok) break;
      // a 64-column tile is one 64-block: one mask for the row
      const long row = (long)t.x * SK_TM + r, col0 = (long)t.y * SK_TN + half * CW;
      if (row < n_pad && (long)t.y <= (row >> 6)) {
        const int ei = eg[row];
        double2 *Kp = reinterpret_cast<double2 *>(K + row * ldk + col0);
#pragma unroll
        for (int q = 0; q < CW / 2; ++q) {
          const double2 o = mode != 0 ? Kp[q] : make_double2(0.0, 0.0);
          double v[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int j = 2 * q + h;
            const double p = ldexp((double)T[j] * 0x1p-32 + (double)F[j], ei + eg[col0 + j] - 14);
            const double old = h ? o.y : o.x;
            v[h] = mode == 0 ? p : (mode == 1 ? old + p : old - p);
          }
          Kp[q] = make_double2(v[0], v[1]);
        }
      }
    }
    if (!ok && lane == 0) note(err, vfail, 33);
  } else if (warp == (SK_NMOV + SK_NEPI) / 32) {
    if (lane == 0) {
      // ---------------- bulk copies: atom a of tile (I, J) into stage st
      int st = 0, use = 0, issued = 0;
      bool ok = true;
      for (int i = 0; i < my_tiles && ok; ++i) {
        int2 t;
        if (!tile_at(tl, (int)blockIdx.x + i * (int)gridDim.x, nc, t)) continue;
        const uint8_t *Abase = Sl + (size_t)t.x * natoms * SK_A_STAGE;
        const uint8_t *Bbase = Sl + (size_t)(t.y >> 1) * natoms * SK_A_STAGE + (size_t)(t.y & 1) * SK_B_SLICE;
        for (int a = 0; a < natoms; ++a) {
          if (use > 0 && !tc_mbar_wait(empty(st), (unsigned)((use - 1) & 1), vfail)) { ok = false; break; }
          const uint32_t dst = sbase + (uint32_t)st * SK_STAGE;
          tc_mbar_arrive_tx(full(st), SK_STAGE);
          tc_bulk_g2s(dst, Abase + (size_t)a * SK_A_STAGE, SK_A_STAGE, full(st));
#pragma unroll
          for (int s = 0; s < SK_NSL; ++s)
            tc_bulk_g2s(dst + SK_A_STAGE + s * SK_B_SLICE, Bbase + (size_t)a * SK_A_STAGE + (size_t)s * SK_A_SLICE,
                        SK_B_SLICE, full(st));
          ++issued;
          if (++st == SK_S) { st = 0; ++use; }
        }
      }
      if (!ok) note(err, vfail, 31);
      // copies already issued must land before the CTA's shared memory goes
      for (int a = (issued > SK_S ? issued - SK_S : 0); a < issued; ++a)
        tc_mbar_wait(full(a % SK_S), (unsigned)((a / SK_S) & 1), nullptr);
    }
  } else {
    // ---------------- MMA issuer (the warp's lanes run together, one is elected to issue)
    const uint32_t idesc = tc_idesc_bf16(SK_TM, SK_TN);
    bool ok = true;
    int st = 0, use = 0, sa = 0, usea = 0, g = 0;       // stages, their use counts, chunk count
    uint32_t dc[SK_NACC];
#pragma unroll
    for (int L = 0; L < SK_NACC; ++L) dc[L] = tmem + (uint32_t)(L * SK_TN);
    for (int i = 0; i < my_tiles && ok; ++i) {
      int2 t;
      if (!tile_at(tl, (int)blockIdx.x + i * (int)gridDim.x, nc, t)) continue;
      for (int c = 0; c < nchunk && ok; ++c, ++g) {
        // the epilogue has read the previous chunk
        if (g > 0 && !wait(tempty, g - 1)) { ok = false; break; }
        tc_fence_after();
        const int ns = 2 * (min(natoms, (c + 1) * SK_CHUNK) - c * SK_CHUNK);
        if (!wait(full(st), use) || !wait(fullA(sa), usea)) { ok = false; break; }
        // the next 16 k are waited for between the halves of this step's MMAs
        for (int s = 0; s < ns; ++s) {
          const int ks = s & 1;
          tc_fence_after();
          const uint32_t aT = tmemA + (uint32_t)(sa * SK_A_COLS);
          const uint64_t bd0 = tc_sdesc64(sbase + (uint32_t)(st * SK_STAGE + SK_A_STAGE) + 32u * ks);
          uint64_t bd[SK_NSL];
#pragma unroll
          for (int j = 0; j < SK_NSL; ++j) bd[j] = bd0 + (uint64_t)(j * (SK_B_SLICE >> 4));
          const bool last = s == ns - 1;
          if (tc_elect()) tc_issue_half<0>(s == 0, dc, aT, bd, idesc);
          __syncwarp();
          const uint32_t eA = emptyA(sa), eS = empty(st);
          if (++sa == SK_SA) { sa = 0; ++usea; }
          if (ks == 1 && ++st == SK_S) { st = 0; ++use; }
          if (!last && ((ks == 1 && !wait(full(st), use)) || !wait(fullA(sa), usea))) ok = false;
          if (tc_elect()) {
            tc_issue_half<1>(s == 0, dc, aT, bd, idesc);
            tc_commit(eA);
            if (ks == 1) tc_commit(eS);
            if (last) tc_commit(tfull);
          }
          __syncwarp();
          if (!ok) break;
        }
      }
    }
    if (!ok && lane == 0) note(err, vfail, 32);
    // every issued MMA complete before TMEM is released
    if (tc_elect()) tc_commit(drain);
    tc_mbar_wait(drain, 0, nullptr);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(512u) : "memory");
}

}  // namespace

// ------------------------------------------------------------------ host side
// the lower 64-block triangle as (128-row tile, 64-column tile): groups of 8
// row tiles, column tile outer, row tile inner
void syrk_tile_list(int n_pad, std::vector<int2> &tl) {
  const int nt = (n_pad + SK_TM - 1) / SK_TM, nc = (n_pad + SK_TN - 1) / SK_TN;
  tl.clear();
  for (int g0 = 0; g0 < nt; g0 += 8) {
    const int g1 = std::min(nt, g0 + 8);
    const int jmax = std::min(nc - 1, 2 * (g1 - 1) + 1);
    for (int J = 0; J <= jmax; ++J)
      for (int I = g0; I < g1; ++I)
        if (J <= 2 * I + 1) tl.push_back(make_int2(I, J));
  }
}

size_t syrk_ws_bytes_per_atom(int n_pad) {
  return (size_t)((n_pad + SK_TM - 1) / SK_TM) * SK_A_STAGE;
}
int syrk_exp_rows(int n_pad) { return (n_pad + SK_TM - 1) / SK_TM * SK_TM; }

// K[i][j] = (G G^T)_ij for the lower 64-block triangle of the n_pad x n_pad
// array K (rows of G >= n are zero); ws holds one panel of slices (a multiple
// of syrk_ws_bytes_per_atom), eg syrk_exp_rows(n_pad) ints, tl the tile list
cudaError_t launch_form_P_tc(const dd *G, long ldg, int n, int kdim, double *K, long ldk, int n_pad,
                             uint8_t *ws, size_t ws_bytes, int *eg, const int2 *tl, int ntl, int *err,
                             cudaStream_t s) {
  if (n <= 0 || n_pad <= 0 || ntl <= 0) return cudaSuccess;
  const int nt = (n_pad + SK_TM - 1) / SK_TM, nrows = nt * SK_TM;
  k_syrk_row_exp<<<(unsigned)(((long)nrows * 32 + 255) / 256), 256, 0, s>>>(G, ldg, n, kdim, eg, nrows);
  count_launches(1);
  const int atoms_total = (kdim + SK_KA - 1) / SK_KA;
  int per_panel = (int)std::min<size_t>(ws_bytes / syrk_ws_bytes_per_atom(n_pad), (size_t)atoms_total);
  if (per_panel > SK_CHUNK) per_panel -= per_panel % SK_CHUNK;
  if (per_panel < 1) return cudaErrorInvalidValue;
  const size_t sm = (size_t)SK_S * SK_STAGE + 1024;
  cudaFuncSetAttribute(k_syrk_sl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = (unsigned)std::max(1, std::min(ntl, nsm));
  for (int a0 = 0; a0 < atoms_total; a0 += per_panel) {
    const int na = std::min(per_panel, atoms_total - a0);
    k_syrk_slice<<<dim3((unsigned)na, (unsigned)nt), 256, 0, s>>>(G, ldg, n, kdim, a0 * SK_KA, eg, ws, na);
    count_launches(1);
    k_syrk_sl<<<grid, SK_NTHR, sm, s>>>(ws, eg, tl, ntl, na, K, ldk, n_pad, a0 == 0 ? 0 : 1, err);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// C -= A A^T for the lower 64-block triangle of the m x m array C (row
// stride ldc; m a multiple of 64), A the m x kdim FP64 panel (row stride lda,
// kdim a multiple of 32): the blocked Cholesky's trailing update, exact
// products on the tensor cores.  ws >= syrk_ws_bytes_per_atom(m) * kdim / 32
// bytes, eg >= syrk_exp_rows(m) ints.
cudaError_t launch_syrk_update_d(const double *A, long lda, int kdim, double *C, long ldc, int m,
                                 uint8_t *ws, size_t ws_bytes, int *eg, int *err, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  const int natoms = kdim / SK_KA;
  if (m % 64 != 0 || kdim % SK_KA != 0 || natoms < 1 || ws_bytes < syrk_ws_bytes_per_atom(m) * natoms)
    return cudaErrorInvalidValue;
  const int nt = (m + SK_TM - 1) / SK_TM, nrows = nt * SK_TM;
  k_syrk_row_exp_d<<<(unsigned)(((long)nrows * 32 + 255) / 256), 256, 0, s>>>(A, lda, m, kdim, eg, nrows);
  count_launches(1);
  k_syrk_slice_d<<<dim3((unsigned)natoms, (unsigned)nt), 256, 0, s>>>(A, lda, m, kdim, eg, ws, natoms);
  count_launches(1);
  const size_t sm = (size_t)SK_S * SK_STAGE + 1024;
  cudaFuncSetAttribute(k_syrk_sl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int ntl = nt * (nt + 1);                 // closed-form row-major order
  const unsigned grid = (unsigned)std::max(1, std::min(ntl, nsm));
  k_syrk_sl<<<grid, SK_NTHR, sm, s>>>(ws, eg, nullptr, ntl, natoms, C, ldc, m, 2, err);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace tw
