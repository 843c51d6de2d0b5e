// trsm_tc.cu -- the batched triangular solves in panels: the bulk of the
// factor is applied by matrix products on the 5th-generation tensor cores.
//
// A sweep z_I = Linv_I d_I - sum_J Lf_IJ z_J (forward; trsm.cu) is cut into
// panels of PW = 12 block rows.  Per panel
//   1. k_trsm (trsm.cu) finishes the panel's rows: within the panel the
//      dependencies are few, so this is the chain of hand-offs alone;
//   2. k_zslice cuts the panel's z into bf16 slices;
//   3. k_trsm_upd adds Lf(rows past the panel, panel) z(panel) to the running
//      sums of every later row, which live in the rows of z not yet solved.
// The backward sweep does the same from the last panel up with Lb^T.
//
// Why.  In k_trsm alone the 64 x 64 blocks are multiplied in double-float on
// the FP32 pipe (15 operations a product), which bounds it: n^2 B / 2 products
// a sweep, 28 ms for 64 right-hand sides at n = 40,000.  Cut into seven exact
// bf16 slices (tc.cuh), a product costs 28 bf16 multiply-adds, which the
// tensor cores do at some 30 times that rate; the factor is then read once
// per 64 right-hand sides.
//
// Accuracy.  As in gemm_sl64.cu: a row of the factor and a column of z have a
// power-of-two exponent per chunk of 192 (three blocks), the level sums of a
// chunk are exact, and chunks are added in double-float; k_trsm rounds its
// running sum after every product.  Loud entries of z that meet small ones of the
// factor leave fewer digits to a sum than double-float does: such sums are found from
// their magnitudes (k_trsm_mag) and formed again in double-float before their row is
// solved (k_trsm_redo).
//
// Panels are separate launches: the products need no flags, and the order of
// every column's sum is fixed by the block rows alone, so a right-hand side
// does not depend on its batch mates.
#include <algorithm>

#include "../../include/tw.h"
#include "dense_api.h"
#include "kernels.h"
#include "tc.cuh"

namespace tw {

namespace {

constexpr int PW = 12;                   // block rows per panel (a multiple of 6)
constexpr int CB = 3;                    // blocks per exact chunk (192 k)
constexpr int NCH = PW / CB;             // chunks per panel
constexpr int PK = PW * NB_;             // k per panel
constexpr int TM = 128;                  // MMA M: factor rows per tile
constexpr int CH_ATOMS = CB * NB_ / 32;  // 32-wide atoms per chunk
constexpr int ATOMS = NCH * CH_ATOMS;    // atoms per panel
constexpr int NSL = TC_NSL, NACC = TC_NACC;
constexpr int A_COLS = NSL * 8;          // TMEM columns of a 16-wide A stage
constexpr int NGRP = 256, NPROD = 2 * NGRP, NEPI = 256;
constexpr int NTHR = NPROD + NEPI + 64;
constexpr int MAXA = 4, SB = 3;          // A stages (at most), B stages
constexpr int RAW_D = 2;                 // raw slots per producer group
constexpr int RAW_ROW = 16 * 8 + 16;     // a row's 16 entries, padded (bank conflicts)
constexpr int RAW_SLOT = TM * RAW_ROW;   // 18 KB
constexpr int NMAX = 64;                 // right-hand sides per tile: 6 x 64 = 384 TMEM columns

__device__ __forceinline__ void note(int *err, volatile int *fail, int info) {
  if (!*fail && atomicCAS(err, 0, TW_ERR_TIMEOUT) == 0) err[1] = info;
  *fail = 1;
}
// largest number of rows any right-hand side's window takes
__device__ __forceinline__ int max_rows(const int *win, int B, int Nd, int Nt) {
  int n = 0;
  for (int b = threadIdx.x & 31; b < B; b += 32) n = max(n, Nd * min(max(__ldg(win + b), 0), Nt));
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) n = max(n, __shfl_xor_sync(0xffffffffu, n, m));
  return n;
}

// ------------------------------------------------ exponents of the factor
// e[c][i] over the blocks J of chunk c (CB c .. CB c + CB-1): row i of Lf_IJ,
// J < I (forward), column i of Lb_JI, J > I (backward).  grid (NB, nchunk)
template <bool FWD>
__global__ void __launch_bounds__(256)
k_upd_exp(const dd *__restrict__ Lx, int8_t *__restrict__ e, int NB) {
  const int I = blockIdx.x, c = blockIdx.y, r = threadIdx.x & 63, q = threadIdx.x >> 6;
  __shared__ float red[4][NB_];
  float mx = 0.f;
  for (int J = c * CB; J < c * CB + CB && J < NB; ++J) {
    if (FWD ? J >= I : J <= I) continue;
    const dd *blk = Lx + (FWD ? packed_index(I, J) : packed_index(J, I)) * NB_ * NB_;
    for (int k = q * 16; k < q * 16 + 16; ++k) mx = fmaxf(mx, fabsf(FWD ? blk[r * NB_ + k].hi : blk[k * NB_ + r].hi));
  }
  red[q][r] = mx;
  __syncthreads();
  if (q == 0)
    e[((size_t)c * NB + I) * NB_ + r] =
        (int8_t)tc_exp_above(fmaxf(fmaxf(red[0][r], red[1][r]), fmaxf(red[2][r], red[3][r])));
}

// ------------------------------------------------ slices of a panel's z
// tiles [nt][chunk][atom][slice][N][32 bf16] (64-byte swizzle), column exponents
// ez[nt][chunk][N] and magnitudes mag[nt][N][PK] (bf16, for the guard); blocks at or
// past NB are zero.  grid (NCH, ntiles, tasks / 256): a CTA cuts 256 pieces of eight
// entries, after the exponents of the columns they lie in
__global__ void __launch_bounds__(256)
k_zslice(const dd *__restrict__ z, long zs, int J0, int NB, int B, int N, uint8_t *__restrict__ tiles,
         int *__restrict__ ez, uint16_t *__restrict__ mag) {
  __shared__ int e_sh[NMAX];
  const int c = blockIdx.x, nt = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long k0 = (long)(J0 + c * CB) * NB_, kend = min((long)NB * NB_, k0 + CB * NB_);
  const int t = blockIdx.z * 256 + threadIdx.x, per_col = 4 * CH_ATOMS;
  for (int n = blockIdx.z * 256 / per_col + warp; n <= (int)(blockIdx.z * 256 + 255) / per_col && n < N; n += 8) {
    const int b = nt * N + n;
    float mx = 0.f;
    if (b < B)
#pragma unroll
      for (long k = k0 + lane; k < kend; k += 32) mx = fmaxf(mx, fabsf(z[(long)b * zs + k].hi));
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
    if (lane == 0) {
      e_sh[n] = tc_exp_above(mx);
      ez[(nt * NCH + c) * N + n] = e_sh[n];
    }
  }
  __syncthreads();
  const size_t slice_bytes = (size_t)N * 64;
  uint8_t *base = tiles + (size_t)(nt * NCH + c) * CH_ATOMS * NSL * slice_bytes;
  if (t < CH_ATOMS * N * 4) {
    // consecutive threads take consecutive 8-entry pieces of a column
    const int q = t & 3, a = (t >> 2) % CH_ATOMS, n = t / (4 * CH_ATOMS), b = nt * N + n;
    const long k = k0 + 32 * a + 8 * q;
    const float sc1 = tc_pow2f(7 - e_sh[n]);
    const f2 sc = f2_make(sc1, sc1);
    Slicer7 sl[4];
    uint32_t mg[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);      // two entries (k is a multiple of 8)
      if (b < B && k < kend) v = *reinterpret_cast<const float4 *>(z + (long)b * zs + k + 2 * u);
      sl[u].init(v.x, v.y, v.z, v.w, sc);
      mg[u] = tc_pack_bf16(fabsf(v.x), fabsf(v.z));
    }
    *reinterpret_cast<uint4 *>(mag + (size_t)(nt * N + n) * PK + c * CB * NB_ + 32 * a + 8 * q) =
        make_uint4(mg[0], mg[1], mg[2], mg[3]);
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

// ------------------------------------------------ the guard (tc.cuh)
// A row's sum runs over all panels before it, so it is judged when its own panel
// is due: se[nt][row][N] holds S and (a bound of) the root of the sum of 192 T^2 so
// far.  S is
// taken from 16 of every 64 k, a quarter of the factor: a lower bound still, and one
// that settles all but a few sums in a thousand (first and last panels apart; panel
// by panel, a tenth to a half of the early panels' sums stayed open).  A CTA takes
// 16 rows and N columns, each of its four warps three of the panel's blocks and a
// quarter of the columns' ends: a panel's latency counts more than its reads.
template <bool FWD>
__global__ void __launch_bounds__(128)
k_trsm_mag(const dd *__restrict__ Lx, const int8_t *__restrict__ ea, const uint16_t *__restrict__ mag,
           const int *__restrict__ ez, float2 *__restrict__ se, const int *__restrict__ win, int Nd, int Nt, int B,
           int N, int J0, int row0, int NB) {
  __shared__ float4 part[4][8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int nmax = max_rows(win, B, Nd, Nt), nt = blockIdx.y;
  const int i0 = row0 + blockIdx.x * 16;                   // 16 rows of one block row
  if ((long)J0 * NB_ >= nmax || i0 >= nmax) return;
  const int ia = i0 + g, I = ia >> 6, nf = N / 8;
  const uint16_t *mw = mag + (size_t)(nt * N + g) * PK + 4 * c;
  float d[8][4] = {};
#pragma unroll
  for (int jj = 0; jj < PW / 4; ++jj) {
    const int J = J0 + warp * (PW / 4) + jj;
    if (J >= NB) continue;
    const dd *blk = Lx + (FWD ? packed_index(I, J) : packed_index(J, I)) * NB_ * NB_;
    const int k0 = 16 * (J & 3), k = k0 + 4 * c;
    float r[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = (ia & 63) + 8 * h;
      if (FWD) {
        const float4 *p = reinterpret_cast<const float4 *>(blk + i * NB_ + k);
        const float4 u = __ldg(p), v = __ldg(p + 1);
        r[h][0] = fabsf(u.x), r[h][1] = fabsf(u.z), r[h][2] = fabsf(v.x), r[h][3] = fabsf(v.z);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) r[h][j] = fabsf(__ldg(&blk[(k + j) * NB_ + i].hi));
      }
    }
    const uint32_t a[4] = {tc_pack_bf16(r[0][0], r[0][1]), tc_pack_bf16(r[1][0], r[1][1]),
                           tc_pack_bf16(r[0][2], r[0][3]), tc_pack_bf16(r[1][2], r[1][3])};
#pragma unroll
    for (int f = 0; f < 8; ++f)
      if (f < nf) {
        const uint2 q = __ldg(reinterpret_cast<const uint2 *>(mw + (size_t)(8 * f) * PK + (J - J0) * NB_ + k0));
        const uint32_t b[2] = {q.x, q.y};
        tc_mma_mag(d[f], a, b);
      }
  }
#pragma unroll
  for (int f = 0; f < 8; ++f) part[warp][f][lane] = make_float4(d[f][0], d[f][1], d[f][2], d[f][3]);
  __syncthreads();
  int er[2][NCH];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int q = 0; q < NCH; ++q) er[h][q] = __ldg(ea + (size_t)(J0 / CB + q) * NB * NB_ + ia + 8 * h);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int f = 2 * warp + u, n = 8 * f + 2 * c;
    if (f >= nf) break;
    float S[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const float4 q = part[v][f][lane];
      S[0] += q.x, S[1] += q.y, S[2] += q.z, S[3] += q.w;
    }
    int ec[2][NCH];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int q = 0; q < NCH; ++q) ec[i][q] = __ldg(ez + (nt * NCH + q) * N + n + i);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 *p = reinterpret_cast<float4 *>(se + ((size_t)nt * NB * NB_ + ia + 8 * h) * N + n);
      float4 o = *p;
      o.x += S[2 * h];
      o.z += S[2 * h + 1];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        int top = -1000;
#pragma unroll
        for (int q = 0; q < NCH; ++q) top = max(top, er[h][q] + ec[i][q]);
        // four chunks of 192, added in quadrature: sqrt(192 v) 2^top with v = sum of 4^(e - top),
        // 1 to 4; sqrt(v) <= (v + 2) / sqrt(8), 6% at most above
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < NCH; ++q) v += tc_pow2f(2 * max(er[h][q] + ec[i][q] - top, -60));
        const float t = top > 120 ? __int_as_float(0x7f800000) : 4.899f * (v + 2.f) * tc_pow2f(max(top, -126));
        float &E = i ? o.w : o.y;
        const float hi = fmaxf(E, t), r = __fdividef(fminf(E, t), hi);
        E = hi * (1.f + 0.5f * r * r);
      }
      *p = o;
    }
  }
}

// before panel I0 .. I1-1 is solved: its rows' sums that fail are formed in double-float
// over all k before the panel (FWD: below I0, else from I1 up), a CTA each.  Of 64
// events of the benchmark about one sum in a thousand does, in the first three panels
// forward and in half of the panels backward; with k_trsm_mag 1.9 ms a sweep.
template <bool FWD>
__global__ void __launch_bounds__(256)
k_trsm_redo(const dd *__restrict__ Lx, const float2 *__restrict__ se, dd *__restrict__ out, long zs,
            const int *__restrict__ win, int Nd, int Nt, int B, int N, int I0, int I1, int NB) {
  __shared__ int list[256], count;
  __shared__ dd sh[8];
  const int lane = threadIdx.x & 31, nmax = max_rows(win, B, Nd, Nt);
  const int kb = FWD ? 0 : I1 * NB_, ke = FWD ? I0 * NB_ : min(NB * NB_, (nmax + NB_ - 1) / NB_ * NB_);
  const int rows = min((I1 - I0) * NB_, nmax - I0 * NB_);
  const long pairs = ke > kb && rows > 0 ? (long)rows * B : 0;
  for (long p0 = blockIdx.x; p0 < pairs; p0 += 256L * gridDim.x) {
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    const long p = p0 + (long)gridDim.x * threadIdx.x;     // a column's rows go to different CTAs
    if (p < pairs) {
      const int b = (int)(p / rows), row = I0 * NB_ + (int)(p % rows);
      const float2 v = se[((size_t)(b / N) * NB * NB_ + row) * N + b % N];
      // the sum itself bounds S as well: where a few k make most of it, the sample may
      // miss them, but they hardly cancel
      const float S = fmaxf(v.x, fabsf(out[(long)b * zs + row].hi));
      if (row < Nd * min(max(__ldg(win + b), 0), Nt) && tc_guard_fails(S, v.y)) list[atomicAdd(&count, 1)] = threadIdx.x;
    }
    __syncthreads();
    const int n = count;
    for (int q = 0; q < n; ++q) {
      const long pq = p0 + (long)gridDim.x * list[q];
      const int b = (int)(pq / rows), row = I0 * NB_ + (int)(pq % rows), I = row >> 6;
      const dd *zb = out + (long)b * zs;
      dd a[4] = {dd_zero(), dd_zero(), dd_zero(), dd_zero()};      // four chains in flight
      for (int k = kb + threadIdx.x; k < ke; k += 1024)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int kk = k + 256 * u, J = kk >> 6;
          if (kk >= ke) continue;
          const dd *blk = Lx + (FWD ? packed_index(I, J) : packed_index(J, I)) * NB_ * NB_;
          a[u] = dd_add(a[u], dd_mul(FWD ? blk[(row & 63) * NB_ + (kk & 63)] : blk[(kk & 63) * NB_ + (row & 63)], zb[kk]));
        }
      const dd y = tc_warp_sum(dd_add(dd_add(a[0], a[1]), dd_add(a[2], a[3])));
      __syncthreads();                   // the sum before is read
      if (lane == 0) sh[threadIdx.x >> 5] = y;
      __syncthreads();
      if (threadIdx.x == 0) {
        dd x = sh[0];
        for (int v = 1; v < 8; ++v) x = dd_add(x, sh[v]);
        out[(long)b * zs + row] = x;
      }
    }
    __syncthreads();                     // the list is read
  }
}

// ------------------------------------------------ the update
template <int N>
struct Cfg {
  static constexpr int nbuf = 2 * NACC * N + 2 * A_COLS <= 512 ? 2 : 1;
  static constexpr int left = (512 - nbuf * NACC * N) / A_COLS;
  static constexpr int SA = left < MAXA ? left : MAXA;
  static constexpr uint32_t b_slice = (uint32_t)N * 64u, b_stage = NSL * b_slice;
  static constexpr uint32_t raw = 2 * RAW_D * RAW_SLOT, acc = N * TM * 8;
  static constexpr size_t smem = 1024 + SB * b_stage + raw + acc;
  static_assert(SA >= 2 && smem <= 227 * 1024, "stages");
};

// out[b][i] += sum_k A(i, k) z[b][k] for the rows i of tiles row0 / 128 + t, t
// < nrt, and the k of panel J0, where A = Lf (FWD) or Lb^T.  Persistent, one
// CTA per SM over (right-hand-side tile, row tile); roles as in gemm_sl64.cu.
// The chunks of a tile are summed in shared memory.
template <int N, bool FWD>
__global__ void __launch_bounds__(NTHR, 1)
k_trsm_upd(const dd *__restrict__ Lx, const int8_t *__restrict__ ea, const uint8_t *__restrict__ Bt,
           const int *__restrict__ ez, dd *__restrict__ out, long zs, const int *__restrict__ win, int Nd,
           int Nt, int B, int ntiles, int J0, int row0, int nrt, int NB, int *err) {
  constexpr int SA = Cfg<N>::SA, nbuf = Cfg<N>::nbuf;
  constexpr uint32_t b_slice = Cfg<N>::b_slice, b_stage = Cfg<N>::b_stage;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * MAXA + 2 * SB + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  // rows at or past the largest window are zero in every column (the whole CTA agrees)
  const int nmax = max_rows(win, B, Nd, Nt);
  if ((long)J0 * NB_ >= nmax) return;
  const int nrt_a = min(nrt, (nmax - row0 + TM - 1) / TM);   // active row tiles (FWD may have none)
  const int T = nrt_a > 0 ? nrt_a * ntiles : 0;
  const int my_tiles = (int)blockIdx.x < T ? (T - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  if (my_tiles == 0) return;
  const uint32_t sB0 = (tc_su32(smem_raw) + 1023u) & ~1023u, sRaw = sB0 + SB * b_stage;
  uint8_t *gRaw = smem_raw + (sRaw - tc_su32(smem_raw));
  float2 *sAcc = reinterpret_cast<float2 *>(gRaw + Cfg<N>::raw);   // [N][128]
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
  constexpr uint32_t tmemA = tmem + (uint32_t)(nbuf * NACC * N);
  volatile int *vfail = &fail;
  // tile i of this CTA: first row and right-hand-side tile (fastest)
  auto tile_of = [&](int i, int &r0, int &nt) {
    const int t = (int)blockIdx.x + i * (int)gridDim.x;
    nt = t % ntiles;
    r0 = row0 + t / ntiles * TM;
  };

  if (warp < NPROD / 32) {
    // ---------------- producers: A slices into TMEM.  Group g fills stage g of
    // every atom; thread = row r, entries 8h .. 8h+7 of the stage's 16 k.
    // Forward: a row's entries are contiguous, so the group copies whole rows
    // (8 threads a row) and exchanges them through shared memory; backward:
    // consecutive rows are contiguous and each thread copies its own entries.
    const int tg = tid & (NGRP - 1), r = tg & (TM - 1), h = tg >> 7, g = tid / NGRP;
    const uint32_t raw0 = sRaw + (uint32_t)(g * RAW_D * RAW_SLOT);
    const uint8_t *rawp = gRaw + g * RAW_D * RAW_SLOT;
    int ii = 0, ia = 0, islot = 0, ir0 = 0, int_;
    tile_of(0, ir0, int_);
    auto load = [&]() {
      if (ii < my_tiles) {
        const int kk = 32 * ia + 16 * g, J = J0 + (kk >> 6), k = kk & 63;
        if (FWD) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int q = u * NGRP + tg, row = q >> 3, ch = q & 7, i = ir0 + row, I = i >> 6;
            const bool in = I < NB;       // J < I: the panel lies left of every row
            const dd *src = in ? Lx + packed_index(I, J) * NB_ * NB_ + (i & 63) * NB_ + k + 2 * ch : Lx;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(raw0 + (uint32_t)(islot * RAW_SLOT + row * RAW_ROW + ch * 16)), "l"(src),
                           "r"(in ? 16 : 0) : "memory");
          }
        } else {
          const int i = ir0 + r, I = i >> 6;
          const bool in = J < NB;         // I < J0: every row lies above the panel
          const dd *src = in ? Lx + packed_index(J, I) * NB_ * NB_ + (k + 8 * h) * NB_ + (i & 63) : Lx;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;"
                         ::"r"(raw0 + (uint32_t)(islot * RAW_SLOT + (u * NGRP + tg) * 8)),
                           "l"(in ? src + u * NB_ : Lx), "r"(in ? 8 : 0) : "memory");
        }
        if (++ia == ATOMS) {
          ia = 0;
          if (++ii < my_tiles) tile_of(ii, ir0, int_);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      islot ^= 1;
    };
    load();
    int slot = 0, st = g, use = 0;
    bool ok = true;
    const uint32_t lane_base = tmemA + ((uint32_t)(32 * (warp & 3)) << 16) + 4u * h;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int r0, nt;
      tile_of(i, r0, nt);
      f2 sc = f2_make(0.f, 0.f);
      for (int a = 0; a < ATOMS; ++a) {
        if (a % CH_ATOMS == 0) {
          const int row = r0 + r;
          const float sc1 =
              tc_pow2f(7 - (row < NB * NB_ ? (int)__ldg(ea + (size_t)(J0 / CB + a / CH_ATOMS) * NB * NB_ + row) : 0));
          sc = f2_make(sc1, sc1);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // the group's copies of this slot are in, and every thread has read the other one
        if (FWD) asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(NGRP) : "memory");
        load();
        Slicer7 sl[4];
        if (FWD) {
          const float4 *p = reinterpret_cast<const float4 *>(rawp + slot * RAW_SLOT + r * RAW_ROW + h * 64);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 v = p[u];
            sl[u].init(v.x, v.y, v.z, v.w, sc);
          }
        } else {
          const float2 *p = reinterpret_cast<const float2 *>(rawp + slot * RAW_SLOT) + tg;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float2 v = p[2 * u * NGRP], v2 = p[(2 * u + 1) * NGRP];
            sl[u].init(v.x, v.y, v2.x, v2.y, sc);
          }
        }
        slot ^= 1;
        if (use > 0) {
          const bool got = tc_mbar_wait(emptyA(st), (unsigned)((use - 1) & 1), vfail);
          if (!__all_sync(0xffffffffu, got)) {
            if (lane == 0) note(err, vfail, 51);
            ok = false;
          }
        }
        if (ok) {      // after a failure the group's barriers still have to be met
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
        }
        st += 2;
        while (st >= SA) { st -= SA; ++use; }
      }
      if (FWD) {       // leave together: a warp that failed must not strand the others at the barrier
        int all;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
                     "barrier.cta.red.and.pred q, %2, %3, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                     : "=r"(all) : "r"((int)ok), "r"(1 + g), "r"(NGRP) : "memory");
        ok = all != 0;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // own copies drained before exit
  } else if (warp < (NPROD + NEPI) / 32) {
    // ---------------- epilogue (two warps a TMEM lane quarter, each half of the columns)
    const int lg = warp & 3, half = (warp - NPROD / 32) >> 2;
    const int r = 32 * lg + lane;
    constexpr int CW = N / 2;
    bool ok = true;
    int bf = 0, use = 0;
    float2 *acc = sAcc + half * CW * TM + r;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int r0, nt;
      tile_of(i, r0, nt);
      const int row = r0 + r, b0 = nt * N + half * CW;
      const bool in = row < NB * NB_;
      for (int c = 0; c < NCH; ++c) {
        const float sa = tc_pow2f((in ? (int)__ldg(ea + (size_t)(J0 / CB + c) * NB * NB_ + row) : 0) - 7);
        const int *ezc = ez + (nt * NCH + c) * N + half * CW;
        const bool got = tc_mbar_wait(tfull(bf), (unsigned)(use & 1), vfail);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) note(err, vfail, 52);
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
            const f2 sc = f2_make(sa * tc_pow2f(__ldg(ezc + c0 + j) - 7), sa * tc_pow2f(__ldg(ezc + c0 + j + 1) - 7));
            xh = mul2(xh, sc);
            xl = mul2(xl, sc);
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
      // the panel's contribution joins the rows' running sums
      if (in) {
        float2 *o = reinterpret_cast<float2 *>(out) + (long)b0 * zs + row;
#pragma unroll 1
        for (int c0 = 0; c0 < CW; c0 += 8) {
          float2 old[8];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            old[j] = b0 + c0 + j < B ? __ldcg(o + (long)(c0 + j) * zs) : make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (b0 + c0 + j >= B) continue;
            const float2 a = acc[(c0 + j) * TM];
            const dd s = dd_add(dd_make_raw(old[j].x, old[j].y), dd_make_raw(a.x, a.y));
            o[(long)(c0 + j) * zs] = make_float2(s.hi, s.lo);
          }
        }
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
    for (int i = 0; i < my_tiles * NCH && ok; ++i) {
      if (used > 0 && !wait(tempty(bf), used - 1)) { ok = false; break; }
      tc_fence_after();
      uint32_t dc[NACC];
#pragma unroll
      for (int L = 0; L < NACC; ++L) dc[L] = tmem + (uint32_t)((bf * NACC + L) * N);
      if (!wait(fullB(sb), useb) || !wait(fullA(sa), usea)) { ok = false; break; }
      // the next stage is waited for between the halves of this one's MMAs
      for (int s = 0; s < 2 * CH_ATOMS; ++s) {
        const int ks = s & 1;
        tc_fence_after();
        const uint32_t aT = tmemA + (uint32_t)(sa * A_COLS);
        const uint64_t bd0 = tc_sdesc64(sB0 + (uint32_t)sb * b_stage + 32u * ks);
        uint64_t bd[NSL];
#pragma unroll
        for (int j = 0; j < NSL; ++j) bd[j] = bd0 + (uint64_t)(j * (b_slice >> 4));
        const bool last = s == 2 * CH_ATOMS - 1;
        if (tc_elect()) tc_issue_half<0>(s == 0, dc, aT, bd, idesc);
        __syncwarp();
        const uint32_t eA = emptyA(sa), eB = emptyB(sb);
        if (++sa == SA) { sa = 0; ++usea; }
        if (ks == 1 && ++sb == SB) { sb = 0; ++useb; }
        if (!last && ((ks == 1 && !wait(fullB(sb), useb)) || !wait(fullA(sa), usea))) ok = false;
        if (tc_elect()) {
          tc_issue_half<1>(s == 0, dc, aT, bd, idesc);
          tc_commit(eA);
          if (ks == 1) tc_commit(eB);
          if (last) tc_commit(tfull(bf));
        }
        __syncwarp();
        if (!ok) break;
      }
      if (++bf == nbuf) { bf = 0; ++used; }
    }
    if (!ok && lane == 0) note(err, vfail, 53);
    // every issued MMA complete before TMEM is released
    if (tc_elect()) tc_commit(drain);
    tc_mbar_wait(drain, 0, nullptr);
  } else if (lane == 0) {
    // ---------------- z slices: one bulk copy per atom
    int st = 0, use = 0, issued = 0;
    bool ok = true;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int r0, nt;
      tile_of(i, r0, nt);
      const uint8_t *Bw = Bt + (size_t)nt * ATOMS * b_stage;
      for (int a = 0; a < ATOMS; ++a) {
        if (use > 0 && !tc_mbar_wait(emptyB(st), (unsigned)((use - 1) & 1), vfail)) { ok = false; break; }
        tc_mbar_arrive_tx(fullB(st), b_stage);
        tc_bulk_g2s(sB0 + (uint32_t)st * b_stage, Bw + (size_t)a * b_stage, b_stage, fullB(st));
        ++issued;
        if (++st == SB) { st = 0; ++use; }
      }
    }
    if (!ok) note(err, vfail, 54);
    // copies already issued must land before the CTA's shared memory goes
    for (int a = (issued > SB ? issued - SB : 0); a < issued; ++a)
      tc_mbar_wait(fullB(a % SB), (unsigned)((a / SB) & 1), nullptr);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(512u) : "memory");
}

// right-hand sides per tile: the fewest tiles of at most NMAX, a multiple of 16
int tile_cols(int B) {
  const int nt = (B + NMAX - 1) / NMAX;
  return ((B + nt - 1) / nt + 15) / 16 * 16;
}
int tile_count(int B) { return (B + tile_cols(B) - 1) / tile_cols(B); }

}  // namespace

// ------------------------------------------------------------------ host side
// Panels against one sweep on the FP32 pipes split over threads (trsm.cu), for
// the reserved batch (not the call's, so that a column's rounding does not
// depend on its batch).  Both pay the chain from row to row; the panels add some 8 us
// a row (five launches and a wave of tiles per 12 rows) up to the largest window, the
// sweep its products, NB / 2 blocks a row for every slice of two right-hand sides,
// up to their own windows.  Measured (us a sweep, panels / split), windows of a quarter
// to the whole: they meet at slices x NB near 4,000 (313 block rows, 24 right-hand
// sides (3,756) 2,525 / 2,489; 132, 64 (4,224) 1,266 / 1,207; 260, 32 (4,160) 2,146 /
// 2,242), above the panels win (188, 48 (4,512) 1,739 / 1,973; 400, 32 (6,400) 3,641 /
// 5,394; 625, 64 (20,000) 8,245 / 22,233), below they lose (260, 24 (3,120) 2,016 /
// 1,671; 188, 24 (2,256) 1,494 / 981).  Windows that are all whole would put the line at
// 2,200 (260, 24 2,165 / 2,731).
bool trsm_tc_applies(int NB, int bmax) { return NB > 2 * PW && (long)((bmax + 1) / 2) * NB > 4096; }

static int exp_chunks(int NB) { return (NB + PW - 1) / PW * NCH; }   // whole panels
size_t trsm_tc_exp_bytes(int NB) { return (size_t)exp_chunks(NB) * NB * NB_; }
// for at most B right-hand sides (tiles hold fewer than 16 unused columns each): one
// panel's slices, magnitudes and exponents, and the guard's sums per row
static size_t z_cols(int B) { return (size_t)B + 16 * ((B + NMAX - 1) / NMAX); }
size_t trsm_tc_ws_bytes(int NB, int B) {
  return z_cols(B) *
         (ATOMS * NSL * 64 + PK * sizeof(uint16_t) + NCH * sizeof(int) + (size_t)NB * NB_ * sizeof(float2));
}

cudaError_t launch_trsm_tc_exp(const dd *Lf, const dd *Lb, int8_t *ef, int8_t *eb, int NB, cudaStream_t s) {
  const dim3 grid(NB, exp_chunks(NB));
  k_upd_exp<true><<<grid, 256, 0, s>>>(Lf, ef, NB);
  k_upd_exp<false><<<grid, 256, 0, s>>>(Lb, eb, NB);
  count_launches(2);
  return cudaGetLastError();
}

struct PanelWs {
  uint8_t *slices;
  uint16_t *mag;
  int *ez;
  float2 *se;
  size_t se_bytes;
};
static PanelWs panel_ws(void *ws, int NB, int B) {
  const size_t cols = (size_t)tile_count(B) * tile_cols(B);
  PanelWs p;
  p.slices = reinterpret_cast<uint8_t *>(ws);
  p.mag = reinterpret_cast<uint16_t *>(p.slices + cols * ATOMS * NSL * 64);
  p.ez = reinterpret_cast<int *>(p.mag + cols * PK);
  p.se = reinterpret_cast<float2 *>(p.ez + cols * NCH);
  p.se_bytes = cols * NB * NB_ * sizeof(float2);
  return p;
}

// one panel's update of the rows past it
template <bool FWD>
static cudaError_t update_panel(const dd *Lx, const int8_t *ea, dd *out, long zs, const int *win, int Nd, int Nt,
                                int B, int NB, int J0, const PanelWs &ws, int nsm, int *err, cudaStream_t s) {
  const int J1 = std::min(NB, J0 + PW);
  const int row0 = FWD ? J1 * NB_ : 0;
  const int nrt = FWD ? ((NB - J1) * NB_ + TM - 1) / TM : J0 * NB_ / TM;
  if (nrt <= 0) return cudaSuccess;
  const int N = tile_cols(B), ntiles = tile_count(B);
  k_zslice<<<dim3(NCH, ntiles, (4 * CH_ATOMS * N + 255) / 256), 256, 0, s>>>(out, zs, J0, NB, B, N, ws.slices, ws.ez, ws.mag);
  k_trsm_mag<FWD><<<dim3(((FWD ? NB - J1 : J0) * NB_) / 16, ntiles), 128, 0, s>>>(Lx, ea, ws.mag, ws.ez, ws.se, win, Nd, Nt, B, N, J0, row0, NB);
  count_launches(2);
  const int grid = std::min(nrt * ntiles, nsm);
  auto run = [&](auto NC) {
    constexpr int NN = NC.value;
    cudaFuncSetAttribute(k_trsm_upd<NN, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<NN>::smem);
    k_trsm_upd<NN, FWD><<<grid, NTHR, Cfg<NN>::smem, s>>>(Lx, ea, ws.slices, ws.ez, out, zs, win, Nd, Nt, B, ntiles, J0,
                                                          row0, nrt, NB, err);
  };
  switch (N) {
    case 16: run(std::integral_constant<int, 16>{}); break;
    case 32: run(std::integral_constant<int, 32>{}); break;
    case 48: run(std::integral_constant<int, 48>{}); break;
    default: run(std::integral_constant<int, 64>{}); break;
  }
  // the next panel's rows have all their products now
  const int p0 = FWD ? J1 : J0 - PW, p1 = FWD ? std::min(NB, J1 + PW) : J0;
  k_trsm_redo<FWD><<<(unsigned)std::min<long>((long)(p1 - p0) * NB_ * B, 4L * nsm), 256, 0, s>>>(
      Lx, ws.se, out, zs, win, Nd, Nt, B, N, p0, p1, NB);
  count_launches(2);
  return cudaGetLastError();
}

cudaError_t launch_trsm_dd_tc(const dd *Lx, const int8_t *ea, const dd *Linv, const void *rhs, int rhs_kind,
                              long rhs_bstride, dd *out, long out_bstride, const int *win, int Nd, int Nt, int B,
                              int NB, int *prog, bool fwd, void *ws, size_t ws_bytes, int *err, int *abort_flag,
                              cudaStream_t s) {
  if (B <= 0 || NB <= 0) return cudaSuccess;
  if (ws_bytes < trsm_tc_ws_bytes(NB, B) || out_bstride < (long)NB * NB_) return cudaErrorInvalidValue;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  nsm = std::max(nsm, 1);
  cudaError_t e = cudaMemsetAsync(prog, 0, sizeof(int) * trsm_prog_ints(B), s);
  const PanelWs w = panel_ws(ws, NB, B);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.se, 0, w.se_bytes, s);
  // the running sums start at zero
  if (e == cudaSuccess)
    e = cudaMemset2DAsync(out, (size_t)out_bstride * sizeof(dd), 0, (size_t)NB * NB_ * sizeof(dd), B, s);
  const int np = (NB + PW - 1) / PW;
  int base = 0;                            // tickets handed out by the panels before
  for (int p = 0; p < np && e == cudaSuccess; ++p) {
    const int J0 = (fwd ? p : np - 1 - p) * PW, J1 = std::min(NB, J0 + PW);
    e = launch_trsm_dd_panel(Lx, Linv, rhs, rhs_kind, rhs_bstride, out, out_bstride, win, Nd, Nt, B, NB, J0, J1,
                             &base, prog, fwd, err, abort_flag, s);
    if (e == cudaSuccess)
      e = fwd ? update_panel<true>(Lx, ea, out, out_bstride, win, Nd, Nt, B, NB, J0, w, nsm, err, s)
              : update_panel<false>(Lx, ea, out, out_bstride, win, Nd, Nt, B, NB, J0, w, nsm, err, s);
  }
  return e;
}

}  // namespace tw
