// autotune.cu -- tile choice of the batched per-frequency products by measurement.
//
// The batched products (the posterior mean's adjoint F^H Y and the
// forecast's forward product F_q X, one matrix product per frequency) have
// tile parameters whose best value depends on the shapes: the number of
// right-hand sides per tensor-core tile of the mixed adjoint (how many tiles
// re-read the operator against the MMA width), the form of each FP64-class
// product (tensor cores, or FP32 pipes: for the adjoint with how many right-hand
// sides per warp), and the lanes per right-hand side of the FP32-pipe forward
// products.  tw_reserve_batch times every legal candidate on the
// context's own operator and workspaces with CUDA events (one warm-up launch,
// then the mean of two) and keeps the fastest; the choice is cached for the
// process by shape, so later contexts of the same shape skip the
// measurement.  TW_AUTOTUNE=0 in the environment keeps the built-in rules.
// None of the parameters changes a result's dependence on its batch mates:
// each column's sums run in an order fixed by the parameters alone.
#include <stdlib.h>
#include <string.h>

#include <array>
#include <map>
#include <mutex>
#include <vector>

#include "ctx.h"

using namespace tw;

namespace {

using Key = std::array<long, 8>;
std::mutex g_mu;
struct Choice {
  tw_tiles t{};
  bool fwd_tc[2] = {true, true};     // FP64-class forward products with F, F_q on the tensor cores
};
std::map<Key, Choice> g_cache;

// (a reservation without the sliced products' tables has other candidates)
Key key_of(const tw_ctx *c, int bmax) {
  return {c->Nd, c->Nq, c->Nx, c->Ny, c->Nt, bmax, (long)c->keep, c->ea64 ? 1L : 0L};
}

// mean device time of fn over two launches after one warm-up (ms; -1 on error)
template <class F>
double time_ms(F fn) {
  cudaEvent_t a = nullptr, b = nullptr;
  if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) return -1.0;
  double ms = -1.0;
  if (fn() == cudaSuccess) {
    cudaEventRecord(a, 0);
    bool ok = fn() == cudaSuccess && fn() == cudaSuccess;
    cudaEventRecord(b, 0);
    float t = 0.f;
    if (ok && cudaEventSynchronize(b) == cudaSuccess && cudaEventElapsedTime(&t, a, b) == cudaSuccess)
      ms = 0.5 * t;
  }
  cudaGetLastError();
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  return ms;
}

void apply(tw_ctx *c, tw_lane &L, const Choice &v) {
  L.sl_tile = v.t.adj_tile;
  L.adj_rw = v.t.adj_rw;
  L.fwd_lpb = v.t.fwd_lanes;
  for (int which = 0; which < 2; ++which) L.fwd_tc[which] = v.fwd_tc[which];
  c->tiles = v.t;
}

// The choice without measuring.  FP64-class products on the tensor cores where that
// was the faster form (60 and 40 steps of 12,500 and 600 points, 1 to 32 right-hand
// sides; us, SIMT less tensor cores): the adjoint from eight sensors on (2: -45, 8: 41,
// 27: 250, 100: 1,090) if it is worth the launches (600 points: 8 sensors -12, 27: 0,
// 100: 35), the forward product from 17 rows on (10: -270, 40: 1,240), with more than
// 16 right-hand sides from three on (1: -370, 3: 40, 10: 300).
Choice rule_tiles(const tw_ctx *c, const tw_lane &L) {
  Choice v;
  tw_tiles &t = v.t;
  t.adj_tile = sl_pick_tile(L.bmax);
  const double work = (double)c->Nd * c->Nm * c->Nf * ((L.bmax + 7) / 8 * 8);
  t.adj_rw = c->Nd >= 8 && work >= 6e6 ? 0 : (L.bmax > 16 ? 4 : (L.bmax > 8 ? 2 : 1));
  for (int which = 0; which < 2; ++which) {
    const int Nr = which == TW_MAP_F ? c->Nd : c->Nq;
    v.fwd_tc[which] = Nr > 16 || (L.bmax > 16 && Nr >= 3);
  }
  t.fwd_lanes = L.bmax <= 16 ? 2 : 1;
  t.adj_tile_ms = t.adj_rw_ms = t.fwd_lanes_ms = -1.0;
  t.tuned = 0;
  return v;
}

}  // namespace

namespace twb {

void copy_tiles(tw_lane &dst, const tw_lane &src) {
  dst.sl_tile = src.sl_tile;
  dst.adj_rw = src.adj_rw;
  dst.fwd_lpb = src.fwd_lpb;
  for (int which = 0; which < 2; ++which) dst.fwd_tc[which] = src.fwd_tc[which];
}

tw_status autotune_lane(tw_ctx *c, tw_lane &L) {
  Choice v = rule_tiles(c, L);
  tw_tiles &t = v.t;
  const char *env = getenv("TW_AUTOTUNE");
  if (env && strcmp(env, "0") == 0) {
    apply(c, L, v);
    return TW_OK;
  }
  const Key key = key_of(c, L.bmax);
  {
    std::lock_guard<std::mutex> g(g_mu);
    auto it = g_cache.find(key);
    if (it != g_cache.end()) {
      apply(c, L, it->second);
      return TW_OK;
    }
  }
  TW_CUDA(c, cudaSetDevice(c->dev));
  TW_CUDA(c, cudaDeviceSynchronize());
  const int Nd = c->Nd, Nq = c->Nq, Nm = c->Nm, Nf = c->Nf, B = L.bmax;
  // inputs of the timed products: zeros (the work does not depend on values)
  TW_CUDA(c, cudaMemset(L.byh, 0, (size_t)B * Nf * c->Rmax * sizeof(cdd)));
  TW_CUDA(c, cudaMemset(L.bxh, 0, (size_t)B * Nf * Nm * sizeof(cdd)));
  // 1) mixed adjoint: right-hand sides per tensor-core tile
  const int fmt = c->op[TW_MAP_F][TW_PREC_C64] ? TW_PREC_C64 : (c->op[TW_MAP_F][TW_PREC_BF16X2] ? TW_PREC_BF16X2 : -1);
  if (fmt > 0 && L.bsl_ws) {
    const void *A = c->opG[fmt] ? c->opG[fmt] : c->op[TW_MAP_F][fmt];
    const int8_t *ea = c->opG[fmt] ? c->eaG[fmt] : c->ea[TW_MAP_F][fmt];
    std::vector<int> cand;
    for (int P = 8; P <= 72 && P <= (B + 7) / 8 * 8; P += 8) cand.push_back(P);
    std::vector<double> ms;
    for (int P : cand)
      ms.push_back(time_ms([&] {
        return launch_gemm_adj_sl(A, fmt, ea, (const cdd *)L.byh, (long)Nf * Nd, (cf *)L.bxh, (long)Nf * Nm, Nf,
                                  Nd, Nm, B, P, L.bsl_ws, L.bsl_ws_n, L.bsl_eb, L.bsl_eb_n, c->d_err, 0);
      }));
    const int k = tw_autotune_pick((int)ms.size(), ms.data());
    if (k >= 0) { t.adj_tile = cand[k]; t.adj_tile_ms = ms[k]; }
  }
  // 2) forward products on the FP32 pipes (the forecast's F_q X): lanes per right-hand side
  {
    const int cand[2] = {1, 2};
    double ms[2];
    const bool f64 = c->op[TW_MAP_FQ][TW_PREC_FP64] != nullptr;
    const int ffmt = f64 ? TW_PREC_FP64 : fmt;
    for (int k = 0; k < 2; ++k)
      ms[k] = ffmt < 0 ? -1.0 : time_ms([&] {
        if (f64)
          return launch_gemm_fwd_dd(c->op[TW_MAP_FQ][0], (const cdd *)L.bxh, (long)Nf * Nm, (cdd *)L.bpart,
                                    (cdd *)L.byh, (long)Nf * Nq, Nf, Nq, Nm, B, 0, cand[k]);
        return launch_gemm_fwd_f(c->op[TW_MAP_FQ][ffmt], ffmt, (const cf *)L.bxh, (long)Nf * Nm, (cf *)L.bpart,
                                 (cf *)L.byh, (long)Nf * Nq, Nf, Nq, Nm, B, 0, cand[k]);
      });
    const int k = tw_autotune_pick(2, ms);
    if (k >= 0) { t.fwd_lanes = cand[k]; t.fwd_lanes_ms = ms[k]; }
  }
  // 3) FP64-class adjoint: on the tensor cores (0), or right-hand sides per warp
  if (c->op[TW_MAP_F][TW_PREC_FP64]) {
    const void *A = c->opG[0] ? c->opG[0] : c->op[TW_MAP_F][0];
    const int cand[4] = {0, 4, 2, 1};
    double ms[4];
    for (int k = 0; k < 4; ++k)
      ms[k] = k == 0 && !c->ea64 ? -1.0 : time_ms([&] {
        if (k == 0)
          return launch_gemm_adj_sl64(A, c->ea64, (const cdd *)L.byh, (long)Nf * Nd, (cdd *)L.bxh, (long)Nf * Nm, Nf,
                                      Nd, Nm, B, L.sl64_ws, L.sl64_ws_n, L.sl64_eb, L.sl64_eb_n, c->d_err, 0);
        return launch_gemm_adj_dd(A, (const cdd *)L.byh, (long)Nf * Nd, (cdd *)L.bxh, (long)Nf * Nm, Nf, Nd, Nm,
                                  B, 0, cand[k]);
      });
    const int k = tw_autotune_pick(4, ms);
    if (k >= 0) { t.adj_rw = cand[k]; t.adj_rw_ms = ms[k]; }
    // 4) FP64-class forward products: the adjoint's choice would not do for them (two
    // sensors and 40 forecast points: FP32 pipes faster by 45 us there, slower by 1,240
    // here; 100 sensors and one point: slower by 1,090 there, faster by 600 here).  Above
    // 16 rows the rule holds at every size measured; there the FP32-pipe form alone would
    // take most of the reservation's time (0.9 s for 100 rows and 64 right-hand sides)
    L.fwd_lpb = t.fwd_lanes;
    for (int which = 0; which < 2; ++which) {
      if ((which == TW_MAP_F ? Nd : Nq) > 16) continue;
      double f[2];
      for (int k = 0; k < 2; ++k) {
        L.fwd_tc[which] = k == 0;
        f[k] = k == 0 && !c->ea64 ? -1.0 : time_ms([&] { return forward_dd(c, L, which, B, 0); });
      }
      const int k2 = tw_autotune_pick(2, f);
      if (k2 >= 0) v.fwd_tc[which] = k2 == 0;
    }
  }
  TW_CUDA(c, cudaDeviceSynchronize());
  tw_status st = tw_check(c, 0);
  if (st != TW_OK) return st;
  t.tuned = 1;
  apply(c, L, v);
  std::lock_guard<std::mutex> g(g_mu);
  g_cache[key] = v;
  return TW_OK;
}

}  // namespace twb

extern "C" {

int tw_autotune_pick(int n, const double *ms) {
  int best = -1;
  for (int k = 0; k < n; ++k)
    if (ms && ms[k] > 0.0 && (best < 0 || ms[k] < ms[best])) best = k;
  return best;
}

tw_status tw_batch_tiles(const tw_ctx *c, tw_tiles *out) {
  if (!c || !out) return TW_ERR_ARG;
  if (c->lane.bmax <= 0) return TW_ERR_STATE;
  *out = c->tiles;
  return TW_OK;
}

tw_status tw_set_batch_tiles(tw_ctx *c, const tw_tiles *t) {
  if (!c || !t) return TW_ERR_ARG;
  if (c->lane.bmax <= 0) return twh::fail(c, TW_ERR_STATE, "tw_reserve_batch must come first");
  if (t->adj_tile < 8 || t->adj_tile > 80 || t->adj_tile % 8 != 0)
    return twh::fail(c, TW_ERR_ARG, "adj_tile must be a multiple of 8 in [8, 80]");
  if (t->adj_rw != 0 && t->adj_rw != 1 && t->adj_rw != 2 && t->adj_rw != 4)
    return twh::fail(c, TW_ERR_ARG, "adj_rw must be 0, 1, 2 or 4");
  if (t->fwd_lanes != 1 && t->fwd_lanes != 2) return twh::fail(c, TW_ERR_ARG, "fwd_lanes must be 1 or 2");
  Choice v;
  v.t = *t;
  v.t.adj_tile_ms = v.t.adj_rw_ms = v.t.fwd_lanes_ms = -1.0;
  v.t.tuned = 2;
  v.fwd_tc[0] = v.fwd_tc[1] = t->adj_rw == 0;
  apply(c, c->lane, v);
  return TW_OK;
}

void tw_autotune_clear_cache(void) {
  std::lock_guard<std::mutex> g(g_mu);
  g_cache.clear();
}

}  // extern "C"
