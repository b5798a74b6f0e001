// pc_price.cuh -- the pricing kernel's body: program staging, the tile
// loop and the per-tile reduction, generic in the payoff evaluator
// (the interpreter eval_path, or a run-time specialised evaluator).
#pragma once

#include "pc_device.cuh"

namespace pc {

// EVAL(P, pool, R, g, live0, live1, Bm, S0) -> float2 payoffs of the lane's
// two paths.
template <int D, bool WRITE, typename EVAL>
__device__ __forceinline__ void price_tiles(const PriceArgs &a, EVAL eval) {
  extern __shared__ __align__(16) uint32_t smem[];
  const Staged st = stage_program(a, smem);
  const uint4 *P = st.P;
  const float *pool = st.pool;
  float2 *R = warp_region(st.regions, layout_of(a).words);
  const float(&Bm)[D * D] = *reinterpret_cast<const float(*)[D * D]>(a.m.Bv);
  const float(&S0)[D] = *reinterpret_cast<const float(*)[D]>(a.m.S0v);
  const int lane = threadIdx.x & 31;
  Rng2 g;
  rng_init(g, a.rk, a.stream, a.path_offset);
  const uint64_t n = walk_paths<WRITE>(a), n_tiles = (n + kTilePaths - 1) / kTilePaths;
  for (;;) {
    const unsigned long long tile = next_unit(a, lane);
    if (tile >= n_tiles) break;
    const uint64_t i0 = tile * kTilePaths + lane, i1 = i0 + 32;
    const bool live0 = i0 < n, live1 = i1 < n;
    rng_path(g, 0, a.path_offset + walk_path<WRITE>(a, i0, live0), a.path_offset);
    rng_path(g, 1, a.path_offset + walk_path<WRITE>(a, i1, live1), a.path_offset);
    const float2 x = eval(P, pool, R, g, live0, live1, Bm, S0);
    if (WRITE && a.list) {
      if (live0) a.out_paths[walk_path<WRITE>(a, i0, true)] = x.x;
      if (live1) a.out_paths[walk_path<WRITE>(a, i1, true)] = x.y;
      continue;
    }
    Moments<2> mo;
    if (live0) {
      mo.set(0, x.x);
      mo.set_prod(1, x.x, x.x);
      if (WRITE) a.out_paths[i0] = x.x;
    }
    if (live1) {
      mo.add(0, x.y);
      mo.add_prod(1, x.y, x.y);
      if (WRITE) a.out_paths[i1] = x.y;
    }
    int index;
    const double tp = mo.warp_total(lane, index);
    finish_tile<2>(a, tile, tp, index, lane);
    if (a.one_pass) break;
  }
  reset_units(a);
}

#if PC_PAIRS == 2
// The same with four paths a lane (two pairs): warps take pairs of
// consecutive tiles (2u, 2u + 1) from the counter; pair h of the lane holds
// tile 2u + h's paths lane and lane + 32, exactly as a one-pair lane holds a
// tile, so every path's value and every tile's partials are those of
// price_tiles.  EVAL(P, pool, R, g, live, Bm, S0) -> PV of the lane's four
// paths.
template <int D, bool WRITE, typename EVAL>
__device__ __forceinline__ void price_tiles2(const PriceArgs &a, EVAL eval) {
  extern __shared__ __align__(16) uint32_t smem[];
  const Staged st = stage_program(a, smem);
  const uint4 *P = st.P;
  const float *pool = st.pool;
  float2 *R = warp_region(st.regions, layout_of(a).words);
  const float(&Bm)[D * D] = *reinterpret_cast<const float(*)[D * D]>(a.m.Bv);
  const float(&S0)[D] = *reinterpret_cast<const float(*)[D]>(a.m.S0v);
  const int lane = threadIdx.x & 31;
  const uint64_t n = walk_paths<WRITE>(a), n_tiles = (n + kTilePaths - 1) / kTilePaths, n_pairs = (n_tiles + 1) / 2;
  RngH<2> g;
  rng_init(g, a.rk, a.stream, a.path_offset);
  for (;;) {
    const unsigned long long u = next_unit(a, lane);
    if (u >= n_pairs) break;
    uint64_t idx[4];
    bool live[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      idx[q] = (2 * u + (q >> 1)) * kTilePaths + lane + 32 * (q & 1);
      live[q] = idx[q] < n;
      rng_path(g, q, a.path_offset + walk_path<WRITE>(a, idx[q], live[q]), a.path_offset);
    }
    const PV x = eval(P, pool, R, g, live, Bm, S0);
    if (WRITE && a.list) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (live[q]) a.out_paths[walk_path<WRITE>(a, idx[q], true)] = pv_get(x, q);
      continue;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint64_t tile = 2 * u + h;
      if (tile >= n_tiles) break;  // warp-uniform
      const float x0 = pv_get(x, 2 * h), x1 = pv_get(x, 2 * h + 1);
      Moments<2> mo;
      if (live[2 * h]) {
        mo.set(0, x0);
        mo.set_prod(1, x0, x0);
        if (WRITE) a.out_paths[idx[2 * h]] = x0;
      }
      if (live[2 * h + 1]) {
        mo.add(0, x1);
        mo.add_prod(1, x1, x1);
        if (WRITE) a.out_paths[idx[2 * h + 1]] = x1;
      }
      int index;
      const double tp = mo.warp_total(lane, index);
      finish_tile<2>(a, tile, tp, index, lane);
    }
    if (a.one_pass) break;
  }
  reset_units(a);
}
#endif

}  // namespace pc
