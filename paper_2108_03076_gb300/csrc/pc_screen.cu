// pc_screen.cu -- the screen and totals kernels (pc_screen.h).
//
// The screen is bound by issue, like the walk: per path four nodes of D
// normals with their Philox blocks computed anew (one or two a node).  Each
// lane takes a tile's two paths; a warp reserves its undecided paths' places
// in the list with one atomic.
#include <cmath>

#include "pc_device.cuh"
#include "pc_screen.h"

namespace pc {

namespace {

template <int D>
__global__ void __launch_bounds__(kBlock, 5) screen_kernel(const __grid_constant__ PriceArgs a,
                                                           const __grid_constant__ Screen s) {
  const int lane = threadIdx.x & 31;
  const float(&Bm)[D * D] = *reinterpret_cast<const float(*)[D * D]>(a.m.Bv);
  const float(&S0)[D] = *reinterpret_cast<const float(*)[D]>(a.m.S0v);
  const LoopTest<D> lt(make_uint4(s.cond.opa, s.cond.b, s.cond.c, s.cond.e));
  Rng2 g;
  rng_init(g, a.rk, a.stream, a.path_offset);
  const uint64_t warps = uint64_t(gridDim.x) * (blockDim.x / 32);
  for (uint64_t tile = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; tile < a.n_tiles; tile += warps) {
    const uint64_t i0 = tile * kTilePaths + lane, i1 = i0 + 32;
    rng_path(g, 0, a.path_offset + i0, a.path_offset);
    rng_path(g, 1, a.path_offset + i1, a.path_offset);
    float2 W[kScreenNodes][D];
    bool c0 = false, c1 = false;
    const float2 zero = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kScreenNodes; ++q) {
      float2 z[1][D];
      op_normals<D>(s.op[q], g, z);
      // nodes: the last date; the middle of (0, last); of (0, middle); of (middle, last)
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const float2 left = q == 3 ? W[1][i] : zero, right = q == 0 ? zero : q == 2 ? W[1][i] : W[0][i];
        W[q][i] = fma_x2(dup2(s.wl[q]), left, fma_x2(dup2(s.wr[q]), right, mul_x2(dup2(s.sd[q]), z[0][i])));
      }
      if (!s.test[q]) continue;
      float2 v[D];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        float2 x = dup2(s.A[q][i]);
#pragma unroll
        for (int k = 0; k <= i; ++k)
          x = make_float2(fmaf(Bm[i * D + k], W[q][k].x, x.x), fmaf(Bm[i * D + k], W[q][k].y, x.y));
        v[i] = make_float2(S0[i] * ex2_approx(x.x), S0[i] * ex2_approx(x.y));
      }
      bool h0, h1;
      lt.test(v, h0, h1);
      c0 = c0 || h0;
      c1 = c1 || h1;
    }
    const bool live0 = i0 < a.n_paths, live1 = i1 < a.n_paths;
    if (live0 && c0) s.payoffs[i0] = s.literal;
    if (live1 && c1) s.payoffs[i1] = s.literal;
    const unsigned m0 = __ballot_sync(kFull, live0 && !c0), m1 = __ballot_sync(kFull, live1 && !c1);
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(s.count, uint32_t(__popc(m0) + __popc(m1)));
    base = __shfl_sync(kFull, base, 0);
    const unsigned below = (1u << lane) - 1;
    if (live0 && !c0) s.list[base + __popc(m0 & below)] = uint32_t(i0);
    if (live1 && !c1) s.list[base + __popc(m0) + __popc(m1 & below)] = uint32_t(i1);
  }
}

__global__ void __launch_bounds__(kBlock) totals_kernel(const __grid_constant__ PriceArgs a, const float *payoffs) {
  const int lane = threadIdx.x & 31;
  const uint64_t warps = uint64_t(gridDim.x) * (blockDim.x / 32);
  for (uint64_t tile = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; tile < a.n_tiles; tile += warps) {
    const uint64_t i0 = tile * kTilePaths + lane, i1 = i0 + 32;
    Moments<2> mo;
    if (i0 < a.n_paths) {
      const float x = payoffs[i0];
      mo.set(0, x);
      mo.set_prod(1, x, x);
    }
    if (i1 < a.n_paths) {
      const float x = payoffs[i1];
      mo.add(0, x);
      mo.add_prod(1, x, x);
    }
    int index;
    const double tp = mo.warp_total(lane, index);
    finish_tile<2>(a, tile, tp, index, lane);
  }
}

// Grid of `per_sm` blocks an SM, or as many as the tiles need.
unsigned tile_grid(uint64_t n_tiles, int sm_count, int per_sm) {
  const uint64_t need = (n_tiles + kBlock / 32 - 1) / (kBlock / 32), cap = uint64_t(sm_count) * per_sm;
  return unsigned(need < cap ? need : cap);
}

}  // namespace

bool screen_program(const Program &p, const ModelHost &H, Screen &s) {
  const size_t n = p.code.size();
  if (n < 4 || H.n < kScreenDates || (p.code[0].opa & 0xffu) != X_LOOPANY) return false;
  const XInsn &L = p.code[0], &C = p.code[1];
  if (L.e >= n || (p.code[L.e].opa & 0xffu) != X_END) return false;
  const uint32_t A = C.opa >> 8, code = (A >> 4) & 7u, leaves = ((A >> 8) & 3u) + 1, rop = A & 3u;
  const bool any = (C.opa & 0xffu) == X_LANY, less = code <= 2;
  if (!((A >> kPlainBit) & 1u) || code < 1 || (C.e & 0x7f800000u) == 0x7f800000u) return false;
  if (!any && leaves > 1 && !(rop == 0 && less) && !(rop == 1 && !less)) return false;
  s = Screen{};
  s.cond = C;
  s.literal = p.pool[L.opa >> 16];
  const int mid = H.n / 2, first = int32_t(C.b) - H.t_now, last = first + int(L.b);
  const int dates[kScreenNodes] = {H.n, mid, mid / 2, (mid + H.n) / 2};
  for (int q = 0; q < kScreenNodes; ++q) {
    const BridgeOp &op = H.nodes[size_t(dates[q])];
    s.wl[q] = op.wl;
    s.wr[q] = op.wr;
    s.sd[q] = op.sd;
    s.op[q] = op.j;
    for (int i = 0; i < H.d; ++i) s.A[q][i] = H.A[size_t(dates[q]) * H.d + i].x;
    s.test[q] = dates[q] >= first && dates[q] <= last;
  }
  return true;
}

double screen_fraction(const ModelHost &H, const Screen &s) {
  const uint32_t A = s.cond.opa >> 8;
  const int leaves = int((A >> 8) & 3u) + 1, mid = H.n / 2;
  const bool less = ((A >> 4) & 7u) <= 2;
  const int dates[kScreenNodes] = {H.n, mid, mid / 2, (mid + H.n) / 2};
  float kf;
  static_assert(sizeof(kf) == sizeof(s.cond.e), "literal bits");
  __builtin_memcpy(&kf, &s.cond.e, sizeof(kf));
  if (!(kf > 0.f)) return 0.0;
  double none = 1.0;
  for (int i = 0; i < leaves && i < H.d; ++i) {
    double best = 0.0;
    for (int q = 0; q < kScreenNodes; ++q) {
      if (!s.test[q]) continue;
      const double t = H.tau[size_t(dates[q])];
      const double sd = H.sigma[size_t(i)] * std::sqrt(t);
      if (!(sd > 0.0)) continue;
      const double x = (std::log(double(kf) / H.S0[size_t(i)]) - (H.r - 0.5 * H.sigma[size_t(i)] * H.sigma[size_t(i)]) * t) / sd;
      const double below = 0.5 * std::erfc(-x / std::sqrt(2.0));
      best = std::max(best, less ? below : 1.0 - below);
    }
    none *= 1.0 - best;
  }
  return 0.8 * (1.0 - none);
}

cudaError_t launch_screen(const PriceArgs &a, const Screen &s, int sm_count, cudaStream_t st) {
  const unsigned grid = tile_grid(a.n_tiles, sm_count, 5);
  switch (a.m.d) {
    case 1: screen_kernel<1><<<grid, kBlock, 0, st>>>(a, s); break;
    case 2: screen_kernel<2><<<grid, kBlock, 0, st>>>(a, s); break;
    case 3: screen_kernel<3><<<grid, kBlock, 0, st>>>(a, s); break;
    case 4: screen_kernel<4><<<grid, kBlock, 0, st>>>(a, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_totals(const PriceArgs &a, const float *payoffs, int sm_count, cudaStream_t st) {
  totals_kernel<<<tile_grid(a.n_tiles, sm_count, 8), kBlock, 0, st>>>(a, payoffs);
  return cudaGetLastError();
}

}  // namespace pc
