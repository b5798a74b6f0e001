// pc_device.cuh -- device building blocks shared by the pricing kernel
// (pc_kernels.cu) and the pathwise-sensitivity kernel (pc_greeks.cu):
// Philox4x32-10 (Salmon et al., SC'11), 24-bit uniforms, Box-Muller, the
// date-ordered Brownian bridge (normals in the order the walk uses them),
// correlated GBM, the fused multi-asset reads, and the deterministic
// reduction (float-pair tile sums, FP64 chunk sums).
//
// Per-thread state lives in shared memory as lane-interleaved slots of the
// warp's own region: slot s of lane l is at region[s * 32 + l] (float2: two
// paths per lane), so the warp-uniform slot indices give conflict-free
// accesses and the stride is a constant (a stride of the block size cost a
// multiply per slot in the interpreting kernels).
#pragma once

#include "pc_types.h"

namespace pc {
namespace {

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;
constexpr unsigned kFull = 0xffffffffu;

// 2*pi*u - pi for u = (k + 1/2) 2^-24, as one FMA in k.
constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr float kThetaScale = float(kTwoPi / 16777216.0);
constexpr float kThetaOffset = float(kTwoPi / 33554432.0 - kTwoPi / 2.0);

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sin_approx(float x) {
  float y;
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float cos_approx(float x) {
  float y;
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed FP32 pairs (f32x2): one instruction for both paths of a lane; each
// half is rounded as the scalar operation rounds it, so results are those
// of two scalar operations.
__device__ __forceinline__ float2 fma_x2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 mul_x2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 add_x2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 sub_x2(float2 a, float2 b) {
  return fma_x2(b, make_float2(-1.f, -1.f), a);  // exact product: rounds as a - b
}
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// Philox4x32-10: ten rounds of two 32x32->64 multiplies, the key bumped by
// the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += kPhiloxW0;
      k1 += kPhiloxW1;
    }
    const uint32_t hi0 = __umulhi(kPhiloxM0, c.x), lo0 = kPhiloxM0 * c.x;
    const uint32_t hi1 = __umulhi(kPhiloxM1, c.z), lo1 = kPhiloxM1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Box-Muller on one word pair of each of the lane's two paths: u_a from the
// even word, u_b from the odd word (path 0 in .x, path 1 in .y); even normal
// r cos(2 pi u_b), odd normal r sin(2 pi u_b) with r = sqrt(q), q = -2 ln u_a.
// u = (k + 1/2) 2^-24 for the 24-bit integer k = word >> 8.  Away from u = 1,
// q = -2 ln 2 lg2.approx(u), whose absolute error (about 7e-8 over (0, 1)) is
// small beside q.  Near 1, where q is tiny and both that error and the
// rounding of u to a float would dominate, q is the series 2v + v^2 +
// (2/3) v^3 of -2 ln(1 - v) in v = 1 - u, which is exact in float for
// u > 1/2 (an odd multiple of 2^-25 below 2^-1); for v < 2^-8 the terms left
// out are below 2^-26 of q.  The angle is reduced to 2 pi u_b - pi in
// (-pi, pi), where cos and sin change sign.  The scalar steps run on packed
// pairs (each lane of a packed operation rounds as the scalar one).
__device__ __forceinline__ void box_muller2(uint32_t a0, uint32_t b0, uint32_t a1, uint32_t b1,
                                            float2 &ze, float2 &zo) {
  const float2 ka = make_float2(__uint2float_rn(a0 >> 8), __uint2float_rn(a1 >> 8));
  const float2 u = fma_x2(ka, dup2(0x1p-24f), dup2(0x1p-25f));
  const float2 v = fma_x2(fma_x2(ka, dup2(-0x1p-24f), dup2(1.0f)), dup2(1.0f), dup2(-0x1p-25f));
  const float2 ql = mul_x2(dup2(-1.3862943611198906f), make_float2(lg2_approx(u.x), lg2_approx(u.y)));
  const float2 qs = mul_x2(v, fma_x2(v, fma_x2(v, dup2(0.6666666666666666f), dup2(1.0f)), dup2(2.0f)));
  const float2 q = make_float2(v.x < 0x1p-8f ? qs.x : ql.x, v.y < 0x1p-8f ? qs.y : ql.y);
  const float2 nr = make_float2(-sqrt_approx(q.x), -sqrt_approx(q.y));
  const float2 kb = make_float2(__uint2float_rn(b0 >> 8), __uint2float_rn(b1 >> 8));
  const float2 th = fma_x2(kb, dup2(kThetaScale), dup2(kThetaOffset));
  ze = mul_x2(nr, make_float2(cos_approx(th.x), cos_approx(th.y)));
  zo = mul_x2(nr, make_float2(sin_approx(th.x), sin_approx(th.y)));
}

// Two paths per lane: every value of the stack machine is a float2 (.x for
// the lane's first path, .y for its second), so each fetched and decoded
// instruction does the work of two paths and the two independent dependency
// chains (Philox rounds, Box-Muller, bridge) overlap in the pipeline.
// A lane with H pairs of paths (H = 2 in a specialised kernel with four
// paths per lane) keeps the generator state of its 2H paths.
//
// Philox at counter (b, p_lo, p_hi, stream), block after block of one path:
// only b changes.  Round 1 multiplies b and p_hi, so its first word,
// mulhi(M1, p_hi) ^ p_lo ^ key, does not depend on b: with PC_ONE_PHI (every
// path of the launch has the same p_hi: the specialised kernels, unless the
// launch's paths cross a multiple of 2^32) round 2's product of it is kept
// per path (hi, lo) in place of the counter words.  Every other word of
// rounds 1 and 2, and one of round 3's two products, then depends on b
// alone and is shared by the lane's paths: a block costs a path 32
// instructions instead of 40.  (The interpreting kernels keep the counter:
// with a third word per path for p_hi they measured 2-6 % slower.)
template <int H>
struct RngH {
#ifdef PC_ONE_PHI
  uint32_t hi[2 * H], lo[2 * H], y;
#else
  uint32_t plo[2 * H], phi[2 * H];
#endif
  uint32_t stream;
  uint32_t rk[20];  // Philox round keys (PriceArgs::rk), copied: the compiler keeps them uniform
};
using Rng2 = RngH<1>;

// Launch-wide state, then path p as the lane's path q.
template <int H>
__device__ __forceinline__ void rng_init(RngH<H> &g, const uint32_t *rk, uint32_t stream, uint64_t path_offset) {
  g.stream = stream;
#pragma unroll
  for (int i = 0; i < 20; ++i) g.rk[i] = rk[i];
#ifdef PC_ONE_PHI
  g.y = kPhiloxM1 * uint32_t(path_offset >> 32);
#else
  (void)path_offset;
#endif
}
template <int H>
__device__ __forceinline__ void rng_path(RngH<H> &g, int q, uint64_t p, uint64_t path_offset) {
#ifdef PC_ONE_PHI
  const uint32_t x = __umulhi(kPhiloxM1, uint32_t(path_offset >> 32)) ^ uint32_t(p) ^ g.rk[0];
  g.hi[q] = __umulhi(kPhiloxM0, x);
  g.lo[q] = kPhiloxM0 * x;
#else
  (void)path_offset;
  g.plo[q] = uint32_t(p);
  g.phi[q] = uint32_t(p >> 32);
#endif
}

// Philox block b of the lane's path q (round keys precomputed: no key
// arithmetic, and in a kernel parameter they come from the constant bank).
template <int H>
__device__ __forceinline__ uint4 philox_path(uint32_t b, const RngH<H> &g, int q) {
#ifdef PC_ONE_PHI
  const uint32_t z1 = __umulhi(kPhiloxM0, b) ^ g.stream ^ g.rk[1];
  uint4 c = make_uint4(__umulhi(kPhiloxM1, z1) ^ g.y ^ g.rk[2], kPhiloxM1 * z1,
                       g.hi[q] ^ ((kPhiloxM0 * b) ^ g.rk[3]), g.lo[q]);
  constexpr int kFirst = 2;
#else
  uint4 c = make_uint4(b, g.plo[q], g.phi[q], g.stream);
  constexpr int kFirst = 0;
#endif
#pragma unroll
  for (int r = kFirst; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(kPhiloxM0, c.x), lo0 = kPhiloxM0 * c.x;
    const uint32_t hi1 = __umulhi(kPhiloxM1, c.z), lo1 = kPhiloxM1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ g.rk[2 * r], lo1, hi0 ^ c.w ^ g.rk[2 * r + 1], lo0);
  }
  return c;
}

// The four normals of Philox block b for each pair h of a lane's 2H paths.
template <int H>
__device__ __forceinline__ void block_normals_h(uint32_t b, const RngH<H> &g, float2 (&e)[H][4]) {
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const uint4 x0 = philox_path<H>(b, g, 2 * h), x1 = philox_path<H>(b, g, 2 * h + 1);
    box_muller2(x0.x, x0.y, x1.x, x1.y, e[h][0], e[h][1]);
    box_muller2(x0.z, x0.w, x1.z, x1.w, e[h][2], e[h][3]);
  }
}

// Slot s of this lane in its warp's region (warp_region).
#define SL(s) R[(s) * 32]

// A specialised kernel's layout is a constant (PC_LAYOUT; a field of -1 comes
// from the arguments: jit_spec), and with a static walk the model's grid too
// (PC_GRID): slot addresses become immediate offsets, and grid checks and
// ordinals fold.
#if defined(PC_LAYOUT)
__device__ __forceinline__ Layout layout_of(const PriceArgs &a) {
  constexpr int32_t v[] = {PC_LAYOUT};
  Layout l = a.lay;
  if (v[0] >= 0) l.stack = v[0];
  if (v[1] >= 0) l.off_bstack = v[1];
  if (v[2] >= 0) l.off_cache = v[2];
  if (v[3] >= 0) l.off_win = v[3];
  if (v[4] >= 0) l.off_xwin = v[4];
  if (v[5] >= 0) l.words = v[5];
  if (v[6] >= 0) l.win = v[6];
  if (v[7] >= 0) l.ids = v[7];
  return l;
}
#else
__device__ __forceinline__ const Layout &layout_of(const PriceArgs &a) { return a.lay; }
#endif
#if defined(PC_GRID)
__device__ __forceinline__ ModelDev model_of(const PriceArgs &a) {
  constexpr int32_t v[] = {PC_GRID};
  ModelDev m = a.m;
  m.n = v[0];
  m.n_hist = v[1];
  m.t_now = v[2];
  return m;
}
#else
__device__ __forceinline__ const ModelDev &model_of(const PriceArgs &a) { return a.m; }
#endif

// This lane's slot 0 in the warp's region of `words` slots, the regions of
// the block's warps one after the other from `base`.  The offset is opaque
// to the compiler, which otherwise recomputes it from the thread index at
// the accesses (76 S2R and as many shifts and adds per tile of the autocall).
__device__ __forceinline__ float2 *warp_region(uint32_t *base, int words) {
  int off = int(threadIdx.x >> 5) * words * 32 + int(threadIdx.x & 31);
  asm volatile("" : "+r"(off));
  return reinterpret_cast<float2 *>(base) + off;
}

// The launch's program and constant pool, staged in shared memory once per
// block; the per-thread regions follow.  A specialised kernel has both in its
// code, and its regions start at once.
struct Staged {
  const uint4 *P;
  const float *pool;
  uint32_t *regions;
};
__device__ __forceinline__ Staged stage_program(const PriceArgs &a, uint32_t *smem) {
#ifdef PC_JIT
  (void)a;
  return {nullptr, nullptr, smem};
#else
  const int prog_words = a.n_insn * 4 + a.n_pool;
  const uint32_t *src = reinterpret_cast<const uint32_t *>(a.prog);
  for (int i = threadIdx.x; i < prog_words; i += blockDim.x) smem[i] = src[i];
  __syncthreads();
  return {reinterpret_cast<const uint4 *>(smem), reinterpret_cast<const float *>(smem + a.n_insn * 4),
          smem + prog_words};
#endif
}

// Window slot w (0 .. win * d - 1) of this thread: in the shared region
// (lane-interleaved after lay.off_win) or, with GW, in the thread's column
// of the HBM window (coalesced across the warp for a uniform slot).
template <bool GW>
__device__ __forceinline__ float2 win_load(const float2 *R, const Layout &lay, int w) {
  if constexpr (GW)
    return lay.gwin[int64_t(w) * lay.gstride + int64_t(blockIdx.x) * blockDim.x + threadIdx.x];
  else
    return SL(lay.off_win + w);
}
template <bool GW>
__device__ __forceinline__ void win_store(float2 *R, const Layout &lay, int w, float2 v) {
  if constexpr (GW)
    lay.gwin[int64_t(w) * lay.gstride + int64_t(blockIdx.x) * blockDim.x + threadIdx.x] = v;
  else
    SL(lay.off_win + w) = v;
}

// Per-path state of a lane's H pairs of paths; the bridge stack holds, per
// level, the D values of pair 0, then of pair 1 (D H slots a level).
template <int D, int H = 1>
struct PathState {
  float2 w[H][D];               // W at the last produced date
  int f;                        // last produced ordinal (frontier), warp-uniform
#ifdef PC_STATIC_DEPTH
  // a static walk (pc_jit.cpp): stack and normals in registers, every index a constant
  float2 bst[PC_STATIC_DEPTH][H][D];
  float2 e[H][4];               // the last Philox block's normals
  int step;                     // steps run so far, warp-uniform
#else
  float2 zc[H][3];              // words 1..3 of the last Philox block (d < 4)
  int bsp;                      // bridge stack size, warp-uniform
  int k;                        // ops run so far (the next op's number), warp-uniform
#endif
  float2 s[H][D];               // S at the last date whose values were formed: with PC_WIN_REGS (a
                                // program that reads no date behind the frontier) the whole window
};

// A path's state at its start; the bottom level of the bridge stack is
// zeroed (the root op reads it with weight 0).
template <int D, int H>
__device__ __forceinline__ void path_state_init(PathState<D, H> &ps, float2 *R, const Layout &lay) {
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int i = 0; i < D; ++i) ps.w[h][i] = make_float2(0.f, 0.f);
  ps.f = 0;
#ifdef PC_STATIC_DEPTH
  ps.step = 0;
#else
#pragma unroll
  for (int i = 0; i < D * H; ++i) SL(lay.off_bstack + i) = make_float2(0.f, 0.f);
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int i = 0; i < 3; ++i) ps.zc[h][i] = make_float2(0.f, 0.f);
  ps.bsp = 0;
  ps.k = 0;
#endif
}

// X_i = sum_k L_ik W_k.
template <int D>
__device__ __forceinline__ float2 correlated(int i, const float2 (&w)[D], const float *Lm) {
  float2 x = mul_x2(dup2(Lm[i * D]), w[0]);
#pragma unroll
  for (int k = 1; k < D; ++k)
    if (k <= i) x = fma_x2(dup2(Lm[i * D + k]), w[k], x);
  return x;
}
// X_l of a read at ordinal o > 0: from the window, or of the frontier date
// from W (a window of one date).
template <int D>
__device__ __forceinline__ float2 read_x(int o, int l, const float2 (&w)[D], const float *Lm, const float2 *R,
                                         const Layout &lay) {
  if (lay.win > 1) return SL(lay.off_xwin + (o & (lay.win - 1)) * D + l);
  float2 x = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < D; ++i)
    if (i == l) x = correlated<D>(i, w, Lm);
  return x;
}

// GBM at date t from W at the frontier into the window slot of t.  With XW
// the correlated Brownian values X = L W of the date are also kept (window
// at lay.off_xwin), which the pathwise sensitivities need.
template <int D, bool XW, bool GW, int H>
__device__ __forceinline__ void date_values(int t, PathState<D, H> &ps, const Layout &lay,
                                            float2 *R, const float (&Bm)[D * D], const float (&S0)[D],
                                            const float *Lm, const float2 (&drift)[D]) {
  static_assert(H == 1 || (!XW && !GW), "several path pairs a lane: no X window, no HBM window");
  const int ws = (t & (lay.win - 1)) * D;
#pragma unroll
  for (int h = 0; h < H; ++h) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      float2 x = drift[i];
#pragma unroll
      for (int k = 0; k <= i; ++k)
        x = make_float2(fmaf(Bm[i * D + k], ps.w[h][k].x, x.x), fmaf(Bm[i * D + k], ps.w[h][k].y, x.y));
      ps.s[h][i] = make_float2(S0[i] * ex2_approx(x.x), S0[i] * ex2_approx(x.y));
#ifdef PC_WIN_REGS
      (void)ws;
#else
      win_store<GW>(R, lay, ws + i, ps.s[h][i]);
#endif
    }
  }
  if constexpr (XW) {
    if (lay.win > 1) {  // (with a window of one date X is formed from W where it is read)
      const int xs = lay.off_xwin + (t & (lay.win - 1)) * D;
#pragma unroll
      for (int i = 0; i < D; ++i) SL(xs + i) = correlated<D>(i, ps.w[0], Lm);
    }
  }
}

#ifdef PC_STATIC_DEPTH
// One op of a static walk: op number K (its normals D K .. D K + D - 1; the
// Philox block computed last is CUR), weights at IDX of the launch's table,
// stack size BSP before it.  The first op is the root.  Everything but the
// values is known to the compiler: no op loads, no phase of the normals, no
// stack in shared memory, no loop.
template <int D, int H, int K, int IDX, int BSP, int CUR>
__device__ __forceinline__ void static_op(PathState<D, H> &ps, const RngH<H> &g, const StaticGrid &sg) {
  constexpr int B0 = (D * K) >> 2, B1 = (D * K + D - 1) >> 2;
  float2 z[H][D];
  if constexpr (B0 != CUR) block_normals_h<H>(B0, g, ps.e);
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int i = 0; i < D; ++i)
      if (((D * K + i) >> 2) == B0) z[h][i] = ps.e[h][(D * K + i) & 3];
  if constexpr (B1 != B0) {
    block_normals_h<H>(B1, g, ps.e);
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int i = 0; i < D; ++i)
        if (((D * K + i) >> 2) == B1) z[h][i] = ps.e[h][(D * K + i) & 3];
  }
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const float2 v = mul_x2(sg.sd[IDX], z[h][i]);
      if constexpr (BSP == 0) ps.bst[0][h][i] = v;
      else ps.bst[BSP][h][i] = fma_x2(sg.wl[IDX], ps.w[h][i], fma_x2(sg.wr[IDX], ps.bst[BSP - 1][h][i], v));
    }
}

// The end of step STEP of a static walk: date t popped (stack level BSP) as
// the frontier, its values formed when the program reads it.
template <int D, int H, bool XW, bool GW, int STEP, int BSP, bool READ>
__device__ __forceinline__ void static_date(int t, PathState<D, H> &ps, const Layout &lay, const StaticGrid &sg,
                                            float2 *R, const float (&Bm)[D * D], const float (&S0)[D],
                                            const float *Lm) {
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int i = 0; i < D; ++i) ps.w[h][i] = ps.bst[BSP][h][i];
  if constexpr (READ) {
    float2 drift[D];
#pragma unroll
    for (int i = 0; i < D; ++i) drift[i] = dup2(sg.A[STEP][i]);
    date_values<D, XW, GW, H>(t, ps, lay, R, Bm, S0, Lm, drift);
  }
  ps.f = t;
  ps.step = STEP + 1;
}
// the generated source defines PC_STEP: a switch on ps.step over the steps
#define NEXT_DATE(XW_, GW_, LM_) PC_STEP(XW_, GW_, LM_)
#else
#define NEXT_DATE(XW_, GW_, LM_) gen_date<D, XW_, GW_>(ps.f + 1, ps, m, lay, g, R, Bm, S0, LM_)

// The normals of op k for every path of the lane: normals D k .. D k + D - 1
// of the path (Philox block m >> 2, word m & 3).  Ops run in order, so the
// block holding normal D k is either new or the last block computed, whose
// words 1..3 the state keeps (zc); a new block is computed at most once per
// op.
template <int D, int H>
__device__ __forceinline__ void node_normals(uint32_t k, const RngH<H> &g, float2 (&zc)[H][3],
                                             float2 (&z)[H][D]) {
  if constexpr (D == 4) {
    float2 e[H][4];
    block_normals_h<H>(k, g, e);
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int i = 0; i < 4; ++i) z[h][i] = e[h][i];
  } else if constexpr (D == 2) {
    if (k & 1) {  // words 2, 3 of block k / 2
#pragma unroll
      for (int h = 0; h < H; ++h) {
        z[h][0] = zc[h][1];
        z[h][1] = zc[h][2];
      }
    } else {
      float2 e[H][4];
      block_normals_h<H>(k >> 1, g, e);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        z[h][0] = e[h][0];
        z[h][1] = e[h][1];
        zc[h][1] = e[h][2];
        zc[h][2] = e[h][3];
      }
    }
  } else if constexpr (D == 1) {
    const uint32_t ph = k & 3;
    if (ph == 0) {
      float2 e[H][4];
      block_normals_h<H>(k >> 2, g, e);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        z[h][0] = e[h][0];
        zc[h][0] = e[h][1];
        zc[h][1] = e[h][2];
        zc[h][2] = e[h][3];
      }
    } else {
#pragma unroll
      for (int h = 0; h < H; ++h) z[h][0] = ph == 1 ? zc[h][0] : ph == 2 ? zc[h][1] : zc[h][2];
    }
  } else {  // D == 3: the first normal is word ph = 3k & 3 of its block
    const uint32_t ph = (3 * k) & 3;
    if (ph == 1) {  // words 1..3 of the last block
#pragma unroll
      for (int h = 0; h < H; ++h) {
        z[h][0] = zc[h][0];
        z[h][1] = zc[h][1];
        z[h][2] = zc[h][2];
      }
    } else {
      float2 e[H][4];
      block_normals_h<H>((3 * k + 2) >> 2, g, e);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        if (ph == 0) {
          z[h][0] = e[h][0];
          z[h][1] = e[h][1];
          z[h][2] = e[h][2];
        } else if (ph == 2) {
          z[h][0] = zc[h][1];
          z[h][1] = zc[h][2];
          z[h][2] = e[h][0];
        } else {
          z[h][0] = zc[h][2];
          z[h][1] = e[h][0];
          z[h][2] = e[h][1];
        }
        zc[h][0] = e[h][1];
        zc[h][1] = e[h][2];
        zc[h][2] = e[h][3];
      }
    }
  }
}

// A bridge op's weights as packed pairs (two 16-byte loads through the
// read-only path: the address is the same in every lane), and in the by-date
// table the op's number and the right end of its interval.
struct OpRegs {
  float2 wl, wr, sd;
  uint32_t j, m;
};
__device__ __forceinline__ OpRegs load_op(const BridgeOp *p) {
  const float4 *q = reinterpret_cast<const float4 *>(p);
  const float4 a = __ldg(q), b = __ldg(q + 1);
  OpRegs o;
  o.wl = make_float2(a.x, a.y);
  o.wr = make_float2(a.z, a.w);
  o.sd = make_float2(b.x, b.y);
  o.j = __float_as_uint(b.z);
  o.m = __float_as_uint(b.w) >> 16;
  return o;
}

// One bridge op: node from W at the frontier and the top of the stack (the
// right end of its interval), pushed.  The root op has wl = wr = 0 and reads
// the bottom level, zeroed at the path's start, as its right end.
// (Branch-free: a push or keep decision per op, and a root test, cost
// register moves at the joins.)
template <int D, int H>
__device__ __forceinline__ void push_node(const OpRegs &op, const float2 (&z)[H][D], PathState<D, H> &ps,
                                          const Layout &lay, float2 *R) {
  const int top = lay.off_bstack + max(ps.bsp - 1, 0) * D * H;
  const int nxt = lay.off_bstack + ps.bsp * D * H;
#pragma unroll
  for (int h = 0; h < H; ++h) {
    float2 nw[D];
#pragma unroll
    for (int i = 0; i < D; ++i)
      nw[i] = fma_x2(op.wl, ps.w[h][i], fma_x2(op.wr, SL(top + h * D + i), mul_x2(op.sd, z[h][i])));
#pragma unroll
    for (int i = 0; i < D; ++i) SL(nxt + h * D + i) = nw[i];
  }
  ++ps.bsp;
}

// The stack's top popped as W of the new frontier date.
template <int D, int H>
__device__ __forceinline__ void pop_date(PathState<D, H> &ps, const Layout &lay, float2 *R) {
  --ps.bsp;
#pragma unroll
  for (int h = 0; h < H; ++h)
#pragma unroll
    for (int i = 0; i < D; ++i) ps.w[h][i] = SL(lay.off_bstack + ps.bsp * D * H + h * D + i);
}

// Produce date t (= frontier + 1) for the lane's paths: the bridge ops of t
// (every op pushes its node; the date's own value, the last node or one
// pushed on an earlier date, is popped), then its values.  The bridge,
// correlation and GBM products run on packed pairs (two paths of the lane);
// with H pairs a lane, each op's schedule and control serve all 2H paths.
template <int D, bool XW = false, bool GW = false, int H = 1>
__device__ __forceinline__ void gen_date(int t, PathState<D, H> &ps, const ModelDev &m,
                                         const Layout &lay, const RngH<H> &g, float2 *R,
                                         const float (&Bm)[D * D], const float (&S0)[D],
                                         const float *Lm = nullptr) {
  const int k1 = __ldg(m.date_ops + t + 1);  // ops of date t: [ps.k, k1)
  for (; ps.k < k1; ++ps.k) {
    const OpRegs op = load_op(m.ops + ps.k);
    float2 z[H][D];
    node_normals<D, H>(uint32_t(ps.k), g, ps.zc, z);
    push_node<D, H>(op, z, ps, lay, R);
  }
  pop_date<D, H>(ps, lay, R);
  float2 drift[D];
#pragma unroll
  for (int i = 0; i < D; ++i) drift[i] = __ldg(m.A + t * D + i);
  date_values<D, XW, GW, H>(t, ps, lay, R, Bm, S0, Lm, drift);
  ps.f = t;
}
#endif

#ifndef PC_JIT
// The normals of op j on their own: its Philox blocks anew, one or two.
template <int D>
__device__ __forceinline__ void op_normals(uint32_t j, const Rng2 &g, float2 (&z)[1][D]) {
  const uint32_t first = D * j;  // normals first .. first + D - 1
  uint32_t blk = first >> 2;
  float2 e[1][4];
  block_normals_h<1>(blk, g, e);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    if (((first + i) >> 2) != blk) {
      blk = (first + i) >> 2;
      block_normals_h<1>(blk, g, e);
    }
    const uint32_t w = (first + i) & 3;
    z[0][i] = w == 0 ? e[0][0] : w == 1 ? e[0][1] : w == 2 ? e[0][2] : e[0][3];
  }
}

// A path's start for an interpreted program that reads no date before t
// (Layout::skip): the frontier straight to t.  From the interval that the
// frontier opens (its right end from the by-date table) bisect while t lies
// inside, pop the right end, and again until t is popped.  Only the nodes
// above t in the bisection tree are computed, each from its own normals (its
// Philox blocks anew, one or two), so the values at t are those of the full
// walk: a contract that reads the last of 365 dates runs one op instead of
// 365.  Afterwards the state is as the full walk leaves it (next op, the words
// kept of its block).  Out of line, at the one place where little else is
// live (called from the reading instructions it cost every program 2-5 % in
// registers and spills).
template <int D, bool XW>
__device__ __noinline__ void skip_to(int t, PathState<D, 1> &ps, const PriceArgs &a, uint4 ids, float2 *R) {
  const ModelDev &m = a.m;
  const Layout &lay = a.lay;
  const float(&Bm)[D * D] = *reinterpret_cast<const float(*)[D * D]>(m.Bv);
  const float(&S0)[D] = *reinterpret_cast<const float(*)[D]>(m.S0v);
  Rng2 g;
  rng_init(g, a.rk, a.stream, 0);
  g.plo[0] = ids.x;
  g.phi[0] = ids.y;
  g.plo[1] = ids.z;
  g.phi[1] = ids.w;
  while (ps.f < t) {
    int r = int(__ldg(reinterpret_cast<const uint32_t *>(m.nodes + ps.f) + 7) >> 16);
    while (t < r) {
      r = (ps.f + r) >> 1;
      const OpRegs op = load_op(m.nodes + r);
      float2 z[1][D];
      op_normals<D>(op.j, g, z);
      push_node<D, 1>(op, z, ps, lay, R);
    }
    pop_date<D, 1>(ps, lay, R);
    ps.f = r;
  }
  float2 drift[D];
#pragma unroll
  for (int i = 0; i < D; ++i) drift[i] = __ldg(m.A + t * D + i);
  date_values<D, XW, false, 1>(t, ps, lay, R, Bm, S0, m.L, drift);
  ps.k = __ldg(m.date_ops + t + 1);
  if (t < m.n && ((D * ps.k) & 3)) {
    float2 e[1][4];
    block_normals_h<1>(uint32_t(D * ps.k) >> 2, g, e);
#pragma unroll
    for (int i = 0; i < 3; ++i) ps.zc[0][i] = e[0][1 + i];
  }
}
#endif

// The evaluators' per-date hook: called after each generated date t with
// the evaluator's reader (read(t, i): S_i at ordinal t of the lane's paths).
// NoDateHook (pricing) does nothing; the control-variate kernel's hook
// accumulates its hedge gains there.
struct NoDateHook {
  static constexpr bool kNone = true;
  template <class RD>
  __device__ __forceinline__ void on_date(int, RD &) {}
};

#if defined(PC_JIT) && !defined(PC_STATIC_DEPTH)
// Dates ps.f + 1 .. o, out of line (the specialised evaluator calls it from
// every instruction that reads a date, so it is not inlined there).
template <int D, bool GW, int H>
__device__ __noinline__ void advance_dates(int o, PathState<D, H> &ps, const ModelDev &m, const Layout &lay,
                                           const RngH<H> &g, float2 *R, const float (&Bm)[D * D],
                                           const float (&S0)[D]) {
  while (ps.f < o) gen_date<D, false, GW>(ps.f + 1, ps, m, lay, g, R, Bm, S0);
}
#endif

template <int D>
__device__ __forceinline__ void load_model_regs(const ModelDev &m, float (&Bm)[D * D],
                                                float (&S0)[D]) {
#pragma unroll
  for (int i = 0; i < D * D; ++i) Bm[i] = m.Bv[i];
#pragma unroll
  for (int i = 0; i < D; ++i) S0[i] = m.S0v[i];
}

__device__ __forceinline__ int bits(float v) { return __float_as_int(v); }
__device__ __forceinline__ float fl(int v) { return __int_as_float(v); }
__device__ __forceinline__ float2 fl2(int a, int b) { return make_float2(fl(a), fl(b)); }

__device__ __forceinline__ float cmp_code(int code, float v, float k) {
  // 1: v < k, 2: v <= k, 3: k < v, 4: k <= v
  const bool r = code == 1 ? v < k : code == 2 ? v <= k : code == 3 ? k < v : k <= v;
  return fl(int(r));
}

// Fused multi-asset value (X_LRED) or test (X_LANY) of instruction I at
// ordinal o for both paths; results of compares are 0/1 int bits.
// rd(l): S of underlying l at o (o > 0).
template <int D, typename RD>
__device__ __forceinline__ float2 fused_value_rd(const uint4 &I, int o, const float *pool, const ModelDev &m,
                                                 RD rd) {
  const uint32_t A = I.x >> 8;
  const int n = int((A >> 8) & 3u) + 1, kind = int((A >> 2) & 3u), code = int((A >> 4) & 7u);
  const bool any = (I.x & 0xffu) == X_LANY, conj = (A & 1u) != 0;
  const int rop = int(A & 3u);
  const float k = __uint_as_float(I.w);
  float2 v = make_float2(0.f, 0.f);
  for (int i = 0; i < n; ++i) {
    int l = int(A >> (10 + 2 * i)) & 3;
    l = l < D ? l : 0;
    float2 s;
    if (o > 0) {
      s = rd(l);
    } else {
      const float sv = __ldg(m.sval + (o + m.n_hist) * D + l);
      s = make_float2(sv, sv);
    }
    if (kind == 1) {
      const float c = pool[I.z + i];
      s = make_float2(__fmul_rn(s.x, c), __fmul_rn(s.y, c));
    } else if (kind == 2) {
      const float c = pool[I.z + i];
      s = make_float2(__fdiv_rn(s.x, c), __fdiv_rn(s.y, c));
    }
    if (any) {
      const float2 p = make_float2(cmp_code(code, s.x, k), cmp_code(code, s.y, k));
      if (i == 0) v = p;
      else if (conj) v = fl2(bits(v.x) & bits(p.x), bits(v.y) & bits(p.y));
      else v = fl2(bits(v.x) | bits(p.x), bits(v.y) | bits(p.y));
    } else if (i == 0) {
      v = s;
    } else if (rop == 0) {
      v = make_float2(fminf(v.x, s.x), fminf(v.y, s.y));
    } else if (rop == 1) {
      v = make_float2(fmaxf(v.x, s.x), fmaxf(v.y, s.y));
    } else {
      v = make_float2(__fadd_rn(v.x, s.x), __fadd_rn(v.y, s.y));
    }
  }
  if (!any && code) v = make_float2(cmp_code(code, v.x, k), cmp_code(code, v.y, k));
  return v;
}

#ifndef PC_JIT
// The interpreter's short form of a plain fused op (kPlainBit): leaf i is
// underlying i, unscaled.  An or of tests v < k (or v <= k) is the test of the
// smallest value, of k < v of the largest (a NaN takes part in neither), so
// every plain op is one min, max or sum and at most one comparison.  The
// general form decodes each leaf's label, scale and comparison: about 185
// instructions for a worst-of test of three against 45.
template <int D, typename RD>
__device__ __forceinline__ float2 fused_plain(const uint4 &I, int o, const ModelDev &m, RD rd) {
  const uint32_t A = I.x >> 8;
  const int n = int((A >> 8) & 3u) + 1, code = int((A >> 4) & 7u);
  const int rop = (I.x & 0xffu) == X_LANY ? (code <= 2 ? 0 : 1) : int(A & 3u);
  float2 s[D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    if (i >= n) break;
    if (o > 0) {
      s[i] = rd(i);
    } else {
      const float sv = __ldg(m.sval + (o + m.n_hist) * D + i);
      s[i] = make_float2(sv, sv);
    }
  }
  float2 v = s[0];
  if (rop == 0) {
#pragma unroll
    for (int i = 1; i < D; ++i)
      if (i < n) v = make_float2(fminf(v.x, s[i].x), fminf(v.y, s[i].y));
  } else if (rop == 1) {
#pragma unroll
    for (int i = 1; i < D; ++i)
      if (i < n) v = make_float2(fmaxf(v.x, s[i].x), fmaxf(v.y, s[i].y));
  } else {
#pragma unroll
    for (int i = 1; i < D; ++i)
      if (i < n) v = make_float2(__fadd_rn(v.x, s[i].x), __fadd_rn(v.y, s[i].y));
  }
  if (code) {
    const float k = __uint_as_float(I.w);
    const bool less = code <= 2, strict = (code & 1) != 0;
    const float ax = less ? v.x : k, bx = less ? k : v.x, ay = less ? v.y : k, by = less ? k : v.y;
    v = make_float2(fl(int(strict ? ax < bx : ax <= bx)), fl(int(strict ? ay < by : ay <= by)));
  }
  return v;
}

// A whole-loop barrier's test on the S just produced, decoded once before the
// loop: path value v of any watched underlying with sgn v < lim.  v <= k is
// v < the next float above k; an unwatched underlying's limit is -inf.  Only
// for plain ops with a finite k that reduce to an or (a min against an upper
// bound, a max against a lower one).
template <int D>
struct LoopTest {
  float lim[D], sgn;
  bool use;
  __device__ __forceinline__ explicit LoopTest(const uint4 &I) {
    const uint32_t A = I.x >> 8;
    const int n = int((A >> 8) & 3u) + 1, code = int((A >> 4) & 7u), rop = int(A & 3u);
    const float k = __uint_as_float(I.w);
    const bool less = code <= 2;
    use = (A >> kPlainBit) & 1u;
    use = use && ((I.x & 0xffu) == X_LANY || n == 1 || (rop == 0 && less) || (rop == 1 && !less));
    use = use && (I.w & 0x7f800000u) != 0x7f800000u;
    sgn = less ? 1.f : -1.f;
    float l = sgn * k;
    if (!(code & 1)) {  // the next float above
      const int b = __float_as_int(l);
      l = l == 0.f ? __int_as_float(1) : __int_as_float(b > 0 ? b + 1 : b - 1);
    }
#pragma unroll
    for (int i = 0; i < D; ++i) lim[i] = i < n ? l : __int_as_float(int(0xff800000u));
  }
  __device__ __forceinline__ void test(const float2 (&s)[D], bool &c0, bool &c1) const {
    c0 = c1 = false;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      c0 = c0 || sgn * s[i].x < lim[i];
      c1 = c1 || sgn * s[i].y < lim[i];
    }
  }
};
#endif

template <int D, bool GW = false>
__device__ __forceinline__ float2 fused_value(const uint4 &I, int o, const float *pool, const float2 *R,
                                              const ModelDev &m, const Layout &lay) {
  const int base = (o & (lay.win - 1)) * D;
#ifndef PC_JIT
  if ((I.x >> (8 + kPlainBit)) & 1u)
    return fused_plain<D>(I, o, m, [&](int l) { return win_load<GW>(R, lay, base + l); });
#endif
  return fused_value_rd<D>(I, o, pool, m, [&](int l) { return win_load<GW>(R, lay, base + l); });
}
// The same with the frontier date's S in registers (cur; a window of one date).
template <int D>
__device__ __forceinline__ float2 fused_value_regs(const uint4 &I, int o, const float *pool,
                                                   const float2 (&cur)[D], const ModelDev &m) {
  return fused_value_rd<D>(I, o, pool, m, [&](int l) { return cur[l]; });
}

// The same instruction as a test only (X_LANY, or X_LRED with a compare),
// as booleans for the lane's two paths: the whole-loop barrier op decides
// its latches from it without the 0/1 value bits.
template <int D, typename RD>
__device__ __forceinline__ void fused_test_rd(const uint4 &I, int o, const float *pool, const ModelDev &m,
                                              RD rd, bool &t0, bool &t1) {
  const uint32_t A = I.x >> 8;
  const int n = int((A >> 8) & 3u) + 1, kind = int((A >> 2) & 3u), code = int((A >> 4) & 7u);
  const bool any = (I.x & 0xffu) == X_LANY, conj = (A & 1u) != 0;
  const int rop = int(A & 3u);
  const float k = __uint_as_float(I.w);
  auto cmp = [&](float v) {
    return code == 1 ? v < k : code == 2 ? v <= k : code == 3 ? k < v : k <= v;
  };
  float2 v = make_float2(0.f, 0.f);
  bool b0 = false, b1 = false;
  for (int i = 0; i < n; ++i) {
    int l = int(A >> (10 + 2 * i)) & 3;
    l = l < D ? l : 0;
    float2 s;
    if (o > 0) {
      s = rd(l);
    } else {
      const float sv = __ldg(m.sval + (o + m.n_hist) * D + l);
      s = make_float2(sv, sv);
    }
    if (kind == 1) {
      const float c = pool[I.z + i];
      s = make_float2(__fmul_rn(s.x, c), __fmul_rn(s.y, c));
    } else if (kind == 2) {
      const float c = pool[I.z + i];
      s = make_float2(__fdiv_rn(s.x, c), __fdiv_rn(s.y, c));
    }
    if (any) {
      const bool p0 = cmp(s.x), p1 = cmp(s.y);
      if (i == 0) {
        b0 = p0;
        b1 = p1;
      } else if (conj) {
        b0 = b0 && p0;
        b1 = b1 && p1;
      } else {
        b0 = b0 || p0;
        b1 = b1 || p1;
      }
    } else if (i == 0) {
      v = s;
    } else if (rop == 0) {
      v = make_float2(fminf(v.x, s.x), fminf(v.y, s.y));
    } else if (rop == 1) {
      v = make_float2(fmaxf(v.x, s.x), fmaxf(v.y, s.y));
    } else {
      v = make_float2(__fadd_rn(v.x, s.x), __fadd_rn(v.y, s.y));
    }
  }
  if (!any) {
    b0 = cmp(v.x);
    b1 = cmp(v.y);
  }
  t0 = b0;
  t1 = b1;
}
template <int D, bool GW = false>
__device__ __forceinline__ void fused_test(const uint4 &I, int o, const float *pool, const float2 *R,
                                           const ModelDev &m, const Layout &lay, bool &t0, bool &t1) {
  const int base = (o & (lay.win - 1)) * D;
  fused_test_rd<D>(I, o, pool, m, [&](int l) { return win_load<GW>(R, lay, base + l); }, t0, t1);
}
template <int D>
__device__ __forceinline__ void fused_test_regs(const uint4 &I, int o, const float *pool, const float2 (&cur)[D],
                                                const ModelDev &m, bool &t0, bool &t1) {
  fused_test_rd<D>(I, o, pool, m, [&](int l) { return cur[l]; }, t0, t1);
}

// The sensitivity evaluators' whole-loop barrier: the descriptor Dsc tested at
// n + 1 dates, ordinal ORDINAL_ at the k-th, the walk brought there by the
// evaluator's LOOP_ADVANCE.  The interpreter decodes a plain test once and
// takes a date just produced from the registers, in a loop of its own (as in
// pc_ops.inc).
#define LOOP_DATES_(ORDINAL_, TEST_)        \
  for (int k = 0;; ++k) {                   \
    int o = ORDINAL_;                       \
    bool c0, c1;                            \
    TEST_                                   \
    if (c0 && !d0) { d0 = true; r0 = lit; } \
    if (c1 && !d1) { d1 = true; r1 = lit; } \
    all = __all_sync(kFull, d0 && d1);      \
    if (all || k == n) break;               \
  }
#define LOOP_GENERAL_                                          \
  {                                                            \
    LOOP_ADVANCE                                               \
    const float2 v_ = fused_value<D>(Dsc, o, pool, R, m, lay); \
    c0 = bits(v_.x) != 0;                                      \
    c1 = bits(v_.y) != 0;                                      \
  }
#ifdef PC_JIT
#define LOOP_TESTS(ORDINAL_) LOOP_DATES_(ORDINAL_, LOOP_GENERAL_)
#else
// S at ordinal o, produced before (in the window) or history.
template <int D>
__device__ __forceinline__ void past_values(int o, const float2 *R, const ModelDev &m, const Layout &lay,
                                            float2 (&s)[D]) {
#pragma unroll
  for (int i = 0; i < D; ++i)
    s[i] = o > 0 ? SL(lay.off_win + (o & (lay.win - 1)) * D + i) : dup2(__ldg(m.sval + (o + m.n_hist) * D + i));
}
#define LOOP_PLAIN_                     \
  {                                     \
    if (ps.f < o) {                     \
      LOOP_ADVANCE                      \
      lt_.test(ps.s[0], c0, c1);        \
    } else {                            \
      LOOP_ADVANCE                      \
      float2 s_[D];                     \
      past_values<D>(o, R, m, lay, s_); \
      lt_.test(s_, c0, c1);             \
    }                                   \
  }
#define LOOP_TESTS(ORDINAL_)               \
  const LoopTest<D> lt_(Dsc);              \
  if (!lt_.use) {                          \
    LOOP_DATES_(ORDINAL_, LOOP_GENERAL_)   \
  } else {                                 \
    LOOP_DATES_(ORDINAL_, LOOP_PLAIN_)     \
  }
#endif

// Values of the stack machine: one per path of the lane, kPL = 2 PC_PAIRS of
// them (PC_PAIRS pairs; a specialised kernel with four paths a lane defines
// PC_PAIRS 2).  pv_get / pv_set take a path index that is a constant once the
// loops over it are unrolled.
#ifndef PC_PAIRS
#define PC_PAIRS 1
#endif
constexpr int kPL = 2 * PC_PAIRS;
#if PC_PAIRS == 2
struct PV {
  float2 a, b;
};
__device__ __forceinline__ float pv_get(const PV &v, int p) {
  return p == 0 ? v.a.x : p == 1 ? v.a.y : p == 2 ? v.b.x : v.b.y;
}
__device__ __forceinline__ void pv_set(PV &v, int p, float x) {
  if (p == 0) v.a.x = x;
  else if (p == 1) v.a.y = x;
  else if (p == 2) v.b.x = x;
  else v.b.y = x;
}
__device__ __forceinline__ PV pv_splat(float x) { return PV{make_float2(x, x), make_float2(x, x)}; }
__device__ __forceinline__ PV pv_pairs(float2 p0, float2 p1) { return PV{p0, p1}; }
#else
typedef float2 PV;
__device__ __forceinline__ float pv_get(const PV &v, int p) { return p ? v.y : v.x; }
__device__ __forceinline__ void pv_set(PV &v, int p, float x) {
  if (p) v.y = x;
  else v.x = x;
}
__device__ __forceinline__ PV pv_splat(float x) { return make_float2(x, x); }
__device__ __forceinline__ PV pv_pairs(float2 p0) { return p0; }
#endif
#define PV_FOR(p) _Pragma("unroll") for (int p = 0; p < kPL; ++p)

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// A tile's moment sums (sum of payoffs, of squares, of products) without
// the FP64 pipe, which issues at a small fraction of the FP32 rate here:
// each sum is an unevaluated pair hi + lo of floats.  An addend enters by
// Knuth's two-sum (hi + x = s + e exactly, e added into lo); a product of
// two floats enters exactly as its rounded value plus the FMA residual.
// Only the low parts round, so a warp's 64-path sums carry a relative
// error of order 2^-45 of the sum of magnitudes (an FP64 sum of the same
// terms: 2^-47), and become doubles once per tile for the chunk sums.
template <int W>
struct Moments {
  float hi[W], lo[W];
  __device__ __forceinline__ Moments() {
#pragma unroll
    for (int v = 0; v < W; ++v) hi[v] = lo[v] = 0.f;
  }
  __device__ __forceinline__ void add(int v, float x) {
    const float s = __fadd_rn(hi[v], x);
    const float b = __fsub_rn(s, hi[v]);
    const float e = __fadd_rn(__fsub_rn(hi[v], __fsub_rn(s, b)), __fsub_rn(x, b));
    hi[v] = s;
    lo[v] = __fadd_rn(lo[v], e);
  }
  __device__ __forceinline__ void add_prod(int v, float x, float y) {
    const float p = __fmul_rn(x, y);
    add(v, p);
    lo[v] = __fadd_rn(lo[v], __fmaf_rn(x, y, -p));
  }
  // The values of the lane's first path: what add and add_prod leave from
  // zero, without the two-sum.
  __device__ __forceinline__ void set(int v, float x) {
    hi[v] = x;
    lo[v] = 0.f;
  }
  __device__ __forceinline__ void set_prod(int v, float x, float y) {
    hi[v] = __fmul_rn(x, y);
    lo[v] = __fmaf_rn(x, y, -hi[v]);
  }
  __device__ __forceinline__ void add(int v, float x, bool first) { first ? set(v, x) : add(v, x); }
  __device__ __forceinline__ void add_prod(int v, float x, float y, bool first) {
    first ? set_prod(v, x, y) : add_prod(v, x, y);
  }
  // Warp totals as doubles, the one value `index` per lane that this lane
  // ends with (the same for several lanes; the total is identical in all).
  // Each butterfly step halves the values a lane carries: a lane keeps one half
  // of them and sends its partner the other, so W values take W - 1 + (5 -
  // log2 W) two-sums and twice as many shuffles in place of 5 W and 10 W (14
  // values: 15 instead of 70), and one conversion to double in place of W.
  // The two-sum's operands may be swapped without changing a bit, so the
  // totals are those of the full butterfly.
  __device__ __forceinline__ double warp_total(int lane, int &index) {
    index = 0;
    halve<W, 16>(lane, index);
    return double(hi[0]) + double(lo[0]);
  }

 private:
  template <int N, int O>
  __device__ __forceinline__ void halve(int lane, int &index) {
    constexpr int K = (N + 1) / 2;  // values kept (of an odd N both lanes keep the middle one)
    const bool up = (lane & O) != 0;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const float kh = N > 1 && up ? hi[N - K + j] : hi[j], kl = N > 1 && up ? lo[N - K + j] : lo[j];
      const float sh = N > 1 && up ? hi[j] : hi[N - K + j], sl = N > 1 && up ? lo[j] : lo[N - K + j];
      const float h = __shfl_xor_sync(kFull, sh, O), l = __shfl_xor_sync(kFull, sl, O);
      const float s = __fadd_rn(kh, h);
      const float b = __fsub_rn(s, kh);
      const float e = __fadd_rn(__fsub_rn(kh, __fsub_rn(s, b)), __fsub_rn(h, b));
      nh[j] = s;
      nl[j] = __fadd_rn(__fadd_rn(kl, l), e);
    }
#pragma unroll
    for (int j = 0; j < K; ++j) {
      hi[j] = nh[j];
      lo[j] = nl[j];
    }
    if (N > 1 && up) index += N - K;
    if constexpr (O > 1) halve<K, O / 2>(lane, index);
  }
  float nh[(W + 1) / 2], nl[(W + 1) / 2];
};

// Deterministic reduction.  Tile t's partials (sum, sum of squares, ...) are
// the warp's Moments totals, in a fixed shuffle order, as doubles.  Tiles form chunks of chunk_tiles
// consecutive tiles; the warp that finishes a chunk's last tile sums the
// chunk's partials in index order (lane l takes tiles l, l+32, ...; then a
// fixed shuffle tree), and the warp that finishes the last chunk sums the
// chunk partials the same way.  So the result depends only on n_paths, not
// on which warp ran which tile.  Counters are consumed and re-zeroed by the
// warps that read them; the tile counter by the last block to exit.
template <int W>
__device__ __forceinline__ void warp_sum_strided(const double *src, uint32_t n, int lane,
                                                 double (&acc)[W]) {
#pragma unroll
  for (int v = 0; v < W; ++v) acc[v] = 0.0;
  if constexpr (W <= 4) {  // four tiles' loads in flight
    uint32_t i = lane;
    for (; i + 96 < n; i += 128) {
      double x[4][W];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < W; ++v) x[u][v] = __ldcg(src + size_t(i + 32 * u) * W + v);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < W; ++v) acc[v] += x[u][v];
    }
    for (; i < n; i += 32)
#pragma unroll
      for (int v = 0; v < W; ++v) acc[v] += __ldcg(src + size_t(i) * W + v);
  } else {
    for (uint32_t i = lane; i < n; i += 32) {
#pragma unroll
      for (int v = 0; v < W; ++v) acc[v] += __ldcg(src + size_t(i) * W + v);
    }
  }
#pragma unroll
  for (int v = 0; v < W; ++v) acc[v] = warp_sum(acc[v]);
}

// The launch's totals: out, then (blocking calls) the ticket and the device
// status to the host's pinned flag, which the host polls instead of waiting
// for a copy and the stream.
template <int W>
__device__ __forceinline__ void finish_launch(const PriceArgs &a, const double (&acc)[W], int lane) {
  if (lane != 0) return;
#pragma unroll
  for (int v = 0; v < W; ++v) a.out[v] = acc[v];
  a.out[W] = double(a.n_paths);
  if (a.done) {
    const uint32_t status = uint32_t(__ldcg(a.status));
    __threadfence_system();
    *reinterpret_cast<volatile unsigned long long *>(a.done) =
        (static_cast<unsigned long long>(a.ticket) << 32) | status;
  }
}

// Tile `tile`'s partials: value `index` is this lane's `tp` (Moments::warp_total).
template <int W>
__device__ __noinline__ void finish_tile(const PriceArgs &a, uint64_t tile, double tp, int index, int lane) {
  unsigned long long *ctr = reinterpret_cast<unsigned long long *>(a.control);
  uint32_t *chunk_cnt = reinterpret_cast<uint32_t *>(a.control + kChunkCountOff);
  double *chunk_part = reinterpret_cast<double *>(a.control + kChunkPartOff);
  const uint32_t chunk = uint32_t(__umul64hi(tile, a.chunk_magic));  // tile / chunk_tiles
  const uint64_t first = uint64_t(chunk) * a.chunk_tiles;
  const uint64_t rest = a.n_tiles - first;
  const uint32_t size = rest < a.chunk_tiles ? uint32_t(rest) : a.chunk_tiles;
  a.tile_partials[tile * W + index] = tp;  // lanes with the same value store the same bits
  __syncwarp();
  uint32_t seen = 0;
  if (lane == 0) {
    // release: the partials are visible before the count that reports them
    asm volatile("atom.release.gpu.global.add.u32 %0, [%1], 1;" : "=r"(seen) : "l"(chunk_cnt + chunk) : "memory");
  }
  seen = __shfl_sync(kFull, seen, 0);
  if (seen != size - 1) return;
  // this warp completed the chunk
  __threadfence();
  double acc[W];
  warp_sum_strided<W>(a.tile_partials + first * W, size, lane, acc);
  if (lane == 0) chunk_cnt[chunk] = 0;
  if (a.n_chunks == 1) {
    finish_launch<W>(a, acc, lane);
    return;
  }
  unsigned long long done = 0;
  if (lane == 0) {
#pragma unroll
    for (int v = 0; v < W; ++v) chunk_part[size_t(chunk) * W + v] = acc[v];
    asm volatile("atom.release.gpu.global.add.u64 %0, [%1], 1;" : "=l"(done) : "l"(ctr + 2) : "memory");
  }
  done = __shfl_sync(kFull, done, 0);
  if (done != a.n_chunks - 1) return;
  // this warp completed the last chunk
  __threadfence();
  warp_sum_strided<W>(chunk_part, a.n_chunks, lane, acc);
  if (lane == 0) ctr[2] = 0;
  finish_launch<W>(a, acc, lane);
}

// The next unit of work (a tile, or a pair) of this warp from the launch's
// counter; with one_pass (no more units than warps) the warp's own number,
// once: no counter to read, none to reset at the end.
__device__ __forceinline__ unsigned long long next_unit(const PriceArgs &a, int lane) {
  if (a.one_pass) return (static_cast<unsigned long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  unsigned long long u = 0;
  if (lane == 0) u = atomicAdd(reinterpret_cast<unsigned long long *>(a.control), 1ull);
  return __shfl_sync(kFull, u, 0);
}

// Paths to walk: all of the launch, or (per-path kernels only) the listed
// ones of a screened launch.
template <bool LIST>
__device__ __forceinline__ uint64_t walk_paths(const PriceArgs &a) {
  return LIST && a.list ? __ldcg(a.list_n) : a.n_paths;
}
// The i-th of them (i below their number, else any).
template <bool LIST>
__device__ __forceinline__ uint64_t walk_path(const PriceArgs &a, uint64_t i, bool live) {
  return !(LIST && a.list) ? i : live ? __ldcg(a.list + i) : 0;
}

// The last block to exit re-zeroes the unit counter: no warp takes units any
// more once every block has left its loop.
__device__ __forceinline__ void reset_units(const PriceArgs &a) {
  if (a.one_pass) return;
  __shared__ int last_block;
  unsigned long long *ctr = reinterpret_cast<unsigned long long *>(a.control);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last_block = atomicAdd(ctr + 1, 1ull) == gridDim.x - 1;
  }
  __syncthreads();
  if (last_block && threadIdx.x == 0) {
    ctr[0] = 0;
    ctr[1] = 0;
  }
}

}  // namespace
}  // namespace pc
