// pc_mlp.cu -- the learned control variate's network on the tensor cores:
// a BF16 multilayer perceptron with FP32 accumulation (forward, backward,
// Adam), and the kernels that turn it into hedge-ratio tables.
//
// Every matrix product is one kernel, mlp_gemm: 64x64 output tiles, 32-deep
// k steps staged in shared memory by cp.async (two stages), fragments read
// with ldmatrix (.trans for operands stored M- or N-major) and multiplied
// with mma.sync m16n8k16 BF16 -> FP32.  Samples are rows: activations are
// [rows, features] BF16, weights [out, in] row-major BF16 copies of FP32
// master weights.  The three products of a layer are
//   forward      Z = H W^T      (A = H, K-major;   B = W,  K-major)
//   data grad    dH = dZ W      (A = dZ, K-major;  B = W,  N-major)
//   weight grad  dW = dZ^T H    (A = dZ, M-major;  B = H,  N-major),
// the last split over the batch (k) into partials summed in a fixed order,
// so every result is deterministic.  Epilogues fuse the bias and softplus
// (forward), the softplus derivative sigma(z) = 1 - exp(-softplus(z)) read
// back from the stored activation (data grad), or write FP32 partials.
#include <cuda_bf16.h>
#include <cstdint>

#include "pc_device.cuh"
#include "pc_mlp.h"

namespace pc {
namespace {

constexpr int BM = 64, BN = 64, BK = 32;
constexpr int SK = BK + 8;   // K-major tile row stride (halves): 80 B rows
constexpr int SC = BM + 8;   // M/N-major tile row stride (halves): 144 B rows
constexpr int kTileHalves = (BM * SK > BK * SC ? BM * SK : BK * SC);

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Stage one k step of an operand: a K-major operand tile is 64 rows of 32
// halves (row r at s + r*SK), an M/N-major one 32 rows (k) of 64 halves
// (row k at s + k*SC).  128 threads, two 16-byte chunks each.
template <bool KMAJOR>
__device__ __forceinline__ void stage(__nv_bfloat16 *s, const __nv_bfloat16 *g, int ld, int row0, int k0) {
#pragma unroll
  for (int c = threadIdx.x; c < 256; c += 128) {
    if (KMAJOR) {
      const int r = c >> 2, col = (c & 3) * 8;
      cp_async16(s + r * SK + col, g + size_t(row0 + r) * ld + k0 + col);
    } else {
      const int k = c >> 3, col = (c & 7) * 8;
      cp_async16(s + k * SC + col, g + size_t(k0 + k) * ld + row0 + col);
    }
  }
}

template <bool A_KM, bool B_KM, int EPI>
__global__ void __launch_bounds__(128) mlp_gemm(const GemmArgs g) {
  __shared__ __align__(16) __nv_bfloat16 sA[2][kTileHalves];
  __shared__ __align__(16) __nv_bfloat16 sB[2][kTileHalves];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = warp >> 1, wn = warp & 1;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kb = blockIdx.z * g.k_split, ke = min(g.K, kb + g.k_split);
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[i][j][v] = 0.f;
  const int steps = (ke - kb) / BK;
  if (steps > 0) {
    stage<A_KM>(sA[0], g.A, g.lda, m0, kb);
    stage<B_KM>(sB[0], g.B, g.ldb, n0, kb);
    cp_async_commit();
  }
  for (int s = 0; s < steps; ++s) {
    const int cur = s & 1;
    if (s + 1 < steps) {
      stage<A_KM>(sA[cur ^ 1], g.A, g.lda, m0, kb + (s + 1) * BK);
      stage<B_KM>(sB[cur ^ 1], g.B, g.ldb, n0, kb + (s + 1) * BK);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const __nv_bfloat16 *a = sA[cur], *b = sB[cur];
#pragma unroll
    for (int ks = 0; ks < BK; ks += 16) {
      uint32_t af[2][4], bf[2][4];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        const int mb = wm * 32 + mi * 16;
        if (A_KM)
          ldsm_x4(af[mi], a + (mb + (lane & 15)) * SK + ks + (lane >> 4) * 8);
        else
          ldsm_x4_t(af[mi], a + (ks + (lane & 7) + (lane >> 4) * 8) * SC + mb + ((lane >> 3) & 1) * 8);
      }
#pragma unroll
      for (int np = 0; np < 2; ++np) {
        const int nb = wn * 32 + np * 16;
        if (B_KM)
          ldsm_x4(bf[np], b + (nb + (lane & 7) + (lane >> 4) * 8) * SK + ks + ((lane >> 3) & 1) * 8);
        else
          ldsm_x4_t(bf[np], b + (ks + (lane & 7) + ((lane >> 3) & 1) * 8) * SC + nb + (lane >> 4) * 8);
      }
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
          mma_bf16(acc[mi][ni], af[mi], bf[ni >> 1][(ni & 1) * 2], bf[ni >> 1][(ni & 1) * 2 + 1]);
    }
    __syncthreads();
  }
  // epilogue: thread holds rows r, r + 8 and columns c, c + 1 of each 16x8 tile
#pragma unroll
  for (int mi = 0; mi < 2; ++mi) {
#pragma unroll
    for (int ni = 0; ni < 4; ++ni) {
      const int c = n0 + wn * 32 + ni * 8 + (lane & 3) * 2;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = m0 + wm * 32 + mi * 16 + (lane >> 2) + h * 8;
        float v0 = acc[mi][ni][2 * h], v1 = acc[mi][ni][2 * h + 1];
        if (EPI == kEpiBiasSoftplus || EPI == kEpiBias) {
          v0 += g.bias[c];
          v1 += g.bias[c + 1];
        }
        if (EPI == kEpiBiasSoftplus) {
          *reinterpret_cast<__nv_bfloat162 *>(g.Cb + size_t(r) * g.ldc + c) =
              __floats2bfloat162_rn(softplus_fast(v0), softplus_fast(v1));
        } else if (EPI == kEpiBias) {
          *reinterpret_cast<float2 *>(g.Cf + size_t(r) * g.ldc + c) = make_float2(v0, v1);
        } else if (EPI == kEpiDSoftplus) {
          const __nv_bfloat162 hv = *reinterpret_cast<const __nv_bfloat162 *>(g.aux + size_t(r) * g.ldaux + c);
          const float2 hf = __bfloat1622float2(hv);
          v0 *= -expm1f(-hf.x);
          v1 *= -expm1f(-hf.y);
          *reinterpret_cast<__nv_bfloat162 *>(g.Cb + size_t(r) * g.ldc + c) = __floats2bfloat162_rn(v0, v1);
        } else {  // kEpiPartial
          float *out = g.Cf + size_t(blockIdx.z) * size_t(g.M) * g.ldc;
          *reinterpret_cast<float2 *>(out + size_t(r) * g.ldc + c) = make_float2(v0, v1);
        }
      }
    }
  }
}

}  // namespace

namespace {

// Rows are padded to kRow = 64 columns (network inputs and outputs); a thread
// takes eight columns of a row and stores them as 16 bytes.  (Indexing by
// 64-bit division over single elements: 12.5 us for 65,536 rows; this 4.5.)
constexpr int kRow = 64;

__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t *>(&h);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__global__ void to_bf16_kernel(const float *x, size_t n, int fin, __nv_bfloat16 *X, size_t rows) {
  pdl_trigger();
  pdl_wait();
  const size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  const size_t r = e >> 3;
  const int c0 = int(e & 7) * 8;
  if (r >= rows) return;
  float v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = r < n && c0 + i < fin ? x[r * fin + c0 + i] : 0.f;
  *reinterpret_cast<uint4 *>(X + r * kRow + c0) = pack8(v);
}

// Eight threads a minibatch row (one thread a row held 64 dependent stores:
// 15 us for 1,024 rows).
__global__ void gather_kernel(const float *x, const float *t, size_t n_data, int fin, int fout,
                              const uint64_t *step, uint32_t s0, uint32_t s1, size_t batch,
                              __nv_bfloat16 *X, float *T) {
  pdl_trigger();
  pdl_wait();
  const size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  const size_t b = e >> 3;
  const int q = int(e & 7), c0 = q * 8;
  if (b >= batch) return;
  const uint64_t st = *step;
  // the first word of Philox4x32-10 at counter (b, step), key (s0, s1)
  const uint32_t u = philox(make_uint4(uint32_t(b), uint32_t(b >> 32), uint32_t(st), uint32_t(st >> 32)), s0, s1).x;
  const size_t src = size_t(u) % n_data;
  float v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = c0 + i < fin ? x[src * fin + c0 + i] : 0.f;
  *reinterpret_cast<uint4 *>(X + b * kRow + c0) = pack8(v);
  for (int c = q; c < fout; c += 8) T[b * fout + c] = t[src * fout + c];
}

// Weighted squared error; rows of kRow columns, thread (tid / 64, tid % 64)
// of block k takes rows 4 k + tid / 64, + 4 gridDim, ... of its column, eight
// at a time so that their loads overlap (65,536 rows: four at a time in 512
// blocks 13.4 us, eight in kLossBlocks 10.6).
constexpr int kLossAhead = 8;
__global__ void loss_kernel(const float *Y, const float *T, const LossWeights w, size_t n, int fout,
                            size_t rows, __nv_bfloat16 *dY, float *part) {
  pdl_trigger();
  pdl_wait();
  __shared__ float red[32];
  float acc = 0.f;
  const float inv = 1.f / float(n);
  const int c = int(threadIdx.x) & (kRow - 1);
  const size_t step = size_t(gridDim.x) * (blockDim.x / kRow);
  const bool col = c < fout;
  const float wc = w.w[c];
  for (size_t r0 = blockIdx.x * size_t(blockDim.x / kRow) + threadIdx.x / kRow; r0 < rows; r0 += kLossAhead * step) {
    float y[kLossAhead], t[kLossAhead];
#pragma unroll
    for (int i = 0; i < kLossAhead; ++i) {
      const size_t r = r0 + size_t(i) * step;
      const bool in = col && r < n;
      y[i] = in ? Y[r * kRow + c] : 0.f;
      t[i] = in ? T[r * fout + c] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < kLossAhead; ++i) {
      const size_t r = r0 + size_t(i) * step;
      if (r >= rows) break;
      float g = 0.f;
      if (col && r < n) {
        const float diff = y[i] - t[i];
        acc += wc * diff * diff * inv;
        g = 2.f * wc * diff * inv;
      }
      dY[r * kRow + c] = __float2bfloat16_rn(g);
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int i = 0; i < int(blockDim.x >> 5); ++i) s += red[i];
    part[blockIdx.x] = s;
  }
}

// Column sums of dZ over chunks of kColChunk rows, in row order: a block
// brings its chunk's 64 columns to shared memory with every load in flight,
// then one thread a column adds the rows (a thread a column straight from
// memory waited on each of its 256 loads: 24 us whatever the row count; this
// 4.6 us for 1,024 rows of 256 columns and 11 for 65,536.  The chunk's chain
// of 256 additions takes about 0.6).
constexpr int kColChunk = 256, kColStride = 64;

__global__ void __launch_bounds__(256) colsum_kernel(const __nv_bfloat16 *dZ, size_t rows, int ld, int cols,
                                                     float *scratch) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) __nv_bfloat16 s[kColChunk * kColStride];
  const int c0 = blockIdx.x * 64;
  const size_t r0 = size_t(blockIdx.y) * kColChunk;
  const int nr = int(min(rows - r0, size_t(kColChunk)));
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int v = threadIdx.x + 256 * j, r = v >> 3, q = (v & 7) * 8;
    if (r < nr)
      *reinterpret_cast<uint4 *>(s + r * kColStride + q) =
          *reinterpret_cast<const uint4 *>(dZ + (r0 + r) * size_t(ld) + c0 + q);
  }
  __syncthreads();
  if (threadIdx.x >= 64) return;
  float a = 0.f;
#pragma unroll 16
  for (int r = 0; r < nr; ++r) a += __bfloat162float(s[r * kColStride + threadIdx.x]);
  scratch[size_t(blockIdx.y) * cols + c0 + threadIdx.x] = a;
}

// Bias corrections of Adam for step *step + 1, once per step (two FP64
// powers in every thread of the update were 66 of a step's 237 us).
__global__ void adam_consts_kernel(const uint64_t *step, float b1, float b2, float *c) {
  const double t = double(*step + 1);
  if (threadIdx.x == 0) c[0] = float(1.0 - pow(double(b1), t));
  if (threadIdx.x == 32) c[1] = float(1.0 - pow(double(b2), t));
}

// Ordered sum of `n` values `stride` apart, kAhead loads in flight (one at a
// time waited a memory latency each).
constexpr int kAhead = 16;
__device__ __forceinline__ float ordered_sum(const float *p, int n, size_t stride) {
  float s = 0.f;
  int z = 0;
  for (; z + kAhead <= n; z += kAhead) {
    float v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) v[u] = p[size_t(z + u) * stride];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) s += v[u];
  }
  float v[kAhead];
#pragma unroll
  for (int u = 0; u < kAhead; ++u) v[u] = z + u < n ? p[size_t(z + u) * stride] : 0.f;
#pragma unroll
  for (int u = 0; u < kAhead; ++u)
    if (z + u < n) s += v[u];
  return s;
}

// A layer's gradient from its partials, in one launch: the weight elements
// (sums over the k splits, in order) by blocks 0 .. wb - 1, then the biases
// (sums over the row chunks of colsum_kernel, in order) 32 columns a block,
// their chunk values staged in shared memory.  With ADAM the parameters are
// updated from the sum in hand and the gradient is not stored.
template <bool ADAM>
__global__ void __launch_bounds__(256) layer_grad_kernel(const LayerGrad g, const AdamStep a) {
  pdl_trigger();
  pdl_wait();
  __shared__ float sh[256][33];
  size_t i;
  float s;
  if (blockIdx.x < g.w_blocks) {
    i = blockIdx.x * size_t(256) + threadIdx.x;
    if (i >= g.count) return;
    s = ordered_sum(g.part + i, g.splits, g.count);
  } else {
    const int c = int(threadIdx.x) & 31, q = int(threadIdx.x) >> 5;
    const int col = int(blockIdx.x - g.w_blocks) * 32 + c;
    s = 0.f;
    for (int z0 = 0; z0 < g.chunks; z0 += 256) {
#pragma unroll
      for (int u = 0; u < 32; ++u) {
        const int z = z0 + q + 8 * u;
        if (z < g.chunks) sh[q + 8 * u][c] = g.colpart[size_t(z) * g.cols + col];
      }
      __syncthreads();
      if (q == 0) {
        const int nz = min(256, g.chunks - z0);
#pragma unroll 16
        for (int z = 0; z < nz; ++z) s += sh[z][c];
      }
      __syncthreads();
    }
    if (q) return;
    i = g.count + size_t(col);
  }
  if (!ADAM) {
    if (i < g.count) {
      const unsigned r = unsigned(i) / unsigned(g.in_w), c = unsigned(i) % unsigned(g.in_w);
      if (r < unsigned(g.w_out) && c < unsigned(g.w_in)) g.out[size_t(r) * g.w_in + c] = s;
    } else if (i - g.count < size_t(g.w_out)) {
      g.out[size_t(g.w_out) * g.w_in + (i - g.count)] = s;
    }
    return;
  }
  const float b1 = a.b1, b2 = a.b2, c1 = a.consts[0], c2 = a.consts[1];
  const float mi = b1 * a.m[i] + (1.f - b1) * s;
  const float vi = b2 * a.v[i] + (1.f - b2) * s * s;
  a.m[i] = mi;
  a.v[i] = vi;
  const float pi = a.p[i] - a.lr * (mi / c1) / (sqrtf(vi / c2) + a.eps);
  a.p[i] = pi;
  a.pb[i] = __float2bfloat16_rn(pi);
}

// The block partials' total in FP64: 32 lanes' strided sums, then a fixed
// shuffle tree (one thread's chain of dependent loads was 43 us for 512).
__global__ void loss_total_kernel(const float *part, int blocks, double *loss, uint64_t *step) {
  pdl_trigger();
  pdl_wait();
  double s = 0.0;
  for (int i = threadIdx.x; i < blocks; i += 32 * 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = i + 32 * u < blocks ? part[i + 32 * u] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) s += double(v[u]);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x != 0) return;
  *loss = s;
  if (step) *step += 1;
}

__global__ void unpad_kernel(const float *Y, int ldy, size_t n, int fout, float *y) {
  pdl_trigger();
  pdl_wait();
  const size_t e = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  if (e >= n * size_t(fout)) return;
  y[e] = Y[(e / fout) * ldy + e % fout];
}

unsigned grid_for(size_t work, int block, unsigned cap = 4096) {
  size_t g = (work + block - 1) / block;
  if (g < 1) g = 1;
  return unsigned(g < cap ? g : cap);
}

}  // namespace

cudaError_t launch_gemm(GemmKind kind, int epi, const GemmArgs &g, int splits, cudaStream_t s) {
  if (g.M % BM || g.N % BN || g.K % BK || g.k_split % BK || splits < 1) return cudaErrorInvalidValue;
  const dim3 grid(unsigned(g.N / BN), unsigned(g.M / BM), unsigned(splits));
  switch (kind) {
    case kGemmForward:
      if (epi == kEpiBiasSoftplus) mlp_gemm<true, true, kEpiBiasSoftplus><<<grid, 128, 0, s>>>(g);
      else if (epi == kEpiBias) mlp_gemm<true, true, kEpiBias><<<grid, 128, 0, s>>>(g);
      else return cudaErrorInvalidValue;
      break;
    case kGemmDataGrad:
      if (epi != kEpiDSoftplus) return cudaErrorInvalidValue;
      mlp_gemm<true, false, kEpiDSoftplus><<<grid, 128, 0, s>>>(g);
      break;
    case kGemmWeightGrad:
      if (epi != kEpiPartial) return cudaErrorInvalidValue;
      mlp_gemm<false, false, kEpiPartial><<<grid, 128, 0, s>>>(g);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_to_bf16(const float *x, size_t n, int fin, __nv_bfloat16 *X, size_t rows, int ld,
                           cudaStream_t s) {
  if (ld != kRow) return cudaErrorInvalidValue;
  to_bf16_kernel<<<unsigned((rows * 8 + 255) / 256), 256, 0, s>>>(x, n, fin, X, rows);
  return cudaGetLastError();
}

cudaError_t launch_gather(const float *x, const float *t, size_t n_data, int fin, int fout,
                          const uint64_t *step, uint32_t s0, uint32_t s1, size_t batch,
                          __nv_bfloat16 *X, int ldx, float *T, cudaStream_t s) {
  if (ldx != kRow) return cudaErrorInvalidValue;
  gather_kernel<<<unsigned((batch * 8 + 127) / 128), 128, 0, s>>>(x, t, n_data, fin, fout, step, s0, s1, batch, X, T);
  return cudaGetLastError();
}

int loss_blocks(size_t rows) { return int(grid_for(rows * kRow, 256, kLossBlocks)); }

cudaError_t launch_loss(const float *Y, int ldy, const float *T, const LossWeights &w, size_t n, int fout,
                        size_t rows, __nv_bfloat16 *dY, int ldd, float *part, int blocks, cudaStream_t s, bool dep) {
  if (ldy != kRow || ldd != kRow) return cudaErrorInvalidValue;
  return launch_chain(dep, loss_kernel, dim3(unsigned(blocks)), dim3(256), 0, s, Y, T, w, n, fout, rows, dY, part);
}

cudaError_t launch_colsum(const __nv_bfloat16 *dZ, size_t rows, int ld, int cols, float *scratch, cudaStream_t s,
                          bool dep) {
  if (cols % 64 || ld % 8) return cudaErrorInvalidValue;
  const unsigned chunks = unsigned((rows + kColChunk - 1) / kColChunk);
  return launch_chain(dep, colsum_kernel, dim3(unsigned(cols / 64), chunks), dim3(256), 0, s, dZ, rows, ld, cols, scratch);
}

cudaError_t launch_layer_grad(LayerGrad g, size_t rows, const AdamStep *adam, cudaStream_t s, bool dep) {
  if (g.cols % 32) return cudaErrorInvalidValue;
  g.chunks = int((rows + kColChunk - 1) / kColChunk);
  g.w_blocks = unsigned((g.count + 255) / 256);
  const unsigned grid = g.w_blocks + unsigned(g.cols / 32);
  if (adam) return launch_chain(dep, layer_grad_kernel<true>, dim3(grid), dim3(256), 0, s, g, *adam);
  return launch_chain(dep, layer_grad_kernel<false>, dim3(grid), dim3(256), 0, s, g, AdamStep{});
}

cudaError_t launch_adam_consts(const uint64_t *step, float b1, float b2, float *consts, cudaStream_t s) {
  adam_consts_kernel<<<1, 64, 0, s>>>(step, b1, b2, consts);
  return cudaGetLastError();
}

cudaError_t launch_loss_total(const float *part, int blocks, double *loss, uint64_t *step, cudaStream_t s,
                              bool dep) {
  return launch_chain(dep, loss_total_kernel, dim3(1), dim3(32), 0, s, part, blocks, loss, step);
}

cudaError_t launch_unpad(const float *Y, int ldy, size_t n, int fout, float *y, cudaStream_t s, bool dep) {
  if (n == 0) return cudaSuccess;
  return launch_chain(dep, unpad_kernel, dim3(unsigned((n * fout + 255) / 256)), dim3(256), 0, s, Y, ldy, n, fout, y);
}

}  // namespace pc
