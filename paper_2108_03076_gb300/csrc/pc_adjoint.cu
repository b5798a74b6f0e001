// pc_adjoint.cu -- the adjoint sensitivity kernel (pc_adjoint.cuh) and its
// launch.
#include <cstdint>

#include "pc_adjoint.cuh"
#include "pc_internal.h"

namespace pc {
namespace {

// SKIP: programs that start at a later date than the first (as price_kernel).
template <int D, bool WRITE, bool SKIP>
__global__ void __launch_bounds__(kBlock, D == 4 ? 4 : 5) adjoint_kernel(const __grid_constant__ PriceArgs a, const TapeArgs t) {
  adjoint_tiles<D, WRITE>(a, t, [&](const uint4 *P, const float *pool, float2 *R, const Rng2 &g, bool live0,
                                   bool live1, const float (&Bm)[D * D], const float (&S0)[D],
                                   const float (&Lm)[D * D], Tape &T, int &res) {
    return eval_adjoint<D, SKIP>(P, pool, R, a, g, live0, live1, Bm, S0, Lm, T, res);
  });
}

template <typename K>
cudaError_t set_smem_a(K kern, size_t smem) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

}  // namespace

cudaError_t launch_adjoint(const PriceArgs &a, const TapeArgs &t, int grid, int block, size_t smem,
                           cudaStream_t s) {
  const bool w = a.out_paths != nullptr;
#define ALAUNCH(DD, WW, SS)                                                        \
  do {                                                                             \
    auto k = adjoint_kernel<DD, WW, SS>;                                           \
    cudaError_t e = set_smem_a(k, smem);                                           \
    if (e != cudaSuccess) return e;                                                \
    k<<<grid, block, smem, s>>>(a, t);                                             \
    return cudaGetLastError();                                                     \
  } while (0)
#define ALAUNCH_D(DD)                                                              \
  do {                                                                             \
    if (a.lay.skip > 1) { if (w) ALAUNCH(DD, true, true); else ALAUNCH(DD, false, true); } \
    else { if (w) ALAUNCH(DD, true, false); else ALAUNCH(DD, false, false); }                  \
  } while (0)
  switch (a.m.d) {
    case 1: ALAUNCH_D(1);
    case 2: ALAUNCH_D(2);
    case 3: ALAUNCH_D(3);
    case 4: ALAUNCH_D(4);
    default: return cudaErrorInvalidValue;
  }
#undef ALAUNCH_D
#undef ALAUNCH
}

namespace {
int adjoint_occupancy(uint64_t v, int block, size_t smem) {
  const int d = int(v & 0xff);
  int nb = 0;
  cudaError_t e = cudaErrorInvalidValue;
#define AOCC(DD)                                                                                 \
  do {                                                                                           \
    e = set_smem_a(adjoint_kernel<DD, false, false>, smem);                                             \
    if (e == cudaSuccess)                                                                        \
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, adjoint_kernel<DD, false, false>, block, smem); \
  } while (0)
  switch (d) {
    case 1: AOCC(1); break;
    case 2: AOCC(2); break;
    case 3: AOCC(3); break;
    case 4: AOCC(4); break;
    default: return 0;
  }
#undef AOCC
  return e == cudaSuccess ? nb : 0;
}
}  // namespace

int adjoint_blocks_per_sm(int d, int block, size_t smem) {
  return occupancy_memo((uint64_t(3) << 32) | uint64_t(d), block, smem, adjoint_occupancy);
}

}  // namespace pc
