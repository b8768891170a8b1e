// tile_ex32.cu -- FP32 transient-distribution instances of the tile chain.
#include "stencil_tile.cuh"

namespace mjp {

cudaError_t tile_ex32(int kind, const ChainParams* p, const TilePlan& tp, cudaStream_t s) {
  const bool cl = tp.cluster > 1;
#define TILE(K, CL, R) \
  if (kind == K && cl == CL && tp.r == R) return tile_one<float, K, false, CL, R, 1>(p, tp, s);
  TILE(MJP_TWOSTATE, false, 1)
  TILE(MJP_TWOSTATE, false, 2)
  TILE(MJP_TWOSTATE, false, 4)
  TILE(MJP_MRNA_PROT2D, false, 1)
  TILE(MJP_MRNA_PROT2D, false, 2)
  TILE(MJP_MRNA_PROT2D, false, 4)
  TILE(MJP_AUTOREG, false, 1)
  TILE(MJP_AUTOREG, false, 2)
  TILE(MJP_AUTOREG, false, 4)
  TILE(MJP_TWOSTATE, true, 1)
  TILE(MJP_TWOSTATE, true, 2)
  TILE(MJP_MRNA_PROT2D, true, 2)
  TILE(MJP_MRNA_PROT2D, true, 3)
  TILE(MJP_MRNA_PROT2D, true, 4)
  TILE(MJP_MRNA_PROT2D, true, 5)
  TILE(MJP_MRNA_PROT2D, true, 6)
  TILE(MJP_AUTOREG, true, 2)
  TILE(MJP_AUTOREG, true, 3)
  TILE(MJP_AUTOREG, true, 4)
  TILE(MJP_AUTOREG, true, 5)
  TILE(MJP_AUTOREG, true, 6)
#undef TILE
  return cudaErrorInvalidValue;
}

}  // namespace mjp
