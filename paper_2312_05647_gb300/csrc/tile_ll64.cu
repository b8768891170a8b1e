// tile_ll64.cu -- FP64 log-likelihood instances of the tile chain.
#include "stencil_tile.cuh"

namespace mjp {

cudaError_t tile_ll64(int kind, const ChainParams* p, const TilePlan& tp, cudaStream_t s) {
  const bool cl = tp.cluster > 1;
#define TILE(K, CL, R)                                                                       \
  if (kind == K && cl == CL && tp.r == R)                                                    \
    return tp.gpt <= 2 ? tile_one<double, K, true, CL, R, 2>(p, tp, s) : tile_one<double, K, true, CL, R, 8>(p, tp, s);
  TILE(MJP_BD1D, false, 1)
  TILE(MJP_BD1D, false, 2)
  TILE(MJP_BD1D, false, 4)
  TILE(MJP_TWOSTATE, false, 1)
  TILE(MJP_TWOSTATE, false, 2)
  TILE(MJP_TWOSTATE, false, 4)
  TILE(MJP_MRNA_PROT2D, false, 1)
  TILE(MJP_MRNA_PROT2D, false, 2)
  TILE(MJP_MRNA_PROT2D, false, 4)
  TILE(MJP_AUTOREG, false, 1)
  TILE(MJP_AUTOREG, false, 2)
  TILE(MJP_AUTOREG, false, 4)
  TILE(MJP_BD1D, true, 1)
  TILE(MJP_BD1D, true, 4)
  TILE(MJP_TWOSTATE, true, 1)
  TILE(MJP_TWOSTATE, true, 4)
  TILE(MJP_MRNA_PROT2D, true, 2)
  TILE(MJP_MRNA_PROT2D, true, 4)
  TILE(MJP_AUTOREG, true, 2)
  TILE(MJP_AUTOREG, true, 4)
#undef TILE
  return cudaErrorInvalidValue;
}

}  // namespace mjp
