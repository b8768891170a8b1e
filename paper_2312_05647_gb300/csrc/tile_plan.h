// tile_plan.h -- launch shape of the register/tile jump chain
// (stencil_tile.cuh): geometry and shared-memory layout used by both sides.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "mjp.h"

namespace mjp {

struct ChainParams;

// Dynamic shared memory of a CTA at most (the rest of the 227 KB is for the
// kernel's few static bytes).
constexpr size_t kTileSmemMax = 226 * 1024;
// Accumulators of transient distributions take shared memory up to here: the
// rest is left to the L1 cache.
constexpr size_t kTileSmemAcc = 192 * 1024;

// What the kernel needs of the launch shape.
struct TileGeo {
  int tx, ty;     // threads along a row and runs per column (row kinds: ty = 1)
  int kc, lgkc;   // jumps per staged chunk of weights, its logarithm
  int nslot;      // transient distributions: accumulators in shared memory
  int halo;       // grid kinds in a cluster: pair rows computed for each neighbour
  int period;     // jumps between two hand-overs of those
};

struct TilePlan {
  int cluster;    // CTAs per instance
  int threads;    // per CTA
  int r;          // pairs per thread
  int gpt;        // observation groups per thread (0: transient distributions)
  size_t smem;    // dynamic shared memory per CTA
  TileGeo geo;
};

// Cells (pairs) of a CTA's tile: row kinds R columns of TX + 2 cells, grid
// kinds TY R + 2 pair rows of M + 2 cells.
__host__ __device__ inline int tile_cells(int kind, int M, int R, int TX, int TY) {
  return (kind == MJP_BD1D || kind == MJP_TWOSTATE) ? R * (TX + 2) : (TY * R + 2) * (M + 2);
}

struct TileSmem {
  size_t cb, up, red, tx, tPL, ttail, pw, twb, tL, tK, tslot, ring, halo, acc, total;
};

// G: observation groups whose accumulators replace the tile at the end;
// nslot x pairs: accumulators of the transient distributions; rows: pair rows
// of a CTA (grid kinds); halo_pairs: halo pairs of one side.
__host__ __device__ inline TileSmem tile_smem(size_t elt, int tiles, int ncell, int nt, int kc, int G, int nslot, int pairs,
                                              int rows, int halo_pairs) {
  TileSmem s;
  auto up = [](size_t v) { return (v + 15) / 16 * 16; };
  size_t o = up(tiles * (size_t)(ncell + 1) * 2 * elt);
  s.cb = o;
  if (elt == 4) o += up((size_t)ncell * 8);
  if (o < up(8 * (size_t)G)) o = up(8 * (size_t)G);
  s.up = o; o += up((size_t)rows * 2 * elt);
  s.red = o; o += 32 * 8;
  s.tx = o; o += up(8 * (size_t)nt);
  s.tPL = o; o += up(8 * (size_t)nt);
  s.ttail = o; o += up(8 * (size_t)nt);
  s.pw = o; o += up(8 * (size_t)nt);
  s.twb = o; o += up(8 * (size_t)nt);
  s.tL = o; o += up(4 * (size_t)nt);
  s.tK = o; o += up(4 * (size_t)nt);
  s.tslot = o; o += up(4 * (size_t)nt);
  s.ring = o; o += up(elt * (size_t)nt * (2 * kc + 4));
  s.halo = o; o += 64 * (size_t)halo_pairs;  // [parity][side] of 16 bytes a pair
  s.acc = o; o += (size_t)nslot * pairs * 16;
  s.total = o;
  return s;
}

// Threads a CTA of the kernel may have: what leaves a thread the registers of
// its R pairs.
__host__ __device__ constexpr int tile_max_threads(size_t elt, bool ll, bool cl, int R) {
  if (elt == 8) return R == 1 && ll ? 640 : R <= 2 ? 512 : 384;
  if (ll) return R <= 2 ? 768 : 512;
  return cl && (R == 3 || R == 4) ? 640 : 512;
}
// Jumps per accumulation of a transient distribution, the depth of its tile
// (stencil_tile.cuh).
__host__ __device__ constexpr int tile_jumps(size_t elt, int R) {
  return elt == 4 ? (R == 1 ? 16 : R == 2 ? 8 : 4) : (R == 1 ? 8 : 4);
}

// Launch shape for B instances of a model (M, P as in ChainParams), or false
// where the kernel does not apply.  overlap: windows of the observation times
// that hold a jump, on average (an estimate that only steers the choice).
bool tile_plan(int kind, int precision, bool ll, int64_t M, int64_t P, int nt, int G, int maxmem, int B,
               double overlap, TilePlan* out);
// Whether log-likelihoods of B thetas take less time in this shape than in
// stencil.cu's (cluster, threads, states and shared memory of a CTA).
bool tile_pays(int kind, int precision, int64_t M, const TilePlan& tp, int nt, int G, int B, double overlap, int cluster,
               int threads, int64_t slab, size_t smem);
cudaError_t launch_chain_tile(int kind, int precision, bool ll, const ChainParams& p, const TilePlan& tp,
                              cudaStream_t s);

// Instantiations by mode and precision (tile_ll32.cu, tile_ll64.cu,
// tile_ex32.cu, tile_ex64.cu).  launch with p == nullptr asks whether a
// cluster of this shape can be resident (cudaSuccess) instead.
cudaError_t tile_ll32(int kind, const ChainParams* p, const TilePlan& tp, cudaStream_t s);
cudaError_t tile_ll64(int kind, const ChainParams* p, const TilePlan& tp, cudaStream_t s);
cudaError_t tile_ex32(int kind, const ChainParams* p, const TilePlan& tp, cudaStream_t s);
cudaError_t tile_ex64(int kind, const ChainParams* p, const TilePlan& tp, cudaStream_t s);

}  // namespace mjp
