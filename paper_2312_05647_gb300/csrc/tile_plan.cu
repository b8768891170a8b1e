// tile_plan.cu -- choice of the launch shape of the register/tile jump chain
// (stencil_tile.cuh) and its dispatch.
#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "tile_plan.h"

namespace mjp {

namespace {

constexpr int kSms = 152;

// Pairs per thread that are instantiated (tile_ll32.cu and its like).
const int* runs_of(int kind, int precision, bool ll, bool cl) {
  static const int bd32[] = {1, 2, 4, 8, 0}, ar32[] = {1, 2, 4, 6, 10, 0}, r124[] = {1, 2, 4, 0};
  static const int r123[] = {1, 2, 3, 0}, r14[] = {1, 4, 0}, r24[] = {2, 4, 0}, r12[] = {1, 2, 0}, r23456[] = {2, 3, 4, 5, 6, 0};
  static const int none[] = {0};
  const bool row = kind == MJP_BD1D || kind == MJP_TWOSTATE;
  if (ll) {
    if (precision == MJP_FP32 && kind == MJP_MRNA_PROT2D) return none;  // stencil_reg.cu
    if (cl) return row ? r14 : r24;
    if (precision == MJP_FP64) return r124;
    return kind == MJP_BD1D ? bd32 : kind == MJP_TWOSTATE ? r124 : ar32;
  }
  if (kind == MJP_BD1D) return none;  // stencil_reg1d.cu
  if (precision == MJP_FP64) return cl && row ? r12 : r123;
  return !cl ? r124 : row ? r12 : r23456;
}

}  // namespace

// The shape with the least estimated time, in cycles per jump.  FP32: a base
// of about 250 (row kinds) or 450 (grid kinds) cycles of latency and 15 per
// pair and warp, 4 more per overlapping window (fitted on the 200 x 200
// mRNA/protein box: 3 to 6 pairs per thread on 13 and 19 warps, 1,530 to 1,920
// cycles without hand-overs, within 2%; the fit dates from sums with one Kahan
// step per J jumps, and 6 per window, nearer to a step per product, leaves all
// but a few shapes as they are).  FP64: every operation holds a
// scheduler's FP64 pipe for 64 cycles per warp.  A cluster barrier adds about
// 1,000 cycles, a hand-over of halo rows about 1,200 (measured: 1,150 on 15
// CTAs).
static bool best_shape(int kind, int precision, bool ll, int64_t M, int64_t P, int nt, int G, int maxmem, int B,
                       double overlap, int max_cluster, TilePlan* out) {
  if (ll && maxmem > 2) return false;  // members beyond the second: stencil.cu's list
  const size_t elt = precision == MJP_FP64 ? 8 : 4;
  const bool row = kind == MJP_BD1D || kind == MJP_TWOSTATE;
  const int64_t total = kind == MJP_BD1D ? (M + 1) / 2 : kind == MJP_TWOSTATE ? M : kind == MJP_AUTOREG ? P / 2 : (P + 1) / 2;
  if (!row && M > 768) return false;
  double best = 0.0;
  bool found = false;
  static const int kClusters[] = {1, 2, 3, 4, 6, 8, 10, 12, 14, 16};
  for (int c : kClusters) {
    if (c > max_cluster) break;
    for (const int* rp = runs_of(kind, precision, ll, c > 1); *rp; ++rp) {
      const int R = *rp, maxt = tile_max_threads(elt, ll, c > 1, R);
      const int64_t part = (total + c - 1) / c;  // columns or pair rows of a CTA
      // Grid kinds in a cluster compute halo pair rows of both neighbours and
      // hand over every `period` jumps.
      for (int h = 1; h <= (row || c == 1 ? 1 : 3); ++h) {
        const int halo = row || c == 1 ? 0 : kind == MJP_AUTOREG ? 2 * h : h;
        const int64_t runs = (part + 2 * halo + R - 1) / R;
        const int64_t owners = row ? runs : runs * M;
        if (owners > maxt) continue;
        const int64_t mine = runs * R - 2 * halo;   // columns or pair rows that are the CTA's own
        const int C = (int)((total + mine - 1) / mine);  // CTAs that hold something
        if (C > c || (C == 1) != (c == 1) || mine < halo) continue;
        TilePlan tp;
        tp.cluster = C;
        tp.r = R;
        tp.geo.tx = (int)(row ? runs : M);
        tp.geo.ty = (int)(row ? 1 : runs);
        int64_t threads = (owners + 31) / 32 * 32;
        tp.gpt = 0;
        if (ll) {
          threads = std::max<int64_t>(threads, ((int64_t)G + 8 * 32 - 1) / (8 * 32) * 32);
          if (threads > maxt) continue;
          tp.gpt = G <= 2 * threads ? 2 : 8;
        }
        tp.threads = (int)threads;
        const int cells = tile_cells(kind, (int)M, R, tp.geo.tx, tp.geo.ty);
        if (2 * cells + 1 > 65535) continue;  // tile positions are kept in 16 bits
        const int J = tile_jumps(elt, R), pairs = R * tp.geo.tx * tp.geo.ty;
        const int kcmin = ll ? 8 : std::max(8, 2 * J);
        int kc = 32;
        while (kc > kcmin && elt * (size_t)nt * (2 * kc + 4) > 40 * 1024) kc /= 2;
        tp.geo.kc = kc;
        tp.geo.lgkc = kc == 32 ? 5 : kc == 16 ? 4 : 3;
        tp.geo.nslot = 0;
        tp.geo.halo = halo;
        tp.geo.period = halo == 0 ? 1 << 30 : kind == MJP_AUTOREG ? halo : 2 * halo;
        const int rows = row ? 0 : tp.geo.ty * R;
        size_t smem = tile_smem(elt, ll ? 2 : J, cells, nt, kc, ll ? G : 0, 0, pairs, rows, halo * (int)M).total;
        if (smem > kTileSmemMax) continue;
        if (!ll) {
          tp.geo.nslot = smem >= kTileSmemAcc ? 0 : (int)std::min<size_t>((size_t)std::min(nt, 64), (kTileSmemAcc - smem) / ((size_t)pairs * 16));
          smem = tile_smem(elt, ll ? 2 : J, cells, nt, kc, 0, tp.geo.nslot, pairs, rows, halo * (int)M).total;
        }
        tp.smem = smem;

        const double warps = threads / 32.0, gact = ll ? std::ceil((double)G / nt * overlap / threads) : 0.0;
        double work, lat;
        if (precision == MJP_FP64) {
          const double ops = kind == MJP_BD1D ? 6 : kind == MJP_TWOSTATE ? 7 : kind == MJP_MRNA_PROT2D ? 10 : 13;
          const double per_warp = R * (ops + (ll ? 0.0 : 2.0 * overlap)) + 2.0 * gact;
          work = warps * per_warp * 16.0;
          lat = 200.0 + 64.0 * per_warp * (double)((threads / 32 + 3) / 4) + 300.0 * (R - 1);
        } else {
          work = warps * (R * (15.0 + (ll ? 0.0 : 4.0 * overlap)) + 5.0 * gact);
          lat = (row ? 250.0 : 450.0) + work + 15.0 * R;
        }
        if (C > 1) lat += halo ? 1200.0 / tp.geo.period : 1000.0;
        // CTAs of one SM share its pipes; clusters beyond the SMs run in waves.
        const double per_sm = std::min({65536.0 / (threads * (elt == 4 && R <= 2 ? 80.0 : 128.0)), 227.0 * 1024 / (smem + 1024), 32.0});
        const double slots = kSms * std::max(1.0, (double)(int)per_sm);
        const double ctas = (double)B * C;
        const double waves = std::max(1.0, (double)(int64_t)((ctas + slots - 1) / slots));
        const double res = std::min(std::max(1.0, ctas / kSms), std::max(1.0, (double)(int)per_sm));
        const double t = waves * std::max(lat, (precision == MJP_FP64 ? 1.0 : 0.75) * work * res);
        if (!found || t < best) {
          best = t;
          found = true;
          *out = tp;
        }
      }
    }
  }
  return found;
}

bool tile_plan(int kind, int precision, bool ll, int64_t M, int64_t P, int nt, int G, int maxmem, int B,
               double overlap, TilePlan* out) {
  if (!best_shape(kind, precision, ll, M, P, nt, G, maxmem, B, overlap, 16, out)) return false;
  if (out->cluster <= 8) return true;
  // More than 8 CTAs only where a GPC holds them.
  const cudaError_t e = precision == MJP_FP64 ? (ll ? tile_ll64(kind, nullptr, *out, 0) : tile_ex64(kind, nullptr, *out, 0))
                                              : (ll ? tile_ll32(kind, nullptr, *out, 0) : tile_ex32(kind, nullptr, *out, 0));
  if (e == cudaSuccess) return true;
  cudaGetLastError();
  return best_shape(kind, precision, ll, M, P, nt, G, maxmem, B, overlap, 8, out);
}

// Log-likelihoods of more CTAs than SMs: what counts is how much of an SM each
// CTA takes, and there the tile kernel's halo pair rows (half of its work where a
// CTA holds four), its cluster barriers, the warps it adds for the observation
// groups and its 80 to 160 registers a thread can cost more than it saves against
// stencil.cu, which holds 2 to 16 times the states per CTA in 64 registers.  Both
// sides are estimated: an SM serves its CTAs in batches of as many as it holds,
// and a batch takes the latency of a jump or the work of its CTAs.  Constants in
// cycles, fitted to 8,000 calls (birth-death models of up to 30,000 states,
// two-state ones of up to 950 columns, mRNA/protein boxes of up to 300 x 300,
// autoregulatory ones of up to 120 x 200, 1 to 8,000 thetas, 1 to 100 times, up to
// 6,000 groups); 80% of the estimates are within 30%.  Of the calls on clusters
// the tile kernel was slower in (at worst, times), and is by this rule:
// mRNA/protein FP64 15.6% (2.1) and 2% (1.3), two-state FP64 13.8% (2.0) and 3%
// (1.3), autoregulatory FP32 28.7% (2.0) and 4% (1.4), FP64 0.6% (1.6) and 0.3%
// (1.2), birth-death FP32 9% (2.9) and 3% (1.4); two-state FP64 on one CTA with
// runs of 2 and more columns 10.7% (1.4) and 4% (1.2).  The shapes without an
// entry gained on average and lost rarely, by at most a fifth.
// Measured: 152 thetas of 120 x 90 mRNA/protein FP64, 13 times, 29.6 (tile) and
// 20.6 ms, 16 thetas 5.3 and 20.5 ms; 1,606 thetas of the 38 x 148 autoregulatory
// network FP32 131 and 64.6 ms; 1,000 thetas of 2 x 131 FP64 3.5 and 2.65 ms.
bool tile_pays(int kind, int precision, int64_t M, const TilePlan& tp, int nt, int G, int B, double overlap, int cluster,
               int threads, int64_t slab, size_t smem) {
  struct Cost {
    double lat, depth, work, group, group_lat;  // a jump; per pair and warp, in latency and work; per group step
    double link;                                // tile: a hand-over or a cluster barrier
  };
  struct Row {
    int kind, precision;
    bool clusters;
    double margin;
    Cost tile, shared;
  };
  static const Row rows[] = {
      {MJP_MRNA_PROT2D, MJP_FP64, true, 1.15, {240, 158, 192, 39, 39, 1270}, {3110, 204, 292, 85, 208, 0}},
      {MJP_TWOSTATE, MJP_FP64, true, 1.1, {820, 0, 138, 45, 45, 1160}, {1140, 112, 159, 66, 414, 0}},
      {MJP_TWOSTATE, MJP_FP64, false, 1.05, {1640, 49, 121, 44, 44, 0}, {1140, 112, 159, 66, 414, 0}},
      {MJP_AUTOREG, MJP_FP64, true, 1.05, {860, 181, 195, 42, 42, 554}, {1800, 344, 432, 68, 183, 0}},
      {MJP_AUTOREG, MJP_FP32, true, 1.15, {830, 4.6, 22.5, 25.7, 25.7, 1560}, {2050, 14.6, 29.4, 38, 198, 0}},
      {MJP_BD1D, MJP_FP32, true, 1.2, {1140, 0, 20.4, 21, 92, 0}, {1560, 12.3, 17.6, 32.6, 133, 0}},
  };
  if ((double)B * tp.cluster <= kSms || (tp.cluster == 1 && tp.r == 1)) return true;
  const Row* row = nullptr;
  for (const Row& r : rows)
    if (r.kind == kind && r.precision == precision && r.clusters == (tp.cluster > 1)) row = &r;
  if (!row) return true;
  // Warps that take a step of the active windows' groups, per jump: 32 groups
  // each, a window's last ones in a warp of their own.
  const double active = (double)G / nt * overlap;
  const double steps = std::min(active, active / 32.0 + 0.5 * std::max(1.0, overlap));
  auto served = [&](const Cost& c, int ctas, int per, double runs, double warps, double extra) {
    // (The FP64 pipe takes a scheduler's warps one after the other.)
    const double work = c.work * runs * warps + c.group * steps;
    const double lat = c.lat + c.depth * runs * (precision == MJP_FP64 ? 4.0 * std::ceil(warps / 4.0) : warps) + extra;
    per = std::max(1, std::min(per, 32));
    const double n = std::ceil((double)B * ctas / kSms), full = std::floor(n / per), rest = n - full * per;
    return full * std::max(lat, work * per) + (rest > 0.0 ? std::max(lat, work * rest) : 0.0);
  };
  const int regs = precision == MJP_FP64 ? (tp.r == 1 ? 96 : tp.r == 2 ? 128 : 160) : tp.r <= 2 ? 80 : 128;
  const double tile = served(row->tile, tp.cluster, std::min(65536 / (tp.threads * regs), (int)(227 * 1024 / (tp.smem + 1024))),
                             tp.r, std::ceil(tp.geo.tx * tp.geo.ty / 32.0),
                             row->tile.link / (tp.geo.halo ? tp.geo.period : 1) +
                                 row->tile.group_lat * steps / std::min(4.0, tp.threads / 32.0));
  // stencil.cu: a thread walks a run of states (birth-death) or of pair rows of its
  // column; from 8 states on one warp sums the observations.
  double runs, warps;
  if (kind == MJP_BD1D) {
    runs = std::ceil((double)slab / (threads - 32));
    warps = std::ceil(std::min<double>((double)slab, threads - 32) / 32.0);
  } else {
    const double ty = std::max<double>(1.0, (double)((threads - 32) / M)), pair_rows = std::ceil(slab / (2.0 * M));
    runs = std::ceil(pair_rows / ty);
    warps = std::ceil(M * std::min(ty, pair_rows) / 32.0);
  }
  const bool one_warp = (kind == MJP_BD1D ? runs : 2.0 * runs) >= 8.0;
  const double shared = served(row->shared, cluster, std::min(1024 / threads, (int)(227 * 1024 / (smem + 1024))), runs, warps,
                               row->shared.group_lat * steps / (one_warp ? 1.0 : threads / 32.0));
  return row->margin * tile < shared;
}

cudaError_t launch_chain_tile(int kind, int precision, bool ll, const ChainParams& p, const TilePlan& tp,
                              cudaStream_t s) {
  if (precision == MJP_FP64) return ll ? tile_ll64(kind, &p, tp, s) : tile_ex64(kind, &p, tp, s);
  return ll ? tile_ll32(kind, &p, tp, s) : tile_ex32(kind, &p, tp, s);
}

}  // namespace mjp
