// stencil_tile.cuh -- jump chain of the stencil models with the states in
// registers and one shared-memory tile for the neighbours' reads (FP32 and
// FP64; every model kind; transient distributions and log-likelihoods).  The
// automatic choice wherever no more special register kernel applies
// (stencil_reg.cu, stencil_reg1d.cu, stencil_regts.cu); stencil.cu stays for
// forced launch shapes, groups of more than two members and boxes that do not
// fit here.  Included by the translation units that instantiate it.
//
// States are pairs (float2 / double2): the two gene states of a column
// (two-state), rows 2j and 2j + 1 of a column (mRNA/protein), both gene
// states of one (n_R, n_P) (autoregulatory), or states c and c + W of a CTA's
// run of 2 W states (birth-death).  A thread owns a run of R pairs: R
// consecutive columns of the one pair row ("row kinds": birth-death and
// two-state) or R consecutive pair rows of one column ("grid kinds").  Its
// values, residuals (FP32) and coefficients stay in registers for all jumps;
// the neighbours along the run are registers too, the other neighbours come
// from the tile, which is double-buffered by jump parity.  Against a kernel
// that keeps everything in shared memory a pair costs 3 shared-memory
// accesses a jump instead of 7 (grid kinds) and no coefficient arithmetic.
//
// Log-likelihoods: every thread owns up to GPT observation groups (group g
// belongs to thread g mod threads), whose members' tile positions and
// accumulators are registers, so a jump costs a group two tile reads, one
// weight and the Kahan step, spread evenly over all warps.  One warp doing
// this beside the others bounded the autoregulatory network: 23,000 of its
// 24,000 cycles per jump.
//
// Transient distributions: the tile is J deep instead of double-buffered, so a
// thread finds its values of the last J jumps there, and takes an output's
// sum through J jumps at a time in registers (FP32: a Kahan step for each
// product P_{k+j} rho_{k+j}; both precisions: the operations of one jump at a
// time in their order.  A jump beyond the window's last one has weight 0; its
// Kahan step leaves sum - compensation as it is).  The accumulators of the windows that overlap stay
// in shared memory while they fit, the others in global memory.
//
// Clusters split row kinds by columns: the pairs at a boundary are pushed into
// the neighbour's tile after every jump and a cluster barrier orders them.
// Grid kinds are split by pair rows with temporal blocking: a CTA also
// computes `halo` pair rows of each neighbour, which stay right for
// halo (autoregulatory: a jump reads a whole pair row beyond) or 2 halo
// (mRNA/protein: one row) jumps; then the neighbours send each other the
// values and residuals of their outermost own pair rows (st.async, counted on
// hand-over mbarriers; every wait is bounded), so that only one jump in
// 2 halo pays the latency between CTAs.
//
// Arithmetic per state is the sequence of stencil.cu, so the chains agree to
// the bit for every layout.
//
// Bound: instruction issue and the latency of a jump (reads behind a barrier,
// the dependent multiply-adds) in FP32, the FP64 pipe (64 cycles per warp
// instruction and scheduler) in FP64; DRAM and L2 are idle (the autoregulatory
// instance below: issue slots 44% busy, L2 0.1%).  Spills: an early version with 90
// bytes spilled inside the jump and nearly all of the shared memory taken ran four
// times slower, its accesses missing the small L1 left.  The thread bounds leave
// some instances with spills all the same (-Xptxas -v, bytes stored): FP32
// log-likelihoods 4 to 16 with R = 1, 8 to 120 with R = 2, 16 with R = 4 on clusters,
// birth-death R = 8 64, autoregulatory R = 10 160 (the 40 x 120 case); FP32 transient
// distributions on clusters 4 (R = 3) to 88 (R = 4); FP64 4.  Theirs stay in the L1
// (the same 0.1% of the L2).
// Measured against the shared-memory kernel (one GB300): autoregulatory
// network 40 x 120, 152 thetas, 50 times, FP32 12.5 -> 2.0 ms; birth-death N =
// 64, 10^4 thetas, FP64 7.61 -> 3.55 ms; two-state N_R = 131, one theta, FP64
// 1.88 -> 1.03 ms; mRNA/protein 200 x 200, 20 times, FP32 463 -> 66 ms (15
// CTAs instead of 4, 0.95 us per jump; sums as multiply-add chains with one
// Kahan step per J jumps took 63 ms, but are held in fewer bits).
#pragma once

#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "chain_common.cuh"
#include "host_util.h"
#include "internal.cuh"
#include "tile_plan.h"

namespace cg = cooperative_groups;

namespace mjp {

namespace {

constexpr bool tile_row_kind(int kind) { return kind == MJP_BD1D || kind == MJP_TWOSTATE; }

template <typename T>
__device__ __forceinline__ typename Pair<T>::type v_zero() {
  return v_make((T)0, (T)0);
}
// Kahan step of a pair, the roundings of the scalar step.
__device__ __forceinline__ void kahan_pair(float2 v, float2& s, float2& c) {
  const float2 m1 = make_float2(-1.0f, -1.0f);
  const float2 y = __ffma2_rn(c, m1, v);
  const float2 t = __fadd2_rn(s, y);
  c = __ffma2_rn(y, m1, __ffma2_rn(s, m1, t));
  s = t;
}

// The value of v, hidden from the optimiser at this place.
__device__ __forceinline__ unsigned tile_opaque(unsigned v) {
  asm volatile("" : "+r"(v));
  return v;
}

// Coefficients of one pair, formed once.  dg: the pair's -e (FP32, delta
// form) or 1 - e (FP64); up: the inflow from the next pair of the run (grid
// kinds: gamma (row + 1) of each half) or from the right (row kinds); bd:
// binding inflow of the autoregulatory model.
template <typename T, int KIND>
struct PairCoef {
  typename Pair<T>::type dg, up;
};

template <typename T, int KIND, bool LL, bool CL, int R, int GPT, int J, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) tile_kernel(const ChainParams p, const TileGeo tg) {
  using T2 = typename Pair<T>::type;
  constexpr bool kComp = sizeof(T) == 4;
  constexpr bool ROW = tile_row_kind(KIND);
  // Long runs read the inflow coefficients from above (they depend on the pair
  // row alone) from a table: their registers are needed for the states.
  constexpr bool kUpTab = !ROW && (R >= 5 || (!LL && CL && R >= 3));
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = CL ? (int)cluster.num_blocks() : 1;
  const int rank = CL ? (int)cluster.block_rank() : 0;
  const int job = p.job_map ? p.job_map[blockIdx.x / C] : (int)(blockIdx.x / C);
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nt = p.ntimes;
  const int N = (int)p.N, M = p.M, P = p.P;
  const int TX = tg.tx, TY = tg.ty, kc = tg.kc;
  constexpr int JB = LL ? 8 : J;  // jumps per block (divides kc)
  const int st = ROW ? TX + 2 : M + 2;  // cells between consecutive pairs of a run
  const int ncell = tile_cells(KIND, M, R, TX, TY);

  constexpr int TB = LL ? 2 : J;  // tiles: rho_k lies in tile k mod TB
  const TileSmem L = tile_smem(sizeof(T), TB, ncell, nt, kc, LL ? p.G : 0, LL ? 0 : tg.nslot, R * TX * TY, ROW ? 0 : TY * R,
                               ROW ? 0 : tg.halo * M);
  T2* const upt = reinterpret_cast<T2*>(smem + L.up);  // inflow coefficients of this CTA's pair rows
  T2* const buf = reinterpret_cast<T2*>(smem);  // [TB][ncell + 1]; cell ncell stays zero
  const int bstride = ncell + 1;
  float2* const cbt = reinterpret_cast<float2*>(smem + L.cb);  // p.renorm x exit defect (FP32)
  double* t_x = reinterpret_cast<double*>(smem + L.tx);
  double* t_PL = reinterpret_cast<double*>(smem + L.tPL);
  double* t_tail = reinterpret_cast<double*>(smem + L.ttail);
  double* pw = reinterpret_cast<double*>(smem + L.pw);  // recurrence state per time
  const T** t_wb = reinterpret_cast<const T**>(smem + L.twb);
  int* t_L = reinterpret_cast<int*>(smem + L.tL);
  int* t_K = reinterpret_cast<int*>(smem + L.tK);
  // Weights of the jumps in slots by k mod 2 kc, 0 outside a window:
  // log-likelihoods [2 kc][nt] (a jump's weights side by side), transient
  // distributions [nt][2 kc + 4], jump k in slot k - 1 (the block of jumps
  // kb + 1 .. kb + J of one time in vector loads).
  T* ring = reinterpret_cast<T*>(smem + L.ring);
  constexpr int K0 = LL ? 0 : 1;  // first jump of the first chunk
  auto ring_at = [&](int i, int k) -> T* {
    const int slot = (k - K0) & (2 * kc - 1);
    return ring + (LL ? slot * nt + i : i * (2 * kc + 4) + slot);
  };
  const T* arena = reinterpret_cast<const T*>(p.arena);

  // ---- prologue ------------------------------------------------------------
  const Win* wj = p.win + (int64_t)job * nt;
  bool rec_mine = false;
  for (int i = tid; i < nt; i += nthr) {
    const Win w = wj[i];
    const bool copy = w.woff >= 0 && arena;
    t_x[i] = w.x;
    t_PL[i] = w.PL;
    t_tail[i] = w.tail;
    t_L[i] = (int)w.L;
    t_K[i] = (int)w.K;
    t_wb[i] = copy ? arena + (w.woff - w.L) : nullptr;
    pw[i] = w.PL;  // P_L; the recurrence of a window that holds jump 0 goes on from it
    rec_mine |= !copy;
  }
  const double omega = p.info[job].omega;
  const int Kmax = (int)p.info[job].Kmax;  // the planner caps K below 2^30 here (tile_plan)
  const Coef<T> co = make_coef<T, KIND>(p.theta + (int64_t)job * p.ntheta, omega);
  const T* rho0 = reinterpret_cast<const T*>(p.rho0);
  for (int j = tid; j < TB * bstride; j += nthr) buf[j] = v_zero<T>();
  if (kComp)
    for (int j = tid; j < ncell; j += nthr) cbt[j] = make_float2(0.0f, 0.0f);

  constexpr bool link = !ROW && CL;  // grid kinds in a cluster: halo pair rows and hand-overs
  // This thread's run.  Row kinds: columns c0 .. c0 + R - 1 of this CTA's
  // W = R TX columns; cell (r, t) at r st + t + 1, so the threads of a warp
  // touch consecutive cells.  Grid kinds: pair rows j0 .. j0 + R - 1 of column
  // tx; cell (row, column) at (row + 1) st + column + 1.
  const bool owner = tid < TX * TY;
  const int tx = ROW ? tid : tid % TX, ty = ROW ? 0 : tid / TX;
  const int W = ROW ? R * TX : M;
  const int D = link ? tg.halo : 0;    // pair rows computed for each neighbour
  const int Hown = TY * R - 2 * D;     // pair rows of this CTA (grid kinds)
  // First column, state or pair row that is computed here (grid kinds: the lower halo's first).
  const int cta0 = ROW ? rank * W * (KIND == MJP_BD1D ? 2 : 1) : rank * Hown - D;
  const int o0 = ROW ? tx + 1 : (ty * R + 1) * st + tx + 1;
  const int Pm = KIND == MJP_AUTOREG ? P / 2 : (P + 1) / 2;  // pair rows of the box (grid kinds)
  // Model index of half h of pair (column c, pair row j) as counted in this
  // CTA's frame: -1 outside the box.
  auto state_of = [&](int c, int j, int h) -> int {
    if (KIND == MJP_BD1D) {  // c: column of this CTA, may be -1 or W (pads)
      const int n = cta0 + c + h * W;
      return n >= 0 && n < N ? n : -1;
    }
    if (KIND == MJP_TWOSTATE) {
      const int m = cta0 + c;
      return m >= 0 && m < M ? m + h * M : -1;
    }
    if (j < 0 || j >= Pm) return -1;
    if (KIND == MJP_AUTOREG) return c + M * j + M * Pm * h;
    const int row = 2 * j + h;
    return row < P ? row * M + c : -1;
  };
  auto rho_of = [&](int n) -> T { return n >= 0 ? rho0[n] : (T)0; };
  auto load_pair = [&](int c, int j) -> T2 { return v_make(rho_of(state_of(c, j, 0)), rho_of(state_of(c, j, 1))); };

  T2 S[R];
  float2 lo[kComp ? R : 1];
  PairCoef<T, KIND> pc[R];
  unsigned vx = 0, vy = 0;  // halves of the run inside the box
  unsigned own = 0;         // pairs of the run that are this CTA's (not a neighbour's)
  const int j0 = ROW ? 0 : cta0 + ty * R;
  const int cfirst = ROW ? tx * R : tx;
  // Column constants of grid kinds.
  const T fcol = (T)tx;
  const T g_cr = KIND == MJP_AUTOREG ? f_mul(co.c, (T)(tx + 1)) : KIND == MJP_MRNA_PROT2D ? f_mul(co.b, (T)(tx + 1)) : (T)0;
  const T g_cd = KIND == MJP_MRNA_PROT2D ? f_mul(co.c, fcol) : KIND == MJP_AUTOREG ? f_mul(co.b, fcol) : (T)0;
  int rtop = -1;  // pair of the run that holds row P - 1 (mRNA/protein)
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int c = ROW ? cfirst + r : tx, j = ROW ? 0 : j0 + r;
    const int n0 = owner ? state_of(c, j, 0) : -1, n1 = owner ? state_of(c, j, 1) : -1;
    if (n0 >= 0) vx |= 1u << r;
    if (n1 >= 0) vy |= 1u << r;
    if (ROW || (ty * R + r >= D && ty * R + r < D + Hown)) own |= 1u << r;
    S[r] = v_make(rho_of(n0), rho_of(n1));
    if (kComp) lo[r] = make_float2(0.0f, 0.0f);
    const T one = (T)1;
    if (KIND == MJP_BD1D) {
      T e[2], cr[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int n = cta0 + c + h * W;
        const T fm = (T)n;
        e[h] = f_add(f_mul(co.b, fm), n + 1 < N ? co.a : (T)0);
        cr[h] = f_mul(co.b, f_add(fm, one));
      }
      pc[r].dg = kComp ? v_make(-e[0], -e[1]) : v_make(f_sub(one, e[0]), f_sub(one, e[1]));
      pc[r].up = v_make(cr[0], cr[1]);
    } else if (KIND == MJP_TWOSTATE) {
      const int m = cta0 + c;
      const T bm = f_mul(co.b, (T)m), cr = f_mul(co.b, (T)(m + 1));
      const T ex = f_add(f_add(bm, m + 1 < M ? co.a : (T)0), co.d), ey = f_add(co.c, bm);
      pc[r].dg = kComp ? v_make(-ex, -ey) : v_make(f_sub(one, ex), f_sub(one, ey));
      pc[r].up = v_make(cr, cr);
    } else if (KIND == MJP_AUTOREG) {
      const T fq = (T)j;
      const bool qtop = j + 1 >= Pm;
      const T a_gm = f_mul(co.c, fcol), a_tx = tx + 1 < M ? co.a : (T)0;
      const T decay = f_add(f_mul(co.d, fq), a_gm);
      const T tr = qtop ? (T)0 : g_cd;
      const T e0 = f_add(f_add(f_add(decay, a_tx), tr), f_mul(co.f, fq));
      const T e1 = f_add(f_add(decay, tr), qtop ? (T)0 : co.e);
      pc[r].dg = kComp ? v_make(-e0, -e1) : v_make(f_sub(one, e0), f_sub(one, e1));
      pc[r].up = v_make(f_mul(co.d, (T)(j + 1)), f_mul(co.f, (T)(j + 1)));  // gamma_P (q+1), lambda_ina (q+1)
    } else {
      const int pp = 2 * j;
      const T e0 = f_add(f_add(f_mul(co.b, fcol), tx + 1 < M ? co.a : (T)0), g_cd);
      const T d0 = kComp ? -e0 : f_sub(one, e0);
      const T2 fpp = v_make((T)pp, (T)(pp + 1));
      T2 dg = v_fma(v_make(-co.d, -co.d), fpp, v_make(d0, d0));
      if (P - 1 == pp || P - 1 == pp + 1) {
        rtop = r;
        if (!kComp) {  // FP64: 1 - e gains the protein birth back in row P - 1
          if (pp == P - 1) dg.x = f_add(dg.x, g_cd);
          else dg.y = f_add(dg.y, g_cd);
        }
      }
      pc[r].dg = dg;
      pc[r].up = v_fma(v_make(co.d, co.d), fpp, v_make(co.d, co.d));
    }
  }
  if (!owner) rtop = -1;
  const bool ptop_y = (P & 1) == 0;  // row P - 1 is the upper half of its pair
  __syncthreads();
  if (owner) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      buf[o0 + r * st] = S[r];
      if (kUpTab && tx == 0) upt[ty * R + r] = pc[r].up;
      if (kComp && p.renorm > 0) {
        const int c = ROW ? cfirst + r : tx, j = ROW ? 0 : j0 + r;
        float b0, b1;
        if (KIND == MJP_BD1D) {
          b0 = exit_defect<KIND>(co, 0, cta0 + c, N, 1);
          b1 = exit_defect<KIND>(co, 0, cta0 + c + W, N, 1);
        } else {
          const int col = KIND == MJP_TWOSTATE ? cta0 + c : c;
          const int row = KIND == MJP_TWOSTATE ? 0 : 2 * j;
          b0 = exit_defect<KIND>(co, row, col, M, P);
          b1 = exit_defect<KIND>(co, row + 1, col, M, P);
        }
        cbt[o0 + r * st] = make_float2((vx >> r & 1) ? (float)p.renorm * b0 : 0.0f,
                                       (vy >> r & 1) ? (float)p.renorm * b1 : 0.0f);
      }
    }
    // rho_0 beyond this CTA's pairs.
    if (ROW) {
      if (tx == 0) buf[(R - 1) * st] = load_pair(-1, 0);
      if (tx == TX - 1) buf[TX + 1] = load_pair(W, 0);
    }
  }
  // Row kinds: the neighbouring CTAs' pads that receive this CTA's boundary pairs.
  T2 *push_dn = nullptr, *push_up = nullptr;  // buffer 0; buffer 1 is bstride cells further
  if (ROW && CL && owner) {
    if (rank > 0 && tx == 0) push_dn = cluster.map_shared_rank(buf, rank - 1) + TX + 1;
    if (rank + 1 < C && tx == TX - 1) push_up = cluster.map_shared_rank(buf, rank + 1) + (R - 1) * st;
  }
  // Grid kinds: halo slots [parity][side][D M] of 16 bytes (FP32: values and
  // residuals of a pair, FP64: its values) and their barriers; side 0 is
  // filled by the CTA below, side 1 by the CTA above.  Armed here for the
  // first two hand-overs.
  __shared__ __align__(8) unsigned long long hbar[2][2];
  const unsigned hb = (unsigned)__cvta_generic_to_shared(&hbar[0][0]);
  unsigned char* const hx = smem + L.halo;
  const unsigned hside = 16u * (unsigned)(D * M);
  if (link && tid == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) hbar_init(hb + 8u * i);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      if (rank > 0) hbar_arm(hb + 8u * par, hside);
      if (rank + 1 < C) hbar_arm(hb + 16u + 8u * par, hside);
    }
  }
  // Which of the run's pairs go to a neighbour and which come from one.
  bool rx_dn = false, rx_up = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    rx_dn |= link && owner && rank > 0 && ty * R + r < D;
    rx_up |= link && owner && rank + 1 < C && ty * R + r >= D + Hown;
  }
  // Halves outside the box and row P - 1 need a look at each jump; most warps have neither.
  const unsigned full = R < 32 ? (1u << R) - 1u : 0xffffffffu;
  const bool edge_w = __any_sync(kFull, owner && (vx != full || vy != full || rtop >= 0));

  // Observation groups of this thread: tile positions of the two members
  // (elements; the zero cell for a state this CTA does not own) and the time.
  unsigned gl[LL ? GPT : 1];
  int gi[LL ? GPT : 1];
  T gs[LL ? GPT : 1];
  float gc[LL && kComp ? GPT : 1];
  unsigned gmask = 0;
  if (LL) {
    auto loc_of = [&](int s) -> unsigned {
      const unsigned none = 2u * (unsigned)ncell;
      if (KIND == MJP_BD1D) {
        const int c = s - cta0;
        if (c < 0 || c >= 2 * W) return none;
        const int h = c >= W ? 1 : 0, cc = c - h * W;
        return 2u * (unsigned)((cc % R) * st + cc / R + 1) + h;
      }
      if (KIND == MJP_TWOSTATE) {
        const int h = s >= M ? 1 : 0, cc = s - h * M - cta0;
        if (cc < 0 || cc >= W) return none;
        return 2u * (unsigned)((cc % R) * st + cc / R + 1) + h;
      }
      int h, j, c;
      if (KIND == MJP_AUTOREG) {
        h = s / (M * Pm);
        const int rem = s - h * M * Pm;
        j = rem / M;
        c = rem - j * M;
      } else {
        const int row = s / M;
        c = s - row * M;
        j = row >> 1;
        h = row & 1;
      }
      j -= cta0;
      if (j < D || j >= D + Hown) return none;
      return 2u * (unsigned)((j + 1) * st + c + 1) + h;
    };
#pragma unroll
    for (int s = 0; s < GPT; ++s) {
      const int g = s * nthr + tid;
      gs[s] = (T)0;
      if (kComp) gc[s] = 0.0f;
      gi[s] = -1;
      gl[s] = 0;
      if (g < p.G) {
        int a = 0, b = nt - 1;  // the time whose groups hold g: last i with gptr[i] <= g
        while (a < b) {
          const int mid = (a + b + 1) >> 1;
          if (p.gptr[mid] <= g) a = mid;
          else b = mid - 1;
        }
        const int q0 = (int)p.mptr[g], q1 = (int)p.mptr[g + 1];
        const unsigned none = 2u * (unsigned)ncell;
        const unsigned la = q1 > q0 ? loc_of(p.members[q0]) : none;
        const unsigned lb = q1 > q0 + 1 ? loc_of(p.members[q0 + 1]) : none;
        gl[s] = la | (lb << 16);
        if (la != none || lb != none) gi[s] = a;
      }
    }
  }
  const bool any_rec = __syncthreads_or(rec_mine) != 0;

  // Weights of jumps [k0, k0 + kc) of every window; 0 where a window does not
  // hold the jump, so that readers need no test.  Windows without a stored
  // copy get theirs from rec_block.
  const int lgc = tg.lgkc;
  auto stage_chunk = [&](int k0) {
    for (int e = tid; e < nt << lgc; e += nthr) {
      const int i = e >> lgc, j = k0 + (e & (kc - 1));  // jump j in [k0, k0 + kc)
      T* d = ring_at(i, j);
      if (j < t_L[i] || j > t_K[i]) *d = (T)0;
      else if (t_wb[i]) cp_async_elem(d, t_wb[i] + j);
    }
    cp_async_commit();
  };
  // Algorithm 2's recurrence P_k = P_{k-1} x / k for the jumps of a block (the
  // tail added at k = K), at least one barrier ahead of their use (warp 0).
  auto rec_block = [&](int k0) {
    for (int i = lane; i < nt; i += 32) {
      if (t_wb[i]) continue;
      double P = pw[i];
      for (int k = max(k0, t_L[i]); k < k0 + JB && k <= t_K[i]; ++k) {
        P = (k == t_L[i]) ? P : __dmul_rn(P, __ddiv_rn(t_x[i], (double)k));
        *ring_at(i, k) = (T)(P + (k == t_K[i] ? t_tail[i] : 0.0));
      }
      pw[i] = P;
    }
  };
  stage_chunk(K0);
  stage_chunk(K0 + kc);
  if (any_rec && warp == 0) rec_block(K0);
  cp_async_wait<0>();
  // Transient distributions: each window takes an accumulator in shared memory
  // that no earlier window still holds (in blocks of J jumps), or works in
  // global memory (-1) when all are taken.
  T2* const accs = reinterpret_cast<T2*>(smem + L.acc);
  int* const t_slot = reinterpret_cast<int*>(smem + L.tslot);
  if (!LL && tid == 0) {
    int* const until = reinterpret_cast<int*>(smem + L.red);  // last block of each accumulator's window (up to 64)
    const int ns = min(tg.nslot, 64);
    for (int q = 0; q < ns; ++q) until[q] = -1;  // blocks are counted from 0
    int q = 0;
    for (int i = 0; i < nt; ++i) {
      int tries = 0;
      while (tries < ns && until[q] >= (t_L[i] - 1) / J) {
        q = q + 1 == ns ? 0 : q + 1;
        ++tries;
      }
      const bool got = ns > 0 && tries < ns;
      t_slot[i] = got ? q : -1;
      if (got) {
        until[q] = (t_K[i] - 1) / J;
        q = q + 1 == ns ? 0 : q + 1;
      }
    }
  }
  if (CL) cluster.sync();
  else __syncthreads();

  // ---- one jump: rho_k (registers and tile `from`) -> rho_{k+1} (tile `to`) ----
  auto update_as = [&](int from, int to, auto EDGEC) {
    constexpr bool EDGE = decltype(EDGEC)::value;
    const T2* src = buf + from * bstride;
    T2* dst = buf + to * bstride;
    if (owner) {
      // Every read of the tile before the first write to the other one: the
      // compiler cannot tell the two apart, and a read behind a write would
      // put the pairs of a run one after another.
      T2 prev = ROW ? src[(R - 1) * st + o0 - 1] : src[o0 - st];
      const T2 nextE = ROW ? src[o0 + 1] : src[o0 + R * st];
      T2 gl_[ROW ? 1 : R], gr_[ROW ? 1 : R];
      if (!ROW) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          gl_[ROW ? 0 : r] = src[o0 + r * st - 1];
          gr_[ROW ? 0 : r] = src[o0 + r * st + 1];
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const T2 cur = S[r];
        const T2 nx = r + 1 < R ? S[r + 1] : nextE;
        const T2 left = ROW ? prev : gl_[ROW ? 0 : r], right = ROW ? nx : gr_[ROW ? 0 : r];
        const T2 dg = pc[r].dg, up = kUpTab ? upt[ty * R + r] : pc[r].up;
        T2 y;
        if constexpr (kComp) {
          float2 l = lo[r], t;
          if (KIND == MJP_BD1D) {
            y = comp_jump(cur, l, v_make(co.a, co.a), left, up, right, dg);
          } else {
            if (KIND == MJP_TWOSTATE) {
              t = v_fma(v_make(co.a, (T)0), left, l);
              t = v_fma(up, right, t);
              t = v_fma(v_make(co.c, co.d), v_make(cur.y, cur.x), t);
              t = v_fma(dg, cur, t);
            } else if (KIND == MJP_AUTOREG) {
              t = l;
              t.x = f_fma(co.a, left.x, t.x);
              t = v_fma(v_make(g_cr, g_cr), right, t);
              t = v_fma(v_make(g_cd, g_cd), prev, t);
              t = v_fma(v_make(up.x, up.x), nx, t);
              t.x = f_fma(co.e, prev.y, t.x);
              t.y = f_fma(up.y, nx.x, t.y);
              t = v_fma(dg, cur, t);
            } else {
              t = v_fma(v_make(co.a, co.a), left, l);
              t = v_fma(v_make(g_cr, g_cr), right, t);
              t.x = f_fma(g_cd, prev.y, t.x);
              t.y = f_fma(g_cd, cur.x, t.y);
              t.x = f_fma(up.x, cur.y, t.x);
              t.y = f_fma(up.y, nx.x, t.y);
              t = v_fma(dg, cur, t);
              if (EDGE && r == rtop) {  // row P - 1: the protein birth does not leave it
                if (ptop_y) t.y = f_fma(g_cd, cur.y, t.y);
                else t.x = f_fma(g_cd, cur.x, t.x);
              }
            }
            y = comp_finish(cur, t, l);
          }
          if (EDGE) {
            if (!(vx >> r & 1)) y.x = l.x = 0.0f;
            if (!(vy >> r & 1)) y.y = l.y = 0.0f;
          }
          lo[r] = l;
        } else {
          if (KIND == MJP_BD1D) {
            y = v_mul(dg, cur);
            y = v_fma(v_make(co.a, co.a), left, y);
            y = v_fma(up, right, y);
          } else if (KIND == MJP_TWOSTATE) {
            y = v_mul(dg, cur);
            y.x = f_fma(co.a, left.x, y.x);
            y = v_fma(up, right, y);
            y = v_fma(v_make(co.c, co.d), v_make(cur.y, cur.x), y);
          } else if (KIND == MJP_AUTOREG) {
            y = v_mul(dg, cur);
            y.x = f_fma(co.a, left.x, y.x);
            y = v_fma(v_make(g_cr, g_cr), right, y);
            y = v_fma(v_make(g_cd, g_cd), prev, y);
            y = v_fma(v_make(up.x, up.x), nx, y);
            y.x = f_fma(co.e, prev.y, y.x);
            y.y = f_fma(up.y, nx.x, y.y);
          } else {
            y = v_fma(v_make(g_cr, g_cr), right, v_fma(v_make(co.a, co.a), left, v_mul(dg, cur)));
            y.x = f_fma(up.x, cur.y, f_fma(g_cd, prev.y, y.x));
            y.y = f_fma(up.y, nx.x, f_fma(g_cd, cur.x, y.y));
          }
          if (EDGE) {
            if (!(vx >> r & 1)) y.x = (T)0;
            if (!(vy >> r & 1)) y.y = (T)0;
          }
        }
        prev = cur;
        S[r] = y;
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        dst[o0 + r * st] = S[r];
      const int po = to * bstride;
      if (KIND == MJP_BD1D) {
        // The halves of a CTA's run meet inside it: state W - 1 precedes state W.
        T* const dl = reinterpret_cast<T*>(dst + (R - 1) * st);  // left pad (x: the CTA below, y: state W - 1)
        T* const dr = reinterpret_cast<T*>(dst + TX + 1);        // right pad (x: state W, y: the CTA above)
        if (tx == 0) dr[0] = S[0].y;
        if (tx == TX - 1) dl[1] = S[R - 1].x;
        if (push_dn) reinterpret_cast<T*>(push_dn + po)[1] = S[0].x;
        if (push_up) reinterpret_cast<T*>(push_up + po)[0] = S[R - 1].y;
      } else {
        if (push_dn) push_dn[po] = S[0];
        if (push_up) push_up[po] = S[R - 1];
      }
    }
  };
  auto update = [&](int from, int to) {
    if (edge_w) update_as(from, to, std::true_type{});
    else update_as(from, to, std::false_type{});
  };
  // The exit defects added back to the residuals.
  auto defect_fix = [&]() {
    if constexpr (kComp) {
      if (!owner) return;
#pragma unroll
      for (int r = 0; r < R; ++r) lo[r] = v_fma(cbt[o0 + r * st], S[r], lo[r]);
    }
  };
  // Observation groups of rho_kp: slot s's group adds w sum_{members} rho.
  auto groups = [&](int kp, int par) {
    if (!gmask) return;
    const T* cur = reinterpret_cast<const T*>(buf + (par ? bstride : 0));
    const T* wr = ring + (kp & (2 * kc - 1)) * nt;
#pragma unroll
    for (int s = 0; s < GPT; ++s) {
      if (!(gmask >> s & 1)) continue;
      const unsigned g = tile_opaque(gl[s]);  // its two positions are unpacked here, not kept in registers
      const T v = f_add(cur[g & 0xffffu], cur[g >> 16]);
      const T w = wr[gi[s]];
      if constexpr (kComp) {
        const float y = __fsub_rn(__fmul_rn(w, v), gc[s]);
        const float t = __fadd_rn(gs[s], y);
        gc[s] = __fsub_rn(__fsub_rn(t, gs[s]), y);
        gs[s] = t;
      } else {
        gs[s] = f_fma(w, v, gs[s]);
      }
    }
  };

  // ---- the jump chain --------------------------------------------------------
  // Jumps come in blocks of JB (at most JB - 1 more than K are formed; their
  // weights are 0), so that everything else is tested once a block: the next
  // chunk of weights is staged at the start of a chunk (log-likelihoods: the
  // slots it takes were last read before the last barrier; transient
  // distributions: after the block's barriers, behind the reads of the chunk
  // before), and has landed before the last barrier of the chunk.  The defect
  // correction (a period of a multiple of 8 jumps) can only fall on the
  // eighth jump of an aligned eight.
  int dleft = p.renorm > 0 ? p.renorm : 0x7fffffff;  // (odd: never reaches 0)
  // Hand-over of the halo pair rows: send the outermost own pairs; then wait
  // for the neighbours' and put them into the registers and the tile that
  // holds the jump.  A hand-over of the same parity reuses the slots and barriers: the
  // neighbour sends it only after it has received this CTA's pairs of the
  // hand-over in between, which left after the slots were read and the
  // barriers armed again (a CTA barrier lies between).  When any thread's wait
  // runs out (kStatusTimeout), the barrier that closes the hand-over tells the
  // whole CTA (threads that send need not receive), and it neither sends, waits
  // nor arms any more.  Its neighbours then run out at the next hand-over at
  // the latest, which they have sent by then: every byte sent falls on a phase
  // armed for it, and no more than these two phases can still be on their way.
  unsigned hpar = 0, hph = 0;  // parity of the hand-over; phase of each parity's barriers
  bool lost = false;           // the same in all threads of the CTA
  auto hand_send = [&]() {
    const unsigned slot0 = (unsigned)__cvta_generic_to_shared(hx) + hpar * 2u * hside;
    if (owner && !lost) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int f = ty * R + r;
        if (rank > 0 && f >= D && f < 2 * D) {
          const unsigned a = cluster_addr(slot0 + hside + 16u * (unsigned)((f - D) * M + tx), rank - 1);
          const unsigned bar = cluster_addr(hb + 16u + 8u * hpar, rank - 1);
          if constexpr (kComp) st_async16(a, S[r], lo[r], bar);
          else st_async16(a, S[r], bar);
        }
        if (rank + 1 < C && f >= Hown && f < Hown + D) {
          const unsigned a = cluster_addr(slot0 + 16u * (unsigned)((f - Hown) * M + tx), rank + 1);
          const unsigned bar = cluster_addr(hb + 8u * hpar, rank + 1);
          if constexpr (kComp) st_async16(a, S[r], lo[r], bar);
          else st_async16(a, S[r], bar);
        }
      }
    }
  };
  // Ends with the CTA barrier after which the tile may be read.
  auto hand_recv = [&](int at) {
    T2* const tile = buf + at * bstride;
    bool out = false;  // this thread's wait ran out
    if (lost) {
      __syncthreads();
      return;
    }
    if (rx_dn || rx_up) {
      const unsigned ph = (hph >> hpar) & 1u;
      bool ok = !rx_dn || hbar_wait(hb + 8u * hpar, ph, p.wait_limit);
      if (ok && rx_up) ok = hbar_wait(hb + 16u + 8u * hpar, ph, p.wait_limit);
      if (ok) {
        // The first thread of the lower halo and the last pair row's first
        // thread of the upper one arm the barriers for the hand-over after next.
        if (rx_dn && tx == 0 && ty == 0) hbar_arm(hb + 8u * hpar, hside);
        if (rx_up && tx == 0 && ty == TY - 1) hbar_arm(hb + 16u + 8u * hpar, hside);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int f = ty * R + r;
          const bool dn = rank > 0 && f < D, up = rank + 1 < C && f >= D + Hown;
          if (!dn && !up) continue;
          const unsigned char* q = hx + hpar * 2u * hside + (dn ? 0u : hside) + 16u * (unsigned)((dn ? f : f - D - Hown) * M + tx);
          if constexpr (kComp) {
            const float4 v = *reinterpret_cast<const float4*>(q);
            S[r] = make_float2(v.x, v.y);
            lo[r] = make_float2(v.z, v.w);
          } else {
            S[r] = *reinterpret_cast<const double2*>(q);
          }
          tile[o0 + r * st] = S[r];
        }
      } else {
        out = true;
        set_status(p.status, kStatusTimeout);
      }
    }
    hph ^= 1u << hpar;
    hpar ^= 1u;
    lost = __syncthreads_or(out) != 0;
  };
  int xleft = tg.period;
  if (LL) {
    // End of a jump whose values lie in tile `at`.
    auto barrier = [&](int at) {
      if (ROW && CL) {
        __syncwarp();  // the cluster barrier wants converged warps
        cluster_arrive();
        cluster_wait();
      } else {
        if (link && --xleft == 0) {
          hand_send();
          hand_recv(at);
          xleft = tg.period;
        } else {
          __syncthreads();
        }
      }
    };
    for (int kb = 0; kb <= Kmax; kb += JB) {
      if ((kb & (kc - 1)) == 0) {
        if (kb > 0 && kb + kc <= Kmax) stage_chunk(kb + kc);
        gmask = 0;  // slots whose window meets this chunk
#pragma unroll
        for (int s = 0; s < GPT; ++s)
          if (gi[s] >= 0 && t_L[gi[s]] < kb + kc && t_K[gi[s]] >= kb) gmask |= 1u << s;
      }
      if (any_rec && warp == 0) rec_block(kb + JB);
      dleft -= JB;
      const bool dblk = dleft == 0;
      if (dblk) dleft = p.renorm;
#pragma unroll 1
      for (int q = 0; q < JB; q += 2) {
        groups(kb + q, 0);
        update(0, 1);
        barrier(1);
        groups(kb + q + 1, 1);
        update(1, 0);
        if (q == JB - 2) {
          if (kComp && dblk) defect_fix();
          cp_async_wait<0>();
        }
        barrier(0);
      }
    }
  } else {
    // P_0 rho_0 opens the windows that hold jump 0 (an accumulator in shared
    // memory or, as the start of the sum, the output itself).
    constexpr int kAcc = kComp ? 2 : 1;  // pairs per accumulator: sum (and compensation)
    const int stride = kAcc * TX * TY;
    auto store_out = [&](int i, int r, T2 s, float2 c, bool last) {
      if (!(own >> r & 1)) return;
      T* const orow = reinterpret_cast<T*>(p.out) + (int64_t)job * p.out_stride + (int64_t)(p.orig ? p.orig[i] : i) * N;
      float* const crow = kComp ? p.comp + (int64_t)job * p.comp_stride + (int64_t)i * N : nullptr;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int n = state_of(ROW ? cfirst + r : tx, ROW ? 0 : j0 + r, h);
        if (n < 0) continue;
        T v = h ? s.y : s.x;
        const float cv = h ? c.y : c.x;
        if (kComp && last) v = (T)__fsub_rn((float)v, cv);
        orow[n] = v;
        if (kComp && !last) crow[n] = cv;
      }
    };
    auto load_out = [&](int i, int r, T2& s, float2& c) {
      if (!(own >> r & 1)) return;
      const T* const orow = reinterpret_cast<const T*>(p.out) + (int64_t)job * p.out_stride + (int64_t)(p.orig ? p.orig[i] : i) * N;
      const float* const crow = kComp ? p.comp + (int64_t)job * p.comp_stride + (int64_t)i * N : nullptr;
      const int n0 = state_of(ROW ? cfirst + r : tx, ROW ? 0 : j0 + r, 0);
      const int n1 = state_of(ROW ? cfirst + r : tx, ROW ? 0 : j0 + r, 1);
      if (n0 >= 0) s.x = orow[n0];
      if (n1 >= 0) s.y = orow[n1];
      if constexpr (kComp) {
        if (n0 >= 0) c.x = crow[n0];
        if (n1 >= 0) c.y = crow[n1];
      }
    };
    auto acc_at = [&](int i) -> T2* { return accs + ((size_t)max(t_slot[i], 0) * R * TX * TY + tid) * kAcc; };
    if (owner)
      for (int i = 0; i < nt; ++i) {
        if (t_L[i] > 0) continue;
        const T w = t_wb[i] ? t_wb[i][0] : (T)(t_PL[i] + (t_K[i] == 0 ? t_tail[i] : 0.0));
        T2* const a = acc_at(i);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const T2 s = v_mul(v_make(w, w), S[r]);
          const float2 z = make_float2(0.0f, 0.0f);
          if (t_slot[i] < 0 || t_K[i] == 0) {
            store_out(i, r, s, z, t_K[i] == 0);
          } else {
            a[(size_t)r * stride] = s;
            if constexpr (kComp) a[(size_t)r * stride + 1] = z;
          }
        }
      }
    int wlo = 0, whi = -1;
    // Block: jumps kb + 1 .. kb + J; rho_{kb+j} is formed in tile j mod J.
    for (int kb = 0; kb < Kmax; kb += J) {
      if (any_rec && warp == 0) rec_block(kb + J + 1);
      if ((kb & (kc - 1)) == 0) cp_async_wait<0>();
      bool sent = false;
#pragma unroll 2
      for (int j = 0; j < J; ++j) {
        const int to = (j + 1) & (J - 1);
        update(j, to);
        if (kComp && ((j & 7) == 7 || j == J - 1)) {
          dleft -= J < 8 ? J : 8;
          if (dleft == 0) {
            dleft = p.renorm;
            defect_fix();
          }
        }
        if (ROW && CL) {
          __syncwarp();
          cluster_arrive();
          cluster_wait();
        } else {
          if (link && --xleft == 0) {
            xleft = tg.period;
            hand_send();
            if (j == J - 1) {
              sent = true;  // received after the block's sums, which hide the way
              break;
            }
            hand_recv(to);
          } else {
            __syncthreads();
          }
        }
      }
      // rho*_i += sum_j P_{kb+j} rho_{kb+j}, j = 1 .. J, for the windows that meet the block.
      while (wlo < nt && t_K[wlo] <= kb) ++wlo;
      while (whi + 1 < nt && t_L[whi + 1] <= kb + J) ++whi;
      if (owner && wlo <= whi) {
        constexpr bool kPre = R <= 2;  // the values of the block stay in registers over all windows
        T2 H[J][kPre ? R : 1];
        auto load_h = [&](int r, int q) {
#pragma unroll
          for (int j = 1; j <= J; ++j) H[j - 1][q] = buf[(j & (J - 1)) * bstride + o0 + r * st];
        };
        if (kPre) {
#pragma unroll
          for (int r = 0; r < R; ++r) load_h(r, kPre ? r : 0);
        }
#pragma unroll 1
        for (int i = wlo; i <= whi; ++i) {
          T w[J];
          const T* wr = ring_at(i, kb + 1);
          if constexpr (kComp) {
#pragma unroll
            for (int q = 0; q < J / 4; ++q) {
              const float4 v = reinterpret_cast<const float4*>(wr)[q];
              w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
            }
          } else {
#pragma unroll
            for (int q = 0; q < J / 2; ++q) {
              const double2 v = reinterpret_cast<const double2*>(wr)[q];
              w[2 * q] = v.x; w[2 * q + 1] = v.y;
            }
          }
          const bool first = t_L[i] > kb, last = t_K[i] <= kb + J, shared = t_slot[i] >= 0;
          const bool plain = shared && !first && !last;
          T2* a = acc_at(i);
#pragma unroll
          for (int r = 0; r < R; ++r, a += stride) {
            if (!kPre) load_h(r, 0);
            T2 s = v_zero<T>();
            float2 c = make_float2(0.0f, 0.0f);
            if (plain) {
              if constexpr (kComp) {
                const float4 v = *reinterpret_cast<const float4*>(a);
                s = make_float2(v.x, v.y);
                c = make_float2(v.z, v.w);
              } else {
                s = a[0];
              }
            } else if (!first) {
              if (shared) {
                s = a[0];
                if constexpr (kComp) c = a[1];
              } else {
                load_out(i, r, s, c);
              }
            }
            constexpr int q = 0;
            if constexpr (kComp) {
#pragma unroll
              for (int j = 0; j < J; ++j) kahan_pair(v_mul(v_make(w[j], w[j]), H[j][kPre ? r : q]), s, c);
            } else {
#pragma unroll
              for (int j = 0; j < J; ++j) s = v_fma(v_make(w[j], w[j]), H[j][kPre ? r : q], s);
            }
            if (plain) {
              if constexpr (kComp) *reinterpret_cast<float4*>(a) = make_float4(s.x, s.y, c.x, c.y);
              else a[0] = s;
            } else if (last || !shared) {
              store_out(i, r, s, c, last);
            } else {
              a[0] = s;
              if constexpr (kComp) a[1] = c;
            }
          }
        }
      }
      if (sent) hand_recv(0);
      // The next chunk of weights, once no one reads the slots it takes (the
      // block's barriers lie behind the reads of the chunk before).
      if ((kb & (kc - 1)) == 0 && kb > 0 && kb + kc < Kmax) stage_chunk(kb + kc + 1);
    }
  }
  cp_async_wait<0>();
  if (link) {
    // No CTA leaves while a neighbour's pairs may be on their way to it: after a
    // wait that ran out, those of that hand-over and of the next one may still
    // come.  Behind this barrier all of them have been sent; the waits (bounded
    // again, 2 ms and more) end as soon as they have landed.
    cluster.sync();
    if (lost) {
      constexpr long long kDrain = 1 << 16;
#pragma unroll 1
      for (int q = 0; q < 2; ++q) {  // the next hand-over, then the one that ran out
        const unsigned par = hpar ^ (unsigned)q, ph = ((hph >> par) & 1u) ^ (unsigned)q;
        if (rx_dn) hbar_wait(hb + 8u * par, ph, kDrain);
        if (rx_up) hbar_wait(hb + 16u + 8u * par, ph, kDrain);
      }
    }
  }
  if (!LL && any_rec && owner) {
    // Times whose K is above the cap (their weight is NaN) have no result.
    for (int i = 0; i < nt; ++i) {
      if (!isnan(t_PL[i])) continue;
      T* const orow = reinterpret_cast<T*>(p.out) + (int64_t)job * p.out_stride + (int64_t)(p.orig ? p.orig[i] : i) * N;
#pragma unroll
      for (int r = 0; r < R; ++r)
        for (int h = 0; h < 2; ++h) {
          const int n = (own >> r & 1) ? state_of(ROW ? cfirst + r : tx, ROW ? 0 : j0 + r, h) : -1;
          if (n >= 0) orow[n] = (T)t_PL[i];
        }
    }
  }

  if (LL) {
    // ---- epilogue: sum_g c_g log(a_g), partial sums of all CTAs --------------
    // Every CTA's accumulators, (sum, compensation) per group, over the tile
    // (no one reads it any more: every phase ended in a barrier).
    T* const es = reinterpret_cast<T*>(smem);
    float* const ec = reinterpret_cast<float*>(smem + 4 * (size_t)p.G);
#pragma unroll
    for (int s = 0; s < GPT; ++s) {
      const int g = s * nthr + tid;
      if (g < p.G) {
        es[g] = gs[s];
        if (kComp) ec[g] = gc[s];
      }
    }
    if (CL) cluster.sync();
    else __syncthreads();
    if (rank == 0) {
      double ll = 0.0;
      bool bad = false;
      for (int g = tid; g < p.G; g += nthr) {
        double a = 0.0;
        for (int r = 0; r < C; ++r) {
          const T* rsum = !CL ? es : cluster.map_shared_rank(es, r);
          double v = (double)rsum[g];
          if (kComp) {
            const float* rc = !CL ? ec : cluster.map_shared_rank(ec, r);
            v -= (double)rc[g];
          }
          a += v;
        }
        const double c = p.counts[g];
        if (c == 0.0) continue;
        if (a > 0.0) ll += c * log(a);
        else if (a > -1e-30) ll = -INFINITY;
        else bad = true;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ll += __shfl_xor_sync(kFull, ll, o);
      double* red = reinterpret_cast<double*>(smem + L.red);
      if (lane == 0) red[warp] = ll;
      __syncthreads();
      if (tid == 0) {
        double tot = 0.0;
        for (int w = 0; w < nthr >> 5; ++w) tot += red[w];
        if (isnan(tot)) set_status(p.status, kStatusNumeric);
        p.ll[job] = tot;
      }
      if (bad) set_status(p.status, kStatusNumeric);
    }
    if (CL) cluster.sync();  // keep every CTA's accumulators alive until rank 0 is done
  }
}

// ---- launch ------------------------------------------------------------------

template <typename T, int KIND, bool LL, bool CL, int R, int GPT>
cudaError_t tile_one(const ChainParams* p, const TilePlan& tp, cudaStream_t s) {
  auto kern = tile_kernel<T, KIND, LL, CL, R, GPT, tile_jumps(sizeof(T), R), tile_max_threads(sizeof(T), LL, CL, R)>;
  // Attributes are set at their largest.
  static std::atomic<uint64_t> done{0};
  cudaError_t e = once_per_device(done, [&] {
    const cudaError_t m = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmemMax);
    return m != cudaSuccess ? m : cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((p ? p->B : 1) * tp.cluster));
  cfg.blockDim = dim3((unsigned)tp.threads);
  cfg.dynamicSmemBytes = tp.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)tp.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = tp.cluster > 1 ? 1 : 0;
  if (p) return cudaLaunchKernelEx(&cfg, kern, *p, tp.geo);
  int n = 0;
  if ((e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg)) != cudaSuccess) {
    cudaGetLastError();
    return e;
  }
  return n > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

}  // namespace
}  // namespace mjp
