// stencil_small.cu -- transient distributions of small birth-death and
// two-state models (FP32 and FP64): one CTA, one state per thread, the sums of
// the observation times on warps of their own.
//
// A solve of some hundred jumps on some dozen states is bound by the latency
// of a jump.  One warp with two states per lane (the register kernel's
// smallest shape) holds its scheduler's FP64 pipe for 64 cycles per operation:
// 6 for the jump and 2 per window that overlaps, 1,480 cycles a jump on 64
// states and five times while three schedulers idle.  Here the chain's warps
// do nothing but the jump (read the neighbours from the ring of the last 16
// jumps, three or four dependent multiply-adds, write, a barrier of the chain
// warps); every 8 jumps they meet the reducer warps, which add the block
// sum_j P_{k+j} rho_{k+j} to the windows that hold it while the chain forms
// the next block.  The two sides touch disjoint slots of the ring: the
// reducers read jumps kb + 1 .. kb + 8, the chain writes kb + 9 .. kb + 16.
//
// Arithmetic per state is the sequence of stencil.cu; the sums are those of
// stencil_tile.cuh (one jump after the other; FP32: a Kahan step for each
// product).
#include <algorithm>

#include "chain_common.cuh"
#include "host_util.h"
#include "internal.cuh"

namespace mjp {

namespace {

constexpr int kJ = 8;            // jumps per block
constexpr int kRing = 2 * kJ;    // jumps the ring holds
constexpr int kWChunk = 32;      // jumps per staged chunk of weights (a multiple of kJ)
constexpr int kWStride = 2 * kWChunk + 4;

struct SmallSmem {
  size_t tx, tPL, ttail, pw, twb, tL, tK, torig, w, acc, total;
};
__host__ __device__ inline SmallSmem small_smem(size_t elt, int cells, int N, int nt) {
  SmallSmem s;
  auto up = [](size_t v) { return (v + 15) / 16 * 16; };
  size_t o = up(elt * kRing * (size_t)cells);
  s.tx = o; o += up(8 * (size_t)nt);
  s.tPL = o; o += up(8 * (size_t)nt);
  s.ttail = o; o += up(8 * (size_t)nt);
  s.pw = o; o += up(8 * (size_t)nt);
  s.twb = o; o += up(8 * (size_t)nt);
  s.tL = o; o += up(4 * (size_t)nt);
  s.tK = o; o += up(4 * (size_t)nt);
  s.torig = o; o += up(4 * (size_t)nt);
  s.w = o; o += up(elt * kWStride * (size_t)nt);
  s.acc = o; o += 8 * (size_t)N * nt;  // FP32: sum and compensation, FP64: sum
  s.total = o;
  return s;
}

__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <typename T, int KIND>
__global__ void __launch_bounds__(1024, 1) chain_small_kernel(const ChainParams p, const int nchain) {
  constexpr bool kComp = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x;
  const int nt = p.ntimes, N = (int)p.N, M = p.M;
  // Cell of state n: BD n + 1; two-state rows of M + 2 cells; the pads stay 0.
  const int cells = KIND == MJP_BD1D ? N + 2 : 2 * (M + 2);
  auto cell = [&](int n) -> int { return KIND == MJP_BD1D ? n + 1 : n + 1 + (n >= M ? 2 : 0); };
  const SmallSmem L = small_smem(sizeof(T), cells, N, nt);
  T* const ring = reinterpret_cast<T*>(smem);
  double* t_x = reinterpret_cast<double*>(smem + L.tx);
  double* t_PL = reinterpret_cast<double*>(smem + L.tPL);
  double* t_tail = reinterpret_cast<double*>(smem + L.ttail);
  double* pw = reinterpret_cast<double*>(smem + L.pw);
  const T** t_wb = reinterpret_cast<const T**>(smem + L.twb);
  int* t_L = reinterpret_cast<int*>(smem + L.tL);
  int* t_K = reinterpret_cast<int*>(smem + L.tK);
  int* t_orig = reinterpret_cast<int*>(smem + L.torig);
  T* const wts = reinterpret_cast<T*>(smem + L.w);  // [nt][kWStride]: jump k in slot (k - 1) mod 64, 0 outside its window
  const T* arena = reinterpret_cast<const T*>(p.arena);
  for (int i = tid; i < nt; i += blockDim.x) {
    const Win w = p.win[i];
    t_x[i] = w.x;
    t_PL[i] = w.PL;
    t_tail[i] = w.tail;
    pw[i] = w.PL;
    t_L[i] = (int)w.L;
    t_K[i] = (int)w.K;
    t_wb[i] = w.woff >= 0 && arena ? arena + (w.woff - w.L) : nullptr;
    t_orig[i] = p.orig[i];
  }
  for (int e = tid; e < kRing * cells; e += blockDim.x) ring[e] = (T)0;
  const int Kmax = (int)p.info[0].Kmax;
  const double omega = p.info[0].omega;
  const T* rho0 = reinterpret_cast<const T*>(p.rho0);
  __syncthreads();
  const bool chain = tid < nchain;
  const bool owner = tid < N;  // chain threads that hold a state
  if (owner) ring[cell(tid)] = rho0[tid];
  __syncthreads();

  if (chain) {
    const Coef<T> co = make_coef<T, KIND>(p.theta, omega);
    const int row = KIND == MJP_TWOSTATE && tid >= M ? 1 : 0, m = tid - row * M;
    const int o = cell(owner ? tid : 0), other = KIND == MJP_TWOSTATE ? (row ? o - (M + 2) : o + (M + 2)) : o;
    T cur = owner ? rho0[tid] : (T)0;
    float lo = 0.0f, cb = 0.0f;
    const T one = (T)1;
    T cl, cr, sw = (T)0, dg;  // inflow from the left, the right, the other row; -e (FP32) or 1 - e (FP64)
    if (KIND == MJP_BD1D) {
      const T fm = (T)m, e = f_add(f_mul(co.b, fm), m + 1 < N ? co.a : (T)0);
      cl = co.a;
      cr = f_mul(co.b, f_add(fm, one));
      dg = kComp ? -e : f_sub(one, e);
    } else {
      const T bm = f_mul(co.b, (T)m);
      const T e = row == 0 ? f_add(f_add(bm, m + 1 < M ? co.a : (T)0), co.d) : f_add(co.c, bm);
      cl = row == 0 ? co.a : (T)0;
      cr = f_mul(co.b, (T)(m + 1));
      sw = row == 0 ? co.c : co.d;
      dg = kComp ? -e : f_sub(one, e);
    }
    if (kComp && p.renorm > 0 && owner) cb = (float)p.renorm * exit_defect<KIND>(co, row, m, KIND == MJP_BD1D ? N : M, 2);
    int dleft = p.renorm > 0 ? p.renorm : 0x7fffffff;  // (odd: never reaches 0)
    for (int kb = 0; kb < Kmax; kb += kJ) {
      const int base = kb & (kRing - 1);  // 0 or 8
#pragma unroll
      for (int j = 0; j < kJ; ++j) {
        const T* src = ring + (base + j) * cells;
        T* dst = ring + ((base + j + 1) & (kRing - 1)) * cells;
        if (owner) {
          const T left = src[o - 1], right = src[o + 1];
          T y;
          if constexpr (kComp) {
            float t = __fmaf_rn(cl, left, lo);
            t = __fmaf_rn(cr, right, t);
            if (KIND == MJP_TWOSTATE) t = __fmaf_rn(sw, src[other], t);
            t = __fmaf_rn(dg, cur, t);
            y = comp_finish(cur, t, lo);
          } else {
            y = f_mul(dg, cur);
            if (KIND == MJP_BD1D || row == 0) y = f_fma(cl, left, y);
            y = f_fma(cr, right, y);
            if (KIND == MJP_TWOSTATE) y = f_fma(sw, src[other], y);
          }
          cur = y;
          dst[o] = y;
        }
        if (kComp && j == kJ - 1) {
          dleft -= kJ;
          if (dleft == 0) {
            dleft = p.renorm;
            lo = __fmaf_rn(cb, (float)cur, lo);
          }
        }
        if (j < kJ - 1) named_barrier(1, nchain);
      }
      __syncthreads();
    }
    return;
  }

  // ---- reducers ----------------------------------------------------------------
  const int rt = tid - nchain, nred = blockDim.x - nchain;
  const int groups = nred / nchain, g = rt / nchain;  // group g takes the times i = g mod groups
  const int n = rt - g * nchain;
  const bool mine = g < groups && n < N;
  const int on = cell(n < N ? n : 0);
  float2* const acc32 = reinterpret_cast<float2*>(smem + L.acc);
  double* const acc64 = reinterpret_cast<double*>(smem + L.acc);
  auto slot = [&](int i, int k) -> T* { return wts + i * kWStride + ((k - 1) & (2 * kWChunk - 1)); };
  auto stage_chunk = [&](int k0) {  // weights of jumps k0 .. k0 + kWChunk - 1
    for (int e = rt; e < nt * kWChunk; e += nred) {
      const int i = e / kWChunk, k = k0 + (e & (kWChunk - 1));
      if (k < t_L[i] || k > t_K[i]) *slot(i, k) = (T)0;
      else if (t_wb[i]) cp_async_elem(slot(i, k), t_wb[i] + k);
    }
    cp_async_commit();
  };
  // Algorithm 2's recurrence for the windows without a stored copy, a block at a time.
  auto rec_block = [&](int k0) {
    for (int i = rt; i < nt; i += nred) {
      if (t_wb[i]) continue;
      double P = pw[i];
      for (int k = max(k0, t_L[i]); k < k0 + kJ && k <= t_K[i]; ++k) {
        P = (k == t_L[i]) ? P : __dmul_rn(P, __ddiv_rn(t_x[i], (double)k));
        *slot(i, k) = (T)(P + (k == t_K[i] ? t_tail[i] : 0.0));
      }
      pw[i] = P;
    }
  };
  T* const out = reinterpret_cast<T*>(p.out);
  auto finish = [&](int i, T s, float c) {
    if (kComp) s = (T)__fsub_rn((float)s, c);
    out[(int64_t)t_orig[i] * N + n] = s;
  };
  stage_chunk(1);
  stage_chunk(1 + kWChunk);
  rec_block(1);
  // P_0 rho_0 opens the windows that hold jump 0.
  if (mine)
    for (int i = g; i < nt; i += groups) {
      if (t_L[i] > 0) continue;
      const T w = t_wb[i] ? t_wb[i][0] : (T)(t_PL[i] + (t_K[i] == 0 ? t_tail[i] : 0.0));
      const T s = f_mul(w, rho0[n]);
      if (t_K[i] == 0) finish(i, s, 0.0f);
      else if constexpr (kComp) acc32[(size_t)i * N + n] = make_float2(s, 0.0f);
      else acc64[(size_t)i * N + n] = s;
    }
  cp_async_wait<0>();
  named_barrier(2, nred);
  int wlo = 0, whi = -1;
  for (int kb = 0; kb < Kmax; kb += kJ) {
    __syncthreads();  // rho_{kb+1} .. rho_{kb+8} are in the ring
    while (wlo < nt && t_K[wlo] <= kb) ++wlo;
    while (whi + 1 < nt && t_L[whi + 1] <= kb + kJ) ++whi;
    if (mine) {
      T H[kJ];
#pragma unroll
      for (int j = 0; j < kJ; ++j) H[j] = ring[((kb + 1 + j) & (kRing - 1)) * cells + on];
      for (int i = wlo + (g - wlo % groups + groups) % groups; i <= whi; i += groups) {
        T w[kJ];
        const T* wr = slot(i, kb + 1);
#pragma unroll
        for (int j = 0; j < kJ; ++j) w[j] = wr[j];
        const bool first = t_L[i] > kb, last = t_K[i] <= kb + kJ;
        if constexpr (kComp) {
          float2 a = first ? make_float2(0.0f, 0.0f) : acc32[(size_t)i * N + n];
#pragma unroll
          for (int j = 0; j < kJ; ++j) {
            const float y = __fsub_rn(__fmul_rn(w[j], H[j]), a.y), s = __fadd_rn(a.x, y);
            a.y = __fsub_rn(__fsub_rn(s, a.x), y);
            a.x = s;
          }
          if (last) finish(i, a.x, a.y);
          else acc32[(size_t)i * N + n] = a;
        } else {
          double s = first ? 0.0 : acc64[(size_t)i * N + n];
#pragma unroll
          for (int j = 0; j < kJ; ++j) s = f_fma(w[j], H[j], s);
          if (last) finish(i, s, 0.0f);
          else acc64[(size_t)i * N + n] = s;
        }
      }
    }
    // The next chunk of weights once a chunk is used up, the next block's
    // recurrences; all reducers meet before anyone reads them.
    const int kn = kb + kJ;
    if (kn < Kmax) {
      named_barrier(2, nred);  // everyone is done with this block's weights
      if ((kn & (kWChunk - 1)) == 0) {
        cp_async_wait<0>();  // the chunk that starts now
        if (kn + kWChunk < Kmax) stage_chunk(kn + kWChunk + 1);
      }
      rec_block(kn + 1);
      named_barrier(2, nred);
    }
  }
  cp_async_wait<0>();
  // Times whose K is above the cap (their weight is NaN) have no result.
  if (mine)
    for (int i = g; i < nt; i += groups)
      if (isnan(t_PL[i])) out[(int64_t)t_orig[i] * N + n] = (T)t_PL[i];
}

template <typename T, int KIND>
cudaError_t launch_small(const ChainParams& p, const SmallPlan& sp, cudaStream_t s) {
  static std::atomic<uint64_t> done{0};
  auto kern = chain_small_kernel<T, KIND>;
  const cudaError_t e = once_per_device(done, [&] {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  });
  if (e != cudaSuccess) return e;
  kern<<<1, sp.threads, sp.smem, s>>>(p, sp.nchain);
  return cudaGetLastError();
}

}  // namespace

// Up to 512 states (16 chain warps, as many reducers).  Two-state FP64 models
// whose windows overlap so much that one SM's FP64 pipe is the bound (about
// 1,200 cycles a jump) go to the tile kernel, which spreads them over a
// cluster; birth-death models have no such alternative.  Measured with K =
// 859 (us a call, planner included), birth-death against stencil_reg1d.cu: N =
// 64 at 5 times FP64 676 -> 181, FP32 415 -> 119, at 20 times FP64 1,490 ->
// 266, FP32 805 -> 142; N = 512 at 5 times FP64 1,121 -> 642, FP32 513 -> 184,
// at 20 times FP64 2,629 -> 1,208, FP32 906 -> 285 (more overlapping windows
// than the shared memory holds accumulators for go to stencil_reg1d.cu).
// Two-state against stencil.cu: N_R = 64 at 5 times FP64 943 -> 258, FP32 852
// -> 125, N_R = 256 FP32 961 -> 185 (against stencil_tile.cuh even there).
bool chain_small_plan(int kind, int precision, int64_t M, int64_t N, int nt, double overlap, SmallPlan* out) {
  if (kind != MJP_BD1D && kind != MJP_TWOSTATE) return false;
  if (N > 512) return false;
  const int nchain = (int)((N + 31) / 32) * 32;
  const int groups = std::max(1, std::min({(1024 - nchain) / nchain, 4, nt}));
  const size_t elt = precision == MJP_FP64 ? 8 : 4;
  const int cells = kind == MJP_BD1D ? (int)N + 2 : 2 * ((int)M + 2);
  const SmallSmem L = small_smem(elt, cells, (int)N, nt);
  if (L.total > 200 * 1024) return false;
  if (precision == MJP_FP64 && kind == MJP_TWOSTATE && (double)N * (3.5 + overlap) / 2.0 > 1200.0) return false;
  out->nchain = nchain;
  out->threads = nchain * (1 + groups);
  out->smem = L.total;
  return true;
}

cudaError_t launch_chain_small(int kind, int precision, const ChainParams& p, const SmallPlan& sp, cudaStream_t s) {
  if (precision == MJP_FP64)
    return kind == MJP_BD1D ? launch_small<double, MJP_BD1D>(p, sp, s) : launch_small<double, MJP_TWOSTATE>(p, sp, s);
  return kind == MJP_BD1D ? launch_small<float, MJP_BD1D>(p, sp, s) : launch_small<float, MJP_TWOSTATE>(p, sp, s);
}

}  // namespace mjp
