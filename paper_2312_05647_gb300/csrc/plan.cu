// plan.cu -- the FP64 planner: Omega, truncation index K and Poisson weight
// window of every (instance, time) pair (Eq. B_def, Algorithm 2).
//
// One CTA per instance (one per window for a single instance).  Omega = 1.1
// max_n e_n: the exit rates grow with every coordinate up to the last but one
// state of an axis (sums of rounded non-negative terms are monotone), so the
// maximum is among the corners of the box (stencil models), or taken from the
// model (CSR).
//
// Paper's rule, in four phases.  A thread per window: K = floor(x + 6 sqrt x)
// + 1 with x = Omega t computed with exactly the roundings of Algorithm 2 (no
// fused multiply-add), the window's bounds and its place in the weight store.
// A warp per window and direction: the Poisson weights around the mode m =
// floor(x) as ratios to w_m = 1, x/k upwards and (k+1)/x downwards, as running
// products of 8 terms per lane joined by a warp-wide product scan.  A thread
// per window: the sum W that normalises the weights, the tail beyond K summed
// explicitly (equal to 1 - sum_{k<=K} P_k, Algorithm 2's last line).  A warp
// per window: the stored weights scaled.  No exp(-x) is ever formed, so nothing
// underflows.
//
// Bound: the FP64 pipe (16 cycles per warp instruction and SM).  Work that all
// lanes of a warp did alike (roots and divisions, about 250 instructions per
// window) runs a thread per window instead, and the FP64 reciprocals of 8
// consecutive k are one reciprocal of their product and 8 multiplications.
// Measured: 256 thetas x 50 times FP32 151 -> 89 us, 10^4 thetas x 5 times
// FP64 756 -> 543 us, one theta x 5 times FP64 20 -> 12 us.
//
// Tolerance rule: a warp per window does everything (K is known only after the
// scans).
#include "internal.cuh"

namespace mjp {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double warp_incl_prod(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    double t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v = __dmul_rn(v, t);
  }
  return v;
}

__device__ __forceinline__ double warp_incl_sum(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    double t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

struct Kahan {
  double s = 0.0, c = 0.0;
  __device__ void add(double v) {
    double y = v - c;
    double t = s + y;
    c = (t - s) - y;
    s = t;
  }
};

// Exit rate e_n = sum_m lambda_nm of a stencil model, summed in ascending
// target order (the column order of the rate matrix row) so that Omega is
// bit-identical to a row sum over a CSR with sorted columns.
__device__ double exit_rate(int kind, int64_t M, int64_t P, int64_t n, const double* th) {
  double e = 0.0;
  if (kind == MJP_BD1D) {  // Eq. BD_def
    if (n >= 1) e = __dadd_rn(e, __dmul_rn(th[1], (double)n));
    if (n + 1 < M) e = __dadd_rn(e, th[0]);
  } else if (kind == MJP_TWOSTATE) {  // Eq. Gene_def, sigma = 0 active
    int64_t sg = n / M, nr = n - sg * M;
    if (sg == 0) {
      if (nr >= 1) e = __dadd_rn(e, __dmul_rn(th[1], (double)nr));
      if (nr + 1 < M) e = __dadd_rn(e, th[0]);
      e = __dadd_rn(e, th[3]);
    } else {
      e = __dadd_rn(e, th[2]);
      if (nr >= 1) e = __dadd_rn(e, __dmul_rn(th[1], (double)nr));
    }
  } else if (kind == MJP_AUTOREG) {  // model index n_R + N_R n_P + N_R N_P sigma; P = 2 N_P tile rows
    const int64_t Pm = P / 2, sg = n / (M * Pm), rem = n - sg * M * Pm, q = rem / M, m = rem - q * M;
    // th = {beta_R, beta_P, gamma_R, gamma_P, lambda_act, lambda_ina}, targets ascending
    if (sg == 1 && q + 1 < Pm) e = __dadd_rn(e, th[4]);
    if (q >= 1) e = __dadd_rn(e, __dmul_rn(th[3], (double)q));
    if (m >= 1) e = __dadd_rn(e, __dmul_rn(th[2], (double)m));
    if (sg == 0 && m + 1 < M) e = __dadd_rn(e, th[0]);
    if (q + 1 < Pm && m >= 1) e = __dadd_rn(e, __dmul_rn(th[1], (double)m));
    if (sg == 0 && q >= 1) e = __dadd_rn(e, __dmul_rn(th[5], (double)q));
  } else {  // MRNA_PROT2D: targets n-M, n-1, n+1, n+M
    int64_t p = n / M, m = n - p * M;
    if (p >= 1) e = __dadd_rn(e, __dmul_rn(th[3], (double)p));
    if (m >= 1) e = __dadd_rn(e, __dmul_rn(th[1], (double)m));
    if (m + 1 < M) e = __dadd_rn(e, th[0]);
    if (p + 1 < P && m >= 1) e = __dadd_rn(e, __dmul_rn(th[2], (double)m));
  }
  return e;
}

__device__ void set_status(int* st, int code) {
  if (st) atomicCAS(st, 0, code);
}

// Window [L, K] of x = Omega t under the paper's rule: Algorithm 2's last k
// and the first k whose left Poisson tail is not negligible; false when
// there is no chain (x = 0) or K exceeds the cap.
__device__ bool window_bounds(const PlanParams& p, double x, int64_t& L, int64_t& K) {
  if (x == 0.0) return false;
  const double s = __dsqrt_rn(x);
  const double kstar = __dadd_rn(x, __dmul_rn(6.0, s));  // Omega t + 6 sqrt(Omega t)
  if (!(kstar + 1.0 <= (double)p.kcap)) return false;
  K = (int64_t)floor(kstar) + 1;
  const double lo = __dsub_rn(x, __dmul_rn(10.0, s));  // Poisson left tail below x - 10 sqrt x is < e^-50
  L = lo > 0.0 ? (int64_t)floor(lo) : 0;
  return true;
}

// A window whose K is above the cap: a NaN weight makes this time's result
// (and a log-likelihood using it) NaN, so a caller that keeps going (a
// sampler) rejects the parameters.
__device__ Win capped_window(double x) {
  Win r;
  r.x = x;
  r.L = 0;
  r.K = 0;
  r.PL = __longlong_as_double(0x7ff8000000000000LL);
  r.tail = 0.0;
  r.woff = -1;
  return r;
}

// Float-float numbers (hi + lo, |lo| <= ulp(hi) / 2: ~48 significant bits)
// on the FP32 pipe, which GB300 runs 64 times faster than its FP64 pipe.
// Error-free transformations: TwoSum (Knuth), FastTwoSum (Dekker, |a| >= |b|)
// and TwoProd with a fused multiply-add; every operation explicitly rounded.
struct FF {
  float hi, lo;
};
__device__ __forceinline__ FF ff_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_from(double d) {
  const float hi = __double2float_rn(d);
  return FF{hi, __double2float_rn(d - (double)hi)};
}
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return ff_fast_two_sum(p, e);
}
// a times an integer-valued float c (exact in FP32).
__device__ __forceinline__ FF ff_mul_int(FF a, float c) {
  const float p = __fmul_rn(a.hi, c);
  float e = __fmaf_rn(a.hi, c, -p);
  e = __fmaf_rn(a.lo, c, e);
  return ff_fast_two_sum(p, e);
}
// 1 / c for an integer-valued float c: r0 rounded, plus r0 times the exact
// residual 1 - c r0.
__device__ __forceinline__ FF ff_rcp_int(float c) {
  const float r0 = __frcp_rn(c);
  const float e = __fmaf_rn(-c, r0, 1.0f);
  return ff_fast_two_sum(r0, __fmul_rn(r0, e));
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float v = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return ff_fast_two_sum(s, e);
}
__device__ __forceinline__ FF ff_shfl_up(FF a, int d) {
  return FF{__shfl_up_sync(kFull, a.hi, d), __shfl_up_sync(kFull, a.lo, d)};
}

// Weights of the paper's rule, ratios to w_m = 1 at the mode m = floor(x), in
// one direction: upward w_k = w_{k-1} x / k over (m, R] (dir 0), downward
// w_k = w_{k+1} (k+1) / x over [L, m) (dir 1).  Each lane forms the running
// product of a run of kRun consecutive terms, one warp-wide product scan joins
// the runs.  The unnormalised weights of [L, K] go to `put` when `store`;
// returns (lane 0) the sum of all weights, that of k > K and, downward, w_L.
//
// FP32 chains: products and a lane's sums in float-float (relative error ~1e-14
// over a window of ~10^4 terms, far below the FP32 weights the chains read); the
// lanes' sums are added as three FP32 numbers each (~72 bits, error-free TwoSums)
// and rounded once to FP64, so they are no further from the exact sum than FP64
// additions, which took 6 of 103 us of a call with 45 times.
constexpr int kRun = 8;
struct Sums64 {
  double all, tail, wL;
};
struct F3 {
  float h, m, l;
};
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}
__device__ __forceinline__ F3 f3_add(F3 a, F3 b) {
  float e1, e2, e3;
  F3 r;
  r.h = two_sum(a.h, b.h, e1);
  const float t = two_sum(a.m, b.m, e2);
  r.m = two_sum(t, e1, e3);
  r.l = __fadd_rn(__fadd_rn(a.l, b.l), __fadd_rn(e2, e3));
  return r;
}
// The lanes' sums of a (returned by lanes 0 to 15) and of b (lanes 16 to 31).
__device__ __forceinline__ F3 lane_sums(FF a, FF b, int lane) {
  const FF mine = lane < 16 ? a : b, theirs = lane < 16 ? b : a;
  F3 v = f3_add(F3{mine.hi, mine.lo, 0.0f},
                F3{__shfl_xor_sync(kFull, theirs.hi, 16), __shfl_xor_sync(kFull, theirs.lo, 16), 0.0f});
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
    v = f3_add(v, F3{__shfl_xor_sync(kFull, v.h, o), __shfl_xor_sync(kFull, v.m, o), __shfl_xor_sync(kFull, v.l, o)});
  return v;
}
__device__ __forceinline__ FF ff_warp_incl_prod(FF v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const FF t = ff_shfl_up(v, o);
    if (lane >= o) v = ff_mul(v, t);
  }
  return v;
}
// I: 32-bit jump counts where they fit (a 64-bit integer's conversion to FP32
// runs at the FP64 pipe's rate, one per weight).
template <class I, class Put>
__device__ Sums64 dir_weights(int dir, FF xf, FF invx, I L, I K, I m, I R, int lane, bool store, Put& put) {
  FF all{0.0f, 0.0f}, tail{0.0f, 0.0f}, wL{1.0f, 0.0f};
  FF carry{1.0f, 0.0f};
  if (dir == 0) {
    for (I base = m + 1; base <= R; base += 32 * kRun) {
      const I k0 = base + lane * kRun;
      FF loc[kRun], pr{1.0f, 0.0f};
#pragma unroll
      for (int b = 0; b < kRun; ++b) {
        const I k = k0 + b;
        const FF term = k <= R ? ff_mul(xf, ff_rcp_int((float)k)) : FF{1.0f, 0.0f};
        pr = ff_mul(pr, term);
        loc[b] = pr;
      }
      const FF incl = ff_warp_incl_prod(pr, lane);
      FF excl = ff_shfl_up(incl, 1);
      if (lane == 0) excl = FF{1.0f, 0.0f};
      const FF pre = ff_mul(carry, excl);
#pragma unroll
      for (int b = 0; b < kRun; ++b) {
        const I k = k0 + b;
        if (k <= R) {
          const FF w = ff_mul(pre, loc[b]);
          all = ff_add(all, w);
          if (k > K) tail = ff_add(tail, w);
          else if (store) put(k, w);
        }
      }
      const FF last = ff_mul(pre, pr);
      carry = FF{__shfl_sync(kFull, last.hi, 31), __shfl_sync(kFull, last.lo, 31)};
    }
  } else {
    for (I base = m - 1; base >= L; base -= 32 * kRun) {
      const I k0 = base - lane * kRun;
      FF loc[kRun], pr{1.0f, 0.0f}, wl{0.0f, 0.0f};
#pragma unroll
      for (int b = 0; b < kRun; ++b) {
        const I k = k0 - b;
        const FF term = k >= L ? ff_mul_int(invx, (float)(k + 1)) : FF{1.0f, 0.0f};
        pr = ff_mul(pr, term);
        loc[b] = pr;
      }
      const FF incl = ff_warp_incl_prod(pr, lane);
      FF excl = ff_shfl_up(incl, 1);
      if (lane == 0) excl = FF{1.0f, 0.0f};
      const FF pre = ff_mul(carry, excl);
#pragma unroll
      for (int b = 0; b < kRun; ++b) {
        const I k = k0 - b;
        if (k >= L) {
          const FF w = ff_mul(pre, loc[b]);
          all = ff_add(all, w);
          if (store) put(k, w);
          if (k == L) wl = w;
        }
      }
      if (base - L < 32 * kRun) {  // the run that holds L
        const int src = (int)((base - L) / kRun);
        wL = FF{__shfl_sync(kFull, wl.hi, src), __shfl_sync(kFull, wl.lo, src)};
      }
      const FF last = ff_mul(pre, pr);
      carry = FF{__shfl_sync(kFull, last.hi, 31), __shfl_sync(kFull, last.lo, 31)};
    }
  }
  F3 v = lane_sums(all, tail, lane);
  if (dir == 1 && lane >= 16) v = F3{wL.hi, wL.lo, 0.0f};
  const double d = (double)v.h + ((double)v.m + (double)v.l), other = __shfl_sync(kFull, d, 16);
  return Sums64{d, other, other};
}

// The same in FP64, for the FP64 chains, whose 1e-12 agreement with the oracle
// needs weights (and P_L, the start of the recurrence of a window without a
// stored copy) to FP64 precision.  Upward, x^b / (k0 (k0+1) ..) for the run's
// positions b comes from one reciprocal of the product of all its k, multiplied
// back from the run's end (products of 8 factors up to 2^40 stay finite).
template <class Put>
__device__ Sums64 dir_weights64(int dir, double x, double invx, int64_t L, int64_t K, int64_t m, int64_t R, int lane,
                                bool store, Put& put) {
  Sums64 r{0.0, 0.0, 1.0};
  double carry = 1.0;
  double xp[kRun];  // x^(b+1), or x^-(b+1)
  xp[0] = dir == 0 ? x : invx;
#pragma unroll
  for (int b = 1; b < kRun; ++b) xp[b] = __dmul_rn(xp[b - 1], xp[0]);
  if (dir == 0) {
    for (int64_t base = m + 1; base <= R; base += 32 * kRun) {
      const int64_t k0 = base + (int64_t)lane * kRun;
      const double kd = (double)k0;
      double loc[kRun], pk = kd;
#pragma unroll
      for (int b = 1; b < kRun; ++b) pk = __dmul_rn(pk, kd + (double)b);
      double inv = __drcp_rn(pk);  // 1 / (k0 .. k0 + 7)
#pragma unroll
      for (int b = kRun - 1; b >= 0; --b) {
        loc[b] = __dmul_rn(xp[b], inv);
        inv = __dmul_rn(inv, kd + (double)b);
      }
      const double incl = warp_incl_prod(loc[kRun - 1], lane);
      double excl = __shfl_up_sync(kFull, incl, 1);
      if (lane == 0) excl = 1.0;
      const double pre = __dmul_rn(carry, excl);
      // The run's sum from its far end: at k = K + 1 it holds the run's tail.
      double run = 0.0, rest = 0.0;
#pragma unroll
      for (int b = kRun - 1; b >= 0; --b) {
        const int64_t k = k0 + b;
        const double w = __dmul_rn(pre, loc[b]);
        if (k <= R) run += w;
        if (k > K) rest = run;
        else if (store && k <= R) put(k, w);
      }
      r.all += run;
      r.tail += rest;
      carry = __dmul_rn(carry, __shfl_sync(kFull, incl, 31));
    }
  } else {
    for (int64_t base = m - 1; base >= L; base -= 32 * kRun) {
      const int64_t k0 = base - (int64_t)lane * kRun;
      const double kd = (double)(k0 + 1);
      double loc[kRun], pk = 1.0, wl = 0.0;
#pragma unroll
      for (int b = 0; b < kRun; ++b) {
        // (Below L the products only feed lanes that hold no weight; below 0
        // the factors are taken as 1 so that they stay finite and positive.)
        pk = __dmul_rn(pk, k0 - b >= L ? kd - (double)b : 1.0);
        loc[b] = __dmul_rn(pk, xp[b]);
      }
      const double incl = warp_incl_prod(loc[kRun - 1], lane);
      double excl = __shfl_up_sync(kFull, incl, 1);
      if (lane == 0) excl = 1.0;
      const double pre = __dmul_rn(carry, excl);
#pragma unroll
      for (int b = 0; b < kRun; ++b) {
        const int64_t k = k0 - b;
        if (k >= L) {
          const double w = __dmul_rn(pre, loc[b]);
          r.all += w;
          if (store) put(k, w);
          if (k == L) wl = w;
        }
      }
      if (base - L < 32 * kRun) r.wL = __shfl_sync(kFull, wl, (int)((base - L) / kRun));
      carry = __dmul_rn(carry, __shfl_sync(kFull, incl, 31));
    }
  }
  r.all = warp_sum(r.all);
  if (dir == 0) r.tail = warp_sum(r.tail);
  return r;
}

// Plan one time on one warp (tolerance rule).
__device__ void plan_time(const PlanParams& p, double omega, double t, Win* dst, int lane) {
  Win r;
  double x = __dmul_rn(omega, t);
  r.x = x;
  if (x == 0.0) {  // t = 0 or no transitions: rho*(t) = rho0
    r.L = 0;
    r.K = 0;
    r.PL = 1.0;
    r.tail = 0.0;
    r.woff = -1;
    if (lane == 0) *dst = r;
    return;
  }
  int64_t K = 0, L = 0;
  if (!window_bounds(p, x, L, K)) {  // K above the cap (also inf / NaN; nothing loops)
    if (lane == 0) {
      set_status(p.status, kStatusKcap);
      *dst = capped_window(x);
    }
    return;
  }
  const double s = __dsqrt_rn(x);
  int64_t m = (int64_t)floor(x);
  int64_t R = (int64_t)floor(x + 10.0 * s) + 10;

  // Tolerance rule.  Upward from the mode: w_k = w_{k-1} x / k, w_m = 1.
  Kahan sum;
  if (lane == 0) sum.add(1.0);
  double carry = 1.0;
  for (int64_t base = m + 1; base <= R; base += 32) {
    int64_t k = base + lane;
    double term = (k <= R) ? __ddiv_rn(x, (double)k) : 1.0;
    double w = __dmul_rn(warp_incl_prod(term, lane), carry);
    carry = __shfl_sync(kFull, w, 31);
    if (k <= R) sum.add(w);
  }
  double wR = carry;
  // Downward from the mode: w_k = w_{k+1} (k+1) / x.
  double wL = (L == m) ? 1.0 : 0.0;
  carry = 1.0;
  for (int64_t base = m - 1; base >= L; base -= 32) {
    int64_t k = base - lane;
    double term = (k >= L) ? __ddiv_rn((double)(k + 1), x) : 1.0;
    double w = __dmul_rn(warp_incl_prod(term, lane), carry);
    carry = __shfl_sync(kFull, w, 31);
    if (k >= L) sum.add(w);
    if (k == L) wL = w;
  }
  double W = warp_sum(sum.s) - warp_sum(sum.c);
  // wL sits in exactly one lane (or lane-uniformly 1.0 when L == m).
  wL = (L == m) ? 1.0 : warp_sum(wL);

  double tail;
  {
    // Smallest K with sum_{j>K} w_j <= tol W: walk down from R with suffix sums.
    double thr = p.tol * W;
    double S = 0.0;   // sum_{j > base}
    double wnext = wR;  // w_{base+1} after the first chunk; starts as w_R for base = R-1
    int64_t Kt = R;
    bool found = false;
    for (int64_t base = R - 1; base >= m && !found; base -= 32) {
      int64_t k = base - lane;
      bool valid = k >= m;
      double term = valid ? __ddiv_rn((double)(k + 1), x) : 1.0;
      double w = __dmul_rn(warp_incl_prod(term, lane), wnext);  // w_k
      // S_k = sum_{j>k} w_j = S + w_{base+1} + ... + w_{k+1}; w_{base+1} = wnext.
      double incl = warp_incl_sum(valid ? w : 0.0, lane);
      double excl = incl - (valid ? w : 0.0);
      double Sk = S + wnext + excl;
      unsigned ok = __ballot_sync(kFull, valid && Sk <= thr);
      unsigned vmask = __ballot_sync(kFull, valid);
      if ((ok & vmask) != vmask) {
        int j = __ffs(~ok) - 1;  // first failing lane: passing lanes form a prefix
        Kt = base - j + 1;
        found = true;
      } else {
        Kt = base - (__popc(vmask) - 1);
      }
      S = S + wnext + __shfl_sync(kFull, incl, 31) - __shfl_sync(kFull, valid ? w : 0.0, 31);
      wnext = __shfl_sync(kFull, w, 31);
    }
    K = Kt;
    // tail = sum_{j > K} w_j / W, recomputed upward from the mode for clarity.
    Kahan ts;
    carry = 1.0;
    for (int64_t base = m + 1; base <= R; base += 32) {
      int64_t k = base + lane;
      double term = (k <= R) ? __ddiv_rn(x, (double)k) : 1.0;
      double w = __dmul_rn(warp_incl_prod(term, lane), carry);
      carry = __shfl_sync(kFull, w, 31);
      if (k <= R && k > K) ts.add(w);
    }
    tail = (warp_sum(ts.s) - warp_sum(ts.c)) / W;
  }
  r.L = L;
  r.K = K;
  r.PL = wL / W;
  r.tail = tail;
  r.woff = -1;
  // P_L..P_K (the tail folded into P_K) in the arena, so the chain reads the
  // weights instead of running the recurrence (K is known only now: the same
  // product scans run again).
  if (p.arena) {
    const int64_t size = K - L + 1;
    unsigned long long off = 0;
    if (lane == 0) off = atomicAdd(p.arena_used, (unsigned long long)size);
    off = __shfl_sync(kFull, off, 0);
    if ((int64_t)off + size <= p.arena_cap) {
      r.woff = (int64_t)off;
      auto put = [&](int64_t k, double w) {
        double v = __ddiv_rn(w, W);
        if (k == K) v = v + tail;
        if (p.arena_fp64) reinterpret_cast<double*>(p.arena)[off + (k - L)] = v;
        else reinterpret_cast<float*>(p.arena)[off + (k - L)] = (float)v;
      };
      if (lane == 0) put(m, 1.0);
      carry = 1.0;
      for (int64_t base = m + 1; base <= K; base += 32) {
        int64_t k = base + lane;
        double term = (k <= R) ? __ddiv_rn(x, (double)k) : 1.0;
        double w = __dmul_rn(warp_incl_prod(term, lane), carry);
        carry = __shfl_sync(kFull, w, 31);
        if (k <= K) put(k, w);
      }
      carry = 1.0;
      for (int64_t base = m - 1; base >= L; base -= 32) {
        int64_t k = base - lane;
        double term = (k >= L) ? __ddiv_rn((double)(k + 1), x) : 1.0;
        double w = __dmul_rn(warp_incl_prod(term, lane), carry);
        carry = __shfl_sync(kFull, w, 31);
        if (k >= L) put(k, w);
      }
    } else if (lane == 0 && p.arena_over) {
      atomicOr(p.arena_over, 1);
    }
  }
  if (lane == 0) *dst = r;
}

// Poisson(L | x) of a window at x <= 250 in FP64, L x / i after another: the start
// of the recurrence of an FP32 window without a stored copy, where w_L is too
// small for float-float (w_L < 1e-30, for x between 70 and 220; its low part
// falls below FP32's range, at x = 106 w_L itself, and every weight of the window
// was off by as much as 1e-3).
__device__ __noinline__ double poisson_start(double x, int64_t L) {
  double P = exp(-x);
  for (int64_t i = 1; i <= L; ++i) P = __dmul_rn(P, __ddiv_rn(x, (double)i));
  return P;
}

// max_n e_n over the corners of the box: the last and last but one state of
// every axis, both gene states (thread c < 8).
__device__ double corner_rate(const PlanParams& p, int64_t M, int64_t N, int c, const double* th) {
  const int64_t m = M - 1 - (c & 1);
  if (p.kind == MJP_BD1D) return c < 2 && m >= 0 ? exit_rate(p.kind, M, 1, m, th) : 0.0;
  if (p.kind == MJP_TWOSTATE) return c < 4 ? exit_rate(p.kind, M, 2, m + (c >> 1) * M, th) : 0.0;
  const int64_t rows = p.kind == MJP_AUTOREG ? p.P / 2 : p.P, q = rows - 1 - ((c >> 1) & 1);
  if (m < 0 || q < 0 || (p.kind != MJP_AUTOREG && c >= 4)) return 0.0;
  return exit_rate(p.kind, M, p.P, m + M * q + M * rows * (c >> 2), th);
}

// (80 registers at 256 threads, 3 CTAs an SM: at 116 registers and 2 CTAs, 10^4
// thetas took 614 us instead of 550.)
template <int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 512 ? 2 : 3) plan_kernel(PlanParams p) {
  const int job = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ double s_omega;
  double omega;
  if (p.omega_fixed >= 0.0) {
    omega = p.omega_fixed;
  } else {
    const double* th = p.theta + (int64_t)job * p.ntheta;
    const int64_t NJ = p.jobN ? (int64_t)p.jobN[job] : p.N;
    if (warp == 0) {
      double mx = lane < 8 ? corner_rate(p, p.jobN ? NJ : p.M, NJ, lane, th) : 0.0;
      if (!(mx > 0.0)) mx = 0.0;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(kFull, mx, o);
        mx = t > mx ? t : mx;
      }
      if (lane == 0) s_omega = mx > 0.0 ? __dmul_rn(p.omega_factor, mx) : 0.0;
    }
    __syncthreads();
    omega = s_omega;
  }
  Win* wj = p.win + (int64_t)job * p.ntimes;
  const double* tj = p.times + (p.times_per_job ? (int64_t)job * p.ntimes : 0);
  const int nt = p.ntimes;
  if (p.trunc_mode != MJP_TRUNC_PAPER) {
    for (int i = warp; i < nt; i += blockDim.x >> 5) plan_time(p, omega, tj[i], wj + i, lane);
    __syncthreads();
    if (tid == 0) {
      int64_t kmax = 0;
      for (int i = 0; i < nt; ++i) kmax = wj[i].K > kmax ? wj[i].K : kmax;
      p.info[job].omega = omega;
      p.info[job].Kmax = kmax;
    }
    return;
  }

  // ---- windows: a thread each ------------------------------------------------
  // s_kind: 0 = a window, 1 = no chain (x = 0), 2 = K above the cap.
  __shared__ double s_x[kMaxTimes], s_invx[kMaxTimes];
  __shared__ long long s_L[kMaxTimes], s_K[kMaxTimes], s_R[kMaxTimes], s_off[kMaxTimes];
  __shared__ signed char s_kind[kMaxTimes];
  // Sums of both directions, the tail and w_L, later 1 / W in s_sum[.][1]; x and
  // 1 / x in float-float (FP32 chains), later 1 / W and the tail.
  __shared__ double s_sum[kMaxTimes][2], s_tail[kMaxTimes], s_wL[kMaxTimes];
  __shared__ FF s_xf[kMaxTimes], s_invxf[kMaxTimes];
  __shared__ long long s_tot;
  static_assert(kMaxTimes <= 256, "a thread per window");
  const bool fp64 = p.fp64_weights || p.arena_fp64;
  if (tid < nt) {
    const double x = __dmul_rn(omega, tj[tid]);
    int64_t L = 0, K = 0;
    long long size = 0;
    signed char kind = x == 0.0 ? 1 : 2;
    s_x[tid] = x;
    if (window_bounds(p, x, L, K)) {
      kind = 0;
      s_R[tid] = (int64_t)floor(x + 10.0 * __dsqrt_rn(x)) + 10;
      s_invx[tid] = fp64 ? __drcp_rn(x) : 1.0 / x;
      if (!fp64) {
        s_xf[tid] = ff_from(x);
        s_invxf[tid] = ff_from(s_invx[tid]);
      }
      size = K - L + 1;
    } else if (kind == 1) {
      K = 1;
    }
    s_L[tid] = L;
    s_K[tid] = K;
    s_kind[tid] = kind;
    s_off[tid] = size;
  }
  __syncthreads();
  // The windows of all this instance's times are reserved in one piece, in time
  // order (the same layout every call, and an instance's windows either all fit
  // or all run the chain's recurrence); a single instance starts at 0.
  if (warp == 0) {
    long long tot = 0, kmax = 0;
    for (int i0 = 0; i0 < nt; i0 += 32) {
      const int i = i0 + lane;
      const long long sz = i < nt ? s_off[i] : 0;
      long long incl = sz;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (i < nt) s_off[i] = sz > 0 ? tot + incl - sz : -1;
      tot += __shfl_sync(kFull, incl, 31);
      const long long k = i < nt ? s_K[i] : 0;
      kmax = k > kmax ? k : kmax;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long t = __shfl_xor_sync(kFull, kmax, o);
      kmax = t > kmax ? t : kmax;
    }
    if (lane == 0) {
      long long base = -1;  // no place
      if (p.arena) {
        base = p.B > 1 && tot > 0 ? (long long)atomicAdd(p.arena_used, (unsigned long long)tot) : 0;
        if (base + tot > (long long)p.arena_cap) {
          base = -1;
          if (p.arena_over) atomicOr(p.arena_over, 1);
        }
      }
      s_tot = base;
      if (blockIdx.y == 0) {
        p.info[job].omega = omega;
        p.info[job].Kmax = kmax;
      }
    }
  }
  __syncthreads();
  const long long abase = s_tot;
  const bool place = abase >= 0;

  // ---- weights: a warp per window and direction --------------------------------
  const int i0 = blockIdx.y, step = gridDim.y;  // this CTA's windows: i0, i0 + step, ...
  const int nw = i0 < nt ? (nt - i0 + step - 1) / step : 0;
  for (int q = warp; q < 2 * nw; q += blockDim.x >> 5) {
    const int i = i0 + (q >> 1) * step, dir = q & 1;
    if (s_kind[i] != 0) continue;
    const double x = s_x[i];
    const int64_t L = s_L[i], K = s_K[i], m = (int64_t)floor(x), R = s_R[i];
    const long long off = abase + s_off[i] - L;
    const bool mode = dir == 0 && lane == 0 && place;  // the mode's own weight
    Sums64 r;
    if (fp64) {
      auto put = [&](int64_t k, double w) {
        if (p.arena_fp64) reinterpret_cast<double*>(p.arena)[off + k] = w;
        else reinterpret_cast<float*>(p.arena)[off + k] = (float)w;
      };
      if (mode) put(m, 1.0);
      r = dir_weights64(dir, x, s_invx[i], L, K, m, R, lane, place, put);
    } else {
      auto put = [&](int64_t k, FF w) { reinterpret_cast<float*>(p.arena)[off + k] = w.hi; };
      if (mode) put(m, FF{1.0f, 0.0f});
      r = R < (1LL << 30)
              ? dir_weights<int>(dir, s_xf[i], s_invxf[i], (int)L, (int)K, (int)m, (int)R, lane, place, put)
              : dir_weights<int64_t>(dir, s_xf[i], s_invxf[i], L, K, m, R, lane, place, put);
    }
    if (lane == 0) {
      s_sum[i][dir] = r.all;
      if (dir == 0) s_tail[i] = r.tail;
      else s_wL[i] = r.wL;
    }
  }
  __syncthreads();

  // ---- normalisation: a thread per window ---------------------------------------
  if (tid < nt && tid % step == i0) {
    Win r;
    if (s_kind[tid] == 2) {
      set_status(p.status, kStatusKcap);
      r = capped_window(s_x[tid]);
    } else {
      r.x = s_x[tid];
      r.L = s_L[tid];
      r.K = s_K[tid];
      r.PL = 1.0;
      r.tail = 0.0;
      r.woff = -1;
      if (s_kind[tid] == 0) {
        const double invW = __ddiv_rn(1.0, 1.0 + s_sum[tid][0] + s_sum[tid][1]);
        r.PL = !fp64 && !place && s_wL[tid] < 1e-30 ? poisson_start(s_x[tid], s_L[tid]) : __dmul_rn(s_wL[tid], invW);
        r.tail = __dmul_rn(s_tail[tid], invW);
        if (place) r.woff = abase + s_off[tid];
        s_tail[tid] = r.tail;
        s_sum[tid][1] = invW;
        if (!fp64) {
          s_xf[tid] = ff_from(invW);
          s_invxf[tid] = ff_from(r.tail);
        }
      }
    }
    wj[tid] = r;
  }
  __syncthreads();  // every raw weight and every factor is visible to the warps that scale them
  if (!place) return;
  for (int q = warp; q < nw; q += blockDim.x >> 5) {
    const int i = i0 + q * step;
    if (s_kind[i] != 0) continue;
    const int64_t size = s_K[i] - s_L[i] + 1;
    if (p.arena_fp64) {
      const double invW = s_sum[i][1], tail = s_tail[i];
      double* a = reinterpret_cast<double*>(p.arena) + abase + s_off[i];
      for (int64_t j = lane; j < size; j += 32) {
        double v = __dmul_rn(a[j], invW);
        if (j == size - 1) v = v + tail;
        a[j] = v;
      }
    } else {  // FP32 weights scaled in float-float on the FP32 pipe
      float* a = reinterpret_cast<float*>(p.arena) + abase + s_off[i];
      const FF invWf = s_xf[i];
      for (int64_t j = lane; j < size; j += 32) {
        FF v = ff_mul(FF{a[j], 0.0f}, invWf);
        if (j == size - 1) v = ff_add(v, s_invxf[i]);
        a[j] = __fadd_rn(v.hi, v.lo);
      }
    }
  }
}

// Longest chain first: map[r] = the job of rank r by decreasing Kmax (ties
// by index), so clusters that start in later waves carry the short chains.
// Each thread ranks one job against all others (a strict total order, so the
// map is a permutation whatever the keys hold).
__global__ void order_jobs_kernel(const JobInfo* info, int B, int32_t* map) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B; i += gridDim.x * blockDim.x) {
    const int64_t ki = info[i].Kmax;
    int r = 0;
    for (int j = 0; j < B; ++j) {
      const int64_t kj = info[j].Kmax;
      r += (kj > ki || (kj == ki && j < i)) ? 1 : 0;
    }
    map[r] = i;
  }
}

}  // namespace

cudaError_t launch_plan(const PlanParams& p, cudaStream_t s) {
  if (p.B <= 0) return cudaSuccess;
  // A single instance by the paper's rule: a CTA per window.
  const int split = p.B == 1 && p.trunc_mode == MJP_TRUNC_PAPER ? (p.ntimes < 64 ? p.ntimes : 64) : 1;
  // A warp per window and direction: above 8 windows, 8 warps take three and
  // more turns at the scans.  Measured with 8 and 16 warps: 256 thetas x 50
  // times 108 and 89 us, 152 thetas x 50 times (smaller x) 63 and 49 us; at 5 times 8 warps
  // have one or two turns, and the third CTA per SM counts for more.
  const int local = (p.ntimes + split - 1) / split;
  const dim3 grid((unsigned)p.B, (unsigned)split);
  if (local > 8) plan_kernel<512><<<grid, 512, 0, s>>>(p);
  else plan_kernel<256><<<grid, 256, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_order_jobs(const JobInfo* info, int B, int32_t* map, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  const int blocks = (B + 255) / 256 < 1024 ? (B + 255) / 256 : 1024;
  order_jobs_kernel<<<blocks, 256, 0, s>>>(info, B, map);
  return cudaGetLastError();
}

}  // namespace mjp
