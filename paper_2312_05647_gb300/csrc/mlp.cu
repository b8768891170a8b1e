// mlp.cu -- the log-likelihood surrogate of include/mjp_surrogate.h: a
// 4 -> 128 -> 128 -> 1 tanh perceptron evaluated and trained (mean squared
// error, Adam of Kingma & Ba 2015) by hand-written FP32 kernels.
//
// Work split of the forward pass: one CTA of 128 threads takes a tile of R
// rows; thread j owns hidden unit j.  W2 (64 KB) sits in shared memory with a
// padded stride, so that reading it is free of bank conflicts; the hidden
// activations of the tile are broadcast from shared memory as float4.
// Gradients have a kernel of their own (grad_kernel below), which writes one
// partial per CTA; a second kernel sums the partials in a fixed order (to
// FP64's accuracy) and applies Adam, so every result is run-to-run identical.  The
// network is tiny (17,281 parameters, 34 kflop per row forward): a step is
// latency-bound, and FP32 FMA on the CUDA cores keeps the gradients exact
// enough to check against FP64 backpropagation.
#include <atomic>
#include <cmath>
#include <cstring>
#include <vector>

#include "host_util.h"
#include "mjp_surrogate.h"
#include "mlp_dev.cuh"
#include "philox.cuh"

using namespace mjp;
using namespace mjp::mlp;

struct mjp_mlp {
  DevBuf P, m, v, norm;
  DevBuf normp;  // column sums of the standardisation (allocated with the network: fitting takes no memory)
  DevBuf partial, loss_part, psi, y, out, losses, grad, scalar;
  int64_t t = 0;
};

namespace {

__global__ void init_kernel(float* __restrict__ P, uint32_t k0, uint32_t k1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPAR) return;
  double a = 0.0;
  if (i < OB1) a = sqrt(6.0 / (D + H));
  else if (i >= OW2 && i < OB2) a = sqrt(6.0 / (H + H));
  else if (i >= OW3 && i < OB3) a = sqrt(6.0 / (H + 1));
  float v = 0.f;
  if (a > 0.0) {
    const uint4 w = philox4x32_10(make_uint4((uint32_t)i, 0u, kInitStream, 0u), k0, k1);
    v = (float)((2.0 * uniform52(w.x, w.y) - 1.0) * a);
  }
  P[i] = v;
}

// Deterministic block sum (FP64): butterfly within warps, then warp 0 over
// the warp partials in warp order.  All threads get the result.
__device__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < nw; ++w) s += red[w];
  return s;
}

// Means and population standard deviations of the 4 input columns and y.
__global__ void __launch_bounds__(256) fit_norm_kernel(const double* __restrict__ psi, const double* __restrict__ y,
                                                        int64_t n, Norm* __restrict__ out) {
  __shared__ double red[8];
  double mean[5], sd[5];
  for (int c = 0; c < 5; ++c) {
    double s = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += blockDim.x) s += c < 4 ? psi[r * 4 + c] : y[r];
    mean[c] = block_sum(s, red) / (double)n;
  }
  for (int c = 0; c < 5; ++c) {
    double s = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += blockDim.x) {
      const double d = (c < 4 ? psi[r * 4 + c] : y[r]) - mean[c];
      s += d * d;
    }
    const double v = block_sum(s, red) / (double)n;
    sd[c] = v > 0.0 ? sqrt(v) : 1.0;
  }
  if (threadIdx.x == 0) {
    Norm nm;
    for (int c = 0; c < 4; ++c) {
      nm.mux[c] = mean[c];
      nm.sdx[c] = sd[c];
    }
    nm.muy = mean[4];
    nm.sdy = sd[4];
    *out = nm;
  }
}

// The same for many rows: column sums of every CTA's share (pass 0: the
// values, pass 1: their squared deviations from the mean that pass 0's sums
// give), each in a fixed order, and a last kernel that adds them up.  One CTA
// over 65,536 rows took 342 us, most of a short training.
constexpr int kNormCtas = 128;
__device__ void norm_sums(const double* part, double inv_n, double* out) {  // [kNormCtas][5] -> 5 (threads 0 .. 4)
  if (threadIdx.x < 5) {
    double s = 0.0;
    for (int b = 0; b < kNormCtas; ++b) s += part[b * 5 + threadIdx.x];
    out[threadIdx.x] = s * inv_n;
  }
  __syncthreads();
}
__global__ void __launch_bounds__(256) norm_part_kernel(const double* __restrict__ psi, const double* __restrict__ y,
                                                        int64_t n, int pass, const double* __restrict__ sums,
                                                        double* __restrict__ part) {
  __shared__ double red[8], mean[5];
  if (pass) norm_sums(sums, 1.0 / (double)n, mean);
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t r = blockIdx.x * 256 + threadIdx.x; r < n; r += (int64_t)gridDim.x * 256) {
    const double2 a = reinterpret_cast<const double2*>(psi)[2 * r], b = reinterpret_cast<const double2*>(psi)[2 * r + 1];
    const double v[5] = {a.x, a.y, b.x, b.y, y[r]};
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const double d = pass ? v[c] - mean[c] : v[c];
      acc[c] += pass ? d * d : d;
    }
  }
  for (int c = 0; c < 5; ++c) {
    const double t = block_sum(acc[c], red);
    if (threadIdx.x == 0) part[blockIdx.x * 5 + c] = t;
  }
}
__global__ void norm_final_kernel(int64_t n, const double* __restrict__ sums, const double* __restrict__ squares,
                                  Norm* __restrict__ out) {
  __shared__ double mean[5], var[5];
  norm_sums(sums, 1.0 / (double)n, mean);
  norm_sums(squares, 1.0 / (double)n, var);
  if (threadIdx.x < 5) {
    const int c = threadIdx.x;
    const double sd = var[c] > 0.0 ? sqrt(var[c]) : 1.0;
    if (c < 4) {
      out->mux[c] = mean[c];
      out->sdx[c] = sd;
    } else {
      out->muy = mean[c];
      out->sdy = sd;
    }
  }
}

struct RowsParams {
  const float* P;
  const Norm* nm;
  const double* psi;
  const double* y;
  int64_t n;      // rows of the data set
  int64_t batch;  // rows evaluated (tile rows beyond it are padding)
  int sample;     // gradient, 1: row r is a Philox draw from the data set, else row r itself
  uint32_t k0, k1, step;
  float inv_batch;
  double* out;        // forward: s(psi) per row
  float* partial;     // gradient: [gridDim.x][NPAR] gradient partials
  double* loss_part;  // gradient: sum of squared residuals per CTA
};

template <int R>
constexpr size_t rows_smem() {
  return sizeof(float) * ((size_t)H * W2S + (size_t)R * H + R * 4 + 4 * R);
}

template <int R>
__global__ void __launch_bounds__(128) rows_kernel(const RowsParams p) {
  extern __shared__ __align__(16) float sm[];
  float* W2s = sm;
  float* h1s = W2s + H * W2S;
  float* xs = h1s + R * H;
  float* red = xs + R * 4;
  const int j = threadIdx.x, lane = j & 31, warp = j >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * R;
  const Norm nm = *p.nm;

  stage_w2(p.P, W2s);
  if (j < R) {
    const int64_t g = r0 + j;
    const bool valid = g < p.batch;
#pragma unroll
    for (int k = 0; k < 4; ++k) xs[j * 4 + k] = valid ? std_input(nm, p.psi + g * 4, k) : 0.f;
  }
  float w1[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w1[k] = p.P[OW1 + k * H + j];
  const float b1 = p.P[OB1 + j], b2 = p.P[OB2 + j], w3 = p.P[OW3 + j], b3 = p.P[OB3];
  __syncthreads();

  // Layer 1 -> h1 (shared), layer 2 -> a[r] = h2 (registers, unit j).
#pragma unroll 4
  for (int r = 0; r < R; ++r) {
    const float x[4] = {xs[r * 4], xs[r * 4 + 1], xs[r * 4 + 2], xs[r * 4 + 3]};
    h1s[r * H + j] = tanhf(layer1(x, w1, b1));
  }
  __syncthreads();
  float a[R];
#pragma unroll
  for (int r = 0; r < R; ++r) a[r] = b2;
  for (int i = 0; i < H; i += 4) {
    const float wa = W2s[i * W2S + j], wb = W2s[(i + 1) * W2S + j];
    const float wc = W2s[(i + 2) * W2S + j], wd = W2s[(i + 3) * W2S + j];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 h = *reinterpret_cast<const float4*>(h1s + r * H + i);
      a[r] = fmaf(h.x, wa, a[r]);
      a[r] = fmaf(h.y, wb, a[r]);
      a[r] = fmaf(h.z, wc, a[r]);
      a[r] = fmaf(h.w, wd, a[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    a[r] = tanhf(a[r]);
    const float v = warp_sum(a[r] * w3);
    if (lane == 0) red[warp * R + r] = v;
  }
  __syncthreads();

  if (j < R && r0 + j < p.batch) {
    const float f = b3 + red[j] + red[R + j] + red[2 * R + j] + red[3 * R + j];
    p.out[r0 + j] = nm.muy + nm.sdy * (double)f;
  }
}

// Gradient partial of a tile of R rows: 256 threads per CTA.  The operations of
// a row and of a partial and their order are those of one thread per unit
// (rows ascending, units ascending, the output sum as a butterfly over 32
// units and then over the four 32-unit parts); only who does them differs:
// W2 comes in by cp.async while the rows are drawn and standardised (a
// division per thread), its rows' 16-byte chunks exchanged by row (chunk c of
// row i at c ^ (i mod 32)), so that both reading a row across columns and a
// chunk across rows hit all banks; activations and deltas are kept
// transposed, [unit][row], so that one vector read serves a thread's rows.
// Layer 2: two units of R / 4 rows per thread.  dL/dW2: one column of 64 rows
// per thread; dL/dh1: one unit of R / 2 rows.  Bound: shared-memory reads
// (about 8,000 wavefronts per CTA at R = 16) and latency.  Measured on 1,024
// rows (64 CTAs): 22.8 -> 14.3 us against one thread per unit; 100 steps with the
// standardisation of 65,536 rows (342 -> ~15 us) and the sums below 4.19 -> 1.82
// ms.
template <int R>
struct GradSmem {
  float W2[H * H];
  float hT[H][R];   // h1
  float aT[H][R];   // h2
  float dzT[H][R];  // dL/dz2, then dL/dz1
  float x[R][4], t[R], dy[R];
  float red[4][R];  // output sums of the four 32-unit parts
};

// Rows [r0, r0 + N) of a transposed row.
template <int N>
__device__ __forceinline__ void load_rows(float (&v)[N], const float* src) {
  if constexpr (N == 2) {
    const float2 a = *reinterpret_cast<const float2*>(src);
    v[0] = a.x; v[1] = a.y;
  } else {
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
      const float4 a = reinterpret_cast<const float4*>(src)[q];
      v[4 * q] = a.x; v[4 * q + 1] = a.y; v[4 * q + 2] = a.z; v[4 * q + 3] = a.w;
    }
  }
}
template <int N>
__device__ __forceinline__ void store_rows(float* dst, const float (&v)[N]) {
  if constexpr (N == 2) {
    *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int q = 0; q < N / 4; ++q)
      reinterpret_cast<float4*>(dst)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  }
}

template <int R>
__global__ void __launch_bounds__(256) grad_kernel(const RowsParams p) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  GradSmem<R>& S = *reinterpret_cast<GradSmem<R>*>(sm_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * R;
  cudaTriggerProgrammaticLaunchCompletion();
  // Row r, component c of the data set (c = 4: the target); independent of the
  // step before, whose Adam update may still be running.
  if (tid < R * 5) {
    const int r = tid / 5, c = tid - 5 * r;
    const int64_t g = r0 + r;
    const bool valid = g < p.batch;
    int64_t src = g;
    if (valid && p.sample) {
      const uint4 w = philox4x32_10(make_uint4((uint32_t)g, p.step, kBatchStream, 0u), p.k0, p.k1);
      src = (int64_t)(((uint64_t)w.x * (uint64_t)p.n) >> 32);
    }
    const double v = valid ? (c < 4 ? p.psi[src * 4 + c] : p.y[src]) : 0.0;
    const double mu = c < 4 ? p.nm->mux[c] : p.nm->muy, sd = c < 4 ? p.nm->sdx[c] : p.nm->sdy;
    const float z = valid ? (float)((v - mu) / sd) : 0.f;
    if (c < 4) S.x[r][c] = z;
    else S.t[r] = z;
  }
  cudaGridDependencySynchronize();  // the parameters are the step before's
  for (int e = tid; e < H * H / 4; e += 256) {
    const int i = e >> 5, c = e & 31;
    const unsigned d = (unsigned)__cvta_generic_to_shared(S.W2 + i * H + 4 * (c ^ (i & 31)));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(p.P + OW2 + 4 * e) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int j = tid & (H - 1), half = tid >> 7;
  float w1[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w1[k] = p.P[OW1 + k * H + j];
  const float b1 = p.P[OB1 + j], b3 = p.P[OB3], w3 = p.P[OW3 + j];
  constexpr int RQ = R / 4, RH = R / 2;
  const int u = tid & 63, c2 = 2 * u, rg = tid >> 6;  // layer 2: units c2, c2 + 1 of rows rg RQ ..
  const float2 b2 = *reinterpret_cast<const float2*>(p.P + OB2 + c2), w3u = *reinterpret_cast<const float2*>(p.P + OW3 + c2);
  __syncthreads();
  // Layer 1, unit j of R / 2 rows.
  {
    float h[RH];
#pragma unroll
    for (int r = 0; r < RH; ++r) {
      const float4 xv = *reinterpret_cast<const float4*>(S.x[RH * half + r]);
      const float x[4] = {xv.x, xv.y, xv.z, xv.w};
      h[r] = tanhf(layer1(x, w1, b1));
    }
    store_rows(&S.hT[j][RH * half], h);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // Layer 2: a[row] = b2 + sum_i h1_i W2[i][unit], i ascending.
  float a0[RQ], a1[RQ];
#pragma unroll
  for (int r = 0; r < RQ; ++r) {
    a0[r] = b2.x;
    a1[r] = b2.y;
  }
#pragma unroll 8
  for (int i = 0; i < H; ++i) {
    const float2 w = *reinterpret_cast<const float2*>(S.W2 + i * H + 4 * ((c2 >> 2) ^ (i & 31)) + (c2 & 3));
    float h[RQ];
    load_rows(h, &S.hT[i][RQ * rg]);
#pragma unroll
    for (int r = 0; r < RQ; ++r) {
      a0[r] = fmaf(h[r], w.x, a0[r]);
      a1[r] = fmaf(h[r], w.y, a1[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < RQ; ++r) {
    a0[r] = tanhf(a0[r]);
    a1[r] = tanhf(a1[r]);
    // Butterfly over the 32 units of a part: unit bits 4 .. 1 are lane bits
    // 3 .. 0, bit 0 is in the thread.
    float v0 = a0[r] * w3u.x, v1 = a1[r] * w3u.y;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      v0 += __shfl_xor_sync(0xffffffffu, v0, o);
      v1 += __shfl_xor_sync(0xffffffffu, v1, o);
    }
    if ((u & 15) == 0) S.red[u >> 4][RQ * rg + r] = v0 + v1;
  }
  store_rows(&S.aT[c2][RQ * rg], a0);
  store_rows(&S.aT[c2 + 1][RQ * rg], a1);
  __syncthreads();
  // dL/df per row and the tile's squared residuals.
  if (warp == 0) {
    double l = 0.0;
    if (lane < R) {
      const bool valid = r0 + lane < p.batch;
      const float f = b3 + S.red[0][lane] + S.red[1][lane] + S.red[2][lane] + S.red[3][lane];
      const float res = f - S.t[lane];
      S.dy[lane] = valid ? 2.f * res * p.inv_batch : 0.f;
      l = valid ? (double)res * (double)res : 0.0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) p.loss_part[blockIdx.x] = l;
  }
  __syncthreads();
  float* out = p.partial + (size_t)blockIdx.x * NPAR;
  float dz[R];  // dL/dz2 of unit j, every row (both halves)
  {
    float a[R];
    load_rows(a, &S.aT[j][0]);
    float gw3 = 0.f, gb2 = 0.f, gb3 = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float dy = S.dy[r];
      gw3 = fmaf(dy, a[r], gw3);
      gb3 += dy;
      dz[r] = dy * w3 * (1.f - a[r] * a[r]);
      gb2 += dz[r];
    }
    if (half == 0) {
      out[OW3 + j] = gw3;
      out[OB2 + j] = gb2;
      if (j == 0) out[OB3] = gb3;
      store_rows(&S.dzT[j][0], dz);
    }
  }
  __syncthreads();
  // dL/dW2[i][j] = sum_r h1[r][i] dz2[r][j], 64 rows i per half.
#pragma unroll 2
  for (int i = 64 * half; i < 64 * half + 64; ++i) {
    float h[R];
    load_rows(h, &S.hT[i][0]);
    float g = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) g = fmaf(h[r], dz[r], g);
    out[OW2 + i * H + j] = g;
  }
  // dL/dh1[r][j] = sum_c dz2[r][c] W2[j][c] for R / 2 rows, then through tanh.
  float d[RH];
#pragma unroll
  for (int r = 0; r < RH; ++r) d[r] = 0.f;
#pragma unroll 2
  for (int c = 0; c < H; c += 4) {
    const float4 w = *reinterpret_cast<const float4*>(S.W2 + j * H + 4 * ((c >> 2) ^ (j & 31)));
    const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float z[RH];
      load_rows(z, &S.dzT[c + q][RH * half]);
#pragma unroll
      for (int r = 0; r < RH; ++r) d[r] = fmaf(z[r], wv[q], d[r]);
    }
  }
  {
    float h[RH];
    load_rows(h, &S.hT[j][RH * half]);
#pragma unroll
    for (int r = 0; r < RH; ++r) d[r] = d[r] * (1.f - h[r] * h[r]);
  }
  __syncthreads();  // everyone is done with dL/dz2
  store_rows(&S.dzT[j][RH * half], d);
  __syncthreads();
  if (half == 0) {
    float z[R], gb1 = 0.f, gw1[4] = {0.f, 0.f, 0.f, 0.f};
    load_rows(z, &S.dzT[j][0]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      gb1 += z[r];
#pragma unroll
      for (int k = 0; k < 4; ++k) gw1[k] = fmaf(S.x[r][k], z[r], gw1[k]);
    }
    out[OB1 + j] = gb1;
#pragma unroll
    for (int k = 0; k < 4; ++k) out[OW1 + k * H + j] = gw1[k];
  }
}

struct AdamParams {
  const float* partial;
  int nblk;
  const double* loss_part;
  double inv_batch;
  float* P;
  float* m;
  float* v;
  float lr, b1, b2, eps, bc1, bc2;
  int apply;      // 1: Adam update, 0: write the gradient only
  float* grad;    // may be null when apply
  double* loss;   // may be null
};

// Gradient = sum of the CTA partials in a fixed order, then Adam.  Four threads
// share a parameter's partials (a quarter each), then the quarters are added in
// order.  Sums are kept as three FP32 numbers (a cascade of Knuth's TwoSum, which
// is error-free: Ogita, Rump and Oishi's SumK with K = 3), ~72 bits, and rounded
// once to FP64 and once to FP32, so they are no further from the exact sum than
// one in FP64.  FP64 additions hold a pipe that is 64 times slower: 100 steps of
// 1,024 rows took 2.17 ms with them, 1.71 ms this way (1.66 ms in two FP32
// numbers).  TwoSum makes an infinity a NaN, so a sum that is not finite is
// formed again in FP64.  The last CTA sums the losses.  The next step's gradient
// may start only when the partials of this one are complete: started while they
// were still being formed, its CTAs shared SMs with them or with each other
// (100 steps of 2,048 rows 2.84 instead of 1.83 ms).
constexpr int kAdamParts = 4, kAdamParams = 64;  // threads per parameter, parameters per CTA
struct Sum3 {
  float hi, mid, lo;
};
// a + b = s + e exactly.
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}
__device__ __forceinline__ void add_to(Sum3& a, float b) {
  float e, f;
  a.hi = two_sum(a.hi, b, e);
  a.mid = two_sum(a.mid, e, f);
  a.lo = __fadd_rn(a.lo, f);
}
__global__ void __launch_bounds__(kAdamParts * kAdamParams) reduce_adam_kernel(const AdamParams q) {
  __shared__ Sum3 part[kAdamParts - 1][kAdamParams];  // of all quarters but the first
  __shared__ double red[8];
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if (blockIdx.x == gridDim.x - 1) {
    if (!q.loss) return;
    double l = 0.0;
    for (int b = threadIdx.x; b < q.nblk; b += blockDim.x) l += q.loss_part[b];
    l = block_sum(l, red);
    if (threadIdx.x == 0) *q.loss = l * q.inv_batch;
    return;
  }
  const int k = threadIdx.x & (kAdamParams - 1), w = threadIdx.x / kAdamParams;
  const int p = blockIdx.x * kAdamParams + k;
  const int per = (q.nblk + kAdamParts - 1) / kAdamParts;
  Sum3 g{0.f, 0.f, 0.f};
  if (p < NPAR) {
    const int b1 = min(q.nblk, (w + 1) * per);
    int b = w * per;
    for (; b + 8 <= b1; b += 8) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = q.partial[(size_t)(b + u) * NPAR + p];
#pragma unroll
      for (int u = 0; u < 8; ++u) add_to(g, v[u]);
    }
    for (; b < b1; ++b) add_to(g, q.partial[(size_t)b * NPAR + p]);
  }
  if (w > 0) part[w - 1][k] = g;
  __syncthreads();
  if (w == 0 && p < NPAR) {
#pragma unroll
    for (int u = 0; u < kAdamParts - 1; ++u) {
      add_to(g, part[u][k].hi);
      add_to(g, part[u][k].mid);
      add_to(g, part[u][k].lo);
    }
    float gf = (float)((double)g.hi + ((double)g.mid + (double)g.lo));
    if (!isfinite(gf)) {
      double d = 0.0;
      for (int b = 0; b < q.nblk; ++b) d += (double)q.partial[(size_t)b * NPAR + p];
      gf = (float)d;
    }
    if (q.grad) q.grad[p] = gf;
    if (q.apply) {
      const float m = q.b1 * q.m[p] + (1.f - q.b1) * gf;
      const float v = q.b2 * q.v[p] + (1.f - q.b2) * gf * gf;
      q.m[p] = m;
      q.v[p] = v;
      q.P[p] -= q.lr * (m / q.bc1) / (sqrtf(v / q.bc2) + q.eps);
    }
  }
}

// Launch of a kernel that may begin while the kernel before it in the stream
// ends (overlap): the kernel itself waits (cudaGridDependencySynchronize)
// before it reads what that one wrote.  Only behind this file's own kernels: a
// gradient reads its rows before the wait, which may be the work of a
// caller's kernel at the first step.
template <typename K, typename P>
cudaError_t launch_after(bool overlap, K kern, int grid, int block, size_t smem, const P& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

cudaError_t launch_adam(const AdamParams& q, cudaStream_t s) {
  return launch_after(true, reduce_adam_kernel, (NPAR + kAdamParams - 1) / kAdamParams + 1, kAdamParts * kAdamParams, 0, q, s);
}

template <int R>
cudaError_t launch_rows(const RowsParams& p, int64_t rows, cudaStream_t s) {
  const size_t smem = rows_smem<R>();
  cudaError_t e = cudaFuncSetAttribute(rows_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  rows_kernel<R><<<(unsigned)((rows + R - 1) / R), 128, smem, s>>>(p);
  return cudaGetLastError();
}

int rows_per_cta(int64_t rows) { return rows <= 512 ? 8 : (rows <= 4096 ? 16 : 32); }

// Up to half as many tiles as SMs ask for more than half of an SM's shared
// memory, so that each has an SM to itself (100 steps of 512 rows, 64 tiles:
// 1.65 -> 1.48 ms; of 1,536 rows, 96 tiles, 1.75 -> 1.83 ms).
template <int R>
cudaError_t launch_grad_rows(const RowsParams& p, int64_t rows, bool overlap, cudaStream_t s) {
  constexpr size_t kAlone = 118 * 1024;
  static_assert(sizeof(GradSmem<R>) <= kAlone, "a tile fits the larger request");
  static std::atomic<uint64_t> done{0};
  const cudaError_t e = once_per_device(done, [] {
    return cudaFuncSetAttribute(grad_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAlone);
  });
  if (e != cudaSuccess) return e;
  const int64_t tiles = (rows + R - 1) / R;
  return launch_after(overlap, grad_kernel<R>, (int)tiles, 256, tiles <= 152 / 2 ? kAlone : sizeof(GradSmem<R>), p, s);
}

cudaError_t launch_grad(const RowsParams& p, int64_t rows, bool overlap, cudaStream_t s) {
  switch (rows_per_cta(rows)) {
    case 8: return launch_grad_rows<8>(p, rows, overlap, s);
    case 16: return launch_grad_rows<16>(p, rows, overlap, s);
    default: return launch_grad_rows<32>(p, rows, overlap, s);
  }
}

// One CTA up to 4,096 rows (or rows that are not aligned to 16 bytes), else
// 128 CTAs in two passes and a last kernel.
int launch_fit_norm(mjp_mlp* net, const double* psi, const double* y, int64_t n, cudaStream_t s) {
  if (n <= 4096 || reinterpret_cast<uintptr_t>(psi) % 16 != 0) {
    fit_norm_kernel<<<1, 256, 0, s>>>(psi, y, n, net->norm.as<Norm>());
    MJP_CUDA(cudaGetLastError());
    return MJP_OK;
  }
  double* sums = net->normp.as<double>();
  double* squares = sums + 5 * kNormCtas;
  norm_part_kernel<<<kNormCtas, 256, 0, s>>>(psi, y, n, 0, nullptr, sums);
  norm_part_kernel<<<kNormCtas, 256, 0, s>>>(psi, y, n, 1, sums, squares);
  norm_final_kernel<<<1, 32, 0, s>>>(n, sums, squares, net->norm.as<Norm>());
  MJP_CUDA(cudaGetLastError());
  return MJP_OK;
}

bool all_finite(const float* v, int64_t n) {
  for (int64_t i = 0; i < n; ++i)
    if (!std::isfinite(v[i])) return false;
  return true;
}

int check_where(int where) {
  if (where != MJP_PTR_HOST && where != MJP_PTR_DEVICE)
    return fail(MJP_ERR_ARG, "where must be MJP_PTR_HOST or MJP_PTR_DEVICE");
  return MJP_OK;
}

// Device copies of the data set (host inputs are uploaded into net scratch).
int stage_data(mjp_mlp* net, const double* psi, const double* y, int64_t n, int where, cudaStream_t s,
               const double** dpsi, const double** dy) {
  *dpsi = psi;
  *dy = y;
  if (where == MJP_PTR_DEVICE) return MJP_OK;
  int rc;
  if ((rc = net->psi.ensure(sizeof(double) * 4 * (size_t)n))) return rc;
  MJP_CUDA(cudaMemcpyAsync(net->psi.p, psi, sizeof(double) * 4 * (size_t)n, cudaMemcpyHostToDevice, s));
  *dpsi = net->psi.as<double>();
  if (y) {
    if ((rc = net->y.ensure(sizeof(double) * (size_t)n))) return rc;
    MJP_CUDA(cudaMemcpyAsync(net->y.p, y, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice, s));
    *dy = net->y.as<double>();
  }
  return MJP_OK;
}

}  // namespace

// Used by the sampler: device parameter vector and standardisation.
namespace mjp {
const float* mlp_params(const mjp_mlp* net) { return net->P.as<float>(); }
const void* mlp_norm(const mjp_mlp* net) { return net->norm.p; }
}  // namespace mjp

extern "C" {

int mjp_mlp_create(mjp_mlp** out, uint64_t seed) try {
  if (!out) return fail(MJP_ERR_ARG, "NULL out");
  *out = nullptr;
  mjp_mlp* net = new mjp_mlp();
  int rc;
  if ((rc = net->P.ensure(sizeof(float) * NPAR)) || (rc = net->m.ensure(sizeof(float) * NPAR)) ||
      (rc = net->v.ensure(sizeof(float) * NPAR)) || (rc = net->norm.ensure(sizeof(Norm))) ||
      (rc = net->normp.ensure(sizeof(double) * 2 * 5 * kNormCtas))) {
    mjp_mlp_destroy(net);
    return rc;
  }
  init_kernel<<<(NPAR + 255) / 256, 256>>>(net->P.as<float>(), (uint32_t)seed, (uint32_t)(seed >> 32));
  Norm id;
  for (int k = 0; k < 4; ++k) {
    id.mux[k] = 0.0;
    id.sdx[k] = 1.0;
  }
  id.muy = 0.0;
  id.sdy = 1.0;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemset(net->m.p, 0, sizeof(float) * NPAR);
  if (e == cudaSuccess) e = cudaMemset(net->v.p, 0, sizeof(float) * NPAR);
  if (e == cudaSuccess) e = cudaMemcpy(net->norm.p, &id, sizeof(Norm), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    cudaGetLastError();
    mjp_mlp_destroy(net);
    return fail(MJP_ERR_CUDA, std::string("mjp_mlp_create: ") + cudaGetErrorString(e));
  }
  *out = net;
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

void mjp_mlp_destroy(mjp_mlp* net) {
  if (!net) return;
  cudaDeviceSynchronize();
  for (DevBuf* b : {&net->P, &net->m, &net->v, &net->norm, &net->normp, &net->partial, &net->loss_part, &net->psi, &net->y,
                    &net->out, &net->losses, &net->grad, &net->scalar})
    b->release();
  delete net;
}

int mjp_mlp_set_params(mjp_mlp* net, const float* params, const double* norm, int where, void* stream) try {
  if (!net) return fail(MJP_ERR_ARG, "NULL network");
  int rc = check_where(where);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<float> hp;
  Norm nm;
  if (params) {
    hp.resize(NPAR);
    MJP_CUDA(cudaMemcpyAsync(hp.data(), params, sizeof(float) * NPAR,
                             where == MJP_PTR_HOST ? cudaMemcpyHostToHost : cudaMemcpyDeviceToHost, s));
  }
  if (norm)
    MJP_CUDA(cudaMemcpyAsync(&nm, norm, sizeof(Norm),
                             where == MJP_PTR_HOST ? cudaMemcpyHostToHost : cudaMemcpyDeviceToHost, s));
  MJP_CUDA(cudaStreamSynchronize(s));
  if (params && !all_finite(hp.data(), NPAR)) return fail(MJP_ERR_ARG, "parameters must be finite");
  if (norm) {
    const double* v = reinterpret_cast<const double*>(&nm);
    for (int i = 0; i < MJP_MLP_NNORM; ++i)
      if (!std::isfinite(v[i])) return fail(MJP_ERR_ARG, "standardisation must be finite");
    for (int k = 0; k < 4; ++k)
      if (!(nm.sdx[k] > 0.0)) return fail(MJP_ERR_ARG, "input deviations must be > 0");
    if (!(nm.sdy > 0.0)) return fail(MJP_ERR_ARG, "output deviation must be > 0");
  }
  if (params) MJP_CUDA(cudaMemcpyAsync(net->P.p, hp.data(), sizeof(float) * NPAR, cudaMemcpyHostToDevice, s));
  if (norm) MJP_CUDA(cudaMemcpyAsync(net->norm.p, &nm, sizeof(Norm), cudaMemcpyHostToDevice, s));
  MJP_CUDA(cudaMemsetAsync(net->m.p, 0, sizeof(float) * NPAR, s));
  MJP_CUDA(cudaMemsetAsync(net->v.p, 0, sizeof(float) * NPAR, s));
  net->t = 0;
  MJP_CUDA(cudaStreamSynchronize(s));
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

int mjp_mlp_get_params(mjp_mlp* net, float* params, double* norm, int where, void* stream) try {
  if (!net) return fail(MJP_ERR_ARG, "NULL network");
  int rc = check_where(where);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const cudaMemcpyKind k = where == MJP_PTR_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  if (params) MJP_CUDA(cudaMemcpyAsync(params, net->P.p, sizeof(float) * NPAR, k, s));
  if (norm) MJP_CUDA(cudaMemcpyAsync(norm, net->norm.p, sizeof(Norm), k, s));
  if (where == MJP_PTR_HOST) MJP_CUDA(cudaStreamSynchronize(s));
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

int mjp_mlp_fit_norm(mjp_mlp* net, const double* psi, const double* y, int64_t n, int where, void* stream) try {
  if (!net || !psi || !y) return fail(MJP_ERR_ARG, "NULL argument");
  if (n < 1) return fail(MJP_ERR_ARG, "n must be >= 1");
  int rc = check_where(where);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const double *dpsi, *dy;
  if ((rc = stage_data(net, psi, y, n, where, s, &dpsi, &dy))) return rc;
  if ((rc = launch_fit_norm(net, dpsi, dy, n, s))) return rc;
  if (where == MJP_PTR_HOST) MJP_CUDA(cudaStreamSynchronize(s));
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

int mjp_mlp_forward(mjp_mlp* net, const double* psi, int64_t n, double* out, int where, void* stream) try {
  if (!net || !psi || !out) return fail(MJP_ERR_ARG, "NULL argument");
  if (n < 1) return fail(MJP_ERR_ARG, "n must be >= 1");
  int rc = check_where(where);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const double *dpsi, *dy;
  if ((rc = stage_data(net, psi, nullptr, n, where, s, &dpsi, &dy))) return rc;
  double* dout = out;
  if (where == MJP_PTR_HOST) {
    if ((rc = net->out.ensure(sizeof(double) * (size_t)n))) return rc;
    dout = net->out.as<double>();
  }
  RowsParams p = {};
  p.P = net->P.as<float>();
  p.nm = net->norm.as<Norm>();
  p.psi = dpsi;
  p.n = n;
  p.batch = n;
  p.out = dout;
  MJP_CUDA(launch_rows<32>(p, n, s));
  if (where == MJP_PTR_HOST) {
    MJP_CUDA(cudaMemcpyAsync(out, dout, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost, s));
    MJP_CUDA(cudaStreamSynchronize(s));
  }
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

int mjp_mlp_loss_grad(mjp_mlp* net, const double* psi, const double* y, int64_t n, double* loss, float* grad,
                      int where, void* stream) try {
  if (!net || !psi || !y) return fail(MJP_ERR_ARG, "NULL argument");
  if (n < 1 || n > 0xFFFFFFFFLL) return fail(MJP_ERR_ARG, "n must be in [1, 2^32)");
  int rc = check_where(where);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const double *dpsi, *dy;
  if ((rc = stage_data(net, psi, y, n, where, s, &dpsi, &dy))) return rc;
  const int R = rows_per_cta(n);
  const int nblk = (int)((n + R - 1) / R);
  if ((rc = net->partial.ensure(sizeof(float) * NPAR * (size_t)nblk))) return rc;
  if ((rc = net->loss_part.ensure(sizeof(double) * (size_t)nblk))) return rc;
  if ((rc = net->grad.ensure(sizeof(float) * NPAR))) return rc;
  if ((rc = net->scalar.ensure(sizeof(double)))) return rc;
  RowsParams p = {};
  p.P = net->P.as<float>();
  p.nm = net->norm.as<Norm>();
  p.psi = dpsi;
  p.y = dy;
  p.n = n;
  p.batch = n;
  p.inv_batch = (float)(1.0 / (double)n);
  p.partial = net->partial.as<float>();
  p.loss_part = net->loss_part.as<double>();
  MJP_CUDA(launch_grad(p, n, false, s));
  AdamParams q = {};
  q.partial = p.partial;
  q.nblk = nblk;
  q.loss_part = p.loss_part;
  q.inv_batch = 1.0 / (double)n;
  q.apply = 0;
  q.grad = (grad && where == MJP_PTR_DEVICE) ? grad : net->grad.as<float>();
  q.loss = (loss && where == MJP_PTR_DEVICE) ? loss : net->scalar.as<double>();
  MJP_CUDA(launch_adam(q, s));
  if (where == MJP_PTR_HOST) {
    if (grad) MJP_CUDA(cudaMemcpyAsync(grad, q.grad, sizeof(float) * NPAR, cudaMemcpyDeviceToHost, s));
    if (loss) MJP_CUDA(cudaMemcpyAsync(loss, q.loss, sizeof(double), cudaMemcpyDeviceToHost, s));
    MJP_CUDA(cudaStreamSynchronize(s));
  }
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

int mjp_mlp_train(mjp_mlp* net, const double* psi, const double* y, int64_t n, const mjp_train_cfg* cfg,
                  double* losses, int where, void* stream) try {
  if (!net || !psi || !y || !cfg) return fail(MJP_ERR_ARG, "NULL argument");
  if (n < 1 || n > 0xFFFFFFFFLL) return fail(MJP_ERR_ARG, "n must be in [1, 2^32)");
  if (cfg->steps < 1 || cfg->steps > 0xFFFFFFFFLL) return fail(MJP_ERR_ARG, "steps must be in [1, 2^32)");
  if (cfg->batch < 1) return fail(MJP_ERR_ARG, "batch must be >= 1");
  if (!(cfg->lr > 0.0) || !std::isfinite(cfg->lr)) return fail(MJP_ERR_ARG, "lr must be > 0");
  if (!(cfg->beta1 >= 0.0 && cfg->beta1 < 1.0) || !(cfg->beta2 >= 0.0 && cfg->beta2 < 1.0))
    return fail(MJP_ERR_ARG, "beta1 and beta2 must be in [0, 1)");
  if (!(cfg->eps > 0.0) || !std::isfinite(cfg->eps)) return fail(MJP_ERR_ARG, "eps must be > 0");
  int rc = check_where(where);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const double *dpsi, *dy;
  if ((rc = stage_data(net, psi, y, n, where, s, &dpsi, &dy))) return rc;
  if (cfg->fit_norm && (rc = launch_fit_norm(net, dpsi, dy, n, s))) return rc;
  const int64_t rows = cfg->batch < n ? cfg->batch : n;
  const int R = rows_per_cta(rows);
  const int nblk = (int)((rows + R - 1) / R);
  if ((rc = net->partial.ensure(sizeof(float) * NPAR * (size_t)nblk))) return rc;
  if ((rc = net->loss_part.ensure(sizeof(double) * (size_t)nblk))) return rc;
  double* dl = losses;
  if (losses && where == MJP_PTR_HOST) {
    if ((rc = net->losses.ensure(sizeof(double) * (size_t)cfg->steps))) return rc;
    dl = net->losses.as<double>();
  }
  RowsParams p = {};
  p.P = net->P.as<float>();
  p.nm = net->norm.as<Norm>();
  p.psi = dpsi;
  p.y = dy;
  p.n = n;
  p.batch = rows;
  p.sample = cfg->batch < n;
  p.k0 = (uint32_t)cfg->seed;
  p.k1 = (uint32_t)(cfg->seed >> 32);
  p.inv_batch = (float)(1.0 / (double)rows);
  p.partial = net->partial.as<float>();
  p.loss_part = net->loss_part.as<double>();
  AdamParams q = {};
  q.partial = p.partial;
  q.nblk = nblk;
  q.loss_part = p.loss_part;
  q.inv_batch = 1.0 / (double)rows;
  q.P = net->P.as<float>();
  q.m = net->m.as<float>();
  q.v = net->v.as<float>();
  q.lr = (float)cfg->lr;
  q.b1 = (float)cfg->beta1;
  q.b2 = (float)cfg->beta2;
  q.eps = (float)cfg->eps;
  q.apply = 1;
  for (int64_t st = 0; st < cfg->steps; ++st) {
    p.step = (uint32_t)st;
    MJP_CUDA(launch_grad(p, rows, st > 0, s));
    const int64_t t = ++net->t;
    q.bc1 = (float)(1.0 - std::pow(cfg->beta1, (double)t));
    q.bc2 = (float)(1.0 - std::pow(cfg->beta2, (double)t));
    q.loss = dl ? dl + st : nullptr;
    MJP_CUDA(launch_adam(q, s));
  }
  if (where == MJP_PTR_HOST) {
    if (losses)
      MJP_CUDA(cudaMemcpyAsync(losses, dl, sizeof(double) * (size_t)cfg->steps, cudaMemcpyDeviceToHost, s));
    MJP_CUDA(cudaStreamSynchronize(s));
  }
  return MJP_OK;
} catch (...) {
  return ::mjp::exception_status();
}

}  // extern "C"
