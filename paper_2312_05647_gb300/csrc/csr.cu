// csr.cu -- the jump chain for a general sparse rate matrix.
//
// Storage (built once per model on the host, see api.cu): the uniformised
// matrix B = I + A/Omega (Eq. B_def) is kept as its transpose -- for every
// target state n the incoming transitions m -> n with weights lambda_mn /
// Omega -- in SELL-32 form: states are renumbered by decreasing in-degree,
// cut into slices of 32 consecutive states, and each slice stores its entries
// column-major (entry j of the slice's 32 states side by side), padded to the
// slice's largest in-degree.  A warp owns a slice; lane i owns state 32s+i,
// so every index and value load is one coalesced 128/256-byte transaction and
// the sorting keeps padding negligible.  The diagonal 1 - e_n/Omega is a
// separate array.  rho (4 MB for 2^20 FP32 states) stays resident in L2;
// neighbour values are gathered with ordinary loads (in the one-launch chain other
// CTAs of the same launch write them, which read-only loads do not allow).
//
// Default: one launch per jump (rho_k = rho_{k-1} B, Algorithm 2's loop body;
// rho_{k+1} depends on all of rho_k, so jumps are separated grid-wide).  Each
// launch may begin while the one before it ends (programmatic dependent
// launch): indices, rates and the diagonal, which do not depend on it, are
// loaded first, so that only the gathers and the multiply-adds follow the wait.
// The last 8 (kCsrBlock) jumps stay in a ring of vectors, and one launch per 8
// jumps adds their terms P_k rho_k to the active times' outputs (FP32: a Kahan
// step per jump), instead of every jump reading and writing every active
// output.
//
// Where only two vectors are held (api.cu: no memory for nine, or a ring that does
// not pay), the launch of a jump adds the vector it reads to the active outputs.
//
// Alternative (MJP_OPT_CHAIN = 2): the whole chain in one cooperative launch
// (all CTAs co-resident), the outputs accumulated at every jump, jumps
// separated by a software grid barrier whose waits are bounded (a CTA that
// polls longer than the limit records kStatusTimeout and leaves, and so do
// the others at their next barrier).  The arithmetic is the same.  The
// Poisson weights of every (time, jump) are the planner's, in FP64.
//
// Bound: one 4-byte gather per lane costs the L1 a tag look-up of its own, one
// a cycle and SM (measured peak 320 G/s), for large matrices; for small ones
// the latency of a launch and of a gather.
#include <algorithm>

#include "internal.cuh"

namespace mjp {

namespace {

__device__ __forceinline__ float fma_t(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_t(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_t(double a, double b) { return __dmul_rn(a, b); }

template <typename T>
__global__ void permute_in_kernel(const T* __restrict__ src, const int32_t* __restrict__ perm, T* __restrict__ dst,
                                  int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    dst[perm[i]] = src[i];
}

template <typename T>
__global__ void permute_out_kernel(const T* __restrict__ src, const int32_t* __restrict__ perm, T* __restrict__ dst,
                                   int64_t n, int ntimes, const int32_t* __restrict__ orig) {
  // dst[orig[i]][s] = src[i][perm[s]]  (row-major ntimes x n)
  const int64_t total = n * ntimes;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = e / n, s = e - i * n;
    dst[(int64_t)orig[i] * n + s] = src[i * n + perm[s]];
  }
}

template <typename T>
__device__ __forceinline__ void csr_jump_body(const CsrJumpParams& p) {
  const int lane = threadIdx.x & 31;
  const int64_t gwarp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const T* cur = reinterpret_cast<const T*>(p.rho_prev);  // (no read-only loads: see above)
  T* nxt = reinterpret_cast<T*>(p.rho_next);
  const T* __restrict__ val = reinterpret_cast<const T*>(p.val);
  const T* __restrict__ diag = reinterpret_cast<const T*>(p.diag);
  T* __restrict__ out = reinterpret_cast<T*>(p.out);
  const int64_t kp = p.k - 1;  // jump whose values are accumulated now
  for (int64_t s = gwarp; s < p.nslices; s += nwarps) {
    const int64_t r = s * 32 + lane;
    const bool valid = r < p.n;
    const T v = valid ? cur[r] : (T)0;
    // rho*_i += P_{k-1} rho_{k-1} for the times whose window holds k-1.
    if (valid) {
      for (int i = p.tlo; i <= p.thi; ++i) {
        const T w = (T)p.wtab[p.woff[i] + (kp - p.L[i])];
        T* o = out + (int64_t)i * p.n + r;
        if (sizeof(T) == 4) {
          float* c = p.comp + (int64_t)i * p.n + r;
          float acc, cc;
          if (kp == p.L[i]) {
            acc = __fmul_rn((float)w, (float)v);
            cc = 0.0f;
          } else {
            acc = (float)*o;
            cc = *c;
            float y = __fsub_rn(__fmul_rn((float)w, (float)v), cc);
            float t = __fadd_rn(acc, y);
            cc = __fsub_rn(__fsub_rn(t, acc), y);
            acc = t;
          }
          if (kp == p.K[i]) *o = (T)__fsub_rn(acc, cc);
          else {
            *o = (T)acc;
            *c = cc;
          }
        } else {
          *o = (kp == p.L[i]) ? mul_t(w, v) : fma_t(w, v, *o);
        }
      }
    }
    if (p.jump && valid) {
      T y = mul_t(diag[r], v);
      const int64_t base = p.slice_ptr[s] + lane;
      const int width = p.slice_len[s];
      // Entries four at a time: the index and value loads of the group, then
      // its four gathers, so each lane has several independent loads in flight
      // (the same multiply-adds in the same order as one at a time).
      int j = 0;
      for (; j + 4 <= width; j += 4) {
        const int64_t e = base + (int64_t)j * 32;
        const int32_t c0 = __ldg(p.col + e), c1 = __ldg(p.col + e + 32), c2 = __ldg(p.col + e + 64),
                      c3 = __ldg(p.col + e + 96);
        const T a0 = __ldg(val + e), a1 = __ldg(val + e + 32), a2 = __ldg(val + e + 64), a3 = __ldg(val + e + 96);
        const T g0 = cur[c0], g1 = cur[c1], g2 = cur[c2], g3 = cur[c3];
        y = fma_t(a0, g0, y);
        y = fma_t(a1, g1, y);
        y = fma_t(a2, g2, y);
        y = fma_t(a3, g3, y);
      }
      for (; j < width; ++j) {
        const int64_t e = base + (int64_t)j * 32;
        const int32_t c = __ldg(p.col + e);
        y = fma_t(__ldg(val + e), cur[c], y);
      }
      nxt[r] = y;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(512) csr_jump_kernel(CsrJumpParams p) {
  csr_jump_body<T>(p);
}

// One jump, a thread per state: its first kCsrPre entries are in registers
// before the wait, and the next ones are loaded while the last ones' gathers
// are on their way.  The multiply-adds run in entry order, as in csr_jump_body.
constexpr int kCsrPre = 8;
template <typename T>
__global__ void __launch_bounds__(256) csr_step_kernel(const CsrStepParams p) {
  const int64_t r = blockIdx.x * (int64_t)256 + threadIdx.x;
  const bool valid = r < p.n;
  const int64_t s = valid ? r >> 5 : 0;
  const int64_t base = p.slice_ptr[s] + (threadIdx.x & 31);
  const int width = valid ? p.slice_len[s] : 0;
  const int32_t* col = p.col + base;
  const T* val = reinterpret_cast<const T*>(p.val) + base;
  const T dg = valid ? reinterpret_cast<const T*>(p.diag)[r] : (T)0;
  const T* rho = reinterpret_cast<const T*>(p.rho_prev);  // (written by the launch before: no read-only loads)
  int32_t c[kCsrPre];
  T a[kCsrPre];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int u = 0; u < kCsrPre; ++u)
      if (j0 + u < width) {
        c[u] = __ldcs(col + (int64_t)(j0 + u) * 32);
        a[u] = __ldcs(val + (int64_t)(j0 + u) * 32);
      }
  };
  fetch(0);
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if (!valid) return;
  T y = mul_t(dg, rho[r]);
  for (int j0 = 0; j0 < width; j0 += kCsrPre) {
    T g[kCsrPre], w[kCsrPre];
#pragma unroll
    for (int u = 0; u < kCsrPre; ++u)
      if (j0 + u < width) {
        g[u] = rho[c[u]];
        w[u] = a[u];
      }
    if (j0 + kCsrPre < width) fetch(j0 + kCsrPre);
#pragma unroll
    for (int u = 0; u < kCsrPre; ++u)
      if (j0 + u < width) y = fma_t(w[u], g[u], y);
  }
  reinterpret_cast<T*>(p.rho_next)[r] = y;
}

// out_i += P_k rho_k for k = k0 .. k0 + count - 1 (count <= kCsrBlock) inside
// the window of time i, for the times [tlo, thi], whose windows meet the block.
template <typename T>
__global__ void __launch_bounds__(256) csr_sum_kernel(const CsrSumParams p) {
  __shared__ double ws[kCsrBlock];
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int64_t r = blockIdx.x * (int64_t)256 + threadIdx.x;
  const bool valid = r < p.n;
  const T* ring = reinterpret_cast<const T*>(p.ring);
  T h[kCsrBlock];
#pragma unroll
  for (int j = 0; j < kCsrBlock; ++j)
    h[j] = valid && j < p.count ? ring[(size_t)((p.k0 + j) % p.nring) * p.n + r] : (T)0;
  for (int i = p.tlo; i <= p.thi; ++i) {
    const int64_t L = p.L[i], K = p.K[i];
    __syncthreads();
    if (threadIdx.x < kCsrBlock) {
      const int64_t k = p.k0 + threadIdx.x;
      ws[threadIdx.x] = (int)threadIdx.x < p.count && k >= L && k <= K ? p.wtab[p.woff[i] + (k - L)] : 0.0;
    }
    __syncthreads();
    if (!valid) continue;
    T* o = reinterpret_cast<T*>(p.out) + (size_t)i * p.n + r;
    const bool first = L >= p.k0, last = K < p.k0 + p.count;
    // The steps of csr_jump_body, a block of them on registers.
    const int j0 = first ? (int)(L - p.k0) : 0, j1 = last ? (int)(K - p.k0) : p.count - 1;
    T sum = first ? (T)0 : *o;
    if constexpr (sizeof(T) == 4) {
      float* cp = p.comp + (size_t)i * p.n + r;
      float c = first ? 0.0f : *cp;
#pragma unroll
      for (int j = 0; j < kCsrBlock; ++j) {
        if (j < j0 || j > j1) continue;
        const float y = __fsub_rn(__fmul_rn((float)ws[j], h[j]), c), t = __fadd_rn(sum, y);
        c = __fsub_rn(__fsub_rn(t, sum), y);
        sum = t;
      }
      *o = last ? __fsub_rn(sum, c) : sum;
      if (!last) *cp = c;
    } else {
#pragma unroll
      for (int j = 0; j < kCsrBlock; ++j)
        if (j >= j0 && j <= j1) sum = fma_t(ws[j], h[j], sum);
      *o = sum;
    }
  }
}

// Grid-wide barrier with a bounded wait.  bar[0] counts arrivals, bar[1] is
// the generation: the last CTA to arrive resets the count and advances the
// generation; the others poll the generation they read before arriving, at
// most `limit` times.  Returns false (and records kStatusTimeout) when the
// wait ran out; every CTA then leaves the chain, the late ones at the latest
// at their next barrier, which can no longer complete.
__device__ bool grid_barrier(unsigned* bar, long long limit, int* status) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u) + 1u;
    int good = 1;
    if (arrived == gridDim.x) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      long long it = 0;
      while (*gen == g) {
        if (it++ >= limit) {
          good = 0;
          break;
        }
        __nanosleep(20);
      }
    }
    __threadfence();
    if (!good) atomicCAS(status, 0, kStatusTimeout);
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

template <typename T>
__global__ void __launch_bounds__(1024) csr_chain_kernel(CsrChainParams c) {
  CsrJumpParams p = c.j;
  const size_t n = (size_t)p.n;
  T* rho = reinterpret_cast<T*>(c.rho);
  int lo = 0, hi = -1;  // times whose window holds jump k-1 (ascending times)
  for (int64_t k = 1; k <= c.kmax + 1; ++k) {
    const int64_t kp = k - 1;
    while (lo < c.ntimes && p.K[lo] < kp) ++lo;
    while (hi + 1 < c.ntimes && p.L[hi + 1] <= kp) ++hi;
    p.k = k;
    p.jump = k <= c.kmax;
    p.tlo = lo;
    p.thi = hi;
    p.rho_prev = rho + ((kp & 1) ? n : 0);
    p.rho_next = rho + ((kp & 1) ? 0 : n);
    csr_jump_body<T>(p);
    if (k <= c.kmax && !grid_barrier(c.bar, c.wait_limit, c.status)) return;
  }
}

// Snapshot log-likelihood from the permuted outputs: one CTA.
__global__ void csr_loglik_kernel(const void* outp, int precision, int64_t n, const int64_t* gptr, int ntimes,
                                  const double* counts, const int64_t* mptr, const int32_t* members,
                                  const int32_t* perm, double* ll, int* status) {
  __shared__ double red[32];
  double acc = 0.0;
  bool bad = false;
  for (int i = 0; i < ntimes; ++i) {
    for (int64_t g = gptr[i] + threadIdx.x; g < gptr[i + 1]; g += blockDim.x) {
      double a = 0.0;
      for (int64_t q = mptr[g]; q < mptr[g + 1]; ++q) {
        int64_t idx = (int64_t)i * n + perm[members[q]];
        a += (precision == MJP_FP64) ? reinterpret_cast<const double*>(outp)[idx]
                                     : (double)reinterpret_cast<const float*>(outp)[idx];
      }
      double c = counts[g];
      if (c == 0.0) continue;
      if (a > 0.0) acc += c * log(a);
      else if (a > -1e-30) acc = -INFINITY;
      else bad = true;
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    *ll = t;
    if (isnan(t) && status) atomicCAS(status, 0, kStatusNumeric);
  }
  if (bad && status) atomicCAS(status, 0, kStatusNumeric);
}

int grid_for(int64_t work, int block) {
  int64_t g = (work + block - 1) / block;
  return (int)(g < 152 * 16 ? (g < 1 ? 1 : g) : 152 * 16);
}

}  // namespace

cudaError_t launch_permute_in(int precision, const void* src, const int32_t* perm, void* dst, int64_t n,
                              cudaStream_t s) {
  if (precision == MJP_FP64)
    permute_in_kernel<double><<<grid_for(n, 256), 256, 0, s>>>((const double*)src, perm, (double*)dst, n);
  else
    permute_in_kernel<float><<<grid_for(n, 256), 256, 0, s>>>((const float*)src, perm, (float*)dst, n);
  return cudaGetLastError();
}

cudaError_t launch_permute_out(int precision, const void* src, const int32_t* perm, void* dst, int64_t n,
                               int ntimes, const int32_t* orig, cudaStream_t s) {
  if (precision == MJP_FP64)
    permute_out_kernel<double><<<grid_for(n * ntimes, 256), 256, 0, s>>>((const double*)src, perm, (double*)dst, n,
                                                                          ntimes, orig);
  else
    permute_out_kernel<float><<<grid_for(n * ntimes, 256), 256, 0, s>>>((const float*)src, perm, (float*)dst, n,
                                                                         ntimes, orig);
  return cudaGetLastError();
}

// Launch that may begin while the one before it in the stream ends.
template <typename P>
static cudaError_t launch_dependent(void (*kern)(P), int64_t grid, const P& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

cudaError_t launch_csr_step(int precision, const CsrStepParams& p, cudaStream_t s) {
  const int64_t grid = (p.n + 255) / 256;
  return precision == MJP_FP64 ? launch_dependent(csr_step_kernel<double>, grid, p, s)
                               : launch_dependent(csr_step_kernel<float>, grid, p, s);
}

cudaError_t launch_csr_sum(int precision, const CsrSumParams& p, cudaStream_t s) {
  const int64_t grid = (p.n + 255) / 256;
  return precision == MJP_FP64 ? launch_dependent(csr_sum_kernel<double>, grid, p, s)
                               : launch_dependent(csr_sum_kernel<float>, grid, p, s);
}

cudaError_t launch_csr_jump(int precision, const CsrJumpParams& p, cudaStream_t s) {
  const int block = 512;
  const int grid = grid_for(p.nslices * 32, block);
  if (precision == MJP_FP64) csr_jump_kernel<double><<<grid, block, 0, s>>>(p);
  else csr_jump_kernel<float><<<grid, block, 0, s>>>(p);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_chain_typed(const CsrChainParams& c, cudaStream_t s) {
  // 1024-thread CTAs: the fewer CTAs meet at each grid barrier, the shorter it is.
  const int block = 1024;
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, csr_chain_kernel<T>, block, 0)) != cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // Every CTA must be resident at once: at most the occupancy limit, and no
  // more than the slices need.
  int grid = std::min<int64_t>((int64_t)per_sm * sms, (c.j.nslices * 32 + block - 1) / block);
  if (grid < 1) grid = 1;
  void* args[] = {const_cast<CsrChainParams*>(&c)};
  return cudaLaunchCooperativeKernel((const void*)csr_chain_kernel<T>, dim3(grid), dim3(block), args, 0, s);
}

cudaError_t launch_csr_chain(int precision, const CsrChainParams& p, cudaStream_t s) {
  return precision == MJP_FP64 ? launch_chain_typed<double>(p, s) : launch_chain_typed<float>(p, s);
}

cudaError_t launch_csr_loglik(const void* outp, int precision, int64_t n, const int64_t* gptr, int ntimes,
                              const double* counts, const int64_t* mptr, const int32_t* members,
                              const int32_t* perm, double* ll, int* status, cudaStream_t s) {
  csr_loglik_kernel<<<1, 1024, 0, s>>>(outp, precision, n, gptr, ntimes, counts, mptr, members, perm, ll, status);
  return cudaGetLastError();
}

}  // namespace mjp
