// Field-wide kernels around the fixed-point map: the inner products and
// tall-skinny projections of the recursive projection method (Section 3,
// Eqs. 3.10-3.13), the Newton step on the unstable subspace, the strain
// combine of Algorithm 2 and the constitutive law sigma = C(x) : eps.
//
// Fields are [6][n] float32 (components 11 22 33 23 13 12).  The inner
// product is the tensor Frobenius product (weights 1,1,1,2,2,2).  Each
// thread accumulates a bounded number of products in float32; the block and
// grid reductions run in float64 with a fixed order (deterministic).
#include <math.h>

#include <atomic>

#include "async_copy.cuh"
#include "rpm_internal.h"

namespace rpm {

constexpr int kRedThreads = 256;
constexpr int kPerThread = 8;        // float4 per thread per dot pass on large grids (32 products)

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Error-free sum a + b = s + e (Knuth's TwoSum, six float32 operations).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// Warp sum of float values as an unevaluated pair hi + lo: every level of the
// shuffle tree is a TwoSum, so the rounding errors of the float32 tree are
// carried exactly in lo (float64 arithmetic is slow on this part; the pair
// gives about 48 significant bits).
__device__ __forceinline__ void warp_sum_compensated(float v, float& hi, float& lo) {
  hi = v;
  lo = 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ohi = __shfl_xor_sync(0xffffffffu, hi, o);
    const float olo = __shfl_xor_sync(0xffffffffu, lo, o);
    float s, e;
    two_sum(hi, ohi, s, e);
    hi = s;
    lo = lo + olo + e;
  }
}

// Block-reduce M float values per thread (acc) into partials[row(j) * nblk + blockIdx.x],
// row(0) = 0 when row0 == 0 (skipped otherwise), row(j) = row0 + j for j >= 1.
// Warp level in compensated float32, warps and blocks combined in float64.
template <int M>
__device__ __forceinline__ void block_store(const float* acc, int m, int row0, double* partials,
                                            int nblk) {
  __shared__ double red[kRedThreads / 32][M];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < M; ++j) {
    if (j < m) {
      float hi, lo;
      warp_sum_compensated(acc[j], hi, lo);
      if (lane == 0) red[warp][j] = (double)hi + (double)lo;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    if (j == 0 && row0 != 0) continue;
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kRedThreads / 32; ++w) s += red[w][j];
    partials[(size_t)(j == 0 ? 0 : row0 + j) * nblk + blockIdx.x] = s;
  }
}

__device__ __forceinline__ float dot4(float4 a, float4 b) {
  return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}

// acc[0] = sum w |x - xm|^2 and acc[1 + j] = sum w (x - xm) . Y_j; without xm,
// sum w |x|^2 and sum w x . Y_j.  The difference is formed per element before
// any product, so Z^T (xi - eps) keeps its accuracy when xi and eps agree to
// many digits (near convergence).
// Partial sums go to rows [0] (the norm) and [1 + row0 + j] of `partials`.
// NX = 2: the same of a second field x2 (no xm), its rows after the first's
// K + 1; every Y_j is read once for both.
// PT: float4 per thread (see dots_per_thread).
template <int KMAX, int PT, int NX>
__device__ __forceinline__ void dots_body(const float4* __restrict__ x,
                                          const float4* __restrict__ x2,
                                          const float4* __restrict__ xm,
                                          const float4* __restrict__ Y, long long ys4, int K,
                                          int row0, long long n4, double* partials, int nblk) {
  // The thread's PT difference vectors stay in registers; each basis vector is
  // then read as PT independent 16-byte loads issued together, and its warp
  // sum is taken at once (no accumulator stays live across the vectors, which
  // keeps the register count at three blocks per SM).
  __shared__ double red[kRedThreads / 32][NX * (KMAX + 1)];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long total = 6 * n4;
  const long long base = (long long)blockIdx.x * kRedThreads * PT + threadIdx.x;
  const float4* xs[2] = {x, x2};
  float4 d[NX][PT];
  float w[PT];
#pragma unroll
  for (int v = 0; v < NX; ++v)
#pragma unroll
    for (int r = 0; r < PT; ++r) {
      const long long q = base + (long long)r * kRedThreads;
      const bool in = q < total;
      w[r] = in ? ((q >= 3 * n4) ? 2.f : 1.f) : 0.f;
      d[v][r] = in ? xs[v][q] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  if (NX == 1 && xm) {
#pragma unroll
    for (int r = 0; r < PT; ++r) {
      const long long q = base + (long long)r * kRedThreads;
      if (q < total) {
        const float4 b = xm[q];
        d[0][r] = make_float4(d[0][r].x - b.x, d[0][r].y - b.y, d[0][r].z - b.z, d[0][r].w - b.w);
      }
    }
  }
#pragma unroll
  for (int v = 0; v < NX; ++v) {
    float a = 0.f, hi, lo;
#pragma unroll
    for (int r = 0; r < PT; ++r) a = fmaf(w[r], dot4(d[v][r], d[v][r]), a);
    warp_sum_compensated(a, hi, lo);
    if (lane == 0) red[warp][v * (K + 1)] = (double)hi + (double)lo;
  }
#pragma unroll
  for (int j = 0; j < KMAX; ++j) {
    if (j < K) {
      const float4* yj = Y + j * ys4;
      float4 y[PT];
#pragma unroll
      for (int r = 0; r < PT; ++r) {
        const long long q = base + (long long)r * kRedThreads;
        y[r] = q < total ? yj[q] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int v = 0; v < NX; ++v) {
        float a = 0.f, hi, lo;
#pragma unroll
        for (int r = 0; r < PT; ++r) a = fmaf(w[r], dot4(d[v][r], y[r]), a);
        warp_sum_compensated(a, hi, lo);
        if (lane == 0) red[warp][v * (K + 1) + 1 + j] = (double)hi + (double)lo;
      }
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < NX * (K + 1); j += blockDim.x) {
    if (j == 0 && row0 != 0) continue;
    double t = 0.0;
#pragma unroll
    for (int v = 0; v < kRedThreads / 32; ++v) t += red[v][j];
    partials[(size_t)(j == 0 ? 0 : row0 + j) * nblk + blockIdx.x] = t;
  }
}

// (bound by HBM: 128^3, K = 20: 174 us, 94 % of the copy rate)
template <int KMAX>
__global__ void __launch_bounds__(kRedThreads, 3) k_dots(const float4* __restrict__ x,
                                                      const float4* __restrict__ xm,
                                                      const float4* __restrict__ Y, long long ys4,
                                                      int K, int row0, long long n4,
                                                      double* partials, int nblk) {
  dots_body<KMAX, kPerThread, 1>(x, nullptr, xm, Y, ys4, K, row0, n4, partials, nblk);
}

// Dots (K <= 32) whose last block to finish also adds the per-block rows in
// a fixed order (a warp per row: lanes take every 32nd block, then a fixed
// shuffle tree) into sums[0..NX (K + 1)) and, when M is given, takes the Newton
// step of k_newton with p = K.  The ticket counter is zero between launches
// (the last block resets it).  One launch instead of three.
// Grids up to about 100^3, bound by latency: 32^3 solve 1.64 -> 0.90 ms, 48^3 1.63 -> 1.16 ms with
// the polled reads, more blocks, launches that overlap and both differences of
// a growth at once; 96^3 cold solve 9.8 -> 8.2 ms.
// With a host block (pinned memory) the sums, and the residual when M is
// given, also go there, followed by the sequence number the host polls: a read
// costs neither a copy nor a stream synchronisation.
template <int KMAX, int PT, int NX>
__global__ void __launch_bounds__(kRedThreads, NX == 2 ? 2 : 3) k_dots_fused(
    const float4* __restrict__ x, const float4* __restrict__ x2, const float4* __restrict__ xm,
    const float4* __restrict__ Y, long long ys4, int K, long long n4, double* partials, int nblk,
    double* sums, unsigned int* ticket, const double* __restrict__ M, double* c, double* res_out,
    double inv_norm, HostRead host) {
  grid_dependency_wait();
  dots_body<KMAX, PT, NX>(x, x2, xm, Y, ys4, K, 0, n4, partials, nblk);
  allow_dependent_launch();
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j = warp; j < NX * (K + 1); j += kRedThreads / 32) {
    // 8 independent chains per lane (loads in flight), added in a fixed order
    const double* row = partials + (size_t)j * nblk;
    double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    int b = lane;
    for (; b + 7 * 32 < nblk; b += 8 * 32) {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] += __ldcg(row + b + q * 32);   // L2, not L1
    }
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (b + q * 32 < nblk) v[q] += __ldcg(row + b + q * 32);
    double t = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    t = warp_sum(t);
    if (lane == 0) {
      sums[j] = t;
      if (host.sums) host.sums[j] = t;
    }
  }
  __syncthreads();
  if (M) {
    __shared__ double d[32];
    for (int j = threadIdx.x; j < K; j += blockDim.x) d[j] = sums[1 + j];
    __syncthreads();
    for (int j = threadIdx.x; j < K; j += blockDim.x) {
      double t = -d[j];
      for (int k = 0; k < K; ++k) t += M[(size_t)j * K + k] * d[k];
      c[j] = t;
    }
    if (threadIdx.x == 0) {
      const double r = sqrt(sums[0]) * inv_norm;   // NaN stays NaN
      res_out[0] = r;
      if (host.res) *host.res = r;
    }
  }
  if (host.sums) __threadfence_system();
  __syncthreads();
  if (threadIdx.x == 0) {
    *ticket = 0u;
    if (host.seq) {
      __threadfence_system();
      *reinterpret_cast<volatile unsigned long long*>(host.seq) = host.value;
    }
  }
}

// float4 per thread of a dots pass: eight where that still gives two blocks per
// SM, fewer on smaller grids, whose passes would leave most SMs idle.
static int dots_per_thread(long long n) {
  const long long total = 6 * (n / 4);
  return total >= 304LL * kRedThreads * 8 ? 8 : (total >= 304LL * kRedThreads * 4 ? 4 : 2);
}

template <int PT, int NX>
static cudaError_t dots_fused_k(const float4* x, const float4* x2, const float4* xm,
                                const float4* Y, long long ys4, int K, long long n4,
                                double* partials, int nblk, double* sums, unsigned int* ticket,
                                const double* M, double* c, double* res_out, double inv_norm,
                                const HostRead& host, cudaStream_t st) {
#define RPM_FUSED(KM)                                                                          \
  launch_pdl(k_dots_fused<KM, PT, NX>, dim3(nblk), kRedThreads, 0, st, x, x2, xm, Y, ys4, K, n4, \
             partials, nblk, sums, ticket, M, c, res_out, inv_norm, host)
  if (K <= 2) return RPM_FUSED(2);
  if (K <= 8) return RPM_FUSED(8);
  if (K <= 16) return RPM_FUSED(16);
  return RPM_FUSED(32);
#undef RPM_FUSED
}

cudaError_t launch_dots_fused(const float* x, const float* x2, const float* x_minus,
                              const float* Y, long long ystride, int K, long long n,
                              double* partials, int nblk, double* sums, unsigned int* ticket,
                              const double* M, double* c, double* res_out, double inv_norm,
                              const HostRead& host, cudaStream_t st) {
  if (K > 32) return cudaErrorInvalidValue;
  const long long n4 = n / 4;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  const float4* z4 = reinterpret_cast<const float4*>(x2);
  const float4* m4 = reinterpret_cast<const float4*>(x_minus);
  const float4* y4 = reinterpret_cast<const float4*>(Y);
  const long long ys4 = ystride / 4;
#define RPM_PT(P)                                                                             \
  (x2 ? dots_fused_k<P, 2>(x4, z4, m4, y4, ys4, K, n4, partials, nblk, sums, ticket, M, c,    \
                           res_out, inv_norm, host, st)                                       \
      : dots_fused_k<P, 1>(x4, z4, m4, y4, ys4, K, n4, partials, nblk, sums, ticket, M, c,    \
                           res_out, inv_norm, host, st))
  switch (dots_per_thread(n)) {
    case 2: return RPM_PT(2);
    case 4: return RPM_PT(4);
    default: return RPM_PT(8);
  }
#undef RPM_PT
}

static int dots_blocks(long long n, int per_thread) {
  const long long total = 6 * (n / 4), per = (long long)kRedThreads * per_thread;
  return (int)((total + per - 1) / per);
}

int dots_fused_blocks_for(long long n) { return dots_blocks(n, dots_per_thread(n)); }
int dots_blocks_for(long long n) { return dots_blocks(n, kPerThread); }

cudaError_t launch_dots(const float* x, const float* x_minus, const float* Y, long long ystride,
                        int K, long long n, double* partials, int nblk, cudaStream_t st) {
  const long long n4 = n / 4;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  const float4* m4 = reinterpret_cast<const float4*>(x_minus);
  const long long ys4 = ystride / 4;
  // K > 32: chunks of 32 basis vectors; the norm row is written by chunk 0
  for (int k0 = 0; k0 == 0 || k0 < K; k0 += 32) {
    const int Kc = K - k0 < 32 ? K - k0 : 32;
    const float4* y4 = reinterpret_cast<const float4*>(Y) + (Y ? k0 * ys4 : 0);
    if (Kc <= 2)
      k_dots<2><<<nblk, kRedThreads, 0, st>>>(x4, m4, y4, ys4, Kc, k0, n4, partials, nblk);
    else if (Kc <= 8)
      k_dots<8><<<nblk, kRedThreads, 0, st>>>(x4, m4, y4, ys4, Kc, k0, n4, partials, nblk);
    else if (Kc <= 16)
      k_dots<16><<<nblk, kRedThreads, 0, st>>>(x4, m4, y4, ys4, Kc, k0, n4, partials, nblk);
    else
      k_dots<32><<<nblk, kRedThreads, 0, st>>>(x4, m4, y4, ys4, Kc, k0, n4, partials, nblk);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int dots_launches(int K) { return K <= 32 ? 1 : (K + 31) / 32; }

// out[j] = sum_b partials[j * nblk + b], one block per j, fixed order.
__global__ void __launch_bounds__(kRedThreads) k_reduce(const double* __restrict__ partials, int nblk,
                                                        double* out) {
  const int j = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += partials[(size_t)j * nblk + b];
  __shared__ double red[kRedThreads / 32];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kRedThreads / 32; ++w) t += red[w];
    out[j] = t;
  }
}

cudaError_t launch_reduce_partials(const double* partials, int nblk, int m, double* out,
                                   cudaStream_t st) {
  k_reduce<<<m, kRedThreads, 0, st>>>(partials, nblk, out);
  return cudaGetLastError();
}

// out = xs * x + sum_j coef[j] * Y_j   (coef in float64 on the device)
// (out may alias x).  The basis vectors are read in groups of 8 so that each
// thread keeps 8 independent 16-byte loads in flight at a modest register count.
// NX = 2: a second field the same way (x2 -> out2, coefficients coef2), every
// basis vector read once for both.
template <int KMAX, int NX>
__global__ void __launch_bounds__(kRedThreads, 3) k_combine(
    float4* out, float4* out2, const float4* x, const float4* x2, float xs,
    const float4* __restrict__ Y, long long ys4, int K, const double* __restrict__ coef,
    const double* __restrict__ coef2, float cscale, long long total4) {
  __shared__ float cf[NX][KMAX > 0 ? KMAX : 1];
  grid_dependency_wait();
  for (int j = threadIdx.x; j < K; j += blockDim.x) {
    cf[0][j] = (float)(coef[j] * (double)cscale);
    if (NX == 2) cf[NX - 1][j] = (float)(coef2[j] * (double)cscale);
  }
  __syncthreads();
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total4;
       q += (long long)gridDim.x * blockDim.x) {
    float4 a[NX];
#pragma unroll
    for (int v = 0; v < NX; ++v) {
      const float4* xv = v ? x2 : x;
      a[v] = xv ? xv[q] : make_float4(0.f, 0.f, 0.f, 0.f);
      a[v] = make_float4(a[v].x * xs, a[v].y * xs, a[v].z * xs, a[v].w * xs);
    }
#pragma unroll 1
    for (int j0 = 0; j0 < K; j0 += 8) {
      float4 y[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j0 + u < K) y[u] = Y[(j0 + u) * ys4 + q];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (j0 + u < K) {
#pragma unroll
          for (int v = 0; v < NX; ++v) {
            const float c = cf[v][j0 + u];
            a[v].x = fmaf(c, y[u].x, a[v].x);
            a[v].y = fmaf(c, y[u].y, a[v].y);
            a[v].z = fmaf(c, y[u].z, a[v].z);
            a[v].w = fmaf(c, y[u].w, a[v].w);
          }
        }
      }
    }
    allow_dependent_launch();
    out[q] = a[0];
    if (NX == 2) out2[q] = a[NX - 1];
  }
}

static int stream_blocks(long long total4) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, v = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    sms = v;
  }
  const long long want = (total4 + kRedThreads - 1) / kRedThreads;
  const long long cap = (long long)sms * 8;
  return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// Grid of a grid-stride kernel: the blocks that are resident at once (so no
// partial last wave), at most one block per 256 threads' worth of work.
// (the occupancy query runs once per kernel instance: `slot` caches it)
template <typename Kern>
static int resident_grid(Kern kernel, long long total4, std::atomic<int>& slot) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, v = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    sms = v;
  }
  int per_sm = slot.load();
  if (per_sm < 1) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kRedThreads, 0) !=
            cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    slot.store(per_sm);
  }
  const long long want = (total4 + kRedThreads - 1) / kRedThreads;
  const long long cap = (long long)sms * per_sm;
  return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

static std::atomic<int> g_combine_occ[2][4];   // resident blocks per SM of k_combine<2, 8, 16, 32>

template <int NX>
static cudaError_t combine_k(float* out, float* out2, const float* x, const float* x2,
                             float xscale, const float* Y, long long ystride, int K,
                             const double* coef, const double* coef2, float cscale, long long n,
                             cudaStream_t st) {
  const long long total4 = 6 * (n / 4);
  float4 *o4 = reinterpret_cast<float4*>(out), *p4 = reinterpret_cast<float4*>(out2);
  const long long ys4 = ystride / 4;
  // K > 32: the first chunk forms xs * x + ..., later chunks accumulate into out
  for (int k0 = 0; k0 == 0 || k0 < K; k0 += 32) {
    const int Kc = K - k0 < 32 ? K - k0 : 32;
    const float4* x4 = k0 == 0 ? reinterpret_cast<const float4*>(x) : o4;
    const float4* z4 = k0 == 0 ? reinterpret_cast<const float4*>(x2) : p4;
    const float xs = k0 == 0 ? xscale : 1.f;
    const float4* y4 = reinterpret_cast<const float4*>(Y) + (Y ? k0 * ys4 : 0);
    const double* cf = coef ? coef + k0 : nullptr;
    const double* cg = coef2 ? coef2 + k0 : nullptr;
#define RPM_COMBINE(KM, SLOT)                                                                  \
  launch_pdl(k_combine<KM, NX>,                                                                \
             dim3(resident_grid(k_combine<KM, NX>, total4, g_combine_occ[NX - 1][SLOT])),      \
             kRedThreads, 0, st, o4, p4, x4, z4, xs, y4, ys4, Kc, cf, cg, cscale, total4)
    const cudaError_t e = Kc <= 2    ? RPM_COMBINE(2, 0)
                          : Kc <= 8  ? RPM_COMBINE(8, 1)
                          : Kc <= 16 ? RPM_COMBINE(16, 2)
                                     : RPM_COMBINE(32, 3);
#undef RPM_COMBINE
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_combine(float* out, const float* x, float xscale, const float* Y,
                           long long ystride, int K, const double* coef, float cscale,
                           long long n, cudaStream_t st) {
  return combine_k<1>(out, nullptr, x, nullptr, xscale, Y, ystride, K, coef, nullptr, cscale, n, st);
}

cudaError_t launch_combine2(float* out, float* out2, const float* Y, long long ystride, int K,
                            const double* coef, const double* coef2, float cscale, long long n,
                            cudaStream_t st) {
  return combine_k<2>(out, out2, out, out2, 1.f, Y, ystride, K, coef, coef2, cscale, n, st);
}

int combine_launches(int K) { return K <= 32 ? 1 : (K + 31) / 32; }

// sigma = C(x) : eps (Eq. 2.2), optionally stored, and per-component sums.
__global__ void __launch_bounds__(kRedThreads) k_stress(const float4* __restrict__ eps,
                                                        const uchar4* __restrict__ phase,
                                                        const float2* __restrict__ cmat,
                                                        float4* __restrict__ sig, long long n4,
                                                        double* partials, int nblk) {
  float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const long long base = (long long)blockIdx.x * kRedThreads * kPerThread + threadIdx.x;
#pragma unroll 1
  for (int r = 0; r < kPerThread; ++r) {
    const long long q = base + (long long)r * kRedThreads;
    if (q >= n4) break;
    const uchar4 ph = phase[q];
    const float2 m0 = cmat[ph.x], m1 = cmat[ph.y], m2 = cmat[ph.z], m3 = cmat[ph.w];
    float4 e[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = eps[c * n4 + q];
    const float4 tr = make_float4(e[0].x + e[1].x + e[2].x, e[0].y + e[1].y + e[2].y,
                                  e[0].z + e[1].z + e[2].z, e[0].w + e[1].w + e[2].w);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      float4 s = make_float4(2.f * m0.y * e[c].x, 2.f * m1.y * e[c].y, 2.f * m2.y * e[c].z,
                             2.f * m3.y * e[c].w);
      if (c < 3) {
        s.x = fmaf(m0.x, tr.x, s.x);
        s.y = fmaf(m1.x, tr.y, s.y);
        s.z = fmaf(m2.x, tr.z, s.z);
        s.w = fmaf(m3.x, tr.w, s.w);
      }
      if (sig) sig[c * n4 + q] = s;
      acc[c] += (s.x + s.y) + (s.z + s.w);
    }
  }
  block_store<6>(acc, 6, 0, partials, nblk);
}

int stress_blocks_for(long long n) {
  const long long n4 = n / 4;
  return (int)((n4 + (long long)kRedThreads * kPerThread - 1) / ((long long)kRedThreads * kPerThread));
}

cudaError_t launch_stress(const GridDev& g, const float* eps, float* sig, double* partials, int nblk,
                          cudaStream_t st) {
  const long long n4 = g.n / 4;
  k_stress<<<nblk, kRedThreads, 0, st>>>(reinterpret_cast<const float4*>(eps),
                                         reinterpret_cast<const uchar4*>(g.phase), g.cmat,
                                         reinterpret_cast<float4*>(sig), n4, partials, nblk);
  return cudaGetLastError();
}

// out = a x + b y (y nullable; out may alias x or y)
__global__ void __launch_bounds__(kRedThreads) k_axpby(float4* out, float a, const float4* x,
                                                       float b, const float4* y, long long total4) {
  grid_dependency_wait();
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total4;
       q += (long long)gridDim.x * blockDim.x) {
    const float4 u = x[q];
    float4 r = make_float4(a * u.x, a * u.y, a * u.z, a * u.w);
    if (y) {
      const float4 v = y[q];
      r = make_float4(fmaf(b, v.x, r.x), fmaf(b, v.y, r.y), fmaf(b, v.z, r.z), fmaf(b, v.w, r.w));
    }
    allow_dependent_launch();
    out[q] = r;
  }
}

cudaError_t launch_axpby(float* out, float a, const float* x, float b, const float* y, long long n,
                         cudaStream_t st) {
  const long long total4 = 6 * (n / 4);
  return launch_pdl(k_axpby, dim3(stream_blocks(total4)), kRedThreads, 0, st,
                    reinterpret_cast<float4*>(out), a, reinterpret_cast<const float4*>(x), b,
                    reinterpret_cast<const float4*>(y), total4);
}

// d0 = a - b, d1 = b - c (five field sweeps for the two differences)
__global__ void __launch_bounds__(kRedThreads) k_diff2(float4* d0, float4* d1, const float4* a,
                                                       const float4* b, const float4* c,
                                                       long long total4) {
  grid_dependency_wait();
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total4;
       q += (long long)gridDim.x * blockDim.x) {
    const float4 u = a[q], v = b[q], w = c[q];
    allow_dependent_launch();
    d0[q] = make_float4(u.x - v.x, u.y - v.y, u.z - v.z, u.w - v.w);
    d1[q] = make_float4(v.x - w.x, v.y - w.y, v.z - w.z, v.w - w.w);
  }
}

cudaError_t launch_diff2(float* d0, float* d1, const float* a, const float* b, const float* c,
                         long long n, cudaStream_t st) {
  const long long total4 = 6 * (n / 4);
  return launch_pdl(k_diff2, dim3(stream_blocks(total4)), kRedThreads, 0, st,
                    reinterpret_cast<float4*>(d0), reinterpret_cast<float4*>(d1),
                    reinterpret_cast<const float4*>(a), reinterpret_cast<const float4*>(b),
                    reinterpret_cast<const float4*>(c), total4);
}

// eps_next = (C + C0)^-1 : (s_a + C0 : eps_b), Algorithm 3, per voxel; the
// inverse of an isotropic stiffness (lam_s, mu_s) maps t to
// (t - k_s tr(t) I) h_s with k_s = lam_s / (3 lam_s + 2 mu_s), h_s = 1 / (2 mu_s),
// both precomputed per phase in the table (lam_a, mu_a, k_s, h_s).
__global__ void __launch_bounds__(kRedThreads) k_pol_post(const float4* __restrict__ eps,
                                                          const float4* __restrict__ epsb,
                                                          const uchar4* __restrict__ phase,
                                                          const float4* __restrict__ post,
                                                          float lam0, float mu0,
                                                          float4* __restrict__ out, long long n4) {
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n4;
       q += (long long)gridDim.x * blockDim.x) {
    const uchar4 ph = phase[q];
    const float4 pm[4] = {post[ph.x], post[ph.y], post[ph.z], post[ph.w]};
    float e[6][4], b[6][4];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float4 u = eps[c * n4 + q], v = epsb[c * n4 + q];
      e[c][0] = u.x; e[c][1] = u.y; e[c][2] = u.z; e[c][3] = u.w;
      b[c][0] = v.x; b[c][1] = v.y; b[c][2] = v.z; b[c][3] = v.w;
    }
    float o[6][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float tre = e[0][k] + e[1][k] + e[2][k];
      const float trb = b[0][k] + b[1][k] + b[2][k];
      float t[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) t[c] = 2.f * pm[k].y * e[c][k] + 2.f * mu0 * b[c][k];
#pragma unroll
      for (int c = 0; c < 3; ++c) t[c] += pm[k].x * tre + lam0 * trb;
      const float trt = t[0] + t[1] + t[2];
      const float sh = pm[k].z * trt, inv2mu = pm[k].w;
#pragma unroll
      for (int c = 0; c < 6; ++c) o[c][k] = (t[c] - (c < 3 ? sh : 0.f)) * inv2mu;
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) out[c * n4 + q] = make_float4(o[c][0], o[c][1], o[c][2], o[c][3]);
  }
}

cudaError_t launch_polarization_post(const GridDev& g, const float4* post, const float* eps,
                                     const float* eps_b, float* out, cudaStream_t st) {
  const long long n4 = g.n / 4;
  k_pol_post<<<stream_blocks(n4), kRedThreads, 0, st>>>(
      reinterpret_cast<const float4*>(eps), reinterpret_cast<const float4*>(eps_b),
      reinterpret_cast<const uchar4*>(g.phase), post, g.lam0, g.mu0,
      reinterpret_cast<float4*>(out), n4);
  return cudaGetLastError();
}

__global__ void k_fill(float4* f, float e0, float e1, float e2, float e3, float e4, float e5,
                       long long n4) {
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < 6 * n4;
       q += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(q / n4);
    const float v = c == 0 ? e0 : c == 1 ? e1 : c == 2 ? e2 : c == 3 ? e3 : c == 4 ? e4 : e5;
    f[q] = make_float4(v, v, v, v);
  }
}

cudaError_t launch_fill(float* f, const double E[6], long long n, cudaStream_t st) {
  const long long n4 = n / 4;
  k_fill<<<stream_blocks(6 * n4), kRedThreads, 0, st>>>(
      reinterpret_cast<float4*>(f), (float)E[0], (float)E[1], (float)E[2], (float)E[3],
      (float)E[4], (float)E[5], n4);
  return cudaGetLastError();
}

// Newton step on the unstable subspace (Eq. 3.11 with H = Z^T F_u Z):
// sums[0] = |xi - eps|^2, sums[1 + j] = zeta_j = <Z_j, xi>;  M = (I - H)^-1.
// z+ = z + M (zeta - z);  c = z+ - zeta (so eps_next = xi + Z c);  z_next = z+
// (z = Z^T eps of the current iterate; z_next = Z^T eps_next).
// res_out = sqrt(sums[0]) * inv_norm.
// Newton step of Eqs. 3.10-3.13 in reduced coordinates.  With
// d = zeta - z = Z^T (xi - eps) (sums[1..p], formed from the difference field)
// and M = (I - H)^-1, the new iterate eps+ = xi + Z (z+ - zeta) with
// z+ = z + M d needs only c = z+ - zeta = (M - I) d.
__global__ void k_newton(const double* __restrict__ sums, int p, const double* __restrict__ M,
                         double* __restrict__ c, double* res_out, double inv_norm) {
  __shared__ double d[kMaxBasis];
  for (int j = threadIdx.x; j < p; j += blockDim.x) d[j] = sums[1 + j];
  __syncthreads();
  for (int j = threadIdx.x; j < p; j += blockDim.x) {
    double s = -d[j];
    for (int k = 0; k < p; ++k) s += M[(size_t)j * p + k] * d[k];
    c[j] = s;
  }
  if (threadIdx.x == 0) res_out[0] = sqrt(sums[0]) * inv_norm;   // NaN stays NaN
}

cudaError_t launch_newton(const double* sums, int p, const double* M, double* c, double* res_out,
                          double inv_norm, cudaStream_t st) {
  if (p > kMaxBasis) return cudaErrorInvalidValue;
  k_newton<<<1, 256, 0, st>>>(sums, p, M, c, res_out, inv_norm);
  return cudaGetLastError();
}

}  // namespace rpm
