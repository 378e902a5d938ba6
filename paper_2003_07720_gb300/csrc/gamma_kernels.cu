// The Lippmann-Schwinger map of Section 2 as three fused passes over HBM.
//
//   pass A (one block per z-plane and tensor component):
//       tau = (C(x) - C0) : eps  (Eq. 2.3, isotropic phases), packed as
//       complex rows z_n = tau_2n + i tau_2n+1, forward FFT along x of
//       length nx/2, real-to-complex untangling, forward FFT along y;
//       writes the half spectrum in slot order.
//   pass B (one block per T consecutive (ky, kx) pencils, all 6 components):
//       forward FFT along z, eps_hat = -Gamma0_hat(xi) : tau_hat per
//       frequency (Eq. 2.5) with the zero frequency set to E n_vox, inverse
//       FFT along z.
//   pass C (one block per z-plane and component): inverse FFT along y,
//       complex-to-real tangling, inverse FFT along x of length nx/2, scale.
//
// These scalar kernels (k_pass_a/b/c, and the z pass k_pencil_green, in which
// the forward z step 2, the Green operator and the inverse z step 1 run in
// registers) run where a caller forces the whole-plane variant or the autotuner
// times it.  By default every grid takes the paired kernels of gamma_pair.cu:
// square planes up to 128 in three passes, 256^2 and nx != ny in five.  The
// dispatch between them is at the end of this file.
//
// The Green operator of the isotropic reference medium is evaluated on the
// fly from the unit wave vector n = xi/|xi|:
//   Gamma0_hat : tau_hat = sym(n (x) w),  w = (v - a n (n.v)) / mu0,
//   v = tau_hat n,  a = (lam0 + mu0) / (lam0 + 2 mu0),
// obtained from div(C0 : eps(u) + tau) = 0 in Fourier space.
#include "async_copy.cuh"
#include "fft_smem.cuh"
#include "rpm_internal.h"

namespace rpm {

constexpr int kThreads = 256;

template <int NX, int NY>
struct PlaneCfg {
  static constexpr int NXH = NX / 2;
  static constexpr int SX = NXH + 1;          // x slots of the half spectrum
  static constexpr int NYP = NY + 1;          // odd column stride in float2
  static constexpr int PLANE_F2 = SX * NYP;
  static constexpr int TAB_F2 = NXH + NY + SX;
};

// X_k from Z_k = a, Z_{M-k} = b (M = nx/2), w = W_nx^k:
// X_k = (a + conj b)/2 - (i/2) w (a - conj b)
__device__ __forceinline__ float2 r2c_post(float2 a, float2 b, float2 w) {
  const float2 s = make_float2(a.x + b.x, a.y - b.y);
  const float2 d = make_float2(a.x - b.x, a.y + b.y);
  const float2 u = cmul(w, d);
  return make_float2(0.5f * (s.x + u.y), 0.5f * (s.y - u.x));
}

// 2 Z_k from X_k = a, X_{M-k} = b, w = W_nx^k:
// 2 Z_k = (a + conj b) + i (a - conj b) conj(w)
__device__ __forceinline__ float2 c2r_pre(float2 a, float2 b, float2 w) {
  const float2 s = make_float2(a.x + b.x, a.y - b.y);
  const float2 d = make_float2(a.x - b.x, a.y + b.y);
  const float2 u = cmulc(d, w);
  return make_float2(s.x - u.y, s.y + u.x);
}

// Block size of the plane passes and the blocks per SM the register budget targets.
constexpr int kPlaneThreads = 256;
constexpr int kPlaneMinBlocks = 3;

template <int NX, int NY>
__global__ void __launch_bounds__(kPlaneThreads, kPlaneMinBlocks)
    k_pass_a(GridDev g, const float* __restrict__ in, float2* __restrict__ spec, int mode) {
  using C = PlaneCfg<NX, NY>;
  extern __shared__ float2 sm[];
  float2* P = sm;
  float2* twx = P + C::PLANE_F2;
  float2* twy = twx + C::NXH;
  float2* r2c = twy + NY;
  float2* dm = r2c + C::SX;
  const int c = blockIdx.x, z = blockIdx.y;
  for (int i = threadIdx.x; i < C::NXH; i += blockDim.x) twx[i] = g.tw_x[i];
  for (int i = threadIdx.x; i < NY; i += blockDim.x) twy[i] = g.tw_y[i];
  for (int i = threadIdx.x; i < C::SX; i += blockDim.x) r2c[i] = g.r2c_w[i];
  for (int i = threadIdx.x; i < 256; i += blockDim.x) dm[i] = g.dmat[i];   // any uint8 id is in range
  __syncthreads();

  const size_t n2 = (size_t)g.n / 2;                     // float2 per component
  const size_t z2 = (size_t)z * NY * C::NXH;             // plane offset in float2
  const float2* in2 = reinterpret_cast<const float2*>(in);
  const uchar2* ph2 = reinterpret_cast<const uchar2*>(g.phase) + z2;
  // Loads are issued in groups of U per thread before any use, so each thread
  // keeps several independent requests in flight (the plane is streamed once).
  constexpr int TOT = NY * C::NXH, U = 4;
  for (int base = threadIdx.x; base < TOT; base += U * kPlaneThreads) {
    float2 a[U], b[U], d[U];
    uchar2 ph[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = base + u * kPlaneThreads;
      if (idx < TOT) {
        const size_t v = z2 + idx;
        if (mode == GM_RAW_TAU || c >= 3) {
          a[u] = in2[c * n2 + v];
        } else {
          a[u] = in2[v];
          b[u] = in2[n2 + v];
          d[u] = in2[2 * n2 + v];
        }
        if (mode != GM_RAW_TAU) ph[u] = ph2[idx];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = base + u * kPlaneThreads;
      if (idx < TOT) {
        const int y = idx / C::NXH, h = idx - y * C::NXH;
        float2 t;
        if (mode == GM_RAW_TAU) {
          t = a[u];
        } else {
          const float2 d0 = dm[ph[u].x], d1 = dm[ph[u].y];
          if (c >= 3) {
            t = make_float2(2.f * d0.y * a[u].x, 2.f * d1.y * a[u].y);
          } else {
            const float2 e = c == 0 ? a[u] : (c == 1 ? b[u] : d[u]);
            t = make_float2(fmaf(d0.x, a[u].x + b[u].x + d[u].x, 2.f * d0.y * e.x),
                            fmaf(d1.x, a[u].y + b[u].y + d[u].y, 2.f * d1.y * e.y));
          }
        }
        P[h * C::NYP + y] = t;
      }
    }
  }
  __syncthreads();
  smem_fft<C::NXH, false, NY, 1, C::NYP>(P, twx);
  for (int t = threadIdx.x; t < NY * (C::NXH / 2 + 1); t += blockDim.x) {
    const int y = t % NY, k = t / NY;
    if (k == 0) {
      const float2 z0 = P[y];
      P[y] = make_float2(z0.x + z0.y, 0.f);
      P[C::NXH * C::NYP + y] = make_float2(z0.x - z0.y, 0.f);
    } else {
      const int kk = C::NXH - k;
      const int sk = slot_of<C::NXH>(k), skk = slot_of<C::NXH>(kk);
      const float2 a = P[sk * C::NYP + y], b = P[skk * C::NYP + y];
      P[sk * C::NYP + y] = r2c_post(a, b, r2c[k]);
      if (kk != k) P[skk * C::NYP + y] = r2c_post(b, a, r2c[kk]);
    }
  }
  __syncthreads();
  smem_fft<NY, false, C::SX, C::NYP, 1>(P, twy);
  float2* out = spec + ((size_t)c * g.nz + z) * g.plane;
  for (int idx = threadIdx.x; idx < NY * C::SX; idx += blockDim.x) {
    const int sy = idx / C::SX, sx = idx - sy * C::SX;
    out[idx] = P[sx * C::NYP + sy];
  }
}

template <int NX, int NY>
__global__ void __launch_bounds__(kPlaneThreads, kPlaneMinBlocks)
    k_pass_c(GridDev g, const float2* __restrict__ spec, float* __restrict__ outp, float scale) {
  using C = PlaneCfg<NX, NY>;
  extern __shared__ float2 sm[];
  float2* P = sm;
  float2* twx = P + C::PLANE_F2;
  float2* twy = twx + C::NXH;
  float2* r2c = twy + NY;
  const int c = blockIdx.x, z = blockIdx.y;
  for (int i = threadIdx.x; i < C::NXH; i += blockDim.x) twx[i] = g.tw_x[i];
  for (int i = threadIdx.x; i < NY; i += blockDim.x) twy[i] = g.tw_y[i];
  for (int i = threadIdx.x; i < C::SX; i += blockDim.x) r2c[i] = g.r2c_w[i];
  const float2* src = spec + ((size_t)c * g.nz + z) * g.plane;
  {
    constexpr int TOT = NY * C::SX, U = 8;
    for (int base = threadIdx.x; base < TOT; base += U * kPlaneThreads) {
      float2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = base + u * kPlaneThreads;
        if (idx < TOT) v[u] = src[idx];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = base + u * kPlaneThreads;
        if (idx < TOT) {
          const int sy = idx / C::SX, sx = idx - sy * C::SX;
          P[sx * C::NYP + sy] = v[u];
        }
      }
    }
  }
  __syncthreads();
  smem_fft<NY, true, C::SX, C::NYP, 1>(P, twy);
  for (int t = threadIdx.x; t < NY * (C::NXH / 2 + 1); t += blockDim.x) {
    const int y = t % NY, k = t / NY;
    if (k == 0) {
      P[y] = c2r_pre(P[y], P[C::NXH * C::NYP + y], make_float2(1.f, 0.f));
    } else {
      const int kk = C::NXH - k;
      const int sk = slot_of<C::NXH>(k), skk = slot_of<C::NXH>(kk);
      const float2 a = P[sk * C::NYP + y], b = P[skk * C::NYP + y];
      P[sk * C::NYP + y] = c2r_pre(a, b, r2c[k]);
      if (kk != k) P[skk * C::NYP + y] = c2r_pre(b, a, r2c[kk]);
    }
  }
  __syncthreads();
  smem_fft<C::NXH, true, NY, 1, C::NYP>(P, twx);
  const size_t n2 = (size_t)g.n / 2;
  float2* out2 = reinterpret_cast<float2*>(outp) + c * n2 + (size_t)z * NY * C::NXH;
  for (int idx = threadIdx.x; idx < NY * C::NXH; idx += blockDim.x) {
    const int y = idx / C::NXH, h = idx - y * C::NXH;
    out2[idx] = cscale(P[h * C::NYP + y], scale);
  }
}

// T consecutive (ky, kx) pencils per pass-B block: TT = 0 takes the default
// for the length (8 pencils = 64-byte rows at nz = 64 and 128; 16 at
// nz = 256, one 512-thread block per SM, measured 0.980 vs 1.012 ms per
// 256^3 apply with 8); the tile autotuner of rpm_create also tries half and
// twice the default (GridDev::pencil_t).
template <int NZ, int TT = 0>
struct PencilCfg {
  static constexpr int T = TT ? TT : (NZ >= 256 ? 16 : (NZ >= 64 ? 8 : 32));
  static constexpr int NZP = (NZ % 2 == 0) ? NZ + 1 : NZ;
};

// eps_hat = -Gamma0_hat(n) : tau_hat for one frequency (components 11 22 33 23 13 12)
__device__ __forceinline__ void green_apply(float2* t, float n1, float n2, float n3, float a,
                                            float inv_mu0) {
  float2 v1, v2, v3;
  v1.x = t[0].x * n1 + t[5].x * n2 + t[4].x * n3;
  v1.y = t[0].y * n1 + t[5].y * n2 + t[4].y * n3;
  v2.x = t[5].x * n1 + t[1].x * n2 + t[3].x * n3;
  v2.y = t[5].y * n1 + t[1].y * n2 + t[3].y * n3;
  v3.x = t[4].x * n1 + t[3].x * n2 + t[2].x * n3;
  v3.y = t[4].y * n1 + t[3].y * n2 + t[2].y * n3;
  const float sx = n1 * v1.x + n2 * v2.x + n3 * v3.x;
  const float sy = n1 * v1.y + n2 * v2.y + n3 * v3.y;
  float2 w1, w2, w3;
  w1.x = (v1.x - a * n1 * sx) * inv_mu0;
  w1.y = (v1.y - a * n1 * sy) * inv_mu0;
  w2.x = (v2.x - a * n2 * sx) * inv_mu0;
  w2.y = (v2.y - a * n2 * sy) * inv_mu0;
  w3.x = (v3.x - a * n3 * sx) * inv_mu0;
  w3.y = (v3.y - a * n3 * sy) * inv_mu0;
  t[0] = make_float2(-n1 * w1.x, -n1 * w1.y);
  t[1] = make_float2(-n2 * w2.x, -n2 * w2.y);
  t[2] = make_float2(-n3 * w3.x, -n3 * w3.y);
  t[3] = make_float2(-0.5f * (n2 * w3.x + n3 * w2.x), -0.5f * (n2 * w3.y + n3 * w2.y));
  t[4] = make_float2(-0.5f * (n1 * w3.x + n3 * w1.x), -0.5f * (n1 * w3.y + n3 * w1.y));
  t[5] = make_float2(-0.5f * (n1 * w2.x + n2 * w1.x), -0.5f * (n1 * w2.y + n2 * w1.y));
}

// Pass B body for NT threads per block (k_pass_b: 256; k_pass_b_wide: 512,
// where shared memory limits a block of 256 to two blocks per SM, nz >= 256,
// so that 32 warps per SM hide the latency).
template <int NZ, int TT, int NT>
__device__ __forceinline__ void pass_b_body(const GridDev& g, float2* __restrict__ spec, int mode,
                                            const GammaArgs& ga) {
  using C = PencilCfg<NZ, TT>;
  constexpr int T = C::T, NZP = C::NZP;
  constexpr int Z1 = Split<NZ>::N1, Z2 = Split<NZ>::N2;
  // two register steps: the first reads the spectrum and the last writes it
  // straight from / to global memory (task q -> pencil t fastest, then
  // component, then n2, so a half-warp covers two components' lines)
  constexpr bool DIRECT = Z2 > 1;
  extern __shared__ float2 sm[];
  float2* B = sm;
  float2* twz = B + 6 * T * NZP;
  __shared__ float4 pen[T];          // per pencil: (xi_x, xi_y, has-Nyquist, non-zero count)
  for (int i = threadIdx.x; i < NZ; i += blockDim.x) twz[i] = g.tw_z[i];
  const int m0 = blockIdx.x * T;
  const int plane = g.plane;
  if (threadIdx.x < T) {
    const int m = m0 + threadIdx.x;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m < plane) {
      const int sxn = g.nxh + 1;
      const int sy = m / sxn, sx = m - sy * sxn;
      const int2 fx = g.fx[sx], fy = g.fy[sy];
      q = make_float4(fx.x * g.inv_lx, fy.x * g.inv_ly, (float)(fx.y | fy.y),
                      (float)((fx.x != 0) + (fy.x != 0)));
    }
    pen[threadIdx.x] = q;
  }
  if constexpr (DIRECT) {
    __syncthreads();
    for (int q = threadIdx.x; q < 6 * T * Z2; q += NT) {
      const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
      const int m = m0 + t;
      const float2* src = spec + ((size_t)c * NZ + n2) * plane + m;
      const size_t zs = (size_t)Z2 * plane;
      float2 v[Z1];
#pragma unroll
      for (int i = 0; i < Z1; ++i) v[i] = m < plane ? src[i * zs] : make_float2(0.f, 0.f);
      RegDft<Z1, false>::run(v);
#pragma unroll
      for (int k1 = 1; k1 < Z1; ++k1) v[k1] = cmul(v[k1], twz[n2 * Z1 + k1]);
      float2* p = B + (c * T + t) * NZP + n2;
#pragma unroll
      for (int i = 0; i < Z1; ++i) p[i * Z2] = v[i];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 6 * T * Z1; q += NT) {   // forward step 2 in shared memory
      const int b = q % (6 * T), k1 = q / (6 * T);
      float2* p = B + b * NZP + k1 * Z2;
      float2 v[Z2];
#pragma unroll
      for (int i = 0; i < Z2; ++i) v[i] = p[i];
      RegDft<Z2, false>::run(v);
#pragma unroll
      for (int i = 0; i < Z2; ++i) p[i] = v[i];
    }
    __syncthreads();
  } else {
    constexpr int TOT = 6 * NZ * T, U = 8;
    for (int base = threadIdx.x; base < TOT; base += U * NT) {
      float2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = base + u * NT;
        const int t = idx % T, r = idx / T, z = r % NZ, c = r / NZ;
        const int m = m0 + t;
        v[u] = (idx < TOT && m < plane) ? spec[((size_t)c * NZ + z) * plane + m]
                                        : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = base + u * NT;
        if (idx < TOT) {
          const int t = idx % T, r = idx / T, z = r % NZ, c = r / NZ;
          B[(c * T + t) * NZP + z] = v[u];
        }
      }
    }
    __syncthreads();
    smem_fft<NZ, false, 6 * T, NZP, 1>(B, twz);
  }
  for (int idx = threadIdx.x; idx < T * NZ; idx += blockDim.x) {
    const int sz = idx % NZ, t = idx / NZ;
    if (m0 + t >= plane) continue;
    const float4 q = pen[t];
    const int kz = freq_of<NZ>(sz);
    const int mz = (2 * kz < NZ) ? kz : kz - NZ;
    const bool nyqz = (NZ % 2 == 0) && NZ > 1 && (2 * kz == NZ);
    float2 tv[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) tv[c] = B[(c * T + t) * NZP + sz];
    const int nnz = (int)q.w + (mz != 0);
    if (nnz == 0) {
#pragma unroll
      for (int c = 0; c < 6; ++c)
        tv[c] = make_float2(mode == GM_FULL_MAP ? ga.En[c] : 0.f, 0.f);
    } else if (g.nyquist == 0 && nnz >= 2 && (q.z != 0.f || nyqz)) {
#pragma unroll
      for (int c = 0; c < 6; ++c) tv[c] = make_float2(0.f, 0.f);
    } else {
      const float x1 = q.x, x2 = q.y, x3 = mz * g.inv_lz;
      const float inv = rsqrtf(x1 * x1 + x2 * x2 + x3 * x3);
      green_apply(tv, x1 * inv, x2 * inv, x3 * inv, ga.a, ga.inv_mu0);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) B[(c * T + t) * NZP + sz] = tv[c];
  }
  __syncthreads();
  if constexpr (DIRECT) {
    for (int q = threadIdx.x; q < 6 * T * Z1; q += NT) {   // inverse step 1 in shared memory
      const int b = q % (6 * T), k1 = q / (6 * T);
      float2* p = B + b * NZP + k1 * Z2;
      float2 v[Z2];
#pragma unroll
      for (int i = 0; i < Z2; ++i) v[i] = p[i];
      RegDft<Z2, true>::run(v);
#pragma unroll
      for (int n2 = 1; n2 < Z2; ++n2) v[n2] = cmulc(v[n2], twz[n2 * Z1 + k1]);
#pragma unroll
      for (int i = 0; i < Z2; ++i) p[i] = v[i];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 6 * T * Z2; q += NT) {   // inverse step 2 -> global
      const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
      const int m = m0 + t;
      const float2* p = B + (c * T + t) * NZP + n2;
      float2 v[Z1];
#pragma unroll
      for (int i = 0; i < Z1; ++i) v[i] = p[i * Z2];
      RegDft<Z1, true>::run(v);
      if (m < plane) {
        float2* dst = spec + ((size_t)c * NZ + n2) * plane + m;
        const size_t zs = (size_t)Z2 * plane;
#pragma unroll
        for (int i = 0; i < Z1; ++i) dst[i * zs] = v[i];
      }
    }
  } else {
    smem_fft<NZ, true, 6 * T, NZP, 1>(B, twz);
    for (int idx = threadIdx.x; idx < 6 * NZ * T; idx += blockDim.x) {
      const int t = idx % T, r = idx / T, z = r % NZ, c = r / NZ;
      const int m = m0 + t;
      if (m < plane) spec[((size_t)c * NZ + z) * plane + m] = B[(c * T + t) * NZP + z];
    }
  }
}

template <int NZ, int TT>
__global__ void __launch_bounds__(kThreads) k_pass_b(GridDev g, float2* __restrict__ spec, int mode,
                                                     GammaArgs ga) {
  pass_b_body<NZ, TT, kThreads>(g, spec, mode, ga);
}

template <int NZ, int TT>
__global__ void __launch_bounds__(2 * kThreads, 2) k_pass_b_wide(GridDev g,
                                                                float2* __restrict__ spec,
                                                                int mode, GammaArgs ga) {
  pass_b_body<NZ, TT, 2 * kThreads>(g, spec, mode, ga);
}


// Pass B with T = 128 / split_n1(nz) pencils per block and 256 threads.
// Forward z step 1 reads the spectrum from global memory; forward step 2, the
// Green operator and inverse step 1 run in registers on one (pencil, k1)
// group per pair of threads, lanes l and l + 16 holding the normal and the
// shear components of the same frequencies and exchanging their partial sums
// of tau_hat n with one shuffle per value; inverse step 2 writes back to
// global memory.
template <int NZ>
struct PencilFused {
  static constexpr int Z1 = Split<NZ>::N1, Z2 = Split<NZ>::N2;
  static constexpr int T = 128 / Z1;
  static constexpr int NZP = NZ + 1;
};

template <int NZ>
__global__ void __launch_bounds__(kThreads, 3) k_pencil_green(GridDev g, float2* __restrict__ spec,
                                                             int mode, GammaArgs ga) {
  using C = PencilFused<NZ>;
  constexpr int Z1 = C::Z1, Z2 = C::Z2, T = C::T, NZP = C::NZP;
  static_assert(T * Z1 * 2 == kThreads, "one thread pair per (pencil, k1) group");
  extern __shared__ __align__(128) float2 sm[];
  float2* B = sm;                       // [6][T][NZP]
  float2* twz = B + 6 * T * NZP;
  __shared__ float4 pen[T];             // per pencil: (xi_x, xi_y, has-Nyquist, non-zero count)
  const int m0 = blockIdx.x * T;
  const int plane = g.plane;
  allow_dependent_launch();
  for (int i = threadIdx.x; i < NZ; i += blockDim.x) twz[i] = g.tw_z[i];
  if (threadIdx.x < T) {
    const int m = m0 + threadIdx.x;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m < plane) {
      const int sxn = g.nxh + 1;
      const int sy = m / sxn, sx = m - sy * sxn;
      const int2 fx = g.fx[sx], fy = g.fy[sy];
      q = make_float4(fx.x * g.inv_lx, fy.x * g.inv_ly, (float)(fx.y | fy.y),
                      (float)((fx.x != 0) + (fy.x != 0)));
    }
    pen[threadIdx.x] = q;
  }
  grid_dependency_wait();
  __syncthreads();
  // forward step 1; task q -> (pencil t fastest, then component, then n2):
  // a half-warp covers two components, whose lines are 16 words apart in banks
  for (int q = threadIdx.x; q < 6 * T * Z2; q += blockDim.x) {
    const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
    const int m = m0 + t;
    const float2* src = spec + ((size_t)c * NZ + n2) * plane + m;
    const size_t zs = (size_t)Z2 * plane;
    float2 v[Z1];
#pragma unroll
    for (int i = 0; i < Z1; ++i) v[i] = m < plane ? src[i * zs] : make_float2(0.f, 0.f);
    RegDft<Z1, false>::run(v);
#pragma unroll
    for (int k1 = 1; k1 < Z1; ++k1) v[k1] = cmul(v[k1], twz[n2 * Z1 + k1]);
    float2* p = B + (c * T + t) * NZP + n2;
#pragma unroll
    for (int i = 0; i < Z1; ++i) p[i * Z2] = v[i];
  }
  __syncthreads();
  {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int pi = w * 16 + (lane & 15);
    const int h = lane >> 4;             // 0: tau11 tau22 tau33, 1: tau23 tau13 tau12
    const int t = pi % T, k1 = pi / T;
    float2 v[3][Z2];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2* p = B + ((3 * h + j) * T + t) * NZP + k1 * Z2;
#pragma unroll
      for (int i = 0; i < Z2; ++i) v[j][i] = p[i];
      RegDft<Z2, false>::run(v[j]);
    }
    const float4 q = pen[t];
#pragma unroll
    for (int k2 = 0; k2 < Z2; ++k2) {
      const int kz = k1 + Z1 * k2;
      const int mz = (2 * kz < NZ) ? kz : kz - NZ;
      const bool nyqz = (NZ % 2 == 0) && (2 * kz == NZ);
      const int nnz = (int)q.w + (mz != 0);
      const bool zero_f = nnz == 0;
      const bool masked = !zero_f && g.nyquist == 0 && nnz >= 2 && (q.z != 0.f || nyqz);
      float n1 = 0.f, n2 = 0.f, n3 = 0.f;
      if (!zero_f) {
        const float x1 = q.x, x2 = q.y, x3 = mz * g.inv_lz;
        const float inv = rsqrtf(x1 * x1 + x2 * x2 + x3 * x3);
        n1 = x1 * inv;
        n2 = x2 * inv;
        n3 = x3 * inv;
      }
      const float2 a0 = v[0][k2], a1 = v[1][k2], a2 = v[2][k2];
      float2 p1, p2, p3;   // this half's share of v = tau_hat n
      if (h == 0) {
        p1 = make_float2(a0.x * n1, a0.y * n1);
        p2 = make_float2(a1.x * n2, a1.y * n2);
        p3 = make_float2(a2.x * n3, a2.y * n3);
      } else {
        p1 = make_float2(a2.x * n2 + a1.x * n3, a2.y * n2 + a1.y * n3);
        p2 = make_float2(a2.x * n1 + a0.x * n3, a2.y * n1 + a0.y * n3);
        p3 = make_float2(a1.x * n1 + a0.x * n2, a1.y * n1 + a0.y * n2);
      }
      p1.x += __shfl_xor_sync(0xffffffffu, p1.x, 16);
      p1.y += __shfl_xor_sync(0xffffffffu, p1.y, 16);
      p2.x += __shfl_xor_sync(0xffffffffu, p2.x, 16);
      p2.y += __shfl_xor_sync(0xffffffffu, p2.y, 16);
      p3.x += __shfl_xor_sync(0xffffffffu, p3.x, 16);
      p3.y += __shfl_xor_sync(0xffffffffu, p3.y, 16);
      const float sx = n1 * p1.x + n2 * p2.x + n3 * p3.x;
      const float sy = n1 * p1.y + n2 * p2.y + n3 * p3.y;
      const float2 w1 = make_float2((p1.x - ga.a * n1 * sx) * ga.inv_mu0,
                                    (p1.y - ga.a * n1 * sy) * ga.inv_mu0);
      const float2 w2 = make_float2((p2.x - ga.a * n2 * sx) * ga.inv_mu0,
                                    (p2.y - ga.a * n2 * sy) * ga.inv_mu0);
      const float2 w3 = make_float2((p3.x - ga.a * n3 * sx) * ga.inv_mu0,
                                    (p3.y - ga.a * n3 * sy) * ga.inv_mu0);
      float2 o0, o1, o2;
      if (h == 0) {
        o0 = make_float2(-n1 * w1.x, -n1 * w1.y);
        o1 = make_float2(-n2 * w2.x, -n2 * w2.y);
        o2 = make_float2(-n3 * w3.x, -n3 * w3.y);
      } else {
        o0 = make_float2(-0.5f * (n2 * w3.x + n3 * w2.x), -0.5f * (n2 * w3.y + n3 * w2.y));
        o1 = make_float2(-0.5f * (n1 * w3.x + n3 * w1.x), -0.5f * (n1 * w3.y + n3 * w1.y));
        o2 = make_float2(-0.5f * (n1 * w2.x + n2 * w1.x), -0.5f * (n1 * w2.y + n2 * w1.y));
      }
      if (zero_f) {
        const bool full = mode == GM_FULL_MAP;
        o0 = make_float2(full ? ga.En[3 * h] : 0.f, 0.f);
        o1 = make_float2(full ? ga.En[3 * h + 1] : 0.f, 0.f);
        o2 = make_float2(full ? ga.En[3 * h + 2] : 0.f, 0.f);
      } else if (masked) {
        o0 = o1 = o2 = make_float2(0.f, 0.f);
      }
      v[0][k2] = o0;
      v[1][k2] = o1;
      v[2][k2] = o2;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      RegDft<Z2, true>::run(v[j]);
#pragma unroll
      for (int n2 = 1; n2 < Z2; ++n2) v[j][n2] = cmulc(v[j][n2], twz[n2 * Z1 + k1]);
      float2* p = B + ((3 * h + j) * T + t) * NZP + k1 * Z2;
#pragma unroll
      for (int i = 0; i < Z2; ++i) p[i] = v[j][i];
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 6 * T * Z2; q += blockDim.x) {   // inverse step 2 -> global
    const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
    const int m = m0 + t;
    const float2* p = B + (c * T + t) * NZP + n2;
    float2 v[Z1];
#pragma unroll
    for (int i = 0; i < Z1; ++i) v[i] = p[i * Z2];
    RegDft<Z1, true>::run(v);
    if (m < plane) {
      float2* dst = spec + ((size_t)c * NZ + n2) * plane + m;
      const size_t zs = (size_t)Z2 * plane;
#pragma unroll
      for (int i = 0; i < Z1; ++i) dst[i * zs] = v[i];
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename K>
static cudaError_t set_smem(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int NX>
static cudaError_t launch_plane_passes(const GridDev& g, const float* in, float* out,
                                       float2* spec, int mode, int which, cudaStream_t st) {
  using C = PlaneCfg<NX, NX>;
  const dim3 grid(6, g.nz);
  if (which == 0) {
    const size_t smem = (size_t)(C::PLANE_F2 + C::TAB_F2 + 256) * sizeof(float2);
    cudaError_t e = set_smem(k_pass_a<NX, NX>, smem);
    if (e != cudaSuccess) return e;
    k_pass_a<NX, NX><<<grid, kPlaneThreads, smem, st>>>(g, in, spec, mode);
  } else {
    const size_t smem = (size_t)(C::PLANE_F2 + C::TAB_F2) * sizeof(float2);
    cudaError_t e = set_smem(k_pass_c<NX, NX>, smem);
    if (e != cudaSuccess) return e;
    k_pass_c<NX, NX><<<grid, kPlaneThreads, smem, st>>>(g, spec, out, 1.0f / (float)g.n);
  }
  return cudaGetLastError();
}

template <int NZ, int TT>
static cudaError_t launch_pencil_tile(const GridDev& g, float2* spec, int mode,
                                      const GammaArgs& ga, cudaStream_t st) {
  using C = PencilCfg<NZ, TT>;
  const size_t smem = (size_t)(6 * C::T * C::NZP + NZ) * sizeof(float2);
  if (TT < 1 || smem > 227 * 1024) return cudaErrorInvalidValue;   // variant not available
  const int blocks = (g.plane + C::T - 1) / C::T;
  cudaError_t e;
  if constexpr (NZ >= 256 && C::T >= 8) {
    if ((e = set_smem(k_pass_b_wide<NZ, TT>, smem)) != cudaSuccess) return e;
    k_pass_b_wide<NZ, TT><<<blocks, 2 * kThreads, smem, st>>>(g, spec, mode, ga);
  } else {
    if ((e = set_smem(k_pass_b<NZ, TT>, smem)) != cudaSuccess) return e;
    k_pass_b<NZ, TT><<<blocks, kThreads, smem, st>>>(g, spec, mode, ga);
  }
  return cudaGetLastError();
}

template <int NZ>
static cudaError_t launch_pencil_pass(const GridDev& g, float2* spec, int mode, const GammaArgs& ga,
                                      cudaStream_t st) {
  constexpr int T0 = PencilCfg<NZ>::T;
  switch (g.pencil_t) {
    case 1: return launch_pencil_tile<NZ, (T0 / 2 > 0 ? T0 / 2 : 1)>(g, spec, mode, ga, st);
    case 2: return launch_pencil_tile<NZ, 2 * T0>(g, spec, mode, ga, st);
    default: return launch_pencil_tile<NZ, T0>(g, spec, mode, ga, st);
  }
}


// nz = 64 takes the 8-pencil tile of the original z pass
#define RPM_FUSED_Z_SIZES(X) X(32) X(48) X(96) X(128)

template <int NZ>
static cudaError_t launch_fused_pencil(const GridDev& g, float2* spec, int mode,
                                       const GammaArgs& ga, cudaStream_t st) {
  using C = PencilFused<NZ>;
  const size_t smem = (size_t)(6 * C::T * C::NZP + NZ) * sizeof(float2);
  cudaError_t e;
  if ((e = set_smem(k_pencil_green<NZ>, smem)) != cudaSuccess) return e;
  return launch_pdl(k_pencil_green<NZ>, dim3((g.plane + C::T - 1) / C::T), kThreads, smem, st, g,
                    spec, mode, ga);
}

static bool fused_pencil_ok(int nz) {
  switch (nz) {
#define RPM_CASE(N) case N:
    RPM_FUSED_Z_SIZES(RPM_CASE)
#undef RPM_CASE
    return true;
    default: return false;
  }
}

static cudaError_t dispatch_fused_pencil(const GridDev& g, float2* spec, int mode,
                                         const GammaArgs& ga, cudaStream_t st) {
  switch (g.nz) {
#define RPM_CASE(N) \
  case N: return launch_fused_pencil<N>(g, spec, mode, ga, st);
    RPM_FUSED_Z_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

// three-pass (whole xy planes in shared memory) when the plane fits
static bool plane_fits(int nx, int ny) { return nx == ny && nx <= 128; }

static bool xy_size_ok(int n) {
  switch (n) {
#define RPM_CASE(N) case N:
    RPM_XY_SIZES(RPM_CASE)
#undef RPM_CASE
    return true;
    default: return false;
  }
}

static bool z_size_ok(int n) {
  switch (n) {
#define RPM_CASE(N) case N:
    RPM_Z_SIZES(RPM_CASE)
#undef RPM_CASE
    return true;
    default: return false;
  }
}

static cudaError_t dispatch_plane(const GridDev& g, const float* in, float* out, float2* spec,
                                  int mode, int which, cudaStream_t st) {
  switch (g.nx) {
#define RPM_CASE(N) \
  case N: return launch_plane_passes<N>(g, in, out, spec, mode, which, st);
    RPM_PLANE_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

static cudaError_t dispatch_pencil(const GridDev& g, float2* spec, int mode, const GammaArgs& ga,
                                   cudaStream_t st) {
  switch (g.nz) {
#define RPM_CASE(N) \
  case N: return launch_pencil_pass<N>(g, spec, mode, ga, st);
    RPM_Z_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

// The plane kernels g.plane_v resolves to on this grid: 0 paired (gamma_pair.cu),
// 1 whole-plane, 2 five-pass.
static int plane_path(const GridDev& g, const float2* spec) {
  if (g.plane_v == 0 && pair_plane_ok(g, spec)) return 0;
  if (g.plane_v <= 1 && plane_fits(g.nx, g.ny)) return 1;
  return 2;
}

static bool fused_z(const GridDev& g) { return g.pencil_t == 0 && fused_pencil_ok(g.nz); }

bool fused_z_pass(const GridDev& g) { return plane_variant(g) == 1 && fused_z(g); }

// (for a spectrum buffer from cudaMalloc, whose alignment is 256 bytes)
int plane_variant(const GridDev& g) { return plane_path(g, nullptr); }

int gamma_launches(const GridDev& g) { return plane_variant(g) == 2 ? 5 : 3; }

int pencil_tile(const GridDev& g) {
  if (plane_variant(g) != 1) return g.nz <= 4 ? 128 : 2 * pair_z_tile(g);
  if (fused_z(g)) return 128 / split_n1(g.nz);
  int t0;
  switch (g.nz) {
#define RPM_CASE(N) \
  case N: t0 = PencilCfg<N>::T; break;
    RPM_Z_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return 0;
  }
  return g.pencil_t == 1 ? (t0 / 2 > 0 ? t0 / 2 : 1) : (g.pencil_t == 2 ? 2 * t0 : t0);
}


bool grid_supported(int nx, int ny, int nz) {
  return xy_size_ok(nx) && xy_size_ok(ny) && z_size_ok(nz);
}

GammaArgs gamma_args(const GridDev& g, const double E[6]) {
  GammaArgs ga;
  for (int c = 0; c < 6; ++c) ga.En[c] = (float)(E ? E[c] * (double)g.n : 0.0);
  const double l0 = g.lam0, m0 = g.mu0;
  ga.a = (float)((l0 + m0) / (l0 + 2.0 * m0));
  ga.inv_mu0 = (float)(1.0 / m0);
  return ga;
}

static cudaError_t z_pass(const GridDev& g, float2* spec, int mode, const GammaArgs& ga,
                          cudaStream_t st) {
  return fused_z(g) ? dispatch_fused_pencil(g, spec, mode, ga, st)
                    : dispatch_pencil(g, spec, mode, ga, st);
}

// the post-step (paired planes) and an added field (paired planes and five
// passes) ride on the last pass, which accesses fields as float2
static bool float2_ok(const float* a, const float* b) {
  return (((uintptr_t)a | (uintptr_t)b) & 7) == 0;
}

int polarization_launches(const GridDev& g, const float* in, const float* out,
                          const float2* spec) {
  return plane_path(g, spec) == 0 && float2_ok(in, out) ? 3 : gamma_launches(g) + 1;
}

cudaError_t launch_polarization_map(const GridDev& g, const float4* post, const float* in,
                                    float* eb, float* out, float2* spec, const double Eb[6],
                                    int mode, cudaStream_t st) {
  if (plane_path(g, spec) == 0 && float2_ok(in, out))
    return launch_pair_polarization(g, post, in, out, spec, Eb, mode, st);
  const cudaError_t e = launch_apply_gamma(g, in, eb, spec, Eb, mode, st);
  if (e != cudaSuccess) return e;
  return launch_polarization_post(g, post, in, eb, out, st);
}

static bool add_rides(const GridDev& g, const float* out, const float* add, const float2* spec) {
  return plane_path(g, spec) != 1 && float2_ok(out, add);
}

int gamma_add_launches(const GridDev& g, const float* out, const float* add, const float2* spec) {
  return gamma_launches(g) + (add && !add_rides(g, out, add, spec) ? 1 : 0);
}

cudaError_t launch_apply_gamma(const GridDev& g, const float* in, float* out, float2* spec,
                               const double E[6], int mode, cudaStream_t st, const float* add) {
  const int path = plane_path(g, spec);
  const float* riding = add && add_rides(g, out, add, spec) ? add : nullptr;
  cudaError_t e;
  if (path == 0) {
    e = launch_pair_map(g, in, out, spec, E, mode, st, riding);
  } else if (path == 2) {
    e = launch_pair_rows_map(g, in, out, spec, E, mode, st, riding);
  } else {
    const GammaArgs ga = gamma_args(g, E);
    if ((e = dispatch_plane(g, in, out, spec, mode, 0, st)) != cudaSuccess) return e;
    if ((e = z_pass(g, spec, mode, ga, st)) != cudaSuccess) return e;
    e = dispatch_plane(g, in, out, spec, mode, 1, st);
  }
  if (e != cudaSuccess || !add || riding) return e;
  return launch_axpby(out, 1.f, out, 1.f, add, g.n, st);
}

}  // namespace rpm
