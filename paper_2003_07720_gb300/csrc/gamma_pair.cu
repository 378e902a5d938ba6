// The Lippmann-Schwinger map on paired lines: the three passes of
// gamma_kernels.cu for square planes nx = ny up to 128, with every
// transform working on two lines at once in packed float32 arithmetic
// (pair_fft.cuh).
//
//   pass A  k_pair_fwd   one block per (z-plane, component): polarization,
//           x transform of rows y and y + ny/2 as one pair, then one radix-2
//           step along y across the two lanes of the pair (even and odd ky),
//           then the ny/2-point y transform of the (even, odd) pair.
//   pass B  k_pair_green z transform, Green operator, inverse z transform of
//           (even ky, odd ky) pencil pairs at one kx.
//   pass C  k_pair_inv   the inverse of pass A; optionally an added field or
//           Algorithm 3's post-step on the way out.
//
// The spectrum is [6][nz][ny/2][nx/2 + 1] float4: real parts of the even and
// the odd ky, then their imaginary parts, in slot order (split_freq).  It
// holds 2 X: the factor 1/2 of the real-to-complex untangling is left out of
// pass A and taken up by the zero frequency (2 E n) and the final scale.
//
// Each kernel lets the next one start when its own last phase begins, not
// earlier: blocks of a kernel two launches on would otherwise sit on every SM
// through a whole pass, holding slots and, by their shared memory, the split
// between shared memory and L1 (256^3: 1046 us a map with the trigger at the
// start of every kernel, 800 us so; 32^3 13.0 and 8.8 us, 24 x 96 x 48 21 and
// 15 us).
//
// What bounds the passes: with one line per thread they were bound by issue
// slots (128^3: 19.1, 21.7 and 13.8 M warp instructions in passes A, B, C,
// 47-61 % issue active).  Pairing brought them to 10.1, 11.7 and 8.5 M; now
// shared-memory bandwidth (70 and 66 % of the L1 pipe's cycles in A and C) and
// the latency of two or three resident blocks bound them.  One map among others
// of 128^3: 96 -> 87 us, of 64^3 20.5 -> 15.2 us, of 48^3 15.3 -> 12.2 us, of
// 16^3 15.8 -> 9.1 us; 96^3 passes A + B + C 71 -> 40 us (single-kernel times).
// A first map on fresh inputs, waited for, gains less, being mostly launches:
// 132 -> 121, 52.9 -> 47.5, 46.1 -> 46.5 and 46.6 -> 41.4 us.
#include <algorithm>
#include <cmath>

#include "async_copy.cuh"
#include "pair_fft.cuh"
#include "rpm_internal.h"

namespace rpm {

namespace {

// Threads per block of the plane passes and the blocks per SM their registers
// are budgeted for.  A block of 256 at 128 registers beats three of 128 at 168
// where a plane fills a third of the SM's shared memory (128^2: 87 against
// 96 us a map) and where one block has few tasks per phase (64^2: 17.1 against
// 23.1 us, 48^2: 13.3 against 16.5 us); at 96^2 four blocks of 128 fit (40.4
// against 47.1 us).  Sides up to 24 take one warp: a thread transforms a whole
// row pair, then a whole column pair, and nothing but the exchange between the
// two goes through shared memory.
constexpr int pair_threads(int n, bool few) {
  return n <= 24 ? 32 : (n == 32 ? 64 : (n == 96 && !few ? 128 : 256));
}
constexpr int pair_blocks(int n, int threads) {
  return n <= 16 ? 16 : (n <= 32 ? 8 : (n == 96 && threads == 128 ? 4 : 2));
}

// The x transform of a block's row pairs: rows nx long, ROWS pairs in shared
// memory as [ROWS][nx/2 + 1], TPB threads.
template <int NX, int ROWS_, int TPB_>
struct PairX {
  static constexpr int NXH = NX / 2, SX = NXH + 1, ROWS = ROWS_, TPB = TPB_;
  static constexpr int X1 = pair_n1(NXH), X2 = NXH / X1;
  static constexpr int NU = X1 / 2 + 1;
  static_assert(X2 == 1 || X1 % 2 == 0, "two-step x splits need an even first factor");
  static_assert(SX % 2 == 1 || X2 == 1, "odd row stride: rows fall in distinct 16-byte banks");
};

template <int N, int TPB_>
struct PairPlane {
  static constexpr int NXH = N / 2, SX = NXH + 1, H = N / 2, PL = H * SX;
  static constexpr int X1 = pair_n1(NXH), X2 = NXH / X1;
  static constexpr int Y1 = pair_n1(H), Y2 = H / Y1;
  static constexpr int TPB = TPB_, MINB = pair_blocks(N, TPB_);
  // two-step x lengths pack the columns 0 and nx/2 into one
  static constexpr bool PACK = X2 > 1;
  static constexpr int COLS = PACK ? NXH : SX;
  using X = PairX<N, H, TPB>;
};

// Task q of an x step that walks rows: (row, n2), n2 fastest.  With X2 = 4
// the two halves of a group of eight lanes take rows 4 apart, so that their
// 16-byte accesses (row stride nx/2 + 1 elements) fall in distinct banks.
template <int X2, int H>
__device__ __forceinline__ void pair_row_task(int q, int& row, int& n2) {
  n2 = q % X2;
  const int g = q / X2;
  if (X2 == 4 && H % 8 == 0)
    row = (g & ~7) + ((g >> 1) & 3) + ((g & 1) << 2);
  else
    row = g;
}

// 2 X_k and 2 X_(M-k) from Z_k = a, Z_(M-k) = b (M = nx/2), w = W_nx^k
__device__ __forceinline__ void pair_r2c(const C2& a, const C2& b, const float4* w, C2& xk,
                                         C2& xm) {
  const C2 s = {f2add(a.re, b.re), f2sub(a.im, b.im)};
  const C2 d = {f2sub(a.re, b.re), f2add(a.im, b.im)};
  const float2 t = f2sub(b.im, a.im);
  const C2 u = c2_mul<false>(d, w);
  xk = {f2add(s.re, u.im), f2sub(s.im, u.re)};
  xm = {f2sub(s.re, u.im), f2sub(t, u.re)};
}

// 2 Z_k and 2 Z_(M-k) from X_k = a, X_(M-k) = b, w = W_nx^k
__device__ __forceinline__ void pair_c2r(const C2& a, const C2& b, const float4* w, C2& zk,
                                         C2& zm) {
  const C2 s = {f2add(a.re, b.re), f2sub(a.im, b.im)};
  const C2 d = {f2sub(a.re, b.re), f2add(a.im, b.im)};
  const C2 u = c2_mul<true>(d, w);
  zk = {f2sub(s.re, u.im), f2add(s.im, u.re)};
  zm = {f2add(s.re, u.im), f2sub(u.re, s.im)};
}

// Lanes (row j, row j + ny/2) -> (even ky, odd ky): the first radix-2 step of
// the y transform, w = W_ny^j.  pair_join_rows is its (doubled) inverse.
__device__ __forceinline__ C2 pair_split_rows(const C2& v, float2 w) {
  const float er = v.re.x + v.re.y, ei = v.im.x + v.im.y;
  const float dr = v.re.x - v.re.y, di = v.im.x - v.im.y;
  return {make_float2(er, fmaf(dr, w.x, -di * w.y)), make_float2(ei, fmaf(dr, w.y, di * w.x))};
}
__device__ __forceinline__ C2 pair_join_rows(const C2& v, float2 w) {
  const float orr = fmaf(v.re.y, w.x, v.im.y * w.y), oi = fmaf(v.im.y, w.x, -v.re.y * w.y);
  return {make_float2(v.re.x + orr, v.re.x - orr), make_float2(v.im.x + oi, v.im.x - oi)};
}

__device__ __forceinline__ float4 splat_twiddle(float2 w) {
  return make_float4(w.x, w.x, w.y, w.y);
}

// Untangling of a row pair held whole in registers (Z_k in v), with the
// radix-2 step along y; X_0 and X_M in slots 0 and M.
template <int M>
__device__ __forceinline__ void pair_untangle_row(const C2* v, const float4* r2c, float2 w,
                                                  float4* p) {
  const float2 zero = f2splat(0.f), x0 = f2add(v[0].re, v[0].im), xm = f2sub(v[0].re, v[0].im);
  c2_store(p, pair_split_rows(C2{f2add(x0, x0), zero}, w));
  c2_store(p + M, pair_split_rows(C2{f2add(xm, xm), zero}, w));
#pragma unroll
  for (int k = 1; k <= M / 2; ++k) {
    C2 xk, xmk;
    pair_r2c(v[k], v[M - k], r2c + k, xk, xmk);
    c2_store(p + k, pair_split_rows(xk, w));
    if (k < M - k) c2_store(p + M - k, pair_split_rows(xmk, w));
  }
}

// (lam, 2 mu) of C - C0.  With at most two phases every thread reads both pairs
// itself and selects (phase ids are < n_phases): no table, and the strain loads
// do not wait for one.  Otherwise a table of all 256 ids in shared memory.
__device__ __forceinline__ float2 pair_material(float2 m) { return make_float2(m.x, 2.f * m.y); }
__device__ __forceinline__ void pair_materials(const GridDev& g, float2* dm, int threads) {
  if (g.n_phases > 2)
    for (int i = threadIdx.x; i < 256; i += threads) dm[i] = pair_material(g.dmat[i]);
}

// x step 1 of pass A: the strain rows j and j + ny/2 are read from global
// memory, the polarization formed on the way in (KIND: one component's rows as
// they are, a shear component, or a normal one, which needs the trace and so
// the other two normal components e1, e2).  Row j + ny/2 lies `low` float2
// after row j; rows past `rows` are skipped.
enum { kRaw, kShear, kNormal };
template <class C, int KIND, bool TWO>
__device__ __forceinline__ void pair_x1(const float2* __restrict__ e0, const float2* __restrict__ e1,
                                        const float2* __restrict__ e2,
                                        const uchar2* __restrict__ phase, int low, int rows,
                                        const float2* __restrict__ dmat, const float2* dm,
                                        float4* P, const float4* twx,
                                        const float4* r2c, const float2* hw) {
  constexpr int NXH = C::NXH, SX = C::SX, X1 = C::X1, X2 = C::X2;
  constexpr int B = KIND == kNormal && X1 > 4 ? 4 : X1;   // voxel pairs loaded per batch
  const float2 dm0 = TWO && KIND != kRaw ? pair_material(dmat[0]) : f2splat(0.f);
  const float2 dm1 = TWO && KIND != kRaw ? pair_material(dmat[1]) : f2splat(0.f);
  auto material = [&](unsigned char id) {
    return TWO ? make_float2(id ? dm1.x : dm0.x, id ? dm1.y : dm0.y) : dm[id];
  };
  // a thread keeps its n2 over its tasks where X2 divides the block size: the
  // twiddles then stay in registers
  constexpr bool KEEP = C::TPB % X2 == 0;
  float2 tw[X1];
  if (KEEP && X2 > 1) {
#pragma unroll
    for (int k1 = 1; k1 < X1; ++k1) {
      const float4 w = twx[k1 * X2 + threadIdx.x % X2];
      tw[k1] = make_float2(w.x, w.z);
    }
  }
  for (int q = threadIdx.x; q < C::ROWS * X2; q += C::TPB) {
    int j, n2;
    pair_row_task<X2, C::ROWS>(q, j, n2);
    if (j >= rows) continue;
    const int rb = j * NXH + n2;
    C2 v[X1];
#pragma unroll
    for (int i0 = 0; i0 < X1; i0 += B) {
      float2 e[B][2], f[B][2], h[B][2];
      uchar2 ph[B][2];
#pragma unroll
      for (int k = 0; k < B; ++k)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int at = rb + r * low + X2 * (i0 + k);
          e[k][r] = __ldcs(e0 + at);
          if (KIND == kNormal) {
            f[k][r] = __ldcs(e1 + at);
            h[k][r] = __ldcs(e2 + at);
          }
          if (KIND != kRaw) ph[k][r] = phase[at];
        }
#pragma unroll
      for (int k = 0; k < B; ++k) {
        float2 t[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          t[r] = e[k][r];
          if (KIND != kRaw) {
            const float2 m0 = material(ph[k][r].x), m1 = material(ph[k][r].y);
            t[r] = make_float2(m0.y * t[r].x, m1.y * t[r].y);
            if (KIND == kNormal) {
              const float2 tr = f2add(f2add(e[k][r], f[k][r]), h[k][r]);
              t[r] = make_float2(fmaf(m0.x, tr.x, t[r].x), fmaf(m1.x, tr.y, t[r].y));
            }
          }
        }
        v[i0 + k] = {make_float2(t[0].x, t[1].x), make_float2(t[0].y, t[1].y)};
      }
    }
    PairDft<X1, false>::run(v);
    float4* p = P + j * SX + n2;
    if constexpr (X2 == 1) {   // the whole row is here: untangle it in registers
      const float2 w = hw[j];
      pair_untangle_row<NXH>(v, r2c, w, p);
      continue;
    }
    c2_store(p, v[0]);
#pragma unroll
    for (int k1 = 1; k1 < X1; ++k1)
      c2_store(p + k1 * X2, KEEP ? c2_mul<false>(v[k1], f2splat(tw[k1].x), f2splat(tw[k1].y))
                                 : c2_mul<false>(v[k1], twx + k1 * X2 + n2));
  }
}

// x step 1 of component c of a block's rows (`in`, `phase`: the first row).
template <class C>
__device__ __forceinline__ void pair_x1_component(const GridDev& g, const float2* in, int c,
                                                  const uchar2* phase, int low, int rows, int mode,
                                                  const float2* dm, float4* P, const float4* twx,
                                                  const float4* r2c, const float2* hw) {
  const size_t nf2 = (size_t)g.n / 2;
  const float2* own = in + c * nf2;
  if (mode == GM_RAW_TAU) {
    pair_x1<C, kRaw, true>(own, in, in, phase, low, rows, g.dmat, dm, P, twx, r2c, hw);
  } else if (c >= 3) {
    if (g.n_phases <= 2)
      pair_x1<C, kShear, true>(own, in, in, phase, low, rows, g.dmat, dm, P, twx, r2c, hw);
    else
      pair_x1<C, kShear, false>(own, in, in, phase, low, rows, g.dmat, dm, P, twx, r2c, hw);
  } else {
    const float2* other = in + (c == 0 ? 1 : 0) * nf2;
    const float2* last = in + (c == 2 ? 1 : 2) * nf2;
    if (g.n_phases <= 2)
      pair_x1<C, kNormal, true>(own, other, last, phase, low, rows, g.dmat, dm, P, twx, r2c, hw);
    else
      pair_x1<C, kNormal, false>(own, other, last, phase, low, rows, g.dmat, dm, P, twx, r2c, hw);
  }
}

// x step 2 (two-step lengths) fused with the untangling and the radix-2 step
// along y.  Slot group k1 holds the frequencies k1 + X1 i; the partner nx/2 - k
// of k lies in group X1 - k1 (groups 0 and X1/2 pair with themselves).  X_0
// and X_nx/2 are both real: with PACK they travel as X_0 + i X_nx/2 in column
// 0, otherwise in columns 0 and nx/2.
template <class C, bool PACK>
__device__ __forceinline__ void pair_x2(float4* P, int rows, const float4* r2c, const float2* hw) {
  constexpr int NXH = C::NXH, SX = C::SX, X1 = C::X1, X2 = C::X2, H = C::ROWS;
  if constexpr (X2 > 1) {
  for (int t = threadIdx.x; t < H * C::NU; t += C::TPB) {
    const int j = t % H, u = t / H;
    if (j >= rows) continue;
    float4* p = P + j * SX;
    const float2 w = hw[j];
    if (u == 0 || u == X1 / 2) {
      C2 v[X2];
#pragma unroll
      for (int i = 0; i < X2; ++i) v[i] = c2_load(p + u * X2 + i);
      PairDft<X2, false>::run(v);
      if (u == 0) {
        const float2 x0 = f2add(v[0].re, v[0].im), xm = f2sub(v[0].re, v[0].im);
        if (PACK) {
          c2_store(p, pair_split_rows(C2{x0, xm}, w));
        } else {
          c2_store(p, pair_split_rows(C2{f2add(x0, x0), f2splat(0.f)}, w));
          c2_store(p + NXH, pair_split_rows(C2{f2add(xm, xm), f2splat(0.f)}, w));
        }
      }
#pragma unroll
      for (int i = 0; i < X2; ++i) {
        // partner of slot i: X2 - i in group 0 (i >= 1), X2 - 1 - i in group X1/2
        if (u == 0) {
          const int ip = X2 - i;
          if (i >= 1 && i <= ip) {
            C2 xk, xm;
            pair_r2c(v[i], v[ip % X2], r2c + X1 * i, xk, xm);
            c2_store(p + i, pair_split_rows(xk, w));
            if (i < ip) c2_store(p + ip, pair_split_rows(xm, w));
          }
        } else {
          const int ip = X2 - 1 - i;
          if (i <= ip) {
            C2 xk, xm;
            pair_r2c(v[i], v[ip], r2c + X1 / 2 + X1 * i, xk, xm);
            c2_store(p + u * X2 + i, pair_split_rows(xk, w));
            if (i < ip) c2_store(p + u * X2 + ip, pair_split_rows(xm, w));
          }
        }
      }
    } else {
      const int up = X1 - u;
      C2 va[X2], vb[X2];
#pragma unroll
      for (int i = 0; i < X2; ++i) {
        va[i] = c2_load(p + u * X2 + i);
        vb[i] = c2_load(p + up * X2 + i);
      }
      PairDft<X2, false>::run(va);
      PairDft<X2, false>::run(vb);
#pragma unroll
      for (int i = 0; i < X2; ++i) {
        const int ip = X2 - 1 - i;
        C2 xk, xm;
        pair_r2c(va[i], vb[ip], r2c + u + X1 * i, xk, xm);
        c2_store(p + u * X2 + i, pair_split_rows(xk, w));
        c2_store(p + up * X2 + ip, pair_split_rows(xm, w));
      }
    }
  }
  }
}

template <int N, int TPB>
__global__ void __launch_bounds__(TPB, PairPlane<N, TPB>::MINB)
    k_pair_fwd(GridDev g, const float* __restrict__ in, float4* __restrict__ spec, int mode) {
  using C = PairPlane<N, TPB>;
  using X = typename C::X;
  constexpr int NXH = C::NXH, SX = C::SX, H = C::H;
  constexpr int Y1 = C::Y1, Y2 = C::Y2;
  extern __shared__ __align__(128) float4 sm4[];
  float4* P = sm4;                     // [H][SX]
  float4* twx = P + C::PL;             // [X1][X2]
  float4* twy = twx + NXH;             // [Y1][Y2]
  float4* r2c = twy + H;               // W_nx^k, k < nx/2
  float2* hw = reinterpret_cast<float2*>(r2c + NXH);   // W_ny^j, j < ny/2
  float2* dm = hw + H;
  const int c = blockIdx.x, z = blockIdx.y;
  for (int i = threadIdx.x; i < NXH; i += TPB) {
    twx[i] = splat_twiddle(g.p_twx[i]);
    r2c[i] = splat_twiddle(g.r2c_w[i]);
  }
  for (int i = threadIdx.x; i < H; i += TPB) {
    twy[i] = splat_twiddle(g.p_twy[i]);
    hw[i] = g.p_hw[i];
  }
  grid_dependency_wait();   // the FFT tables are fixed; everything below may be in flight
  pair_materials(g, dm, TPB);
  __syncthreads();
  pair_x1_component<X>(g, reinterpret_cast<const float2*>(in) + (size_t)z * N * NXH, c,
                       reinterpret_cast<const uchar2*>(g.phase) + (size_t)z * N * NXH,
                                H * NXH, H, mode, dm, P, twx, r2c, hw);
  __syncthreads();
  float4* out = spec + ((size_t)c * g.nz + z) * C::PL;
  if constexpr (!C::PACK) {   // one y step, straight to global memory
    static_assert(Y2 == 1, "single-step x and y lengths go together");
    allow_dependent_launch();
    for (int b = threadIdx.x; b < C::COLS; b += TPB) {
      C2 v[Y1];
#pragma unroll
      for (int i = 0; i < Y1; ++i) v[i] = c2_load(P + i * SX + b);
      PairDft<Y1, false>::run(v);
#pragma unroll
      for (int i = 0; i < Y1; ++i) c2_store(out + i * SX + b, v[i]);
    }
    return;
  }
  pair_x2<X, true>(P, H, r2c, hw);
  __syncthreads();
  for (int t = threadIdx.x; t < NXH * Y2; t += TPB) {   // y step 1
    const int b = t % NXH, n2 = t / NXH;
    float4* p = P + b + n2 * SX;
    C2 v[Y1];
#pragma unroll
    for (int i = 0; i < Y1; ++i) v[i] = c2_load(p + i * Y2 * SX);
    PairDft<Y1, false>::run(v);
    c2_store(p, v[0]);
#pragma unroll
    for (int k1 = 1; k1 < Y1; ++k1)
      c2_store(p + k1 * Y2 * SX, c2_mul<false>(v[k1], twy + k1 * Y2 + n2));
  }
  __syncthreads();
  allow_dependent_launch();
  for (int t = threadIdx.x; t < NXH * Y1; t += TPB) {   // y step 2 -> global
    const int b = t % NXH, k1 = t / NXH;
    float4* p = P + b + k1 * Y2 * SX;
    C2 v[Y2];
#pragma unroll
    for (int i = 0; i < Y2; ++i) v[i] = c2_load(p + i * SX);
    PairDft<Y2, false>::run(v);
    float4* d = b == 0 ? p : out + (size_t)k1 * Y2 * SX + b;
#pragma unroll
    for (int i = 0; i < Y2; ++i) c2_store(d + i * SX, v[i]);
  }
  __syncthreads();
  // separate the packed column: 2 X_0 = C_k + conj C_-k, 2 X_nx/2 = (C_k - conj C_-k) / i;
  // -k of an even ky = 2q is the even line's ny/2 - q, of 2q + 1 the odd line's ny/2 - 1 - q
  for (int s = threadIdx.x; s < H; s += TPB) {
    const int q = split_freq(H, C::Y1, s);
    const C2 a = c2_load(P + s * SX);
    const C2 be = c2_load(P + split_slot(H, C::Y1, (H - q) % H) * SX);
    const C2 bo = c2_load(P + split_slot(H, C::Y1, H - 1 - q) * SX);
    const C2 b = {make_float2(be.re.x, bo.re.y), make_float2(be.im.x, bo.im.y)};
    c2_store(out + (size_t)s * SX, C2{f2add(a.re, b.re), f2sub(a.im, b.im)});
    c2_store(out + (size_t)s * SX + NXH, C2{f2add(a.im, b.im), f2sub(b.re, a.re)});
  }
}

// The reverse of pair_untangle_row: 2 Z_k of a row pair from its M + 1 slots.
template <int M>
__device__ __forceinline__ void pair_tangle_row(const float4* p, const float4* r2c, float2 w,
                                                C2* v) {
  const float2 x0 = pair_join_rows(c2_load(p), w).re, xm = pair_join_rows(c2_load(p + M), w).re;
  v[0] = {f2add(x0, xm), f2sub(x0, xm)};
#pragma unroll
  for (int k = 1; k <= M / 2; ++k) {
    C2 zk, zm;
    const C2 a = pair_join_rows(c2_load(p + k), w), b = pair_join_rows(c2_load(p + M - k), w);
    pair_c2r(a, b, r2c + k, zk, zm);
    v[k] = zk;
    if (k < M - k) v[M - k] = zm;
  }
}

// The last radix-2 step along y and the tangling, fused into x step 1 of the
// inverse (two-step lengths); the reverse of pair_x2.
template <class C, bool PACK>
__device__ __forceinline__ void pair_x1_inv(float4* P, int rows, const float4* twx,
                                            const float4* r2c, const float2* hw) {
  constexpr int NXH = C::NXH, SX = C::SX, X1 = C::X1, X2 = C::X2, H = C::ROWS;
  if constexpr (X2 > 1) {
  for (int t = threadIdx.x; t < H * C::NU; t += C::TPB) {
    const int j = t % H, u = t / H;
    if (j >= rows) continue;
    float4* p = P + j * SX;
    const float2 w = hw[j];
    if (u == 0 || u == X1 / 2) {
      C2 v[X2], o[X2];
#pragma unroll
      for (int i = 0; i < X2; ++i) v[i] = pair_join_rows(c2_load(p + u * X2 + i), w);
      if (u == 0) {
        const float2 xm = PACK ? v[0].im : pair_join_rows(c2_load(p + NXH), w).re;
        o[0] = {f2add(v[0].re, xm), f2sub(v[0].re, xm)};   // from X_0 and X_nx/2, both real
#pragma unroll
        for (int i = 1; i < X2; ++i) {
          const int ip = X2 - i;
          if (i <= ip) {
            C2 zk, zm;
            pair_c2r(v[i], v[ip], r2c + X1 * i, zk, zm);
            o[i] = zk;
            if (i < ip) o[ip] = zm;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < X2; ++i) {
          const int ip = X2 - 1 - i;
          if (i <= ip) {
            C2 zk, zm;
            pair_c2r(v[i], v[ip], r2c + X1 / 2 + X1 * i, zk, zm);
            o[i] = zk;
            if (i < ip) o[ip] = zm;
          }
        }
      }
      PairDft<X2, true>::run(o);
      c2_store(p + u * X2, o[0]);
#pragma unroll
      for (int n2 = 1; n2 < X2; ++n2)
        c2_store(p + u * X2 + n2, c2_mul<true>(o[n2], twx + u * X2 + n2));
    } else {
      const int up = X1 - u;
      C2 va[X2], vb[X2];
#pragma unroll
      for (int i = 0; i < X2; ++i) {
        va[i] = pair_join_rows(c2_load(p + u * X2 + i), w);
        vb[i] = pair_join_rows(c2_load(p + up * X2 + i), w);
      }
#pragma unroll
      for (int i = 0; i < X2; ++i) {
        const int ip = X2 - 1 - i;
        C2 zk, zm;
        pair_c2r(va[i], vb[ip], r2c + u + X1 * i, zk, zm);
        va[i] = zk;
        vb[ip] = zm;
      }
      PairDft<X2, true>::run(va);
      PairDft<X2, true>::run(vb);
      c2_store(p + u * X2, va[0]);
      c2_store(p + up * X2, vb[0]);
#pragma unroll
      for (int n2 = 1; n2 < X2; ++n2) {
        c2_store(p + u * X2 + n2, c2_mul<true>(va[n2], twx + u * X2 + n2));
        c2_store(p + up * X2 + n2, c2_mul<true>(vb[n2], twx + up * X2 + n2));
      }
    }
  }
  }
}

// Algorithm 3's last step at one voxel: out = (C + C0)^-1 : (s_a + C0 : eps_b)
// with s_a = lam_a tr(eps) I + 2 mu_a eps and (C + C0) = (lam_s, mu_s); the
// inverse of an isotropic stiffness maps t to (t - k_s tr(t) I) h_s with
// k_s = lam_s / (3 lam_s + 2 mu_s), h_s = 1 / (2 mu_s).  pm = (lam_a, mu_a,
// k_s, h_s) of the voxel's phase.
__device__ __forceinline__ void post_normal(const float e[3], const float b[3], float4 pm,
                                            float lam0, float mu0, float o[3]) {
  const float tre = e[0] + e[1] + e[2];
  const float trb = b[0] + b[1] + b[2];
  float t[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    t[k] = 2.f * pm.y * e[k] + 2.f * mu0 * b[k];
    t[k] += pm.x * tre + lam0 * trb;
  }
  const float sh = pm.z * (t[0] + t[1] + t[2]);
#pragma unroll
  for (int k = 0; k < 3; ++k) o[k] = (t[k] - sh) * pm.w;
}

__device__ __forceinline__ float post_shear(float e, float b, float4 pm, float mu0) {
  return (2.f * pm.y * e + 2.f * mu0 * b) * pm.w;
}

// Pass C, one block per (component, z).  The spectrum plane arrives by one
// bulk asynchronous copy; the fields leave with streaming stores, so that they
// do not push the spectrum of the next map out of L2 (128^3: 95 -> 91 us).  Without POST a non-null `eps` is a field added to
// the output on the way out (the defect of a re-centred iterate).
//
// POST: the pass ends with Algorithm 3's post-step instead (Section 5.5),
// the transformed planes being eps_b and `eps` the map's input.  Blocks are
// numbered z * 6 + c and run in clusters of three: the shear blocks apply
// the post-step to their own component on the way out; the three normal
// blocks of a plane, which need tr(eps_b), keep their real planes in shared
// memory and each finishes all three normal components on a third of the
// plane, reading the other two planes from the cluster's shared memory.
template <int N, int TPB, bool POST>
__global__ void __launch_bounds__(TPB, PairPlane<N, TPB>::MINB)
    k_pair_inv(GridDev g, const float4* __restrict__ spec, float* __restrict__ outp, float scale,
               const float* __restrict__ eps, const float4* __restrict__ post) {
  using C = PairPlane<N, TPB>;
  using X = typename C::X;
  constexpr int NXH = C::NXH, SX = C::SX, H = C::H, PL = C::PL;
  constexpr int X1 = C::X1, X2 = C::X2, Y1 = C::Y1, Y2 = C::Y2;
  extern __shared__ __align__(128) float4 sm4[];
  float4* P = sm4;
  float4* twx = P + PL;
  float4* twy = twx + NXH;
  float4* r2c = twy + H;
  float4* pt = r2c + NXH;              // POST
  float2* hw = reinterpret_cast<float2*>(pt + (POST ? 256 : 0));
  __shared__ __align__(8) uint64_t bar;
  __shared__ int fail;
  const int c = POST ? (int)blockIdx.x % 6 : (int)blockIdx.x / g.nz;
  const int z = POST ? (int)blockIdx.x / 6 : (int)blockIdx.x - c * g.nz;
  const bool gather = POST && c < 3;   // a normal block of a post-step cluster
  if (threadIdx.x == 0) {
    fail = 0;
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  for (int i = threadIdx.x; i < NXH; i += TPB) {
    twx[i] = splat_twiddle(g.p_twx[i]);
    r2c[i] = splat_twiddle(g.r2c_w[i]);
  }
  for (int i = threadIdx.x; i < H; i += TPB) {
    twy[i] = splat_twiddle(g.p_twy[i]);
    hw[i] = g.p_hw[i];
  }
  if (POST)
    for (int i = threadIdx.x; i < 256; i += TPB) pt[i] = post[i];
  grid_dependency_wait();
  if (threadIdx.x == 0) {
    mbar_arrive_expect_tx(&bar, PL * 16);
    bulk_load(P, spec + ((size_t)c * g.nz + z) * PL, PL * 16, &bar);
  }
  __syncthreads();
  if (!mbar_wait(&bar, 0)) fail = 1;
  __syncthreads();
  if (fail) {   // the copy never completed: record it and leave the plane alone
    if (threadIdx.x == 0) {
      atomicExch(g.err, 1);
      mbar_wait(&bar, 0);
    }
    if (gather) {   // the cluster's two barriers are still met
      cluster_sync();
      cluster_sync();
    }
    return;
  }
  if constexpr (!C::PACK) {
    for (int b = threadIdx.x; b < C::COLS; b += TPB) {
      C2 v[Y1];
#pragma unroll
      for (int i = 0; i < Y1; ++i) v[i] = c2_load(P + i * SX + b);
      PairDft<Y1, true>::run(v);
#pragma unroll
      for (int i = 0; i < Y1; ++i) c2_store(P + i * SX + b, v[i]);
    }
  } else {
  for (int t = threadIdx.x; t < NXH * Y1; t += TPB) {   // y step 1 (inverse)
    const int b = t % NXH, k1 = t / NXH;
    float4* p = P + k1 * Y2 * SX + b;
    C2 v[Y2];
#pragma unroll
    for (int i = 0; i < Y2; ++i) v[i] = c2_load(p + i * SX);
    if (b == 0) {   // X_0 + i X_nx/2: their inverse y transforms are real
#pragma unroll
      for (int i = 0; i < Y2; ++i) v[i] = c2_add_mi<true>(v[i], c2_load(p + i * SX + NXH));
    }
    PairDft<Y2, true>::run(v);
    c2_store(p, v[0]);
#pragma unroll
    for (int n2 = 1; n2 < Y2; ++n2) c2_store(p + n2 * SX, c2_mul<true>(v[n2], twy + k1 * Y2 + n2));
  }
  __syncthreads();
  for (int t = threadIdx.x; t < NXH * Y2; t += TPB) {   // y step 2 (inverse)
    const int b = t % NXH, n2 = t / NXH;
    float4* p = P + b + n2 * SX;
    C2 v[Y1];
#pragma unroll
    for (int i = 0; i < Y1; ++i) v[i] = c2_load(p + i * Y2 * SX);
    PairDft<Y1, true>::run(v);
#pragma unroll
    for (int i = 0; i < Y1; ++i) c2_store(p + i * Y2 * SX, v[i]);
  }
  __syncthreads();
  pair_x1_inv<X, true>(P, H, twx, r2c, hw);
  }
  __syncthreads();
  allow_dependent_launch();
  constexpr int LOW = H * NXH;         // row j + ny/2 lies LOW float2 after row j
  const size_t nf2 = (size_t)g.n / 2, zoff = (size_t)z * N * NXH;
  float2* out2 = reinterpret_cast<float2*>(outp) + zoff;
  const float2* e2 = reinterpret_cast<const float2*>(eps) + zoff;
  const uchar2* ph2 = reinterpret_cast<const uchar2*>(g.phase) + zoff;
  const bool addend = !POST && eps != nullptr;
  for (int q = threadIdx.x; q < H * X2; q += TPB) {   // x step 2 (inverse)
    int j, n2;
    pair_row_task<X2, H>(q, j, n2);
    float4* p = P + j * SX + n2;
    const int r = j * NXH + n2;
    float2 ea[X1], eb[X1];   // the added field, or the shear post-step's input and phases,
    uchar2 pa[X1], pb[X1];   // loaded ahead of the transform
    if ((POST || addend) && !gather) {
#pragma unroll
      for (int i = 0; i < X1; ++i) {
        ea[i] = e2[c * nf2 + r + i * X2];
        eb[i] = e2[c * nf2 + r + LOW + i * X2];
        if (POST) {
          pa[i] = ph2[r + i * X2];
          pb[i] = ph2[r + LOW + i * X2];
        }
      }
    }
    C2 v[X1];
    if constexpr (X2 == 1) {
      pair_tangle_row<NXH>(p, r2c, hw[j], v);
    } else {
#pragma unroll
      for (int i = 0; i < X1; ++i) v[i] = c2_load(p + i * X2);
    }
    PairDft<X1, true>::run(v);
    float2* o = out2 + c * nf2 + r;
    if (gather) {   // -> the block's own slots, for the cluster's post-step
      const float2 sc = f2splat(scale);
#pragma unroll
      for (int i = 0; i < X1; ++i)
        c2_store(p + i * X2, C2{f2mul(v[i].re, sc), f2mul(v[i].im, sc)});
      continue;
    }
#pragma unroll
    for (int i = 0; i < X1; ++i) {
      float2 a = make_float2(v[i].re.x * scale, v[i].im.x * scale);
      float2 b = make_float2(v[i].re.y * scale, v[i].im.y * scale);
      if (POST) {   // shear component: post-step on the way out
        a = make_float2(post_shear(ea[i].x, a.x, pt[pa[i].x], g.mu0),
                        post_shear(ea[i].y, a.y, pt[pa[i].y], g.mu0));
        b = make_float2(post_shear(eb[i].x, b.x, pt[pb[i].x], g.mu0),
                        post_shear(eb[i].y, b.y, pt[pb[i].y], g.mu0));
      } else if (addend) {
        a = make_float2(a.x + ea[i].x, a.y + ea[i].y);
        b = make_float2(b.x + eb[i].x, b.y + eb[i].y);
      }
      __stcs(o + i * X2, a);
      __stcs(o + LOW + i * X2, b);
    }
  }
  if (!gather) return;
  // eps_b of the three normal components sits in the cluster's blocks 0, 1, 2
  // (rank = c), at slot j * SX + h for the float2 pair h of rows j (lanes x)
  // and j + ny/2 (lanes y).  Each thread takes U such elements (four voxels
  // each) at a time, all loads issued before any use, the map's input and the
  // phases one batch ahead.
  constexpr int U = 2, STRIDE = 3 * TPB, TOT = H * NXH;
  float2 e[U][2][3];
  uchar2 ph[U][2];
  auto load_input = [&](int f0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int f = f0 + u * STRIDE;
      if (f < TOT) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
#pragma unroll
          for (int k = 0; k < 3; ++k) e[u][r][k] = e2[k * nf2 + f + r * LOW];
          ph[u][r] = ph2[f + r * LOW];
        }
      }
    }
  };
  int f0 = threadIdx.x + c * TPB;
  load_input(f0);   // in flight while the cluster meets
  cluster_sync();
  uint32_t rb[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) rb[k] = cluster_map(P, (uint32_t)k);
  while (f0 < TOT) {
    float4 b[U][3];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int f = f0 + u * STRIDE;
      if (f < TOT) {
        const int s = f + f / NXH;   // j * SX + h
#pragma unroll
        for (int k = 0; k < 3; ++k) b[u][k] = ld_cluster_f4(rb[k] + 16u * (uint32_t)s);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int f = f0 + u * STRIDE;
      if (f < TOT) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float ex[3] = {e[u][r][0].x, e[u][r][1].x, e[u][r][2].x};
          const float ey[3] = {e[u][r][0].y, e[u][r][1].y, e[u][r][2].y};
          float bx[3], by[3], ox[3], oy[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            bx[k] = r ? b[u][k].y : b[u][k].x;
            by[k] = r ? b[u][k].w : b[u][k].z;
          }
          post_normal(ex, bx, pt[ph[u][r].x], g.lam0, g.mu0, ox);
          post_normal(ey, by, pt[ph[u][r].y], g.lam0, g.mu0, oy);
#pragma unroll
          for (int k = 0; k < 3; ++k)
            __stcs(out2 + k * nf2 + f + r * LOW, make_float2(ox[k], oy[k]));
        }
      }
    }
    f0 += U * STRIDE;
    load_input(f0);
  }
  cluster_sync();   // no block leaves while another still reads its planes
}

// ---------------------------------------------------------------------------
// The same map in five passes, for planes that do not fit in shared memory
// (256^2) and for nx != ny: x rows, y lines, the z pass, y lines and x rows
// back.  Same spectrum; the columns 0 and nx/2 are not packed.
// ---------------------------------------------------------------------------

// x rows, one block per (component, R row pairs, z): both x steps, the rows
// j and j + ny/2 of a pair side by side; the finished rows leave in one bulk
// copy.  Inverse: one bulk copy in, both steps, the rows straight to global
// memory.  Bound by DRAM back (256^3: 182 -> 122 us, one pass over the field
// and one over the spectrum take 119 us at the copy rate) and by the L1 pipe
// forward (246 -> 183 us: a normal component reads three strain fields).
// 160 threads, one round for both x steps, leave room for three blocks an SM
// instead of four: 200 and 132 us.
template <int NX, int R>
struct PairRows {
    static constexpr int TPB = PairX<NX, R, 1>::X2 == 1 ? (R < 32 ? 32 : R) : 8 * R;
  static constexpr int MINB = 512 / TPB;
  using X = PairX<NX, R, TPB>;
  static size_t smem(bool table) {
    return (size_t)(R * X::SX + 2 * X::NXH) * sizeof(float4) + R * sizeof(float2) +
           (table ? 256 * sizeof(float2) : 0);
  }
};

template <int NX, int R>
__global__ void __launch_bounds__(PairRows<NX, R>::TPB, PairRows<NX, R>::MINB)
    k_pair_rows_fwd(GridDev g, const float* __restrict__ in, float4* __restrict__ spec, int mode) {
  using X = typename PairRows<NX, R>::X;
  constexpr int NXH = X::NXH, SX = X::SX, TPB = X::TPB;
  extern __shared__ __align__(128) float4 sm4[];
  float4* P = sm4;                     // [R][SX]
  float4* twx = P + R * SX;
  float4* r2c = twx + NXH;
  float2* hw = reinterpret_cast<float2*>(r2c + NXH);
  float2* dm = hw + R;
  const int c = blockIdx.x, j0 = blockIdx.y * R, z = blockIdx.z;
  const int h = g.ny / 2, rows = min(R, h - j0);
  for (int i = threadIdx.x; i < NXH; i += TPB) {
    twx[i] = splat_twiddle(g.p_twx[i]);
    r2c[i] = splat_twiddle(g.r2c_w[i]);
  }
  for (int i = threadIdx.x; i < rows; i += TPB) hw[i] = g.p_hw[j0 + i];
  grid_dependency_wait();
  pair_materials(g, dm, TPB);
  __syncthreads();
  const size_t row0 = ((size_t)z * g.ny + j0) * NXH;
  pair_x1_component<X>(g, reinterpret_cast<const float2*>(in) + row0, c,
                              reinterpret_cast<const uchar2*>(g.phase) + row0, h * NXH, rows,
                              mode, dm, P, twx, r2c, hw);
  __syncthreads();
  allow_dependent_launch();
  pair_x2<X, false>(P, rows, r2c, hw);
  fence_async_smem();
  __syncthreads();
  if (threadIdx.x == 0) {
    bulk_store(spec + (((size_t)c * g.nz + z) * h + j0) * SX, P, (uint32_t)rows * SX * 16);
    bulk_commit();
    bulk_wait_all();
  }
}

template <int NX, int R>
__global__ void __launch_bounds__(PairRows<NX, R>::TPB, PairRows<NX, R>::MINB)
    k_pair_rows_inv(GridDev g, const float4* __restrict__ spec, float* __restrict__ outp,
                    float scale, const float* __restrict__ add) {
  using X = typename PairRows<NX, R>::X;
  constexpr int NXH = X::NXH, SX = X::SX, TPB = X::TPB, X1 = X::X1, X2 = X::X2;
  extern __shared__ __align__(128) float4 sm4[];
  float4* P = sm4;
  float4* twx = P + R * SX;
  float4* r2c = twx + NXH;
  float2* hw = reinterpret_cast<float2*>(r2c + NXH);
  __shared__ __align__(8) uint64_t bar;
  __shared__ int fail;
  const int c = blockIdx.x, j0 = blockIdx.y * R, z = blockIdx.z;
  const int h = g.ny / 2, rows = min(R, h - j0);
  if (threadIdx.x == 0) {
    fail = 0;
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  for (int i = threadIdx.x; i < NXH; i += TPB) {
    twx[i] = splat_twiddle(g.p_twx[i]);
    r2c[i] = splat_twiddle(g.r2c_w[i]);
  }
  for (int i = threadIdx.x; i < rows; i += TPB) hw[i] = g.p_hw[j0 + i];
  grid_dependency_wait();
  if (threadIdx.x == 0) {
    mbar_arrive_expect_tx(&bar, (uint32_t)rows * SX * 16);
    bulk_load(P, spec + (((size_t)c * g.nz + z) * h + j0) * SX, (uint32_t)rows * SX * 16, &bar);
  }
  __syncthreads();
  if (!mbar_wait(&bar, 0)) fail = 1;
  __syncthreads();
  if (fail) {   // the copy never completed: record it and leave the rows alone
    if (threadIdx.x == 0) {
      atomicExch(g.err, 1);
      mbar_wait(&bar, 0);
    }
    return;
  }
  pair_x1_inv<X, false>(P, rows, twx, r2c, hw);
  if (X2 > 1) __syncthreads();
  allow_dependent_launch();
  const size_t nf2 = (size_t)g.n / 2;
  const int low = h * NXH;
  const size_t at0 = c * nf2 + ((size_t)z * g.ny + j0) * NXH;
  float2* out2 = reinterpret_cast<float2*>(outp) + at0;
  const float2* a2 = reinterpret_cast<const float2*>(add) + at0;
  for (int q = threadIdx.x; q < R * X2; q += TPB) {   // x step 2 (inverse)
    int j, n2;
    pair_row_task<X2, R>(q, j, n2);
    if (j >= rows) continue;
    const float4* p = P + j * SX + n2;
    const int r = j * NXH + n2;
    C2 v[X1];
    if constexpr (X2 == 1) {
      pair_tangle_row<NXH>(p, r2c, hw[j], v);
    } else {
#pragma unroll
      for (int i = 0; i < X1; ++i) v[i] = c2_load(p + i * X2);
    }
    PairDft<X1, true>::run(v);
#pragma unroll
    for (int i = 0; i < X1; ++i) {
      float2 a = make_float2(v[i].re.x * scale, v[i].im.x * scale);
      float2 b = make_float2(v[i].re.y * scale, v[i].im.y * scale);
      if (add) {
        const float2 ea = a2[r + i * X2], eb = a2[r + low + i * X2];
        a = make_float2(a.x + ea.x, a.y + ea.y);
        b = make_float2(b.x + eb.x, b.y + eb.y);
      }
      __stcs(out2 + r + i * X2, a);
      __stcs(out2 + r + low + i * X2, b);
    }
  }
}

// (Splitting the map into slabs of z planes so that the spectrum of a slab
// stays in L2 between the x and the y pass loses more at the kernel boundaries
// than it saves: 256^3 826 us whole, 862 / 929 / 1086 us in slabs of 64 / 32 / 16.)

// y lines of H = ny/2 pairs: T columns of the spectrum per block, numbered
// over all planes (column = (component, z) plane * (nx/2 + 1) + x slot), so
// that only the last block is ragged.  The first register step reads global
// memory, the second writes it; shared memory holds the exchange between the
// two (none for single-step lengths).
// T: 256-byte rows forward, 128-byte rows back (256^3: 126 and 122 us a pass;
// the other way round 139 and 139 us).
template <int H, bool INV>
struct PairLines {
  static constexpr int Y1 = pair_n1(H), Y2 = H / Y1;
  static constexpr bool ONE = H <= 16;   // a thread takes a whole line
  static constexpr int TPB = 128, T = ONE ? TPB : (INV ? 8 : 16), HP = H | 1;
  static constexpr size_t SMEM = ONE ? 0 : (size_t)(T * HP + H) * sizeof(float4);
};

template <int H, bool INV>
__global__ void __launch_bounds__(PairLines<H, INV>::TPB, 4)
    k_pair_lines(GridDev g, float4* __restrict__ spec) {
  using C = PairLines<H, INV>;
  constexpr int Y1 = C::Y1, Y2 = C::Y2, T = C::T, TPB = C::TPB, HP = C::HP;
  extern __shared__ __align__(128) float4 sm4[];
  float4* B = sm4;                     // [T][HP]
  float4* twy = B + T * HP;
  const int SX = g.nxh + 1, cols = 6 * g.nz * SX;
  const int m0 = blockIdx.x * T;
  if (!C::ONE)
    for (int i = threadIdx.x; i < H; i += TPB) twy[i] = splat_twiddle(g.p_twy[i]);
  grid_dependency_wait();
  if (!C::ONE) __syncthreads();
  auto column = [&](int t) {   // first element of column m0 + t (rows SX apart)
    const int m = m0 + t, pl = m / SX;
    return spec + (size_t)pl * H * SX + (m - pl * SX);
  };
  if constexpr (C::ONE) {
    if (m0 + (int)threadIdx.x < cols) {
      float4* p = column(threadIdx.x);
      C2 v[H];
#pragma unroll
      for (int i = 0; i < H; ++i) v[i] = c2_load(p + (size_t)(INV ? split_slot(H, Y1, i) : i) * SX);
      allow_dependent_launch();
      PairDft<H, INV>::run(v);
#pragma unroll
      for (int i = 0; i < H; ++i) c2_store(p + (size_t)(INV ? i : split_slot(H, Y1, i)) * SX, v[i]);
    }
    return;
  }
  constexpr int A1 = INV ? Y2 : Y1, A2 = INV ? Y1 : Y2;   // points of the first, second step
  for (int q = threadIdx.x; q < T * A2; q += TPB) {   // A2 tasks a column
    const int t = q % T, k = q / T;   // k: n2 forward, k1 inverse
    if (m0 + t >= cols) continue;
    const float4* p = column(t) + (size_t)(INV ? k * Y2 : k) * SX;
    C2 v[A1];
#pragma unroll
    for (int i = 0; i < A1; ++i) v[i] = c2_load(p + (size_t)(INV ? i : i * Y2) * SX);
    PairDft<A1, INV>::run(v);
    float4* b = B + t * HP + (INV ? k * Y2 : k);
    c2_store(b, v[0]);
#pragma unroll
    for (int i = 1; i < A1; ++i)
      c2_store(b + (INV ? i : i * Y2), c2_mul<INV>(v[i], twy + (INV ? k * Y2 + i : i * Y2 + k)));
  }
  __syncthreads();
  allow_dependent_launch();
  for (int q = threadIdx.x; q < T * A1; q += TPB) {
    const int t = q % T, k = q / T;   // k: k1 forward, n2 inverse
    if (m0 + t >= cols) continue;
    const float4* b = B + t * HP + (INV ? k : k * Y2);
    C2 v[A2];
#pragma unroll
    for (int i = 0; i < A2; ++i) v[i] = c2_load(b + (INV ? i * Y2 : i));
    PairDft<A2, INV>::run(v);
    float4* p = column(t) + (size_t)(INV ? k : k * Y2) * SX;
#pragma unroll
    for (int i = 0; i < A2; ++i) c2_store(p + (size_t)(INV ? i * Y2 : i) * SX, v[i]);
  }
}

// Threads per z block and blocks per SM: with few pencils a block, 192 threads
// take the first and last z steps in one round (nz = 64, T = 4: 5.6 us, 128
// threads 7.0 us; nz = 48, T = 2: 4.2 against 4.9 us).
constexpr int pair_z_threads(int nz, int t) {
  return nz * t >= 2048 ? 512 : (t >= 8 ? 256 : (nz <= 64 ? 192 : 128));
}
constexpr int pair_z_blocks(int nz, int t) {
  return nz * t >= 2048 ? 1 : (t >= 8 || nz <= 64 ? 2 : 3);
}

template <int NZ, int TT>
struct PairZ {
  static constexpr int Z1 = pair_z1(NZ), Z2 = NZ / Z1, T = TT;
  static constexpr int TPB = pair_z_threads(NZ, T), MINB = pair_z_blocks(NZ, T);
  // Element (component c, pencil t, k1, i) at c CS + t TS + k1 Z2P + i.  A
  // phase of eight lanes covers eight pencils (T >= 8: odd TS), or T pencils
  // of 8/T components (forward step 1) or 8/T groups k1 (middle step).
  static constexpr int Z2P = (T >= 8 || Z2 % 2) ? Z2 : Z2 + 1;
  static constexpr int LZ = Z1 * Z2P;
  static constexpr int want = T >= 8 ? 1 : 8 / T;     // TS mod 8
  static constexpr int TS = T >= 8 ? (LZ | 1) : LZ + ((want - LZ % 8) + 8) % 8;
  static constexpr int CS = T >= 8 ? T * TS : T * TS + ((1 - T * TS % 8) + 8) % 8;
  static constexpr size_t SMEM = (size_t)(6 * CS + NZ) * sizeof(float4);
};

// Unit wave vectors of one frequency of a pencil pair (lanes: even, odd ky).
// n = 0 at the zero frequency; `special`: a lane is the zero frequency or a
// masked (mixed Nyquist) one, whose result pair_green_special replaces.
struct PairFreq {
  float2 n1, n2, n3;
  bool zero, masked_e, masked_o, special;
};

template <int NZ>
__device__ __forceinline__ PairFreq pair_freq_vector(const GridDev& g, float4 q, int fl, int kz) {
  const int mz = (2 * kz < NZ) ? kz : kz - NZ;
  const bool nyqz = (NZ % 2 == 0) && (2 * kz == NZ);
  const int ne = (fl & 3) + (mz != 0), no = ((fl >> 2) & 3) + (mz != 0);
  const float x3 = mz * g.inv_lz;
  const float2 x2 = make_float2(q.y, q.z);
  const float2 sq = f2fma(x2, x2, f2splat(fmaf(q.x, q.x, x3 * x3)));
  float2 inv = make_float2(rsqrtf(sq.x), rsqrtf(sq.y));
  PairFreq f;
  f.zero = ne == 0;   // an odd ky is never zero
  f.masked_e = g.nyquist == 0 && ne >= 2 && ((fl & 16) || nyqz);
  f.masked_o = g.nyquist == 0 && no >= 2 && ((fl & 32) || nyqz);
  f.special = f.zero | f.masked_e | f.masked_o;
  if (f.zero) inv.x = 0.f;
  f.n1 = f2mul(f2splat(q.x), inv);
  f.n2 = f2mul(x2, inv);
  f.n3 = f2mul(f2splat(x3), inv);
  return f;
}

__device__ __forceinline__ C2 pair_dot2(const C2& a, float2 m, const C2& b, float2 n) {
  return {f2fma(a.re, m, f2mul(b.re, n)), f2fma(a.im, m, f2mul(b.im, n))};
}
__device__ __forceinline__ C2 pair_dot3(const C2& a, float2 l, const C2& b, float2 m, const C2& c,
                                        float2 n) {
  return {f2fma(a.re, l, f2fma(b.re, m, f2mul(c.re, n))),
          f2fma(a.im, l, f2fma(b.im, m, f2mul(c.im, n)))};
}

// Three components (HALF 0: 11 22 33, 1: 23 13 12) of -sym(n (x) w), w = (p - a n (n.p)) / mu0
template <int HALF>
__device__ __forceinline__ void pair_green_w(const PairFreq& f, const C2& p1, const C2& p2,
                                             const C2& p3, const GammaArgs& ga, C2* o) {
  C2 s = pair_dot3(p1, f.n1, p2, f.n2, p3, f.n3);
  const float2 ma = f2splat(-ga.a);
  s = {f2mul(s.re, ma), f2mul(s.im, ma)};
  const C2 w1 = {f2fma(f.n1, s.re, p1.re), f2fma(f.n1, s.im, p1.im)};
  const C2 w2 = {f2fma(f.n2, s.re, p2.re), f2fma(f.n2, s.im, p2.im)};
  const C2 w3 = {f2fma(f.n3, s.re, p3.re), f2fma(f.n3, s.im, p3.im)};
  const float2 m = f2splat(HALF == 0 ? -ga.inv_mu0 : -0.5f * ga.inv_mu0);
  const float2 g1 = f2mul(f.n1, m), g2 = f2mul(f.n2, m), g3 = f2mul(f.n3, m);
  if (HALF == 0) {
    o[0] = {f2mul(g1, w1.re), f2mul(g1, w1.im)};
    o[1] = {f2mul(g2, w2.re), f2mul(g2, w2.im)};
    o[2] = {f2mul(g3, w3.re), f2mul(g3, w3.im)};
  } else {
    o[0] = pair_dot2(w3, g2, w2, g3);
    o[1] = pair_dot2(w3, g1, w1, g3);
    o[2] = pair_dot2(w2, g1, w1, g2);
  }
}

__device__ __forceinline__ void pair_green_special(const PairFreq& f, bool full, const float* En,
                                                   C2* o) {
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (f.zero || f.masked_e) {
      o[j].re.x = f.zero && full ? En[j] : 0.f;
      o[j].im.x = 0.f;
    }
    if (f.masked_o) o[j].re.y = o[j].im.y = 0.f;
  }
}

// All six components at one frequency: o = -Gamma0_hat : a.
__device__ __forceinline__ void pair_green_all(const PairFreq& f, const C2* a, bool full,
                                               const GammaArgs& ga, C2* o) {
  const C2 p1 = pair_dot3(a[0], f.n1, a[5], f.n2, a[4], f.n3);
  const C2 p2 = pair_dot3(a[5], f.n1, a[1], f.n2, a[3], f.n3);
  const C2 p3 = pair_dot3(a[4], f.n1, a[3], f.n2, a[2], f.n3);
  pair_green_w<0>(f, p1, p2, p3, ga, o);
  pair_green_w<1>(f, p1, p2, p3, ga, o + 3);
  if (f.special) {
    pair_green_special(f, full, ga.En, o);
    pair_green_special(f, full, ga.En + 3, o + 3);
  }
}

// Wave vector of pencil pair m: *pen = (xi_x, xi_y even, xi_y odd, 0); *flag:
// bits 0-1, 2-3 count the non-zero (x, y) components of the even and the odd
// line, bits 4, 5 are their x or y Nyquist flags.
__device__ __forceinline__ void pair_pencil(const GridDev& g, int m, int plane, float4* pen,
                                            int* flag) {
  float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
  int f = 0;
  if (m < plane) {
    const int sxn = g.nxh + 1, j = m / sxn, sx = m - j * sxn;
    const int2 fx = g.p_fx[sx];
    const int4 fy = g.p_fy[j];
    q = make_float4(fx.x * g.inv_lx, fy.x * g.inv_ly, fy.z * g.inv_ly, 0.f);
    f = ((fx.x != 0) + (fy.x != 0)) | (((fx.x != 0) + (fy.z != 0)) << 2) |
        ((fx.y | fy.y) << 4) | ((fx.y | fy.w) << 5);
  }
  *pen = q;
  *flag = f;
}

// Forward z step 2, the Green operator and inverse step 1 on the T pencil
// pairs of a block (layout of PairZ), in place.
template <int NZ, int T, int TPB>
__device__ __forceinline__ void pair_z_middle(const GridDev& g, float4* B, const float4* twz,
                                              const float4* pen, const int* flag, int mode,
                                              const GammaArgs& ga) {
  using C = PairZ<NZ, T>;
  constexpr int Z1 = C::Z1, Z2 = C::Z2, Z2P = C::Z2P, TS = C::TS, CS = C::CS;
  if constexpr (Z2 > 8) {
    // three components of a 16-point middle step do not fit a thread's
    // registers: forward step 2, Green operator and inverse step 1 separately
    for (int q = threadIdx.x; q < 6 * T * Z1; q += TPB) {
      const int t = q % T, c = (q / T) % 6, k1 = q / (6 * T);
      float4* p = B + c * CS + t * TS + k1 * Z2P;
      C2 v[Z2];
#pragma unroll
      for (int i = 0; i < Z2; ++i) v[i] = c2_load(p + i);
      PairDft<Z2, false>::run(v);
#pragma unroll
      for (int i = 0; i < Z2; ++i) c2_store(p + i, v[i]);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < T * NZ; q += TPB) {
      const int t = q % T, s = q / T, k1 = s / Z2, k2 = s % Z2;
      float4* p = B + t * TS + k1 * Z2P + k2;
      const PairFreq f = pair_freq_vector<NZ>(g, pen[t], flag[t], k1 + Z1 * k2);
      C2 a[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) a[c] = c2_load(p + c * CS);
      C2 o[6];
      pair_green_all(f, a, mode == GM_FULL_MAP, ga, o);
#pragma unroll
      for (int c = 0; c < 6; ++c) c2_store(p + c * CS, o[c]);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 6 * T * Z1; q += TPB) {
      const int t = q % T, c = (q / T) % 6, k1 = q / (6 * T);
      float4* p = B + c * CS + t * TS + k1 * Z2P;
      C2 v[Z2];
#pragma unroll
      for (int i = 0; i < Z2; ++i) v[i] = c2_load(p + i);
      PairDft<Z2, true>::run(v);
      c2_store(p, v[0]);
#pragma unroll
      for (int n2 = 1; n2 < Z2; ++n2) c2_store(p + n2, c2_mul<true>(v[n2], twz + k1 * Z2 + n2));
    }
  } else {
  const int lane = threadIdx.x & 31, h = lane >> 4;   // h = 0: tau11 22 33, 1: tau23 13 12
  for (int wg = threadIdx.x >> 5; wg < (T * Z1 + 15) / 16; wg += TPB / 32) {
    const int pi = wg * 16 + (lane & 15);
    const bool have = (T * Z1) % 16 == 0 || pi < T * Z1;
    const int t = pi % T, k1 = have ? pi / T : 0;
    float4* base = B + 3 * h * CS + t * TS + k1 * Z2P;
    C2 v[3][Z2];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
      for (int i = 0; i < Z2; ++i) v[j][i] = c2_load(base + j * CS + i);
      PairDft<Z2, false>::run(v[j]);
    }
    const float4 q = pen[t];
    const int fl = flag[t];
#pragma unroll
    for (int k2 = 0; k2 < Z2; ++k2) {
      const PairFreq f = pair_freq_vector<NZ>(g, q, fl, k1 + Z1 * k2);
      const C2 a0 = v[0][k2], a1 = v[1][k2], a2 = v[2][k2];
      C2 p1, p2, p3;   // this half's share of v = tau_hat n
      if (h == 0) {
        p1 = {f2mul(a0.re, f.n1), f2mul(a0.im, f.n1)};
        p2 = {f2mul(a1.re, f.n2), f2mul(a1.im, f.n2)};
        p3 = {f2mul(a2.re, f.n3), f2mul(a2.im, f.n3)};
      } else {
        p1 = pair_dot2(a2, f.n2, a1, f.n3);
        p2 = pair_dot2(a2, f.n1, a0, f.n3);
        p3 = pair_dot2(a1, f.n1, a0, f.n2);
      }
      p1 = c2_add(p1, c2_shfl16(p1));
      p2 = c2_add(p2, c2_shfl16(p2));
      p3 = c2_add(p3, c2_shfl16(p3));
      C2 o[3];
      if (h == 0)
        pair_green_w<0>(f, p1, p2, p3, ga, o);
      else
        pair_green_w<1>(f, p1, p2, p3, ga, o);
      if (f.special) pair_green_special(f, mode == GM_FULL_MAP, ga.En + 3 * h, o);
#pragma unroll
      for (int j = 0; j < 3; ++j) v[j][k2] = o[j];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      PairDft<Z2, true>::run(v[j]);
      if (have) {
        c2_store(base + j * CS, v[j][0]);
#pragma unroll
        for (int n2 = 1; n2 < Z2; ++n2)
          c2_store(base + j * CS + n2, c2_mul<true>(v[j][n2], twz + k1 * Z2 + n2));
      }
    }
  }
  }
}

// Pass B: T pencil pairs per block.  Forward z step 1 reads the spectrum from
// global memory; forward step 2, the Green operator and inverse step 1 run in
// registers on one (pencil pair, k1) group per pair of threads, lanes l and
// l + 16 holding the normal and the shear components of the same frequencies
// and exchanging their partial sums of tau_hat n by shuffles; inverse step 2
// writes back to global memory.
template <int NZ, int T>
__global__ void __launch_bounds__(PairZ<NZ, T>::TPB, PairZ<NZ, T>::MINB)
    k_pair_green(GridDev g, float4* __restrict__ spec, int mode, GammaArgs ga) {
  using C = PairZ<NZ, T>;
  constexpr int Z1 = C::Z1, Z2 = C::Z2, Z2P = C::Z2P, TS = C::TS, CS = C::CS, TPB = C::TPB;
  extern __shared__ __align__(128) float4 sm4[];
  float4* B = sm4;
  float4* twz = B + 6 * CS;            // [Z1][Z2]
  __shared__ float4 pen[T];            // see pair_pencil
  __shared__ int flag[T];
  const int m0 = blockIdx.x * T;
  const int plane = (g.ny / 2) * (g.nxh + 1);   // pencil pairs
  for (int i = threadIdx.x; i < NZ; i += TPB) twz[i] = splat_twiddle(g.p_twz[i]);
  if (threadIdx.x < T) pair_pencil(g, m0 + threadIdx.x, plane, pen + threadIdx.x, flag + threadIdx.x);
  grid_dependency_wait();
  __syncthreads();
  // forward step 1; task q -> (pencil t fastest, then component, then n2)
  for (int q = threadIdx.x; q < 6 * T * Z2; q += TPB) {
    const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
    const int m = m0 + t;
    const float4* src = spec + ((size_t)c * NZ + n2) * plane + m;
    const size_t zs = (size_t)Z2 * plane;
    C2 v[Z1];
#pragma unroll
    for (int i = 0; i < Z1; ++i)
      v[i] = m < plane ? c2_load(src + i * zs) : C2{f2splat(0.f), f2splat(0.f)};
    PairDft<Z1, false>::run(v);
    float4* p = B + c * CS + t * TS + n2;
    c2_store(p, v[0]);
#pragma unroll
    for (int k1 = 1; k1 < Z1; ++k1)
      c2_store(p + k1 * Z2P, Z2 > 1 ? c2_mul<false>(v[k1], twz + k1 * Z2 + n2) : v[k1]);
  }
  __syncthreads();
  pair_z_middle<NZ, T, TPB>(g, B, twz, pen, flag, mode, ga);
  __syncthreads();
  allow_dependent_launch();
  for (int q = threadIdx.x; q < 6 * T * Z2; q += TPB) {   // inverse step 2 -> global
    const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
    const int m = m0 + t;
    const float4* p = B + c * CS + t * TS + n2;
    C2 v[Z1];
#pragma unroll
    for (int i = 0; i < Z1; ++i) v[i] = c2_load(p + i * Z2P);
    PairDft<Z1, true>::run(v);
    if (m < plane) {
      float4* dst = spec + ((size_t)c * NZ + n2) * plane + m;
      const size_t zs = (size_t)Z2 * plane;
#pragma unroll
      for (int i = 0; i < Z1; ++i) c2_store(dst + i * zs, v[i]);
    }
  }
}

// The z pass of up to four planes (a 2D cell: one): a thread holds its pencil
// pair's six lines; no shared memory (256 x 256 x 1: 4.7 -> 2.6 us a pass).
constexpr int kShortTPB = 64;
template <int NZ>
__global__ void __launch_bounds__(kShortTPB) k_pair_green_short(GridDev g,
                                                                float4* __restrict__ spec, int mode,
                                                                GammaArgs ga) {
  const int plane = (g.ny / 2) * (g.nxh + 1), m = blockIdx.x * kShortTPB + threadIdx.x;
  float4 q;
  int fl;
  pair_pencil(g, m, plane, &q, &fl);
  grid_dependency_wait();
  if (m >= plane) return;
  C2 v[6][NZ];
#pragma unroll
  for (int c = 0; c < 6; ++c)
#pragma unroll
    for (int i = 0; i < NZ; ++i) v[c][i] = c2_load(spec + ((size_t)c * NZ + i) * plane + m);
  allow_dependent_launch();
#pragma unroll
  for (int c = 0; c < 6; ++c) PairDft<NZ, false>::run(v[c]);
#pragma unroll
  for (int k = 0; k < NZ; ++k) {
    const PairFreq f = pair_freq_vector<NZ>(g, q, fl, k);
    C2 a[6], o[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) a[c] = v[c][k];
    pair_green_all(f, a, mode == GM_FULL_MAP, ga, o);
#pragma unroll
    for (int c = 0; c < 6; ++c) v[c][k] = o[c];
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    PairDft<NZ, true>::run(v[c]);
#pragma unroll
    for (int i = 0; i < NZ; ++i) c2_store(spec + ((size_t)c * NZ + i) * plane + m, v[c][i]);
  }
}

// The z pass for lines whose tile fills an SM (nz = 256): one persistent block
// per SM; the next tile travels into a raw buffer [6][nz][T] by 16-byte
// asynchronous copies while the present one is transformed in the work buffer
// (the layout of PairZ).  Two resident blocks of k_pair_green hide less of the
// loads (256^3: 298 us a pass, this one 238 us; T = 2 with two blocks 296 us).
// At nz = 128, where three blocks fit, k_pair_green is the faster one (28.5
// against 33.8 us).  The last and first steps have 6 T 16 tasks, the threads.
template <int NZ, int T>
struct PairZStream {
  using Z = PairZ<NZ, T>;
  static constexpr int TPB = 6 * T * Z::Z2, RAW = 6 * NZ * T;
  static constexpr size_t SMEM = (size_t)(RAW + 6 * Z::CS + NZ) * sizeof(float4);
};

template <int NZ, int T>
__global__ void __launch_bounds__(PairZStream<NZ, T>::TPB, 1)
    k_pair_green_stream(GridDev g, float4* __restrict__ spec, int mode, GammaArgs ga) {
  using C = PairZ<NZ, T>;
  constexpr int Z1 = C::Z1, Z2 = C::Z2, Z2P = C::Z2P, TS = C::TS, CS = C::CS;
  constexpr int TPB = PairZStream<NZ, T>::TPB, RAW = PairZStream<NZ, T>::RAW;
  extern __shared__ __align__(128) float4 sm4[];
  float4* raw = sm4;                   // [6][NZ][T]
  float4* B = raw + RAW;
  float4* twz = B + 6 * CS;            // [Z1][Z2]
  __shared__ float4 pen[T];
  __shared__ int flag[T];
  const int plane = (g.ny / 2) * (g.nxh + 1), tiles = (plane + T - 1) / T;
  for (int i = threadIdx.x; i < NZ; i += TPB) twz[i] = splat_twiddle(g.p_twz[i]);
  grid_dependency_wait();
  auto prefetch = [&](int tile) {
    for (int q = threadIdx.x; q < RAW; q += TPB) {
      const int t = q % T, cz = q / T;
      if (tile * T + t < plane) async_copy16(raw + q, spec + (size_t)cz * plane + tile * T + t);
    }
    async_copy_commit();
  };
  prefetch(blockIdx.x);
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int m0 = tile * T;
    if (threadIdx.x < T) pair_pencil(g, m0 + threadIdx.x, plane, pen + threadIdx.x, flag + threadIdx.x);
    async_copy_wait();
    __syncthreads();
    for (int q = threadIdx.x; q < 6 * T * Z2; q += TPB) {   // forward step 1
      const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
      const float4* src = raw + (c * NZ + n2) * T + t;
      C2 v[Z1];
#pragma unroll
      for (int i = 0; i < Z1; ++i) v[i] = c2_load(src + i * Z2 * T);
      PairDft<Z1, false>::run(v);
      float4* p = B + c * CS + t * TS + n2;
      c2_store(p, v[0]);
#pragma unroll
      for (int k1 = 1; k1 < Z1; ++k1) c2_store(p + k1 * Z2P, c2_mul<false>(v[k1], twz + k1 * Z2 + n2));
    }
    __syncthreads();
    if (tile + (int)gridDim.x < tiles) prefetch(tile + gridDim.x);
    else
      allow_dependent_launch();   // the block's last tile
    pair_z_middle<NZ, T, TPB>(g, B, twz, pen, flag, mode, ga);
    __syncthreads();
    for (int q = threadIdx.x; q < 6 * T * Z2; q += TPB) {   // inverse step 2 -> global
      const int t = q % T, c = (q / T) % 6, n2 = q / (6 * T);
      const float4* p = B + c * CS + t * TS + n2;
      C2 v[Z1];
#pragma unroll
      for (int i = 0; i < Z1; ++i) v[i] = c2_load(p + i * Z2P);
      PairDft<Z1, true>::run(v);
      if (m0 + t < plane) {
        float4* dst = spec + ((size_t)c * NZ + n2) * plane + m0 + t;
        const size_t zs = (size_t)Z2 * plane;
#pragma unroll
        for (int i = 0; i < Z1; ++i) c2_store(dst + i * zs, v[i]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
      v = 148;
    return v;
  }();
  return n;
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int N>
size_t plane_smem(bool table) {
  using C = PairPlane<N, 32>;
  return (size_t)(C::PL + 2 * C::NXH + C::H) * sizeof(float4) + C::H * sizeof(float2) +
         (table ? 256 * sizeof(float2) : 0);
}

template <int N, int TPB>
cudaError_t launch_fwd(const GridDev& g, const float* in, float4* spec, int mode, cudaStream_t st) {
  const size_t smem = plane_smem<N>(true);
  cudaError_t e = set_smem(k_pair_fwd<N, TPB>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_pair_fwd<N, TPB>, dim3(6, g.nz), TPB, smem, st, g, in, spec, mode);
}

// pass C, or with a post table its form with Algorithm 3's post-step (clusters
// of three blocks, `eps` being the map's input)
template <int N, int TPB>
cudaError_t launch_inv(const GridDev& g, float* out, const float4* spec, const float* eps,
                       const float4* post, cudaStream_t st) {
  const float scale = 0.5f / (float)g.n;
  cudaError_t e;
  if (post) {
    const size_t smem = plane_smem<N>(false) + 256 * sizeof(float4);
    if ((e = set_smem(k_pair_inv<N, TPB, true>, smem)) != cudaSuccess) return e;
    return launch_pdl_cluster(k_pair_inv<N, TPB, true>, dim3(6 * g.nz), TPB, smem, st, 3u, g, spec,
                              out, scale, eps, post);
  }
  const size_t smem = plane_smem<N>(false);
  if ((e = set_smem(k_pair_inv<N, TPB, false>, smem)) != cudaSuccess) return e;
  return launch_pdl(k_pair_inv<N, TPB, false>, dim3(6 * g.nz), TPB, smem, st, g, spec, out, scale,
                    eps, post);
}

// At 96^2, blocks of 128 threads pay once there are enough of them for two per
// SM; below, a block of 256 finishes its plane sooner (24 x 96 x 96: map 25 -> 19 us).
bool few_planes(const GridDev& g) { return 6 * g.nz <= 304; }

// Row pairs per block: enough for four blocks an SM, or few where the grid is small.
template <int NX>
struct RowsTile {
  static constexpr bool ONE = PairX<NX, 1, 1>::X2 == 1;
  static constexpr int BIG = ONE ? 64 : 16, SMALL = ONE ? 16 : 4;
};

template <int NX, int R>
cudaError_t launch_rows_r(const GridDev& g, const float* in, float* out, float4* spec, int mode,
                          bool inv, const float* add, cudaStream_t st) {
  using C = PairRows<NX, R>;
  const dim3 grid(6, (g.ny / 2 + R - 1) / R, g.nz);
  const size_t smem = C::smem(!inv);
  cudaError_t e;
  if (inv) {
    if ((e = set_smem(k_pair_rows_inv<NX, R>, smem)) != cudaSuccess) return e;
    return launch_pdl(k_pair_rows_inv<NX, R>, grid, C::TPB, smem, st, g, (const float4*)spec, out,
                      0.5f / (float)g.n, add);
  }
  if ((e = set_smem(k_pair_rows_fwd<NX, R>, smem)) != cudaSuccess) return e;
  return launch_pdl(k_pair_rows_fwd<NX, R>, grid, C::TPB, smem, st, g, in, spec, mode);
}

template <int NX>
cudaError_t launch_rows(const GridDev& g, const float* in, float* out, float4* spec, int mode,
                        bool inv, const float* add, cudaStream_t st) {
  using T = RowsTile<NX>;
  if ((long long)6 * g.nz * (g.ny / 2) >= 140LL * T::BIG)
    return launch_rows_r<NX, T::BIG>(g, in, out, spec, mode, inv, add, st);
  return launch_rows_r<NX, T::SMALL>(g, in, out, spec, mode, inv, add, st);
}

template <int H, bool INV>
cudaError_t launch_lines(const GridDev& g, float4* spec, cudaStream_t st) {
  using C = PairLines<H, INV>;
  cudaError_t e = set_smem(k_pair_lines<H, INV>, C::SMEM);
  if (e != cudaSuccess) return e;
  const int cols = 6 * g.nz * (g.nxh + 1);
  const dim3 grid((cols + C::T - 1) / C::T);
  return launch_pdl(k_pair_lines<H, INV>, grid, C::TPB, C::SMEM, st, g, spec);
}

template <int NZ, int T>
cudaError_t launch_green(const GridDev& g, float4* spec, int mode, const GammaArgs& ga,
                         cudaStream_t st) {
  using C = PairZ<NZ, T>;
  if constexpr (NZ <= 4) {
    const int pencils = (g.ny / 2) * (g.nxh + 1);
    return launch_pdl(k_pair_green_short<NZ>, dim3((pencils + kShortTPB - 1) / kShortTPB), kShortTPB,
                      0, st, g, spec, mode, ga);
  } else if constexpr (NZ == 256 && T == 4) {
    using S = PairZStream<NZ, T>;
    cudaError_t e = set_smem(k_pair_green_stream<NZ, T>, S::SMEM);
    if (e != cudaSuccess) return e;
    const int pencils = (g.ny / 2) * (g.nxh + 1), tiles = (pencils + T - 1) / T;
    return launch_pdl(k_pair_green_stream<NZ, T>, dim3(std::min(tiles, sm_count())), S::TPB,
                      S::SMEM, st, g, spec, mode, ga);
  } else if constexpr (C::SMEM <= 227 * 1024) {
    cudaError_t e = set_smem(k_pair_green<NZ, T>, C::SMEM);
    if (e != cudaSuccess) return e;
    const int pencils = (g.ny / 2) * (g.nxh + 1);
    return launch_pdl(k_pair_green<NZ, T>, dim3((pencils + T - 1) / T), C::TPB, C::SMEM, st, g,
                      spec, mode, ga);
  } else {
    return cudaErrorInvalidValue;   // variant not available
  }
}

template <int NZ>
cudaError_t launch_green_tile(const GridDev& g, float4* spec, int mode, const GammaArgs& ga,
                              cudaStream_t st) {
  switch (pair_z_tile(g)) {
    case 2: return launch_green<NZ, 2>(g, spec, mode, ga, st);
    case 4: return launch_green<NZ, 4>(g, spec, mode, ga, st);
    case 8: return launch_green<NZ, 8>(g, spec, mode, ga, st);
    default: return launch_green<NZ, 16>(g, spec, mode, ga, st);
  }
}

cudaError_t pass_fwd(const GridDev& g, const float* in, float4* spec, int mode, cudaStream_t st) {
  if (g.nx == 96 && few_planes(g))
    return launch_fwd<96, pair_threads(96, true)>(g, in, spec, mode, st);
  switch (g.nx) {
#define RPM_CASE(N) case N: return launch_fwd<N, pair_threads(N, false)>(g, in, spec, mode, st);
    RPM_PLANE_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t pass_inv(const GridDev& g, float* out, const float4* spec, const float* eps,
                     const float4* post, cudaStream_t st) {
  if (g.nx == 96 && few_planes(g))
    return launch_inv<96, pair_threads(96, true)>(g, out, spec, eps, post, st);
  switch (g.nx) {
#define RPM_CASE(N) case N: return launch_inv<N, pair_threads(N, false)>(g, out, spec, eps, post, st);
    RPM_PLANE_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t pass_green(const GridDev& g, float4* spec, int mode, const double E[6],
                       cudaStream_t st) {
  GammaArgs ga = gamma_args(g, E);
  for (float& v : ga.En) v *= 2.f;   // the spectrum holds 2 X
  switch (g.nz) {
#define RPM_CASE(N) case N: return launch_green_tile<N>(g, spec, mode, ga, st);
    RPM_Z_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t pass_rows(const GridDev& g, const float* in, float* out, float4* spec, int mode,
                      bool inv, const float* add, cudaStream_t st) {
  switch (g.nx) {
#define RPM_CASE(N) case N: return launch_rows<N>(g, in, out, spec, mode, inv, add, st);
    RPM_XY_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t pass_lines(const GridDev& g, float4* spec, bool inv, cudaStream_t st) {
  switch (g.ny) {
#define RPM_CASE(N) \
  case N: return inv ? launch_lines<N / 2, true>(g, spec, st) : launch_lines<N / 2, false>(g, spec, st);
    RPM_XY_SIZES(RPM_CASE)
#undef RPM_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

bool pair_plane_ok(const GridDev& g, const float2* spec) {
  if (g.nx != g.ny || ((uintptr_t)spec & 15) != 0) return false;   // 16-byte spectrum elements
  switch (g.nx) {
#define RPM_CASE(N) case N:
    RPM_PLANE_SIZES(RPM_CASE)
#undef RPM_CASE
    return true;
    default: return false;
  }
}

// Pencil pairs per z block T: the largest that still gives every SM a block or
// two (measured: a second, partly filled round of blocks costs more than 32- or
// 64-byte rows do).  64^3: T = 4, 264 blocks, 5.6 us a pass (T = 2 9.0, T = 8
// 7.7); 64 x 24 x 128: T = 4, 195 blocks, 5.3 us (T = 2 8.2); 48^3: T = 2, 300
// blocks, 4.2 us (T = 4 4.4).  nz = 96, where three blocks of T = 4 fit an SM:
// T = 8 from 290 blocks on (96^3 11.7 us, T = 4 15.2; 96 x 64 x 96 T = 4 10.2,
// T = 8 11.6).  nz = 128: never above 4, the last pass cannot start while the
// 100 KB blocks drain.  nz = 256: T = 4 is the persistent kernel, worth it from
// one tile per SM on (256 x 48 x 48: 9.2 us, T = 2 12.8).
int pair_z_tile(const GridDev& g) {
  const int pencils = (g.ny / 2) * (g.nxh + 1);
  const int blocks = g.nz == 96 ? 290 : (g.nz == 256 ? 140 : 190);
  int t = g.nz <= 16 ? 16 : (g.nz >= 128 ? 4 : 8);
  while (t > 2 && pencils < blocks * t) t /= 2;
  if (g.pencil_t == 1) t = t > 2 ? t / 2 : 2;
  if (g.pencil_t == 2) t = t < 16 ? 2 * t : 16;
  return t;
}

cudaError_t launch_pair_map(const GridDev& g, const float* in, float* out, float2* spec,
                            const double E[6], int mode, cudaStream_t st, const float* add) {
  float4* s4 = reinterpret_cast<float4*>(spec);
  cudaError_t e;
  if ((e = pass_fwd(g, in, s4, mode, st)) != cudaSuccess) return e;
  if ((e = pass_green(g, s4, mode, E, st)) != cudaSuccess) return e;
  return pass_inv(g, out, s4, add, nullptr, st);
}

cudaError_t launch_pair_rows_map(const GridDev& g, const float* in, float* out, float2* spec,
                                 const double E[6], int mode, cudaStream_t st, const float* add) {
  if ((uintptr_t)spec & 15) return cudaErrorInvalidValue;   // as in pair_plane_ok: no other kernels
  float4* s4 = reinterpret_cast<float4*>(spec);
  cudaError_t e;
  if ((e = pass_rows(g, in, nullptr, s4, mode, false, nullptr, st)) != cudaSuccess) return e;
  if ((e = pass_lines(g, s4, false, st)) != cudaSuccess) return e;
  if ((e = pass_green(g, s4, mode, E, st)) != cudaSuccess) return e;
  if ((e = pass_lines(g, s4, true, st)) != cudaSuccess) return e;
  return pass_rows(g, nullptr, out, s4, mode, true, add, st);
}

cudaError_t launch_pair_polarization(const GridDev& g, const float4* post, const float* in,
                                     float* out, float2* spec, const double Eb[6], int mode,
                                     cudaStream_t st) {
  float4* s4 = reinterpret_cast<float4*>(spec);
  cudaError_t e;
  if ((e = pass_fwd(g, in, s4, mode, st)) != cudaSuccess) return e;
  if ((e = pass_green(g, s4, mode, Eb, st)) != cudaSuccess) return e;
  return pass_inv(g, out, s4, in, post, st);
}

void pair_tables(int nx, int ny, int nz, PairTables* t) {
  *t = PairTables{};
  auto root = [](int k, int n) {
    const double a = -2.0 * M_PI * (double)k / (double)n;
    return make_float2((float)std::cos(a), (float)std::sin(a));
  };
  auto twiddles = [&](int len, int n1, float2* out) {   // W_len^(n2 k1) at k1 * N2 + n2
    for (int k1 = 0; k1 < n1; ++k1)
      for (int n2 = 0; n2 < len / n1; ++n2) *out++ = root(n2 * k1, len);
  };
  const int nxh = nx / 2, nyh = ny / 2;
  twiddles(nxh, pair_n1(nxh), t->twx);
  twiddles(nyh, pair_n1(nyh), t->twy);
  twiddles(nz, pair_z1(nz), t->twz);
  for (int j = 0; j < nyh; ++j) t->hw[j] = root(j, ny);
  for (int s = 0; s <= nxh; ++s) {
    const int k = s < nxh ? split_freq(nxh, pair_n1(nxh), s) : nxh;
    t->fx[s] = k == nxh ? make_int2(-k, 1) : make_int2(k, 0);
  }
  auto signed_y = [&](int k) { return 2 * k < ny ? k : k - ny; };
  for (int s = 0; s < nyh; ++s) {
    const int e = 2 * split_freq(nyh, pair_n1(nyh), s), o = e + 1;
    t->fy[s] = make_int4(signed_y(e), 2 * e == ny, signed_y(o), 2 * o == ny);
  }
}

void set_pair_tables(GridDev* g, const PairTables* dev) {
  g->p_twx = dev->twx;
  g->p_twy = dev->twy;
  g->p_twz = dev->twz;
  g->p_hw = dev->hw;
  g->p_fx = dev->fx;
  g->p_fy = dev->fy;
}

}  // namespace rpm
