// Register DFTs on pairs of complex lines (sm_103a packed float32 arithmetic).
//
// Two lines that take the same transform -- the even and the odd ky of a
// plane, or rows y and y + ny/2 -- travel as one pair: `re` holds the two
// real parts, `im` the two imaginary parts, each in one 64-bit register pair.
// Every butterfly then is one packed instruction (add/sub/mul/fma.f32x2) for
// both lines, rotations by +-i are renamings, and an element is one 16-byte
// shared-memory access (float4: re.x re.y im.x im.y).  The packed
// instructions run at the same rate per lane as the scalar ones (measured:
// 120 lane operations per clock and SM either way), so what they save is
// issue slots, which bound the transforms.
#pragma once
#include <cuda_runtime.h>

namespace rpm {

__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\t"
      "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "sub.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 f2splat(float s) { return make_float2(s, s); }

// A pair of complex numbers.
struct C2 {
  float2 re, im;
};

__device__ __forceinline__ C2 c2_load(const float4* p) {
  const float4 v = *p;
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ float4 c2_pack(const C2& a) {
  return make_float4(a.re.x, a.re.y, a.im.x, a.im.y);
}
__device__ __forceinline__ void c2_store(float4* p, const C2& a) { *p = c2_pack(a); }

__device__ __forceinline__ C2 c2_add(const C2& a, const C2& b) {
  return {f2add(a.re, b.re), f2add(a.im, b.im)};
}
__device__ __forceinline__ C2 c2_sub(const C2& a, const C2& b) {
  return {f2sub(a.re, b.re), f2sub(a.im, b.im)};
}
// a -+ i b (the rotation of the forward / inverse transform), and a +- i b
template <bool INV>
__device__ __forceinline__ C2 c2_add_mi(const C2& a, const C2& b) {
  return INV ? C2{f2sub(a.re, b.im), f2add(a.im, b.re)} : C2{f2add(a.re, b.im), f2sub(a.im, b.re)};
}
template <bool INV>
__device__ __forceinline__ C2 c2_add_pi(const C2& a, const C2& b) {
  return c2_add_mi<!INV>(a, b);
}
// a * w (CONJ: a * conj w) for a twiddle held as w.x = {wr, wr}, w.y = {wi, wi}
template <bool CONJ>
__device__ __forceinline__ C2 c2_mul(const C2& a, float2 wr, float2 wi) {
  if (CONJ)
    return {f2fma(a.im, wi, f2mul(a.re, wr)), f2sub(f2mul(a.im, wr), f2mul(a.re, wi))};
  return {f2sub(f2mul(a.re, wr), f2mul(a.im, wi)), f2fma(a.re, wi, f2mul(a.im, wr))};
}
// the same with the twiddle from a table of (wr, wr, wi, wi)
template <bool CONJ>
__device__ __forceinline__ C2 c2_mul(const C2& a, const float4* w) {
  const float4 v = *w;
  return c2_mul<CONJ>(a, make_float2(v.x, v.y), make_float2(v.z, v.w));
}
// a * (c - i s) forward, a * (c + i s) inverse, c and s constants
template <bool INV>
__device__ __forceinline__ C2 c2_rot(const C2& a, float c, float s) {
  const float2 c2 = f2splat(c), p = f2splat(INV ? -s : s), m = f2splat(INV ? s : -s);
  return {f2fma(a.im, p, f2mul(a.re, c2)), f2fma(a.re, m, f2mul(a.im, c2))};
}

// the element of lane ^ 16
__device__ __forceinline__ C2 c2_shfl16(const C2& a) {
  return {make_float2(__shfl_xor_sync(0xffffffffu, a.re.x, 16), __shfl_xor_sync(0xffffffffu, a.re.y, 16)),
          make_float2(__shfl_xor_sync(0xffffffffu, a.im.x, 16), __shfl_xor_sync(0xffffffffu, a.im.y, 16))};
}

template <int R, bool INV>
struct PairDft;

template <bool INV>
struct PairDft<1, INV> {
  __device__ __forceinline__ static void run(C2*) {}
};

template <bool INV>
struct PairDft<2, INV> {
  __device__ __forceinline__ static void run(C2* v) {
    const C2 a = v[0], b = v[1];
    v[0] = c2_add(a, b);
    v[1] = c2_sub(a, b);
  }
};

template <bool INV>
struct PairDft<3, INV> {
  __device__ __forceinline__ static void run(C2* v) {
    const C2 a = v[0], t = c2_add(v[1], v[2]), d = c2_sub(v[1], v[2]);
    const float2 h = f2splat(-0.5f), s3 = f2splat(0.866025403784438646763723170753f);
    const C2 m = {f2fma(t.re, h, a.re), f2fma(t.im, h, a.im)};
    const C2 e = {f2mul(d.re, s3), f2mul(d.im, s3)};
    v[0] = c2_add(a, t);
    v[1] = c2_add_mi<INV>(m, e);
    v[2] = c2_add_pi<INV>(m, e);
  }
};

template <bool INV>
struct PairDft<4, INV> {
  __device__ __forceinline__ static void run(C2* v) {
    const C2 t0 = c2_add(v[0], v[2]), t1 = c2_sub(v[0], v[2]);
    const C2 t2 = c2_add(v[1], v[3]), t3 = c2_sub(v[1], v[3]);
    v[0] = c2_add(t0, t2);
    v[2] = c2_sub(t0, t2);
    v[1] = c2_add_mi<INV>(t1, t3);
    v[3] = c2_add_pi<INV>(t1, t3);
  }
};

template <bool INV>
struct PairDft<8, INV> {
  __device__ __forceinline__ static void run(C2* v) {
    C2 e[4] = {v[0], v[2], v[4], v[6]};
    C2 o[4] = {v[1], v[3], v[5], v[7]};
    PairDft<4, INV>::run(e);
    PairDft<4, INV>::run(o);
    const float2 h = f2splat(0.707106781186547524400844362105f);
    // o1 W8 = h (o1 -+ i o1),  o3 W8^3 = -h (o3 +- i o3)
    C2 p = c2_add_mi<INV>(o[1], o[1]);
    p = {f2mul(p.re, h), f2mul(p.im, h)};
    C2 q = c2_add_pi<INV>(o[3], o[3]);
    q = {f2mul(q.re, h), f2mul(q.im, h)};
    v[0] = c2_add(e[0], o[0]);
    v[4] = c2_sub(e[0], o[0]);
    v[1] = c2_add(e[1], p);
    v[5] = c2_sub(e[1], p);
    v[2] = c2_add_mi<INV>(e[2], o[2]);
    v[6] = c2_add_pi<INV>(e[2], o[2]);
    v[3] = c2_sub(e[3], q);
    v[7] = c2_add(e[3], q);
  }
};

// Two-level DFT of length A * B in registers: A-point DFTs over the stride-B
// subsequences, twiddles, B-point DFTs; natural output order.
// cos(2 pi m / 48) for the multiples the 6, 12 and 16 point transforms use
__device__ __forceinline__ float pair_cos(int m) {
  switch (m) {
    case 0: return 1.f;
    case 3: return 0.923879532511286756128183189397f;
    case 4: return 0.866025403784438646763723170753f;
    case 6: return 0.707106781186547524400844362105f;
    case 8: return 0.5f;
    case 9: return 0.382683432365089771728459984030f;
    case 12: return 0.f;
    case 16: return -0.5f;
    case 18: return -0.707106781186547524400844362105f;
    case 24: return -1.f;
    case 27: return -0.923879532511286756128183189397f;
    default: return 0.f;   // not used
  }
}
__device__ __forceinline__ float pair_sin(int m) {
  switch (m) {
    case 0: case 24: return 0.f;
    case 3: return 0.382683432365089771728459984030f;
    case 4: return 0.5f;
    case 6: case 18: return 0.707106781186547524400844362105f;
    case 8: case 16: return 0.866025403784438646763723170753f;
    case 9: return 0.923879532511286756128183189397f;
    case 12: return 1.f;
    case 27: return -0.382683432365089771728459984030f;
    default: return 0.f;   // not used
  }
}

template <int A, int B, bool INV>
__device__ __forceinline__ void pair_dft_2level(C2* v) {
  C2 y[B][A];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
    C2 t[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) t[n1] = v[n1 * B + n2];
    PairDft<A, INV>::run(t);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      const int m = 48 / (A * B) * n2 * k1;
      if (m == 0)
        y[n2][k1] = t[k1];
      else if (m == 12)   // -i forward, +i inverse
        y[n2][k1] = INV ? C2{f2sub(f2splat(0.f), t[k1].im), t[k1].re}
                        : C2{t[k1].im, f2sub(f2splat(0.f), t[k1].re)};
      else
        y[n2][k1] = c2_rot<INV>(t[k1], pair_cos(m), pair_sin(m));
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    C2 t[B];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) t[n2] = y[n2][k1];
    PairDft<B, INV>::run(t);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = t[k2];
  }
}

template <bool INV>
struct PairDft<6, INV> {
  __device__ __forceinline__ static void run(C2* v) { pair_dft_2level<3, 2, INV>(v); }
};
template <bool INV>
struct PairDft<12, INV> {
  __device__ __forceinline__ static void run(C2* v) { pair_dft_2level<4, 3, INV>(v); }
};
template <bool INV>
struct PairDft<16, INV> {
  __device__ __forceinline__ static void run(C2* v) { pair_dft_2level<4, 4, INV>(v); }
};

// Split of a paired line into its two register steps, L = n1 * (L / n1).  Plane
// lines (x: nx/2, y: ny/2): one step up to 12 points, 4 x 4 at 16 (four times
// the threads of one 16-point step: 32^3 map 17.9 -> 14.0 us), then radix 8 first, 32 data
// registers a thread.  z lines:
// a 16-point first step, so that the middle step of the z pass, which holds
// three components of each frequency, stays short (nz = 64: 16 x 4 points
// 5.6 us a pass, 8 x 8 points 7.9 us; nz = 48: 16 x 3 4.9 us, 8 x 6 5.1 us).
__host__ __device__ constexpr int pair_n1(int L) {
  return L <= 12 ? L : (L == 16 ? 4 : (L <= 64 ? 8 : 16));
}
__host__ __device__ constexpr int pair_z1(int L) { return L <= 16 ? L : (L <= 32 ? 8 : 16); }
// Slot s = k1 * n2 + k2 of a line with first factor n1 holds frequency k1 + n1 * k2.
__host__ __device__ constexpr int split_freq(int L, int n1, int s) {
  return s / (L / n1) + n1 * (s % (L / n1));
}
__host__ __device__ constexpr int split_slot(int L, int n1, int k) {
  return (k % n1) * (L / n1) + k / n1;
}

}  // namespace rpm
