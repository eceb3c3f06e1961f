// Two complex64 values as one element: the two components (u1, u3) of a field at one point.
//
// Every transform of the 2D operator runs on both components with the same twiddles, so a thread
// holds them as packed pairs: re = (re of component 0, re of component 1), im likewise. Blackwell
// adds and multiplies such a pair of FP32 values with one instruction (add/sub/mul/fma.rn.f32x2,
// each half rounded as the scalar instruction would). A pair instruction occupies the FP32 lanes as
// long as two scalar ones (probe: 38.5 T FP32 adds/s packed against 34.5 T scalar), so the lanes'
// floor stays where it was; what it saves is the issue slot, and these kernels issue far more than
// they multiply. The element is 16 bytes, so exchanges through shared memory and the
// spectra in global memory move with one 16-byte access where the separate components took two of
// 8 bytes.
//
// Twiddle products are scalar: a pair product would need every twiddle duplicated into both
// halves (two moves each), as many instructions as it saves.
#pragma once

#include <cstring>

#include "fft.cuh"

namespace dbi {

using pair64 = unsigned long long;  // two floats: component 0 in the low half

__host__ __device__ __forceinline__ pair64 pk(float lo, float hi) {
#ifdef __CUDA_ARCH__
  pair64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
#else
  pair64 r;
  const float f[2] = {lo, hi};
  std::memcpy(&r, f, sizeof(r));
  return r;
#endif
}
__host__ __device__ __forceinline__ float2 unpk(pair64 v) {
  float2 r;
#ifdef __CUDA_ARCH__
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
#else
  std::memcpy(&r, &v, sizeof(v));
#endif
  return r;
}
__host__ __device__ __forceinline__ pair64 add2(pair64 a, pair64 b) {
#ifdef __CUDA_ARCH__
  pair64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
#else
  const float2 x = unpk(a), y = unpk(b);
  return pk(x.x + y.x, x.y + y.y);
#endif
}
__host__ __device__ __forceinline__ pair64 sub2(pair64 a, pair64 b) {
#ifdef __CUDA_ARCH__
  pair64 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
#else
  const float2 x = unpk(a), y = unpk(b);
  return pk(x.x - y.x, x.y - y.y);
#endif
}
__host__ __device__ __forceinline__ pair64 fma2(pair64 a, pair64 b, pair64 c) {
#ifdef __CUDA_ARCH__
  pair64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
#else
  const float2 x = unpk(a), y = unpk(b), z = unpk(c);
  return pk(fmaf(x.x, y.x, z.x), fmaf(x.y, y.y, z.y));
#endif
}

struct alignas(16) cpair {
  pair64 re, im;
};

template <> struct RealOf<cpair> { using type = float; };

__host__ __device__ __forceinline__ cpair pzero() { return cpair{0ull, 0ull}; }
// Both components at one point, and one of them.
__host__ __device__ __forceinline__ cpair mkpair(float2 c0, float2 c1) {
  return cpair{pk(c0.x, c1.x), pk(c0.y, c1.y)};
}
__host__ __device__ __forceinline__ float2 comp0(const cpair &v) {
  float2 r;
  r.x = unpk(v.re).x;
  r.y = unpk(v.im).x;
  return r;
}
__host__ __device__ __forceinline__ float2 comp1(const cpair &v) {
  float2 r;
  r.x = unpk(v.re).y;
  r.y = unpk(v.im).y;
  return r;
}
__host__ __device__ __forceinline__ cpair hadd(cpair a, cpair b) { return cpair{add2(a.re, b.re), add2(a.im, b.im)}; }
__host__ __device__ __forceinline__ cpair hsub(cpair a, cpair b) { return cpair{sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a +- (-i) b (forward) or a +- (+i) b (inverse): the quarter turn is a choice of operands.
template <bool INV> __host__ __device__ __forceinline__ cpair hadd_mi(cpair a, cpair b) {
  return INV ? cpair{sub2(a.re, b.im), add2(a.im, b.re)} : cpair{add2(a.re, b.im), sub2(a.im, b.re)};
}
template <bool INV> __host__ __device__ __forceinline__ cpair hsub_mi(cpair a, cpair b) {
  return hadd_mi<!INV>(a, b);
}
// both components times one complex factor
__host__ __device__ __forceinline__ cpair hmul(cpair a, float2 w) {
  const float2 r = unpk(a.re), i = unpk(a.im);
  return cpair{pk(r.x * w.x - i.x * w.y, r.y * w.x - i.y * w.y), pk(r.x * w.y + i.x * w.x, r.y * w.y + i.y * w.x)};
}

// R-point DFTs, R = 2, 4, 8 (the plans of fft.cuh on pairs). HALF: the second half of the inputs is
// zero and not read.
template <bool INV> __host__ __device__ __forceinline__ void pdft4(cpair *v) {
  const cpair t0 = hadd(v[0], v[2]), t1 = hsub(v[0], v[2]);
  const cpair t2 = hadd(v[1], v[3]), t3 = hsub(v[1], v[3]);
  v[0] = hadd(t0, t2);
  v[2] = hsub(t0, t2);
  v[1] = hadd_mi<INV>(t1, t3);
  v[3] = hsub_mi<INV>(t1, t3);
}
template <bool INV> __host__ __device__ __forceinline__ void pdft8_join(cpair *v, const cpair (&e)[4], const cpair (&o)[4]) {
  const float h = 0.70710678118654752440f;  // 1 / sqrt(2)
  const pair64 P = pk(h, h), N = pk(-h, -h);
  v[0] = hadd(e[0], o[0]);
  v[4] = hsub(e[0], o[0]);
  v[2] = hadd_mi<INV>(e[2], o[2]);
  v[6] = hsub_mi<INV>(e[2], o[2]);
  // e1 +- o1 W8 and e3 +- o3 W8^3: with s = re + im and d = im - re, o W8 = h (s, d) and
  // o W8^3 = h (d, -s) forward; h (-d, s) and h (-s, -d) inverse
  const pair64 s1 = add2(o[1].re, o[1].im), d1 = sub2(o[1].im, o[1].re);
  const pair64 s3 = add2(o[3].re, o[3].im), d3 = sub2(o[3].im, o[3].re);
  if constexpr (!INV) {
    v[1] = cpair{fma2(s1, P, e[1].re), fma2(d1, P, e[1].im)};
    v[5] = cpair{fma2(s1, N, e[1].re), fma2(d1, N, e[1].im)};
    v[3] = cpair{fma2(d3, P, e[3].re), fma2(s3, N, e[3].im)};
    v[7] = cpair{fma2(d3, N, e[3].re), fma2(s3, P, e[3].im)};
  } else {
    v[1] = cpair{fma2(d1, N, e[1].re), fma2(s1, P, e[1].im)};
    v[5] = cpair{fma2(d1, P, e[1].re), fma2(s1, N, e[1].im)};
    v[3] = cpair{fma2(s3, N, e[3].re), fma2(d3, N, e[3].im)};
    v[7] = cpair{fma2(s3, P, e[3].re), fma2(d3, P, e[3].im)};
  }
}
template <int R, bool INV, bool HALF> __host__ __device__ __forceinline__ void pair_dft(cpair *v) {
  static_assert(R == 2 || R == 4 || R == 8, "radix");
  if constexpr (R == 2) {
    const cpair a = v[0];
    if constexpr (HALF) {
      v[1] = a;
    } else {
      const cpair b = v[1];
      v[0] = hadd(a, b);
      v[1] = hsub(a, b);
    }
  } else if constexpr (R == 4) {
    if constexpr (HALF) {
      const cpair a = v[0], b = v[1];
      v[0] = hadd(a, b);
      v[1] = hadd_mi<INV>(a, b);
      v[2] = hsub(a, b);
      v[3] = hsub_mi<INV>(a, b);
    } else {
      pdft4<INV>(v);
    }
  } else {
    cpair e[4], o[4];
    if constexpr (HALF) {
      e[0] = hadd(v[0], v[2]); e[1] = hadd_mi<INV>(v[0], v[2]);
      e[2] = hsub(v[0], v[2]); e[3] = hsub_mi<INV>(v[0], v[2]);
      o[0] = hadd(v[1], v[3]); o[1] = hadd_mi<INV>(v[1], v[3]);
      o[2] = hsub(v[1], v[3]); o[3] = hsub_mi<INV>(v[1], v[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        e[i] = v[2 * i];
        o[i] = v[2 * i + 1];
      }
      pdft4<INV>(e);
      pdft4<INV>(o);
    }
    pdft8_join<INV>(v, e, o);
  }
}

}  // namespace dbi
