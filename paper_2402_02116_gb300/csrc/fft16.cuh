// Transforms of pairs (fft_pair.cuh) with 16 points per thread: L = 16 R2 (R2 = 2 .. 16) as a
// radix-16 pass, one exchange and a radix-R2 pass, by the L / 16 threads of a line, which are lanes of
// one warp.
//
// With 8 points per thread a line crosses shared memory twice per transform (82 % of the peak wavefront
// rate in the column stage of L = 512) and, beyond 256 points, meets at block barriers; here it
// crosses once and only its warp waits for it. The price is registers: 64 for the points alone.
//
// Thread t holds the points t + m T (T = L / 16, m < 16) before and after (natural order). Pass 1:
// the 16-point DFT of the thread's points, outputs to positions 16 t + r. Pass 2: butterflies
// j = t + i T (i < 16 / R2) over the points j + 16 r, times W_L^{rj}, outputs to j + 16 r = t + (i + r 16 /
// R2) T, the thread's own points again.
// A line's positions are stored with one padding slot per 16 points (pitch L + L / 16): a
// quarter warp's 16-byte stores (positions 16 t + r) and loads (consecutive points) hit 8 distinct
// bank slots, with several lines per warp too (pitch 4 mod 8 at L = 64, 2 mod 8 at L = 32).
#pragma once

#include "fft_reg.cuh"

namespace dbi {

__host__ __device__ __forceinline__ pair64 mul2(pair64 a, pair64 b) {
#ifdef __CUDA_ARCH__
  pair64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
#else
  const float2 x = unpk(a), y = unpk(b);
  return pk(x.x * y.x, x.y * y.y);
#endif
}
// a (wr + i wi), or a (wr - i wi) for an inverse transform, with a constant factor
template <bool INV> __host__ __device__ __forceinline__ cpair pmulc(cpair a, float wr, float wi_fwd) {
  const float wi = INV ? -wi_fwd : wi_fwd;
  const pair64 R = pk(wr, wr), I = pk(wi, wi), N = pk(-wi, -wi);
  return cpair{fma2(a.re, R, mul2(a.im, N)), fma2(a.im, R, mul2(a.re, I))};
}

// 16-point DFT in natural order as 4 x 4. HALF: v[8 .. 15] are zero and not read.
template <bool INV, bool HALF> __host__ __device__ __forceinline__ void pdft16(cpair (&v)[16]) {
  constexpr float c = 0.92387953251128675613f, s = 0.38268343236508977173f, h = 0.70710678118654752440f;
  cpair y[4][4];  // y[a] = 4-point DFT of v[a + 4 b] over b
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    if constexpr (HALF) {
      y[a][0] = hadd(v[a], v[a + 4]);
      y[a][1] = hadd_mi<INV>(v[a], v[a + 4]);
      y[a][2] = hsub(v[a], v[a + 4]);
      y[a][3] = hsub_mi<INV>(v[a], v[a + 4]);
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b) y[a][b] = v[a + 4 * b];
      pdft4<INV>(y[a]);
    }
  }
  // times W16^{a k}, then 4-point DFTs over a: X[k + 4 l]
  y[1][1] = pmulc<INV>(y[1][1], c, -s);
  y[2][1] = pmulc<INV>(y[2][1], h, -h);
  y[3][1] = pmulc<INV>(y[3][1], s, -c);
  y[1][2] = pmulc<INV>(y[1][2], h, -h);
  y[3][2] = pmulc<INV>(y[3][2], -h, -h);
  y[1][3] = pmulc<INV>(y[1][3], s, -c);
  y[2][3] = pmulc<INV>(y[2][3], -h, -h);
  y[3][3] = pmulc<INV>(y[3][3], -c, s);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    cpair z[4] = {y[0][k], y[1][k], y[2][k], y[3][k]};
    if (k == 2) {  // W16^4 = -i (forward): the quarter turn folded into the first butterflies
      const cpair t0 = hadd_mi<INV>(z[0], z[2]), t1 = hsub_mi<INV>(z[0], z[2]);
      const cpair t2 = hadd(z[1], z[3]), t3 = hsub(z[1], z[3]);
      z[0] = hadd(t0, t2);
      z[2] = hsub(t0, t2);
      z[1] = hadd_mi<INV>(t1, t3);
      z[3] = hsub_mi<INV>(t1, t3);
    } else {
      pdft4<INV>(z);
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) v[k + 4 * l] = z[l];
  }
}

// w^1 .. w^15 from the table's values of w, w^4 and w^8, by at most four products in sequence (w^15 = w^8 w^7).
__host__ __device__ __forceinline__ void powers16(float2 w1, float2 w4, float2 w8, float2 (&w)[16]) {
  w[1] = w1;
  w[2] = hmul(w1, w1);
  w[3] = hmul(w[2], w1);
  w[4] = w4;
#pragma unroll
  for (int r = 5; r < 8; ++r) w[r] = hmul(w4, w[r - 4]);
  w[8] = w8;
#pragma unroll
  for (int r = 9; r < 16; ++r) w[r] = hmul(w8, w[r - 8]);
}

template <int L> struct Fft16 {
  static constexpr int R2 = L / 16, T = L / 16, NB = 16 / R2, LP = L + L / 16;
  static_assert(R2 == 2 || R2 == 4 || R2 == 8 || R2 == 16, "L = 32 .. 256");

  // The thread's base twiddles of the second pass, read once per kernel: W_L^j of its NB butterflies
  // j = t + i T, or at R2 = 16 (one butterfly) W_L^j, W_L^{4j} and W_L^{8j}, from which the powers take
  // at most four products in sequence (from W_L^j alone the operator's error grew by a tenth).
  static constexpr int kBase = R2 == 16 ? 3 : NB;
  struct Base {
    float2 w[kBase];
    __host__ __device__ __forceinline__ Base(int t, const float2 *__restrict__ tw) {
      constexpr int S = kTwiddleN / L;
      if constexpr (R2 == 16) {
        w[0] = tw[t * S];
        w[1] = tw[4 * t * S];
        w[2] = tw[8 * t * S];
      } else {
#pragma unroll
        for (int i = 0; i < NB; ++i) w[i] = tw[(t + i * T) * S];
      }
    }
  };

  // Transforms the line held by the lanes of its warp; `line` is the line's shared memory (LP pairs).
  // sync() must order the accesses of the line's lanes (a warp barrier).
  template <bool INV, bool HALF, typename Sync>
  __host__ __device__ __forceinline__ static void run(cpair (&v)[16], cpair *line, int t, const Base &base, Sync &&sync) {
    pdft16<INV, HALF>(v);
    cpair *d = line + 17 * t;  // position 16 t + r, padded
#pragma unroll
    for (int r = 0; r < 16; ++r) d[r] = v[r];
    sync();
    // position t + m T, padded: the multiple of 16 below it is that of m T (t < T divides 16)
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = line[t + m * T + (m * T) / 16];
    sync();  // the line may be written again
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      float2 w1 = base.w[i];
      if (INV) w1.y = -w1.y;
      if constexpr (R2 == 16) {
        float2 w[16], w4 = base.w[1], w8 = base.w[2];
        if (INV) { w4.y = -w4.y; w8.y = -w8.y; }
        powers16(w1, w4, w8, w);
#pragma unroll
        for (int r = 1; r < 16; ++r) v[r] = hmul(v[r], w[r]);
        pdft16<INV, false>(v);
      } else {
        float2 w[R2];
        twiddle_powers<float2, R2>(w1, w);
        cpair x[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) x[r] = r ? hmul(v[i + r * NB], w[r]) : v[i];
        pair_dft<R2, INV, false>(x);
#pragma unroll
        for (int r = 0; r < R2; ++r) v[i + r * NB] = x[r];
      }
    }
  }
};

}  // namespace dbi
