// Complex128 operator stages for batches too small to fill the GPU, FFT lengths up to 128: 32-thread
// CTAs whose lanes hold one component each (T = L / 8 lanes per line, the two components of a row
// or column side by side). FP64 runs at about two lanes a cycle and SM, so a warp's FP64 instruction
// count is its time: with both components per thread the three stages of one 32 x 32 problem took 24,
// 19 and 15 us and its BiCGSTAB solve 1.10 ms, with one component 0.84 ms. The spectra T[c][kx][z]
// are read and written from registers (strided, but they stay in L2).
#pragma once

#include "op_tiles.cuh"

namespace dbi {

template <int L> struct Small64 {
  static constexpr int T = L / 8, UNITS = 16 / T;  // rows or columns per CTA (two lines each)
  static constexpr int LP = RegFFT<double2, L>::LP;
  static_assert(T <= 16, "both lines of a unit in one warp");
  static constexpr size_t lines = size_t(2) * UNITS * LP * sizeof(double2);
};
template <int LX> inline size_t small64_forward_smem(int nx, bool stencil) {
  constexpr int U = Small64<LX>::UNITS;
  const size_t st = stencil ? size_t(3 * (U + 2) + 2 * (U + 4)) * (nx + 2) * sizeof(double2) : 0;
  return std::max(Small64<LX>::lines, st);
}

// Rows z0 .. z0 + UNITS - 1: the contrast source (or the scaled input), forward FFT along x.
template <int LX, bool STENCIL, int V, typename A>
__device__ __forceinline__ void small64_rows_forward(const A &a, int tile, double2 *smem) {
  using C = double2;
  using S = Small64<LX>;
  constexpr int T = S::T, U = S::UNITS, RS = U + 4, RG = U + 2;
  const int lane = threadIdx.x, g = lane / T, t = lane % T, rr = g >> 1, c = g & 1;
  const int nz = a.nz(), nx = a.nx(), z0 = tile * U, z = z0 + rr, W = nx + 2;
  const size_t plane = size_t(nz) * nx;
  const C *u1 = a.in();
  const double isc = a.isc();
  const TwReg<C, LX, V> tr(t, a.tw());
  C v[1][8];
  if constexpr (STENCIL) {
    C *sg = smem, *su = smem + size_t(3) * RG * W;  // stress rows z0 - 1 .., u rows z0 - 2 ..
    for (int i = lane; i < 2 * RS * W; i += 32) {
      const int k = i / W, xx = i - k * W - 1, cc = k >= RS, zz = z0 - 2 + k - cc * RS;
      const bool in = unsigned(zz) < unsigned(nz) && unsigned(xx) < unsigned(nx);
      su[i] = in ? cscale(__ldg(u1 + cc * plane + size_t(zz) * nx + xx), isc) : czero<C>();
    }
    __syncwarp();
    const double ms = a.ms(), w2 = a.w2(), f = a.inv2h();
    for (int i = lane; i < RG * W; i += 32) {
      const int k = i / W, xx = i - k * W - 1;
      C s1, s3, s5;
      stress_at(a, su, RS, W, z0, z0 - 1 + k, xx, ms, s1, s3, s5);
      sg[i] = s1;
      sg[RG * W + i] = s3;
      sg[2 * RG * W + i] = s5;
    }
    __syncwarp();
    // component 0: d1 sigma1 + d3 sigma5, component 1: d1 sigma5 + d3 sigma3
    const C *px = sg + size_t(c ? 2 : 0) * RG * W + (rr + 1) * W + 1, *pz = sg + size_t(c ? 1 : 2) * RG * W + (rr + 1) * W + 1;
    const C *pu = su + size_t(c * RS + rr + 2) * W + 1;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int x = t + m * T;
      v[0][m] = czero<C>();
      if (m < kHalf && z < nz && x < nx) {
        const C o = cscale(cadd(csub(px[x + 1], px[x - 1]), csub(pz[x + W], pz[x - W])), f);
        const double wr = w2 * (__ldg(a.m() + size_t(z) * nx + x) - a.ref(0)) * ms;
        v[0][m] = cadd(o, cscale(pu[x], wr));
      }
    }
    __syncwarp();  // the lines reuse the buffers
  } else {
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int x = t + m * T;
      v[0][m] = m < kHalf && z < nz && x < nx ? cscale(__ldg(u1 + c * plane + size_t(z) * nx + x), isc) : czero<C>();
    }
  }
  C *const line[1] = {smem + size_t(g) * S::LP};
  RegPlan<LX, V>::template run<C, 1, false, true>(v, line, t, tr, RowSync<T>{0});
  if (z < nz) {
    C *o = a.T() + size_t(c) * LX * nz + z;
#pragma unroll
    for (int m = 0; m < 8; ++m) o[size_t(t + m * T) * nz] = v[0][m];
  }
}

// Columns: forward FFT along z, the product (the other component's lane has its point), inverse FFT.
template <int LZ, int V, typename A>
__device__ __forceinline__ void small64_cols(const A &a, int tile, double2 *smem) {
  using C = double2;
  using S = Small64<LZ>;
  constexpr int T = S::T;
  const int lane = threadIdx.x, g = lane / T, t = lane % T, c = g & 1, kx = tile * S::UNITS + (g >> 1);
  const int nz = a.nz(), lx = a.lx();
  const bool live = kx < lx;
  C *p = a.T() + (size_t(c) * lx + (live ? kx : 0)) * nz;
  const TwReg<C, LZ, V> tr(t, a.tw());
  const size_t plane = size_t(lx) * LZ;
  const C *G = a.G() + size_t(live ? kx : 0) * LZ, *Gd = G + (c ? 2 * plane : 0);
  C v[1][8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int z = t + m * T;
    v[0][m] = m < kHalf && live && z < nz ? p[z] : czero<C>();
  }
  C *const line[1] = {smem + size_t(g) * S::LP};
  RegPlan<LZ, V>::template run<C, 1, false, true>(v, line, t, tr, RowSync<T>{0});
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int kz = t + m * T;
    const C own = v[0][m];
    const C other = mk<C>(__shfl_xor_sync(0xffffffffu, own.x, T), __shfl_xor_sync(0xffffffffu, own.y, T));
    v[0][m] = cadd(cmul(__ldg(Gd + kz), own), cmul(__ldg(G + plane + kz), other));
  }
  RegPlan<LZ, V>::template run<C, 1, true>(v, line, t, tr, RowSync<T>{0});
  if (live) {
#pragma unroll
    for (int m = 0; m < kHalf; ++m) {
      const int z = t + m * T;
      if (z < nz) p[z] = v[0][m];
    }
  }
}

// Rows back: inverse FFT along x and the epilogue of rows_inverse_tile.
template <int LX, int EPI, int V, typename A>
__device__ __forceinline__ void small64_rows_inverse(const A &a, int tile, double2 *smem) {
  using C = double2;
  using S = Small64<LX>;
  constexpr int T = S::T;
  const int lane = threadIdx.x, g = lane / T, t = lane % T, c = g & 1, z = tile * S::UNITS + (g >> 1);
  const int nz = a.nz(), nx = a.nx();
  const bool row = z < nz;
  const TwReg<C, LX, V> tr(t, a.tw());
  const C *p = a.T() + size_t(c) * LX * nz + (row ? z : 0);
  const size_t base = size_t(c) * nz * nx + size_t(row ? z : 0) * nx;
  C v[1][8], id[kHalf], h[kHalf];
#pragma unroll
  for (int m = 0; m < 8; ++m) v[0][m] = row ? p[size_t(t + m * T) * nz] : czero<C>();
#pragma unroll
  for (int m = 0; m < kHalf; ++m) {
    const int x = t + m * T;
    const bool in = row && x < nx;
    id[m] = a.ident() && in ? __ldg(a.ident() + base + x) : czero<C>();
    h[m] = EPI == 1 && in ? __ldg(a.krhat() + base + x) : czero<C>();
  }
  C *const line[1] = {smem + size_t(g) * S::LP};
  RegPlan<LX, V>::template run<C, 1, true>(v, line, t, tr, RowSync<T>{0});
  const double osc = a.osc();
  double acc[3] = {0, 0, 0};
#pragma unroll
  for (int m = 0; m < kHalf; ++m) {
    const int x = t + m * T;
    if (!row || x >= nx) continue;
    const C r = cscale(v[0][m], osc), w = a.ident() ? csub(id[m], r) : r;
    a.out()[base + x] = w;
    if constexpr (EPI == 1) {  // conj(rhat) w
      acc[0] += h[m].x * w.x + h[m].y * w.y;
      acc[1] += h[m].x * w.y - h[m].y * w.x;
    } else if constexpr (EPI == 2) {  // conj(w) id and |w|^2
      acc[0] += w.x * id[m].x + w.y * id[m].y;
      acc[1] += w.x * id[m].y - w.y * id[m].x;
      acc[2] += w.x * w.x + w.y * w.y;
    }
  }
  if constexpr (EPI == 1) {
    double two[2] = {acc[0], acc[1]};
    block_sum_store<2>(two, a.part() + size_t(tile) * kRedSlots);
  } else if constexpr (EPI == 2) {
    block_sum_store<3>(acc, a.part() + size_t(tile) * kRedSlots);
  }
}

}  // namespace dbi
