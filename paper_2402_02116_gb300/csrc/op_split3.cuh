// LS-operator stages for the FFT length L = 3M = 768 (complex64), for grids of up to 384 cells
// along the axis (L >= 2N - 1). Every transform of the operator is half-pruned (N <= L/2 = 1.5 M
// non-zero inputs, or the first N outputs only), and a length-3M transform is three M-point
// transforms. Forward, with x_j = 0 for j >= 1.5 M:
//   X[3m + q] = sum_{i<M} W_L^{iq} (x_i + W_3^q x_{i+M}) W_M^{im},   q = 0, 1, 2,
// (x_{i+M} is non-zero only for i < M/2). Inverse, for the first 1.5 M outputs:
//   y_j = sum_q W_L^{-jq} v_q[j mod M],   v_q = the unnormalised inverse M-point DFT of Y[3m + q].
// With M = 256 a line is one warp (32 threads x 8 points), so its exchanges need only warp
// barriers; each warp takes one residue q of one row or column, and the three residues of a row
// or column meet once, through shared memory. Compared with L = 1024 the FFT grid of a 384-cell
// axis shrinks by a quarter, and the transforms by more (three 256-point lines instead of two
// 512-point ones).
#pragma once

#include "op_split.cuh"

namespace dbi {

constexpr int kS3L = 768, kS3M = 256;
constexpr int kS3T = kS3M / 8;                    // threads per line: one warp
constexpr int kS3Units = 4;                       // rows or columns per CTA
constexpr int kS3Threads = kS3Units * 3 * kS3T;   // 384: a warp per (unit, residue)
// Padded line of pairs in shared memory; at 2 mod 8 the lines of one residue of four rows (6 mod 8
// apart) hit distinct bank slots with two consecutive points each.
constexpr int kS3LP = row_pitch<kS3M, kS3Units>;
constexpr int kS3UnitThreads = 3 * kS3T;          // 96 threads per row or column
constexpr int kS3Tw = kTwiddleN / kS3L;           // W_L^j = tw[j * kS3Tw]
constexpr int kS3Third = kTwiddleN / 3;           // W_3 = tw[kS3Third]

// Shared memory (bytes): a line of pairs per warp; the residues' inverse transforms that the combine
// step reads reuse it. Every stage takes the same amount.
__host__ __device__ constexpr size_t s3_smem() { return size_t(kS3Units) * 3 * kS3LP * sizeof(cpair); }

// Warp barrier: a line's exchanges stay inside its warp.
struct WarpSync {
  __device__ __forceinline__ void operator()() const { __syncwarp(); }
};

// The folded, twiddled input of residue q (both components) at the thread's points
// i = t + m T (m < 8): W_L^{iq} (x(i) + W_3^q x(i + M)), from a reader x(j) of the line's
// points (zero where j >= n). W_L^{iq} = W_L^{tq} W_24^{mq} (T = 32 = L / 24): one per-thread table
// load and a warp-uniform one per m, instead of a 32-byte-strided load per point.
template <typename Read>
__device__ __forceinline__ void s3_fold(cpair (&v)[8], int t, int q, int n, const float2 *tw, Read &&x) {
  using C = float2;
  const C w3 = __ldg(tw + q * kS3Third);                  // W_3^q
  const C wt = __ldg(tw + ((t * q) % kS3L) * kS3Tw);      // W_L^{tq}
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int i = t + m * kS3T;
    const C wm = cmul(wt, __ldg(tw + ((m * q) % 24) * (kTwiddleN / 24)));  // W_L^{iq}
    cpair a = i < n ? x(i) : pzero();
    if (m < 4 && i + kS3M < n) a = hadd(a, hmul(x(i + kS3M), w3));
    v[m] = hmul(a, wm);
  }
}

// A value of the twiddle table.
__host__ __device__ __forceinline__ float2 s3_tw(const float2 *p) {
#ifdef __CUDA_ARCH__
  return __ldg(p);
#else
  return *p;
#endif
}

// The residues' inverse transforms of one row or column (held by its three warps in natural
// order) combined: y_j = sum_q W_L^{-jq} v_q[j mod M] for the unit's points j = u + 96 i (i < 4) of
// thread u = 32 (w mod 3) + t. The warps first store v_q into their own lines, behind a barrier of their lanes
// (`warp`): the transform before may leave the last exchange's reads of the line unordered
// (run_regrouped). One CTA barrier (`all`) later every thread reads the three residues of its points.
// Every thread of the CTA must call it.
template <typename Warp, typename All>
__host__ __device__ __forceinline__ void s3_combine(const cpair (&v)[8], cpair *smem, int w, int t, const float2 *tw,
                                                    cpair (&y)[4], Warp &&warp, All &&all) {
  using C = float2;
  cpair *own = smem + size_t(w) * kS3LP;
  warp();
#pragma unroll
  for (int m = 0; m < 8; ++m) own[t + m * kS3T] = v[m];
  all();
  const int unit = w / 3, u = (w - 3 * unit) * kS3T + t;
  const cpair *base = smem + size_t(3 * unit) * kS3LP;  // lines of warps 3 unit + q
  // W_L^{-j} = W_L^{-u} W_8^{-i} and W_L^{-2j} = W_L^{-2u} W_4^{-i} for j = u + 96 i (96 = L / 8)
  const C wu1 = cconj(s3_tw(tw + u * kS3Tw)), wu2 = cconj(s3_tw(tw + 2 * u * kS3Tw));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int j = u + i * kS3UnitThreads, jm = j & (kS3M - 1);
    const C w1 = i ? cmulc(wu1, s3_tw(tw + i * (kTwiddleN / 8))) : wu1;
    const C w2 = i ? cmulc(wu2, s3_tw(tw + i * (kTwiddleN / 4))) : wu2;
    y[i] = hadd(base[jm], hadd(hmul(base[kS3LP + jm], w1), hmul(base[2 * kS3LP + jm], w2)));
  }
}

// Inverse transform of the four rows of a tile, thread `tid` of the CTA: on entry v holds the points
// tq + 32 m (m < 8) of residue qs of row r as the thread read them from memory (s3_place), afterwards y the
// outputs x = u + 96 i of row w / 3.
struct S3Place {
  int r, tq, qs;
};
__host__ __device__ __forceinline__ S3Place s3_place(int tid) {
  return {tid % kS3Units, tid / kS3Units % kS3T, tid / (kS3Units * kS3T)};
}
template <typename Warp, typename All>
__host__ __device__ __forceinline__ void s3_rows_inverse(cpair (&v)[1][8], cpair *smem, int tid,
                                                         const TwReg<float2, kS3M, 0> &tr, const float2 *tw,
                                                         cpair (&y)[4], Warp &&warp, All &&all) {
  const S3Place p = s3_place(tid);
  const int w = tid / kS3T, t = tid % kS3T;
  cpair *const lines[1] = {smem + size_t(3 * p.r + p.qs) * kS3LP}, *const lines2[1] = {smem + size_t(w) * kS3LP};
  RegPlan<kS3M, 0>::template run_regrouped<cpair, 1, true, 0>(v, lines, p.tq, lines2, t, tr, warp, all);
  s3_combine(v[0], smem, w, t, tw, y, warp, all);
}

// Columns kx = 4 tile .. 4 tile + 3: warp (column, q) folds the column's nz points (both
// components), transforms them forward (the spectra at kz = 3k + q), multiplies by Ghat(kz, kx) and
// transforms back; the three residues are combined into the nz outputs, written back in place.
// Ghat at lz = 768 is stored residue-major (slot q M + k holds kz = 3k + q), so a warp reads its
// residue's entries contiguously.
template <typename A>
__device__ __forceinline__ void cols_tile_s3(const A &a, int tile, float2 *smem) {
  using C = float2;
  const int w = threadIdx.x >> 5, t = threadIdx.x & 31;
  const int cc = w / 3, q = w - 3 * cc;
  const int kx = tile * kS3Units + cc;
  const int nz = a.nz(), lx = a.lx();
  const bool live = kx < lx;
  const C *tw = a.tw();
  cpair *col = reinterpret_cast<cpair *>(a.T()) + size_t(kx) * nz;
  cpair *ps = reinterpret_cast<cpair *>(smem);
  const TwReg<C, kS3M, 0> tr(t, tw);
  const int n = live ? nz : 0;
  cpair v[1][8];
  s3_fold(v[0], t, q, n, tw, [&](int j) { return col[j]; });
  cpair *const lines[1] = {ps + size_t(w) * kS3LP};
  RegPlan<kS3M, 0>::template run<cpair, 1, false>(v, lines, t, tr, WarpSync{});
  if (live) {
    const size_t plane = size_t(lx) * kS3L;
    const C *G = a.G() + size_t(kx) * kS3L + q * kS3M;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int k = t + m * kS3T;
      v[0][m] = green_product(v[0][m], __ldg(G + k), __ldg(G + plane + k), __ldg(G + 2 * plane + k));
    }
  }
  RegPlan<kS3M, 0>::template run<cpair, 1, true>(v, lines, t, tr, WarpSync{});
  cpair y[4];
  s3_combine(v[0], ps, w, t, tw, y, WarpSync{}, CtaSync{});
  if (live) {
    const int u = threadIdx.x - cc * kS3UnitThreads;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int z = u + i * kS3UnitThreads;
      if (z < nz) col[z] = y[i];
    }
  }
}

// Rows z0 .. z0 + 3: warp (row, q) folds the row (the source rows from the stencil kernel, or the
// raw input times its scale) and transforms it (the spectra at kx = 3k + q); the threads of the
// regrouped last pass store the pairs into the column-major spectra T[kx][z] in runs of four rows.
template <typename A>
__device__ __forceinline__ void rows_forward_tile_s3(const A &a, int tile, float2 *smem, const float2 *src,
                                                     float scale) {
  using C = float2;
  const int w = threadIdx.x >> 5, t = threadIdx.x & 31;
  const int rr = w / 3, q = w - 3 * rr;
  const int z0 = tile * kS3Units, z = z0 + rr;
  const int nz = a.nz(), nx = a.nx();
  const size_t plane = size_t(nz) * nx;
  const C *tw = a.tw();
  const auto [r, tq, qs] = s3_place(threadIdx.x);  // of the stores: row z0 + r, residue qs
  const TwReg<C, kS3M, 0> tr(t, tq, tw);
  const int n = z < nz ? nx : 0;
  const C *row = src + size_t(z < nz ? z : 0) * nx;
  cpair *ps = reinterpret_cast<cpair *>(smem);
  cpair v[1][8];
  s3_fold(v[0], t, q, n, tw,
          [&](int j) { return mkpair(cscale(__ldg(row + j), scale), cscale(__ldg(row + plane + j), scale)); });
  cpair *const lines[1] = {ps + size_t(w) * kS3LP}, *const lines2[1] = {ps + size_t(3 * r + qs) * kS3LP};
  RegPlan<kS3M, 0>::template run_regrouped<cpair, 1, false, 1>(v, lines, t, lines2, tq, tr, WarpSync{}, CtaSync{});
  if (z0 + r < nz) {
    cpair *Tp = reinterpret_cast<cpair *>(a.T()) + z0 + r;
#pragma unroll
    for (int m = 0; m < 8; ++m) Tp[size_t(3 * (tq + m * kS3T) + qs) * nz] = v[0][m];
  }
}

// Rows z0 .. z0 + 3: the spectra T[kx][z0 .. z0 + 3] by warp (row, q) the inverse transform of residue q, the residues combined
// into y_x for x < nx, then the epilogue of rows_inverse_tile: out = ident - scale * y (or the
// scaled y) with the fused inner products.
template <int EPI, typename A>
__device__ __forceinline__ void rows_inverse_tile_s3(const A &a, int tile, float2 *smem) {
  using C = float2;
  const int w = threadIdx.x >> 5, t = threadIdx.x & 31;
  const int rr = w / 3;
  const int z0 = tile * kS3Units, z = z0 + rr;
  const int nz = a.nz(), nx = a.nx();
  const C *tw = a.tw();
  const TwReg<C, kS3M, 0> tr(t, tw);
  cpair *ps = reinterpret_cast<cpair *>(smem);
  cpair v[1][8];
  {
    const S3Place at = s3_place(threadIdx.x);
    const bool in = z0 + at.r < nz;
    const cpair *T0 = reinterpret_cast<const cpair *>(a.T()) + (in ? z0 + at.r : 0);
#pragma unroll
    for (int m = 0; m < 8; ++m)
      v[0][m] = in ? load_spectrum(T0 + size_t(3 * (at.tq + m * kS3T) + at.qs) * nz) : pzero();
  }
  prefetch_rows<kS3Threads>(a, a.ident(), z0, kS3Units, sizeof(C));
  if constexpr (EPI == 1) prefetch_rows<kS3Threads>(a, a.krhat(), z0, kS3Units, sizeof(C));
  cpair yp[4];
  s3_rows_inverse(v, ps, threadIdx.x, tr, tw, yp, WarpSync{}, CtaSync{});
  C y[2][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    y[0][i] = comp0(yp[i]);
    y[1][i] = comp1(yp[i]);
  }
  const int u = threadIdx.x - rr * kS3UnitThreads;
  const float osc = a.osc();
  const size_t base = size_t(z) * nx, fplane = size_t(nz) * nx;
  float a0 = 0, a1 = 0, a2 = 0;
  if (z < nz) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      C id[4], h[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int x = u + i * kS3UnitThreads;
        const size_t o = base + c * fplane + x;
        id[i] = (a.ident() && x < nx) ? __ldg(a.ident() + o) : czero<C>();
        if constexpr (EPI == 1) h[i] = x < nx ? __ldg(a.krhat() + o) : czero<C>();
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int x = u + i * kS3UnitThreads;
        if (x < nx) {
          const size_t o = base + c * fplane + x;
          const C rv = cscale(y[c][i], osc);
          const C wv = a.ident() ? csub(id[i], rv) : rv;
          a.out()[o] = wv;
          if constexpr (EPI == 1) {  // conj(rhat) w
            a0 += h[i].x * wv.x + h[i].y * wv.y;
            a1 += h[i].x * wv.y - h[i].y * wv.x;
          } else if constexpr (EPI == 2) {  // conj(w) id and |w|^2
            a0 += wv.x * id[i].x + wv.y * id[i].y;
            a1 += wv.x * id[i].y - wv.y * id[i].x;
            a2 += wv.x * wv.x + wv.y * wv.y;
          }
        }
      }
    }
  }
  if constexpr (EPI == 1) {
    float acc[2] = {a0, a1};
    block_sum_store<2>(acc, a.part() + size_t(tile) * kRedSlots);
  } else if constexpr (EPI == 2) {
    float acc[3] = {a0, a1, a2};
    block_sum_store<3>(acc, a.part() + size_t(tile) * kRedSlots);
  }
}

}  // namespace dbi
