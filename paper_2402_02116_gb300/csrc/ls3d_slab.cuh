// The complex64 3D operator with its y and z transforms fused per kx slab (ls3d.cu runs it where it
// applies, slab_fits; the separate passes elsewhere):
//   k3_stress       sigma = dC : eps(u)                                                   -> T2
//   k3_src_x        w^2 drho u + div sigma of 2 x 128 / T rows, forward FFT along x, stored kx-major
//   k3_yz           per (slot, kx): forward FFTs along y and z of the slab [3][nz][ny], the symmetric
//                   3 x 3 product, inverse FFTs along z and y; in place
//   k3_x_inv        inverse FFT along x, out = ident - result
// The spectra between the x passes are T'[slot][kx][c][r], r = z ny + y (Rp = nz ny rounded up to even
// rows), so that a slab is one contiguous block read and written once: the separate y and z passes moved
// the padded spectra [3][nz][ly][lx] through memory three times in each direction (8.9 GB per pass of 64
// wavefields of 80 x 40 x 32 cells, 2.8 GB now). The Green's tables are copied kx-major
// once per solve, G'[f][kx][e][kz][ky / 2] in pairs of neighbouring ky, and the contrasts rounded to FP32
// once (the values the separate passes form per cell and wavefield in FP64). Both live in the part of
// the spectral scratch that T' leaves free.
//
// Transforms run on pairs (fft_pair.cuh) of lines with the same twiddles: two rows along x, two depths
// along y, two neighbouring ky along z.
#pragma once

#include <algorithm>

#include "fft16.cuh"
#include "operator.cuh"
#include "op_tiles.cuh"

namespace dbi {

constexpr int kSlabXThreads = 128;

struct WarpBarrier {
  __device__ __forceinline__ void operator()() const { __syncwarp(); }
};
__device__ __forceinline__ cpair ldpair(const cpair *p) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(p));
  return cpair{v.x, v.y};
}

struct SlabP {
  int nb, nz, ny, nx, lx, nf, nzp, rows;  // nzp: nz rounded up to even; rows: nz ny
  size_t Rp;                              // row stride of T' (rows rounded up to even)
  float inv2h;
  const double *omega;
  const int *fidx, *plist, *active;
  const float2 *u, *sig, *ident;
  const double *in_scale, *out_scale;
  float2 *out, *T;
  const float *wr, *dc;  // [nf][cells] w^2 drho and [5][cells] dC (rounded)
  const cpair *G;
  const float2 *tw;
  int ahead;  // kx distance at which k3_yz fetches a later slab's input and tables into L2
  int spare;  // slab rows of k3_yz before the spare lines of lanes without work
};

__device__ __forceinline__ int slab_problem(const SlabP &p, int slot) {
  const int b = p.plist ? p.plist[slot] : slot;
  return (p.active && !p.active[b]) || unsigned(p.fidx[b]) >= unsigned(p.nf) ? -1 : b;
}

// Starts fetching `bytes` (a multiple of 16, 16-byte aligned) into L2; one thread's work.
__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}

// Copies of the tables: G'[f][kx][e][kz][ky / 2], one 32 x 32 tile (ky, kx) of one (f, e, kz) per CTA.
static __global__ void __launch_bounds__(256) k3_tables_kx(int lz, int ly, int lx, const float2 *G, cpair *Gp) {
  pdl_begin();
  __shared__ float2 tile[32][33];
  const int kx0 = blockIdx.x * 32, ky0 = blockIdx.y * 32, fekz = blockIdx.z;  // (f * 6 + e) * lz + kz
  const int fe = fekz / lz, kz = fekz - fe * lz, f = fe / 6, e = fe - f * 6;
  const float2 *src = G + size_t(fekz) * ly * lx;
  for (int i = threadIdx.x >> 5; i < 32; i += 8) {
    const int ky = ky0 + i, kx = kx0 + (threadIdx.x & 31);
    if (ky < ly && kx < lx) tile[i][threadIdx.x & 31] = src[size_t(ky) * lx + kx];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 32 * 16; i += 256) {
    const int kx = kx0 + (i >> 4), k = i & 15;  // pair ky0 + 2 k
    if (kx < lx && ky0 + 2 * k < ly)
      Gp[(((size_t(f) * lx + kx) * 6 + e) * lz + kz) * (ly / 2) + ky0 / 2 + k] =
          mkpair(tile[2 * k][i >> 4], tile[2 * k + 1][i >> 4]);
  }
}

// The contrasts as FP32 values: w^2 (rho - rho0) per frequency, C - C0 per parameter.
static __global__ void k3_contrast(size_t cells, int nf, const double *omega, const float *m, double r0, double r1,
                                   double r2, double r3, double r4, double r5, float *wr, float *dc) {
  pdl_begin();
  const size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= cells) return;
  const double dr = double(m[i]) - r0;
  for (int f = 0; f < nf; ++f) {
    const double w = omega[f];
    wr[size_t(f) * cells + i] = float(w * w * dr);
  }
  const double ref[5] = {r1, r2, r3, r4, r5};
  for (int q = 0; q < 5; ++q) dc[q * cells + i] = float(double(m[(q + 1) * cells + i]) - ref[q]);
}

// Rows r0 .. of one component: the source (STENCIL: w^2 drho u_c + the divergence of sigma; else the
// scaled input), forward FFT along x, transposed into T'[kx][c][r] in runs of 2 x 128 / T rows.
template <int LX, bool STENCIL>
__global__ void __launch_bounds__(kSlabXThreads) k3_src_x(SlabP p) {
  pdl_begin();
  using F = Fft16<LX>;
  constexpr int T = F::T, LINES = kSlabXThreads / T, KP = LX + 1;  // KP odd: reads down the tile hit distinct banks
  const int b = slab_problem(p, blockIdx.z);
  if (b < 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpair *s = reinterpret_cast<cpair *>(smem_raw);
  const int g = threadIdx.x / T, t = threadIdx.x % T, c = blockIdx.y;
  const int r0 = blockIdx.x * 2 * LINES, ny = p.ny, nx = p.nx, nz = p.nz;
  const size_t cells = size_t(p.rows) * nx;
  const float sc = p.in_scale ? float(p.in_scale[b]) : 1.0f;
  const float2 *uc = p.u + (size_t(b) * 3 + c) * cells;
  const typename F::Base base(t, p.tw);
  // sigma components differentiated along x, y, z for component c (Voigt: s11 s22 s33 s23 s13 s12)
  const int kx_ = c == 0 ? 0 : c == 1 ? 5 : 4, ky_ = c == 0 ? 5 : c == 1 ? 1 : 3, kz_ = c == 0 ? 4 : c == 1 ? 3 : 2;
  const float2 *sb = STENCIL ? p.sig + size_t(blockIdx.z) * 6 * cells : nullptr;
  const float *wr = STENCIL ? p.wr + size_t(p.fidx[b]) * cells : nullptr;
  float2 w[2][8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = r0 + 2 * g + h, z = r / ny, y = r - z * ny;
    const bool row = r < p.rows;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int x = t + m * T;
      w[h][m] = make_float2(0.f, 0.f);
      if (!row || x >= nx) continue;
      const size_t cell = size_t(r) * nx + x;
      if constexpr (STENCIL) {
        auto D = [&](int k, bool hi, bool lo, int step) {
          const float2 *q = sb + k * cells + cell;
          const float2 a = hi ? __ldg(q + step) : make_float2(0.f, 0.f), d = lo ? __ldg(q - step) : make_float2(0.f, 0.f);
          return cscale(csub(a, d), p.inv2h);
        };
        const float2 dv = cadd(cadd(D(kx_, x + 1 < nx, x > 0, 1), D(ky_, y + 1 < ny, y > 0, nx)),
                               D(kz_, z + 1 < nz, z > 0, ny * nx));
        w[h][m] = cadd(dv, cscale(__ldg(uc + cell), __ldg(wr + cell) * sc));
      } else {
        w[h][m] = cscale(__ldg(uc + cell), sc);
      }
    }
  }
  cpair v[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) v[m] = m < 8 ? mkpair(w[0][m], w[1][m]) : pzero();
  F::template run<false, true>(v, s + size_t(g) * F::LP, t, base, WarpBarrier{});
  __syncthreads();  // the tile reuses the lines
#pragma unroll
  for (int m = 0; m < 16; ++m) s[size_t(g) * KP + t + m * T] = v[m];
  __syncthreads();
  float2 *o = p.T + (size_t(blockIdx.z) * p.lx * 3 + c) * p.Rp + r0;
  const int pl = threadIdx.x % LINES;
  if (r0 + 2 * pl < p.rows) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int kx = threadIdx.x / LINES + i * T;
      const cpair e = s[size_t(pl) * KP + kx];
      const float2 a = comp0(e), d = comp1(e);
      *reinterpret_cast<float4 *>(o + size_t(kx) * 3 * p.Rp + 2 * pl) = make_float4(a.x, a.y, d.x, d.y);
    }
  }
}

// The same rows back: T'[kx][c][r] through the tile, inverse FFT along x, out = ident - osc y for x < nx.
template <int LX> __global__ void __launch_bounds__(kSlabXThreads) k3_x_inv(SlabP p) {
  pdl_begin();
  using F = Fft16<LX>;
  constexpr int T = F::T, LINES = kSlabXThreads / T, KP = LX + 1;
  const int b = slab_problem(p, blockIdx.z);
  if (b < 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpair *s = reinterpret_cast<cpair *>(smem_raw);
  const int g = threadIdx.x / T, t = threadIdx.x % T, c = blockIdx.y;
  const int r0 = blockIdx.x * 2 * LINES, nx = p.nx;
  const float2 *in = p.T + (size_t(blockIdx.z) * p.lx * 3 + c) * p.Rp;
  {
    const int pl = threadIdx.x % LINES;
    const bool ok = r0 + 2 * pl < p.rows;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int kx = threadIdx.x / LINES + i * T;
      cp_async16z(s + size_t(pl) * KP + kx, in + (ok ? size_t(kx) * 3 * p.Rp + r0 + 2 * pl : 0), ok);
    }
  }
  const typename F::Base base(t, p.tw);
  cp_async_wait_all();
  __syncthreads();
  cpair v[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const float4 e = reinterpret_cast<const float4 *>(s)[size_t(g) * KP + t + m * T];
    v[m] = mkpair(make_float2(e.x, e.y), make_float2(e.z, e.w));
  }
  __syncthreads();  // the lines reuse the tile
  F::template run<true, false>(v, s + size_t(g) * F::LP, t, base, WarpBarrier{});
  const size_t cells = size_t(p.rows) * nx, o0 = (size_t(b) * 3 + c) * cells;
  const float osc = p.out_scale ? float(p.out_scale[b]) : 1.0f;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = r0 + 2 * g + h;
    if (r >= p.rows) continue;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int x = t + m * T;
      if (x >= nx) continue;
      const size_t o = o0 + size_t(r) * nx + x;
      const float2 y = cscale(h ? comp1(v[m]) : comp0(v[m]), osc);
      p.out[o] = p.ident ? csub(__ldg(p.ident + o), y) : y;
    }
  }
}

// Slab geometry of k3_yz: rows [c nzp + z] of P complex values, ky contiguous. P = ly + ly / 16 at least
// (two neighbouring rows hold the exchange line of their pair) and 8 mod 16, so that the z transforms'
// 16-byte accesses (ky pairs of a column, rows P / 2 = 4 mod 8 slots apart) spread over the banks.
template <int LY> constexpr int kSlabP = ((LY + LY / 16 + 7) / 16) * 16 + 8;
// Threads per slab: as many as the z transforms have lanes, 64 to 256. (With 256 on every slab most of a
// CTA idled at short lengths: one pass over 160 wavefields of 9 x 11 x 13 cells, ly = lz = 32, took 219 us, now
// 121 us, and 205 us as separate passes; of 16^3 305, 209 and 304 us.)
template <int LY, int LZ> constexpr int kSlabThreads = std::clamp(LY / 2 * (LZ / 8), 64, 256);
// Slab rows: 3 nzp, or the z exchange's line if that is longer, rounded up to even.
template <int LZ> inline int slab_rows(int nzp) {
  const int lp = RegFFT<cpair, LZ>::LP;
  return std::max(3 * nzp, (lp + 1) / 2 * 2);
}
template <int LY, int LZ> inline size_t slab_smem(int nzp) {
  const bool spare = (3 * nzp / 2) % (32 / (LY / 16)) != 0;  // a warp's last lines without work
  return (size_t(slab_rows<LZ>(nzp)) * kSlabP<LY> + (spare ? size_t(32 / (LY / 16)) * 2 * Fft16<LY>::LP : 0)) *
         sizeof(float2);
}

// acc += g v on both halves; nim = -v.im
__device__ __forceinline__ cpair pmad(cpair acc, cpair g, cpair v, pair64 nim) {
  return cpair{fma2(g.im, nim, fma2(g.re, v.re, acc.re)), fma2(g.im, v.re, fma2(g.re, v.im, acc.im))};
}

// One slab (slot, kx), in place in T'. y: T lanes per pair of depths, exchanges in the two rows' own memory;
// z: T lanes per pair of ky, exchanges in the column's own memory, which holds nothing else between the
// reads and the final writes. Only the lanes of one warp ever share a line: the CTA meets twice.
// Slots are the fastest grid index, so the slots of one frequency find each kx's tables in L2; they would
// all wait for the same first read of them from memory (with two 107 KB slabs per SM and 128 registers a
// thread has few loads in flight), so every CTA also starts the L2 fetch of the slab that follows its own
// wave and of an eighth of that slab's tables.
template <int LY, int LZ>
__global__ void __launch_bounds__(kSlabThreads<LY, LZ>, 512 / kSlabThreads<LY, LZ>) k3_yz(SlabP p) {
  pdl_begin();
  using F = Fft16<LY>;
  constexpr int P = kSlabP<LY>, TY = F::T, TZ = LZ / 8, KPW = 32 / TZ, NT = kSlabThreads<LY, LZ>;
  const int slot = int(blockIdx.x % unsigned(p.nb)), kx = int(blockIdx.x / unsigned(p.nb));
  const int b = slab_problem(p, slot);
  if (b < 0) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *slab = reinterpret_cast<float2 *>(smem_raw);
  const int nz = p.nz, ny = p.ny, nzp = p.nzp, half = nzp / 2, nlines = 3 * half;
  float2 *io = p.T + (size_t(slot) * p.lx + kx) * 3 * p.Rp;
  constexpr size_t kTable = size_t(6) * LZ * (LY / 2);  // G' entries of one (f, kx)
  if (threadIdx.x == 0 && kx + p.ahead < p.lx) {
    prefetch_l2(io + size_t(p.ahead) * 3 * p.Rp, unsigned(3 * p.Rp * sizeof(float2)));
    prefetch_l2(p.G + (size_t(p.fidx[b]) * p.lx + kx + p.ahead) * kTable + (slot & 7) * (kTable / 8),
                unsigned(kTable / 8 * sizeof(cpair)));
  }
  const int ty = threadIdx.x % TY;
  const typename F::Base base(ty, p.tw);
  // along y: line l = (c, z / 2), all lanes of a warp take part in its exchanges
  auto lines_y = [&](auto &&body) {
    for (int l0 = (threadIdx.x >> 5) * (32 / TY); l0 < nlines; l0 += NT / TY) {
      const int l = l0 + (threadIdx.x & 31) / TY;
      const bool live = l < nlines;
      const int c = live ? l / half : 0, z0 = live ? 2 * (l - c * half) : 0;
      float2 *row = live ? slab + size_t(c * nzp + z0) * P
                         : slab + size_t(p.spare) * P + size_t((threadIdx.x & 31) / TY) * 2 * F::LP;
      body(live, row, io + c * p.Rp + size_t(z0) * ny, live && z0 + 1 < nz);
    }
  };
  lines_y([&](bool live, float2 *row, float2 *g, bool two) {
    cpair v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int y = ty + m * TY;
      const float2 zero = make_float2(0.f, 0.f);
      v[m] = m < 8 ? mkpair(live && y < ny ? g[y] : zero, two && y < ny ? g[ny + y] : zero) : pzero();
    }
    F::template run<false, true>(v, reinterpret_cast<cpair *>(row), ty, base, WarpBarrier{});
    if (live) {
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        row[ty + m * TY] = comp0(v[m]);
        row[P + ty + m * TY] = comp1(v[m]);
      }
    }
  });
  __syncthreads();
  {
    const int lane = threadIdx.x & 31, tz = lane / KPW;
    const TwReg<float2, LZ, 0> tr(tz, p.tw);
    const cpair *Gk = p.G + (size_t(p.fidx[b]) * p.lx + kx) * kTable;
    for (int k0 = (threadIdx.x >> 5) * KPW; k0 < LY / 2; k0 += NT / 32 * KPW) {
      const int kp = k0 + lane % KPW;
      cpair *col = reinterpret_cast<cpair *>(slab) + kp;  // row i at col[i P / 2]
      const StridedLine<cpair> line[1] = {{col, P / 2}};
      cpair v[3][8];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const int z = tz + m * TZ;
          v[c][m] = pzero();
          if (m < 4 && z < nz) {
            const float4 e = *reinterpret_cast<const float4 *>(col + size_t(c * nzp + z) * (P / 2));
            v[c][m] = mkpair(make_float2(e.x, e.y), make_float2(e.z, e.w));
          }
        }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 3; ++c)
        RegPlan<LZ, 0>::template run<cpair, 1, false, true>(reinterpret_cast<cpair(&)[1][8]>(v[c]), line, tz, tr,
                                                            WarpBarrier{});
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const cpair *G = Gk + size_t(tz + m * TZ) * (LY / 2) + kp;
        constexpr size_t E = size_t(LZ) * (LY / 2);
        const cpair g11 = ldpair(G), g12 = ldpair(G + E), g13 = ldpair(G + 2 * E);
        const cpair g22 = ldpair(G + 3 * E), g23 = ldpair(G + 4 * E), g33 = ldpair(G + 5 * E);
        const cpair a = v[0][m], d = v[1][m], e = v[2][m];
        const pair64 neg = pk(-1.f, -1.f);
        const pair64 na = mul2(a.im, neg), nd = mul2(d.im, neg), ne = mul2(e.im, neg);
        v[0][m] = pmad(pmad(pmad(pzero(), g11, a, na), g12, d, nd), g13, e, ne);
        v[1][m] = pmad(pmad(pmad(pzero(), g12, a, na), g22, d, nd), g23, e, ne);
        v[2][m] = pmad(pmad(pmad(pzero(), g13, a, na), g23, d, nd), g33, e, ne);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c)
        RegPlan<LZ, 0>::template run<cpair, 1, true>(reinterpret_cast<cpair(&)[1][8]>(v[c]), line, tz, tr, WarpBarrier{});
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int z = tz + m * TZ;
          if (z < nz) {
            const float2 a = comp0(v[c][m]), d = comp1(v[c][m]);
            *reinterpret_cast<float4 *>(col + size_t(c * nzp + z) * (P / 2)) = make_float4(a.x, a.y, d.x, d.y);
          }
        }
    }
  }
  __syncthreads();
  lines_y([&](bool live, float2 *row, float2 *g, bool two) {
    cpair v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m)
      v[m] = mkpair(row[ty + m * TY], row[(live ? P : 0) + ty + m * TY]);
    __syncwarp();  // the rows have been read: the exchange may overwrite them
    F::template run<true, false>(v, reinterpret_cast<cpair *>(row), ty, base, WarpBarrier{});
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int y = ty + m * TY;
      if (live && y < ny) g[y] = comp0(v[m]);
      if (two && y < ny) g[ny + y] = comp1(v[m]);
    }
  });
}

}  // namespace dbi
