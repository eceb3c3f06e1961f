// The batched LS operator A u = u - h^2 G * (w^2 drho u + div(dC : eps(u))) (Eq. 6, 10) and the
// plain Green's convolution, both evaluated by Eq. 12 on the zero-padded lz x lx grid, for a batch
// of problems on one grid: three kernels per batch (the tile bodies are in op_tiles.cuh), each
// with one CTA per (tile, problem):
//   k_rows_forward : contrast source and forward FFT along x of a few rows -> T[b][c][kx][z]
//   k_cols         : column FFTs, 2x2 Ghat multiply, inverse column FFTs, in place in T
//   k_rows_inverse : inverse FFT along x of a few rows, out = ident - result (or the result)
#include <algorithm>

#include "fft16.cuh"
#include "group.cuh"
#include "krylov_finish.cuh"
#include "op_split.cuh"
#include "op_split3.cuh"
#include "op_tiles.cuh"
#include "operator.cuh"
#include "rows_stream.cuh"
#include "small64.cuh"
#include "tune.cuh"

namespace dbi {

template <typename C> struct OpP {
  using Rl = typename RealOf<C>::type;
  int nz, nx, lz, lx, nf;
  Rl inv2h;
  const double *omega;
  const int *fidx;
  const Rl *m;
  Rl ref[5];
  const C *in;
  const C *ident;
  C *out;
  C *T;
  const C *Ghat;
  const C *tw;
  const int *active;
  const int *plist;  // slot -> problem (NULL: problem = s0 + slot)
  int s0;            // first slot of this launch
  int nb;            // slots in this launch
  const double *in_scale, *m_scale, *out_scale;
  const C *krhat;
  double *part_out;
  int part_count;
  KrylovFinish fin;  // the solver's scalar steps, done by the last inverse row tile of a problem
  C *S;  // [slots][2][nz][nx] contrast-source scratch of the split row stages (L = 1024, 768), or NULL
};

// Problem of this CTA's launch slot y (blockIdx.y, or reversed_y()); the spectral scratch is indexed by the slot.
template <typename C> __device__ __forceinline__ int problem_of(const OpP<C> &p, int y = blockIdx.y) {
  const int sl = p.s0 + y;
  return p.plist ? p.plist[sl] : sl;
}

// Tile accessor of problem b in launch slot `slot`: every value is read from the kernel's
// parameters where the tile body uses it (kernel parameters live in constant memory, so they cost
// no registers until then; a reference to the parameter would force generic loads through its
// address instead).
template <typename C> struct BatchTile {
  using Rl = typename RealOf<C>::type;
  OpP<C> p;  // a copy of the kernel parameter: its fields stay parameter reads (no address taken)
  int b, slot, f;
  __device__ __forceinline__ size_t fld() const { return size_t(b) * 2 * p.nz * p.nx; }
  __device__ __forceinline__ int nz() const { return p.nz; }
  __device__ __forceinline__ int nx() const { return p.nx; }
  __device__ __forceinline__ int lx() const { return p.lx; }
  __device__ __forceinline__ Rl inv2h() const { return p.inv2h; }
  __device__ __forceinline__ Rl ref(int i) const { return p.ref[i]; }
  __device__ __forceinline__ const Rl *m() const { return p.m; }
  __device__ __forceinline__ const C *in() const { return p.in + fld(); }
  __device__ __forceinline__ const C *ident() const { return p.ident ? p.ident + fld() : nullptr; }
  __device__ __forceinline__ C *out() const { return p.out + fld(); }
  __device__ __forceinline__ C *T() const { return p.T + size_t(slot) * 2 * p.lx * p.nz; }
  __device__ __forceinline__ const C *G() const { return p.Ghat + size_t(f) * 3 * p.lx * p.lz; }
  __device__ __forceinline__ const C *tw() const { return p.tw; }
  __device__ __forceinline__ const C *krhat() const { return p.krhat + fld(); }
  __device__ __forceinline__ C *S() const { return p.S + size_t(slot) * 2 * p.nz * p.nx; }
  __device__ __forceinline__ double *part() const { return p.part_out + size_t(b) * p.part_count * kRedSlots; }
  __device__ __forceinline__ Rl w2() const {
    const double om = p.omega[f];
    return Rl(om * om);
  }
  __device__ __forceinline__ Rl isc() const { return p.in_scale ? Rl(p.in_scale[b]) : Rl(1); }
  __device__ __forceinline__ Rl osc() const { return p.out_scale ? Rl(p.out_scale[b]) : Rl(1); }
  __device__ __forceinline__ Rl ms() const { return p.m_scale ? Rl(p.m_scale[0]) : Rl(1); }
};

template <typename C, int LX, bool STENCIL, int V, int NTT>
__global__ void __launch_bounds__(NTT, NTT == kTileThreads ? Cfg<C>::rowFwdMinBlocks(LX) : 1) k_rows_forward(OpP<C> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  rows_forward_tile<C, LX, STENCIL, V, NTT>(BatchTile<C>{p, b, int(blockIdx.y), f}, blockIdx.x,
                                       reinterpret_cast<C *>(smem_raw));
}

// Lengths whose forward row stage walks down the rows (with the stencil).
template <typename C, int LX> constexpr bool kRowsStream = kPairSpectra<C> && LX >= 128 && LX <= 512;

// The forward row stage of complex64 lengths 128 to 512 in chunks of `chunk` rows (rows_stream.cuh). 768
// threads per SM (80 registers each); with 512 the stage was no faster.
#ifndef DBI_STREAM_THREADS
#define DBI_STREAM_THREADS 768
#endif
template <int LX, int V>
__global__ void __launch_bounds__(LX / 2, DBI_STREAM_THREADS / (LX / 2)) k_rows_stream(OpP<float2> p, int chunk) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int zb = blockIdx.x * chunk;
  rows_stream<LX, V>(BatchTile<float2>{p, b, int(blockIdx.y), f}, zb, min(zb + chunk, p.nz),
                     reinterpret_cast<float4 *>(smem_raw));
}

template <typename C, int LZ, int V, int NTT>
__global__ void __launch_bounds__(NTT, NTT == kTileThreads ? Cfg<C>::colMinBlocks : 1) k_cols(OpP<C> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cols_tile<C, LZ, V, NTT>(BatchTile<C>{p, b, int(blockIdx.y), f}, blockIdx.x, reinterpret_cast<C *>(smem_raw));
}

// The complex64 column stage of length 512: a CTA takes the columns kx of SL launch slots at a time (units
// of T threads: unit u = column u / SL, slot u % SL). With SL = 4 the columns' Green's tables of the
// first slot's frequency are staged in shared memory by asynchronous copies issued before the
// forward transforms; slots of that frequency (consecutive slots share it, problems being
// frequency-major) read them there, others from global memory. SL = 1 (few slots) reads the
// tables from global memory. Bound by shared memory (82 % of the wavefront rate at L = 512, 80
// registers, 3 CTAs per SM): 256 problems of 256^2 take 422 us, against 462 us with the components as
// separate 8-byte lines and the tables read from L2 by every slot.
template <int LZ, int V, int SL>
__global__ void __launch_bounds__(kTileThreads, Cfg<float2>::colMinBlocks) k_cols_pairs(OpP<float2> p) {
  pdl_begin();
  using CF = ColCfg<float2, LZ>;
  constexpr int COLS = CF::CC / SL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpair *lines = reinterpret_cast<cpair *>(smem_raw);
  float2 *Gs = reinterpret_cast<float2 *>(lines + size_t(CF::CC) * CF::PLP);
  const int u = threadIdx.x / CF::T, t = threadIdx.x - u * CF::T;
  const int kx = blockIdx.x * COLS + u / SL, sl0 = SL * reversed_y(), sl = sl0 + u % SL;
  auto prob = [&](int slot) { return p.plist ? p.plist[p.s0 + slot] : p.s0 + slot; };
  auto freq = [&](int slot) {  // the slot's table, or -1 when it has no work
    if (slot >= p.nb) return -1;
    const int b = prob(slot), f = p.fidx[b];
    return ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) ? -1 : f;
  };
  const int f0 = freq(sl0), f = SL == 1 ? f0 : freq(sl);
  if constexpr (SL == 1) {
    if (f0 < 0) return;  // uniform over the CTA
  } else if (f0 >= 0) {
    const size_t plane = size_t(p.lx) * LZ;
    const float2 *G = p.Ghat + size_t(f0) * 3 * plane;
    constexpr int N16 = COLS * 3 * LZ / 2;  // 16-byte copies
#pragma unroll
    for (int i = 0; i < (N16 + kTileThreads - 1) / kTileThreads; ++i) {
      const int e = threadIdx.x + i * kTileThreads, ct = e / (LZ / 2), k = e - ct * (LZ / 2);  // ct = column * 3 + table
      const int gx = blockIdx.x * COLS + ct / 3;
      if (e < N16 && gx < p.lx) cp_async16(Gs + 2 * e, G + (ct % 3) * plane + size_t(gx) * LZ + 2 * k);
    }
  }
  const bool live = f >= 0 && kx < p.lx;
  const int b = live ? prob(sl) : 0;
  cols_unit_pairs<LZ, V, SL != 1>(BatchTile<float2>{p, b, live ? sl : 0, live ? f : 0}, kx, u, t, live, lines,
                                  f == f0 ? Gs + size_t(u / SL) * 3 * LZ : nullptr);
}
template <int LZ, int SL> constexpr size_t cols_pairs_smem() {
  using CF = ColCfg<float2, LZ>;
  return size_t(CF::CC) * CF::PLP * sizeof(cpair) + (SL == 1 ? 0 : size_t(CF::CC / SL) * 3 * LZ * sizeof(float2));
}

// The complex64 column stage of lengths 128 and 256 with 16 points per thread (fft16.cuh): T lanes of one
// warp take one column of one slot, every exchange stays inside them, and the CTA meets at no
// barrier. SL slots of a column sit side by side, so that their warp or CTA finds the column's Green's
// tables in L1. 168 registers, 3 CTAs per SM (128 spill). Against 8 points per thread (k_cols) the whole
// operator pass took, on 256 problems, 64.3 against 73.1 us of 64^2 (lz = 128) and 214 against 237 us of
// 128^2 (lz = 256); on one problem both take the same. At lengths 32 and 64, with 2 and 4 lanes per
// line, it is k_cols that is faster: 16 BiCGSTAB iterations on 1, 16 and 256 problems of 32^2 (lz = 64) 864,
// 929 and 1196 us against 893, 950 and 1240 us, of 16 x 64 (lz = 32) 664, 683 and 1020 against 696, 709 and
// 996 us, of 16^2 790, 809 and 1182 against 809, 838 and 1181 us. At length 512
// (two 256-point transforms per half-pruned one, the two half warps combining by lane exchanges) the
// 16-point form took 408 to 444 us for 256 problems of 256^2 with more rounding error or more table loads,
// against 422 us of the 8-point form above, which stays there.
constexpr int kCols16Threads = 128;
template <int LZ> constexpr size_t kCols16Smem = size_t(kCols16Threads / (LZ / 16)) * Fft16<LZ>::LP * sizeof(cpair);
template <int LZ, int SL>
__global__ void __launch_bounds__(kCols16Threads, 3) k_cols16(OpP<float2> p) {
  pdl_begin();
  using F = Fft16<LZ>;
  constexpr int T = F::T, COLS = kCols16Threads / T / SL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int u = threadIdx.x / T, t = threadIdx.x % T;
  cpair *line = reinterpret_cast<cpair *>(smem_raw) + size_t(u) * F::LP;
  const int kx = blockIdx.x * COLS + u / SL, sl = SL * reversed_y() + u % SL;
  int f = -1;
  if (sl < p.nb && kx < p.lx) {
    const int b = p.plist ? p.plist[p.s0 + sl] : p.s0 + sl;
    f = p.fidx[b];
    if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) f = -1;
  }
  const bool live = f >= 0;
  const int nz = p.nz;
  cpair *c = reinterpret_cast<cpair *>(p.T) + (live ? (size_t(sl) * p.lx + kx) * nz : 0);
  const typename F::Base base(t, p.tw);
  cpair v[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int j = t + m * T;
    v[m] = m < 8 && live && j < nz ? c[j] : pzero();
  }
  F::template run<false, true>(v, line, t, base, WarpSync{});
  if (live) {
    const size_t plane = size_t(p.lx) * LZ;
    const float2 *G = p.Ghat + size_t(f) * 3 * plane + size_t(kx) * LZ;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int k = t + m * T;
      v[m] = green_product(v[m], __ldg(G + k), __ldg(G + plane + k), __ldg(G + 2 * plane + k));
    }
  }
  F::template run<true, false>(v, line, t, base, WarpSync{});
  if (live) {
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int j = t + m * T;
      if (j < nz) c[j] = v[m];
    }
  }
}

template <typename C, int LX, int EPI, int V, int NTT>
__global__ void __launch_bounds__(NTT, NTT == kTileThreads ? Cfg<C>::rowInvMinBlocks : 1) k_rows_inverse(OpP<C> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<C> a{p, b, int(blockIdx.y), f};
  rows_inverse_tile<C, LX, EPI, V, NTT>(a, blockIdx.x, reinterpret_cast<C *>(smem_raw));
  if constexpr (EPI != 0) finish_tile<EPI>(p.fin, b, a.part(), gridDim.x);
}

// The stages of small complex128 batches at lengths up to 128 (small64.cuh).
template <int LX, bool STENCIL, int V> __global__ void __launch_bounds__(32) k_rows_forward_small(OpP<double2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  small64_rows_forward<LX, STENCIL, V>(BatchTile<double2>{p, b, int(blockIdx.y), f}, blockIdx.x,
                                       reinterpret_cast<double2 *>(smem_raw));
}
template <int LZ, int V> __global__ void __launch_bounds__(32) k_cols_small(OpP<double2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  small64_cols<LZ, V>(BatchTile<double2>{p, b, int(blockIdx.y), f}, blockIdx.x, reinterpret_cast<double2 *>(smem_raw));
}
template <int LX, int EPI, int V> __global__ void __launch_bounds__(32) k_rows_inverse_small(OpP<double2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<double2> a{p, b, int(blockIdx.y), f};
  small64_rows_inverse<LX, EPI, V>(a, blockIdx.x, reinterpret_cast<double2 *>(smem_raw));
  if constexpr (EPI != 0) finish_tile<EPI>(p.fin, b, a.part(), gridDim.x);
}

// Stages of the L = 1024 complex64 operator as pairs of 512-point transforms (op_split.cuh).
__global__ void __launch_bounds__(kSrcThreads) k_source_split(OpP<float2> p) {
  pdl_begin();
  const int b = problem_of(p, reversed_y()), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<float2> a{p, b, reversed_y(), f};
  source_rows(a, blockIdx.x, reinterpret_cast<float2 *>(smem_raw), a.S());
}

template <bool STENCIL>
__global__ void __launch_bounds__(kTileThreads, 2) k_rows_forward_split(OpP<float2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<float2> a{p, b, int(blockIdx.y), f};
  float2 *smem = reinterpret_cast<float2 *>(smem_raw);
  if constexpr (STENCIL) rows_forward_tile_split(a, blockIdx.x, smem, a.S(), 1.0f);
  else rows_forward_tile_split(a, blockIdx.x, smem, a.in(), a.isc());
}

// Column kx = blockIdx.x of the four launch slots 4 y .. + 3 (y = reversed_y()) (64 threads each). The
// column's Green's tables of the first slot's frequency are staged in shared memory by
// asynchronous copies issued before the forward transforms, so their latency is hidden; slots of
// that frequency (consecutive slots share it, problems being frequency-major) read them there,
// others from global memory.
__global__ void __launch_bounds__(kTileThreads, 2) k_cols_split(OpP<float2> p) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *smem = reinterpret_cast<float2 *>(smem_raw);
  float4 *Gs = reinterpret_cast<float4 *>(smem + split_cols_lines_smem() / sizeof(float2));
  const int g = threadIdx.x / kSplitT, kx = blockIdx.x;
  const int sl0 = 4 * reversed_y(), sl = sl0 + g;
  auto prob = [&](int slot) { return p.plist ? p.plist[p.s0 + slot] : p.s0 + slot; };
  auto freq = [&](int slot) {  // the slot's table, or -1 when it has no work
    if (slot >= p.nb) return -1;
    const int b = prob(slot), f = p.fidx[b];
    return ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) ? -1 : f;
  };
  const int f0 = freq(sl0), f = freq(sl);
  if (f0 >= 0) {  // Ghat(:, kx) of table f0: 3 x 1024 points, six 16-byte copies per thread
    const float2 *G = p.Ghat + size_t(f0) * 3 * p.lx * kSplitL + size_t(kx) * kSplitL;
    const size_t plane = size_t(p.lx) * kSplitL;
#pragma unroll
    for (int i = 0; i < 3 * kSplitL / 2 / kTileThreads; ++i) {
      const int e = threadIdx.x + i * kTileThreads, tb = e / (kSplitL / 2), k = e - tb * (kSplitL / 2);
      cp_async16(Gs + e, G + tb * plane + 2 * k);
    }
  }
  const int b = f >= 0 ? prob(sl) : 0;
  cols_column_split<true>(BatchTile<float2>{p, b, sl, f >= 0 ? f : 0}, kx, g, f >= 0, smem,
                          f == f0 ? Gs : nullptr);
}

template <int EPI>
__global__ void __launch_bounds__(kTileThreads, 2) k_rows_inverse_split(OpP<float2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<float2> a{p, b, int(blockIdx.y), f};
  rows_inverse_tile_split<EPI>(a, blockIdx.x, reinterpret_cast<float2 *>(smem_raw));
  if constexpr (EPI != 0) finish_tile<EPI>(p.fin, b, a.part(), gridDim.x);
}

// Stages of the L = 768 complex64 operator as triples of 256-point transforms (op_split3.cuh);
// the contrast source comes from k_source_split.
template <bool STENCIL>
__global__ void __launch_bounds__(kS3Threads, 2) k_rows_forward_s3(OpP<float2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<float2> a{p, b, int(blockIdx.y), f};
  float2 *smem = reinterpret_cast<float2 *>(smem_raw);
  if constexpr (STENCIL) rows_forward_tile_s3(a, blockIdx.x, smem, a.S(), 1.0f);
  else rows_forward_tile_s3(a, blockIdx.x, smem, a.in(), a.isc());
}

__global__ void __launch_bounds__(kS3Threads, 2) k_cols_s3(OpP<float2> p) {
  pdl_begin();
  const int b = problem_of(p, reversed_y()), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cols_tile_s3(BatchTile<float2>{p, b, reversed_y(), f}, blockIdx.x, reinterpret_cast<float2 *>(smem_raw));
}

template <int EPI>
__global__ void __launch_bounds__(kS3Threads, 2) k_rows_inverse_s3(OpP<float2> p) {
  pdl_begin();
  const int b = problem_of(p), f = p.fidx[b];
  if ((p.active && !p.active[b]) || unsigned(f) >= unsigned(p.nf)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const BatchTile<float2> a{p, b, int(blockIdx.y), f};
  rows_inverse_tile_s3<EPI>(a, blockIdx.x, reinterpret_cast<float2 *>(smem_raw));
  if constexpr (EPI != 0) finish_tile<EPI>(p.fin, b, a.part(), gridDim.x);
}

// Threads per CTA of the ordinary stages: 256, or for complex128 batches too small to give every SM a
// 256-thread tile, as few as hold whole lines and warps (beyond length 128; up to it the kernels of
// small64.cuh run). FP64 runs at two lanes a cycle and SM, so what counts there is the SM with the most
// rows or columns: a 32 x 32 grid of one problem was one row tile and two column tiles (68, 40 and 24 us for
// the stages).
template <int L> constexpr int kSmallThreads = L / 8 > 32 ? L / 8 : 32;
inline size_t ceil_div(size_t a, size_t b) { return (a + b - 1) / b; }
// The row stages on small tiles, of one row each from length 128 on. Such a tile also forms the stress of
// its own halo rows, about as much work as 0.35 (length 128) or 0.6 rows; so they pay where the busiest SM has
// less to do with them. Measured, as shares of the pass: with 80 to 112 of the 256-thread tiles (of 152 SMs) -9
// to -2 % at length 128, -2 to +10 at 256, +7 at 1024; with 128 to 152 of them up to +21 %; with 156 to 182
// -13 to 0 %; with 240 to 304 up to +27 %; with fewer than 76 -25 to -50 %. Up to length 64 they win up to two
// waves (-12 % at 128, -8 % at 152 tiles of 32^2). A pass without the stencil has no halo (16 convolutions of 100^2
// 345 us on small tiles, 374 us on the others).
inline bool small_rows(int B, int nz, int lx, int precision, bool stencil) {
  if (precision != DBI_C128 || lx > 1024) return false;
  const size_t rows = size_t(2048 / lx), tiles = size_t(B) * ceil_div(nz, rows);
  const size_t halo = !stencil ? 0 : lx <= 128 ? 7 : 12;  // in 1/20 rows
  if (tiles >= 2 * kSMs) return false;
  return lx <= 64 || ceil_div(size_t(B) * nz, kSMs) * (20 + halo) < ceil_div(tiles, kSMs) * (20 * rows + halo);
}
// The column stage on small tiles: no halo, but fewer warps behind each other's latency. They pay unless the
// last wave of 256-thread tiles is nearly full: -22 to -10 % of the pass with 16 to 76 tiles, -9 % at 96,
// -5 to 0 % at 128, +1 to +3 % at 144 to 152; -17 % at 160 to 176, -6 to 0 % at 256, up to +3 % at 272 to 304;
// -11 % at 320, -4 % at 384.
inline bool small_cols(int B, int lz, int lx, int precision) {
  if (precision != DBI_C128 || lz > 1024) return false;
  const size_t tiles = size_t(B) * ceil_div(lx, 2048 / lz);
  return tiles < 4 * kSMs && 8 * tiles <= 7 * kSMs * ceil_div(tiles, kSMs);
}
template <typename C, int L, typename F> inline void with_tile(bool small, F &&f) {
  if constexpr (sizeof(C) == sizeof(double2) && L > 128) {
    if (small) {
      f.template operator()<kSmallThreads<L>>();
      return;
    }
  }
  f.template operator()<kTileThreads>();
}

// Calls f.template operator()<V>() with the radix plan chosen for length L (plans differ only
// when L is not a power of 8).
template <int L, typename F> inline void with_plan(int precision, F &&f) {
  if constexpr (L == 64 || L == 512) f.template operator()<0>();
  else if (radix_plan(precision, L) == 1) f.template operator()<1>();
  else f.template operator()<0>();
}

// The three kernels for launch slots [s0, s0 + nb) (problems plist[slot], or the slots themselves),
// each slot using its own part of the spectral scratch.
template <typename C> static int run_chunk(const OpArgs &a, int s0, int nb, int cap, cudaStream_t s) {
  using Rl = typename RealOf<C>::type;
  OpP<C> p;
  p.nz = a.nz; p.nx = a.nx; p.lz = a.lz; p.lx = a.lx; p.nf = a.nf;
  p.inv2h = Rl(1.0 / (2.0 * a.h));
  p.omega = a.omega; p.fidx = a.fidx;
  p.m = static_cast<const Rl *>(a.m);
  for (int i = 0; i < 5; ++i) p.ref[i] = Rl(a.ref[i]);
  p.in = static_cast<const C *>(a.in);
  p.ident = static_cast<const C *>(a.ident);
  p.out = static_cast<C *>(a.out);
  p.T = static_cast<C *>(a.T);
  p.Ghat = static_cast<const C *>(a.Ghat);
  p.tw = static_cast<const C *>(a.tw);
  p.active = a.active;
  p.plist = a.plist;
  p.s0 = s0;
  p.nb = nb;
  p.in_scale = a.in_scale;
  p.m_scale = a.m_scale;
  p.out_scale = a.out_scale;
  p.part_count = operator_parts(a.B, a.nz, a.lx, a.precision);
  p.fin = KrylovFinish{};
  if (a.finish && a.epi != 0) p.fin = *a.finish;
  p.krhat = static_cast<const C *>(a.krhat);
  p.part_out = a.part_out;
  p.S = nullptr;
  int rc = DBI_OK;
  const bool stencil = a.stencil;
  const bool small_r = small_rows(a.B, a.nz, a.lx, a.precision, stencil);
  const bool small_c = small_cols(a.B, a.lz, a.lx, a.precision);
  const int kr = split_kind(a.lx, a.precision), kc = split_kind(a.lz, a.precision);
  const bool split_r = kr != 0, split_c = kc != 0;
  if (split_r) p.S = p.T + size_t(cap) * 2 * a.lx * a.nz;  // after the chunk's spectra
  prof_mark(PROF_ROWS_FORWARD, false, s);
  if constexpr (sizeof(C) == sizeof(float2)) {
    if (split_r) {
      OpP<float2> &q = reinterpret_cast<OpP<float2> &>(p);
      cudaError_t e = cudaSuccess;
      if (stencil) {
        const int chunks = (a.nz + kSrcRows - 1) / kSrcRows;
        e = allow_smem(k_source_split, source_smem());
        if (e == cudaSuccess) launch_pdl(k_source_split, dim3(chunks, nb), kSrcThreads, source_smem(), s, q);
        rc = e != cudaSuccess ? cuda_fail("k_source_split smem", e) : check_launch("k_source_split");
        if (rc) return rc;
      }
      if (kr == kSplitPair) {
        const dim3 grid((a.nz + kSplitRows - 1) / kSplitRows, nb);
        auto kern = stencil ? k_rows_forward_split<true> : k_rows_forward_split<false>;
        e = allow_smem(kern, split_rows_smem());
        if (e == cudaSuccess) launch_pdl(kern, grid, kTileThreads, split_rows_smem(), s, q);
        rc = e != cudaSuccess ? cuda_fail("k_rows_forward_split smem", e) : check_launch("k_rows_forward_split");
      } else {
        const dim3 grid((a.nz + kS3Units - 1) / kS3Units, nb);
        auto kern = stencil ? k_rows_forward_s3<true> : k_rows_forward_s3<false>;
        e = allow_smem(kern, s3_smem());
        if (e == cudaSuccess) launch_pdl(kern, grid, kS3Threads, s3_smem(), s, q);
        rc = e != cudaSuccess ? cuda_fail("k_rows_forward_s3 smem", e) : check_launch("k_rows_forward_s3");
      }
    }
  }
  if (!split_r) dispatch_len(a.lx, [&]<int LX>() {
    if constexpr (!kPairSpectra<C> || LX <= 512)  // (complex64 of length 1024 is split)
    with_plan<LX>(a.precision, [&]<int V>() {
      cudaError_t e;
      if constexpr (kRowsStream<C, LX>) {
        if (stencil) {
          // rows per CTA: 32 while that leaves four waves of CTAs, at least 4
          int chunk = 32;
          const int wave = DBI_STREAM_THREADS / (LX / 2) * int(kSMs);
          while (chunk > 4 && long((a.nz + chunk - 1) / chunk) * nb < 4L * wave) chunk /= 2;
          const size_t bytes = StreamCfg<LX>::smem;
          e = allow_smem(k_rows_stream<LX, V>, bytes);
          if (e == cudaSuccess)
            launch_pdl(k_rows_stream<LX, V>, dim3((a.nz + chunk - 1) / chunk, nb), LX / 2, bytes, s, p, chunk);
          rc = e != cudaSuccess ? cuda_fail("k_rows_stream smem", e) : check_launch("k_rows_stream");
          return;
        }
      }
      if constexpr (sizeof(C) == sizeof(double2) && LX <= 128) {
        if (small_r) {
          const size_t bytes = small64_forward_smem<LX>(a.nx, stencil);
          constexpr int U = Small64<LX>::UNITS;
          auto kern = stencil ? k_rows_forward_small<LX, true, V> : k_rows_forward_small<LX, false, V>;
          e = allow_smem(kern, bytes);
          if (e == cudaSuccess) launch_pdl(kern, dim3((a.nz + U - 1) / U, nb), 32, bytes, s, p);
          rc = e != cudaSuccess ? cuda_fail("k_rows_forward_small smem", e) : check_launch("k_rows_forward_small");
          return;
        }
      }
      with_tile<C, LX>(small_r, [&]<int NTT>() {
        using RC = RowCfg<C, LX, NTT>;
        const size_t bytes = rows_forward_smem<C, LX, NTT>(a.nx, stencil);
        dim3 grid((a.nz + RC::ROWS - 1) / RC::ROWS, nb);
        auto launch = [&](auto kernel) {
          e = allow_smem(kernel, bytes);
          if (e == cudaSuccess) launch_pdl(kernel, grid, RC::NT, bytes, s, p);
        };
        if constexpr (kRowsStream<C, LX>) launch(k_rows_forward<C, LX, false, V, NTT>);
        else if (stencil) launch(k_rows_forward<C, LX, true, V, NTT>);
        else launch(k_rows_forward<C, LX, false, V, NTT>);
      });
      rc = e != cudaSuccess ? cuda_fail("k_rows_forward smem", e) : check_launch("k_rows_forward");
    });
  });
  prof_mark(PROF_ROWS_FORWARD, true, s);
  if (rc) return rc;
  prof_mark(PROF_COLS, false, s);
  if constexpr (sizeof(C) == sizeof(float2)) {
    if (kc == kSplitPair) {
      OpP<float2> &q = reinterpret_cast<OpP<float2> &>(p);
      const dim3 grid(a.lx, (nb + 3) / 4);
      cudaError_t e = allow_smem(k_cols_split, split_cols_staged_smem());
      if (e == cudaSuccess) launch_pdl(k_cols_split, grid, kTileThreads, split_cols_staged_smem(), s, q);
      rc = e != cudaSuccess ? cuda_fail("k_cols_split smem", e) : check_launch("k_cols_split");
    } else if (kc == kSplitTriple) {
      OpP<float2> &q = reinterpret_cast<OpP<float2> &>(p);
      const dim3 grid((a.lx + kS3Units - 1) / kS3Units, nb);
      cudaError_t e = allow_smem(k_cols_s3, s3_smem());
      if (e == cudaSuccess) launch_pdl(k_cols_s3, grid, kS3Threads, s3_smem(), s, q);
      rc = e != cudaSuccess ? cuda_fail("k_cols_s3 smem", e) : check_launch("k_cols_s3");
    }
  }
  if (!split_c) dispatch_len(a.lz, [&]<int LZ>() {
    with_plan<LZ>(a.precision, [&]<int V>() {
      using CF = ColCfg<C, LZ>;
      if constexpr (kPairSpectra<C>) {
        cudaError_t e = cudaSuccess;
        // four slots per CTA unless the last group would leave much of its CTAs idle
        [[maybe_unused]] const bool four = nb % 4 == 0 || nb >= 16;
        if constexpr (LZ == 512) {
          auto launch = [&]<int SL>() {
            constexpr int COLS = CF::CC / SL;
            const size_t bytes = cols_pairs_smem<LZ, SL>();
            e = allow_smem(k_cols_pairs<LZ, V, SL>, bytes);
            if (e == cudaSuccess)
              launch_pdl(k_cols_pairs<LZ, V, SL>, dim3((a.lx + COLS - 1) / COLS, (nb + SL - 1) / SL), CF::NT, bytes, s, p);
          };
          if (four) launch.template operator()<4>();
          else launch.template operator()<1>();
        } else if constexpr (LZ >= 128 && LZ <= 256) {
          auto launch = [&]<int SL>() {
            constexpr int COLS = kCols16Threads / (LZ / 16) / SL;
            e = allow_smem(k_cols16<LZ, SL>, kCols16Smem<LZ>);
            if (e == cudaSuccess)
              launch_pdl(k_cols16<LZ, SL>, dim3((a.lx + COLS - 1) / COLS, (nb + SL - 1) / SL), kCols16Threads,
                         kCols16Smem<LZ>, s, p);
          };
          if (four) launch.template operator()<4>();
          else launch.template operator()<1>();
        } else if constexpr (LZ <= 64) {
          const size_t bytes = cols_smem<C, LZ>();
          e = allow_smem(k_cols<C, LZ, V, kTileThreads>, bytes);
          if (e == cudaSuccess)
            launch_pdl(k_cols<C, LZ, V, kTileThreads>, dim3((a.lx + CF::CC - 1) / CF::CC, nb), CF::NT, bytes, s, p);
        }  // 1024 runs as pairs of 512-point transforms
        rc = e != cudaSuccess ? cuda_fail("k_cols smem", e) : check_launch("k_cols");
      } else {
        cudaError_t e = cudaSuccess;
        if constexpr (LZ <= 128) {
          if (small_c) {
            constexpr int U = Small64<LZ>::UNITS;
            launch_pdl(k_cols_small<LZ, V>, dim3((a.lx + U - 1) / U, nb), 32, Small64<LZ>::lines, s, p);
            rc = check_launch("k_cols_small");
            return;
          }
        }
        with_tile<C, LZ>(small_c, [&]<int NTT>() {
          using CN = ColCfg<C, LZ, NTT>;
          const size_t bytes = cols_smem<C, LZ, NTT>();
          dim3 grid((a.lx + CN::CC - 1) / CN::CC, nb);
          e = allow_smem(k_cols<C, LZ, V, NTT>, bytes);
          if (e == cudaSuccess) launch_pdl(k_cols<C, LZ, V, NTT>, grid, CN::NT, bytes, s, p);
        });
        rc = e != cudaSuccess ? cuda_fail("k_cols smem", e) : check_launch("k_cols");
      }
    });
  });
  prof_mark(PROF_COLS, true, s);
  if (rc) return rc;
  prof_mark(PROF_ROWS_INVERSE, false, s);
  if constexpr (sizeof(C) == sizeof(float2)) {
    if (kr == kSplitPair) {
      OpP<float2> &q = reinterpret_cast<OpP<float2> &>(p);
      const dim3 grid((a.nz + kSplitRows - 1) / kSplitRows, nb);
      auto kern = a.epi == 1 ? k_rows_inverse_split<1> : a.epi == 2 ? k_rows_inverse_split<2> : k_rows_inverse_split<0>;
      cudaError_t e = allow_smem(kern, split_rows_inverse_smem());
      if (e == cudaSuccess) launch_pdl(kern, grid, kTileThreads, split_rows_inverse_smem(), s, q);
      rc = e != cudaSuccess ? cuda_fail("k_rows_inverse_split smem", e) : check_launch("k_rows_inverse_split");
    } else if (kr == kSplitTriple) {
      OpP<float2> &q = reinterpret_cast<OpP<float2> &>(p);
      const dim3 grid((a.nz + kS3Units - 1) / kS3Units, nb);
      auto kern = a.epi == 1 ? k_rows_inverse_s3<1> : a.epi == 2 ? k_rows_inverse_s3<2> : k_rows_inverse_s3<0>;
      cudaError_t e = allow_smem(kern, s3_smem());
      if (e == cudaSuccess) launch_pdl(kern, grid, kS3Threads, s3_smem(), s, q);
      rc = e != cudaSuccess ? cuda_fail("k_rows_inverse_s3 smem", e) : check_launch("k_rows_inverse_s3");
    }
  }
  if (!split_r) dispatch_len(a.lx, [&]<int LX>() {
    if constexpr (!kPairSpectra<C> || LX <= 512)  // (complex64 of length 1024 is split)
    with_plan<LX>(a.precision, [&]<int V>() {
      cudaError_t e;
      if constexpr (sizeof(C) == sizeof(double2) && LX <= 128) {
        if (small_r) {
          constexpr int U = Small64<LX>::UNITS;
          auto kern = a.epi == 1 ? k_rows_inverse_small<LX, 1, V> : a.epi == 2 ? k_rows_inverse_small<LX, 2, V>
                                                                               : k_rows_inverse_small<LX, 0, V>;
          launch_pdl(kern, dim3((a.nz + U - 1) / U, nb), 32, Small64<LX>::lines, s, p);
          rc = check_launch("k_rows_inverse_small");
          return;
        }
      }
      with_tile<C, LX>(small_r, [&]<int NTT>() {
        using RC = RowCfg<C, LX, NTT>;
        const size_t bytes = rows_inverse_smem<C, LX, NTT>();
        dim3 grid((a.nz + RC::ROWS - 1) / RC::ROWS, nb);
        auto launch = [&](auto kernel) {
          e = allow_smem(kernel, bytes);
          if (e == cudaSuccess) launch_pdl(kernel, grid, RC::NT, bytes, s, p);
        };
        if (a.epi == 1) launch(k_rows_inverse<C, LX, 1, V, NTT>);
        else if (a.epi == 2) launch(k_rows_inverse<C, LX, 2, V, NTT>);
        else launch(k_rows_inverse<C, LX, 0, V, NTT>);
      });
      rc = e != cudaSuccess ? cuda_fail("k_rows_inverse smem", e) : check_launch("k_rows_inverse");
    });
  });
  prof_mark(PROF_ROWS_INVERSE, true, s);
  return rc;
}

template <typename C> static int run_typed(const OpArgs &a, cudaStream_t s) {
  const int nb = a.plist ? a.nb : a.B;
  if (nb <= 0) return DBI_OK;
  dbi_grid g{a.nz, a.nx, a.lz, a.lx, a.h};
  const int chunk = spectral_chunk(&g, a.B, a.precision);
  int rc = DBI_OK;
  prof_mark(PROF_OPERATOR, false, s);
  for (int s0 = 0; s0 < nb && rc == DBI_OK; s0 += chunk)
    rc = run_chunk<C>(a, s0, std::min(chunk, nb - s0), chunk, s);
  prof_mark(PROF_OPERATOR, true, s);
  return rc;
}

int operator_parts(int B, int nz, int lx, int precision) {
  static_assert(kS3Units == kSplitRows, "split row tiles hold the same number of rows");
  if (split_rows(lx, precision)) return (nz + kSplitRows - 1) / kSplitRows;
  if (small_rows(B, nz, lx, precision, true)) {
    int rows = 1;
    dispatch_len(lx, [&]<int LX>() {
      if constexpr (LX <= 128) rows = Small64<LX>::UNITS;
      else rows = RowCfg<double2, LX, kSmallThreads<LX>>::ROWS;
    });
    return (nz + rows - 1) / rows;
  }
  return operator_parts_k(nz, lx, precision);
}

int operator_parts_k(int nz, int lx, int precision) {
  int rows = 1;
  auto pick = [&](auto tag) {
    using C = decltype(tag);
    dispatch_len(lx, [&]<int LX>() { rows = RowCfg<C, LX>::ROWS; });
  };
  if (precision == DBI_C64) pick(float2{});
  else pick(double2{});
  return (nz + rows - 1) / rows;
}

int run_operator(const OpArgs &a, cudaStream_t s) {
  if (a.ny > 0) return run_operator_3d(a, s);
  if (a.group) return run_group_operator(a, s);
  if (a.Dhat) return run_form_k(a, s);
  return a.precision == DBI_C64 ? run_typed<float2>(a, s) : run_typed<double2>(a, s);
}

}  // namespace dbi

using namespace dbi;

// Common validation of the operator entry points.
static int check_op(const dbi_grid *g, const dbi_batch *batch, const void *Ghat, const void *in,
                    const void *out, int precision, void *work, size_t work_bytes, int op) {
  int rc;
  if ((rc = check_grid(g, precision)) || (rc = check_batch(batch)) || (rc = check_precision(precision))) return rc;
  if (batch->B > 0 && (!Ghat || !in || !out)) { set_error("NULL Ghat, input or output"); return DBI_ERR_ARG; }
  if (in == out && batch->B > 0) { set_error("input and output must be distinct buffers"); return DBI_ERR_ARG; }
  const size_t need = dbi_workspace_bytes(g, batch->B, precision, op);
  if (batch->B > 0 && (!work || work_bytes < need)) {
    set_error("work buffer of %zu bytes, need %zu", work_bytes, need);
    return DBI_ERR_WORKSPACE;
  }
  return DBI_OK;
}

extern "C" int green_convolve(const dbi_grid *g, const dbi_batch *batch, const void *Ghat,
                              const void *src, void *out, int precision, void *work,
                              size_t work_bytes, dbi_stream stream) {
  clear_error();
  int rc = check_op(g, batch, Ghat, src, out, precision, work, work_bytes, DBI_OP_CONVOLVE);
  if (rc || batch->B == 0) return rc;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  Arena ar(work, work_bytes);
  void *tw = ar.take(bytes_twiddles(precision));
  void *T = ar.take(bytes_spectral(g, batch->B, precision));
  Scales sc = carve_scales(ar, batch->B);
  if ((rc = ar.check(__func__))) return rc;
  if ((rc = launch_twiddles(tw, precision, s))) return rc;
  if ((rc = pow2_scales(src, precision, false, batch->B, size_t(2) * g->nz * g->nx, sc.part, sc.scale, sc.inv,
                        nullptr, s)))
    return rc;
  OpArgs a{};
  a.precision = precision; a.nz = g->nz; a.nx = g->nx; a.lz = g->lz; a.lx = g->lx; a.h = g->h;
  a.B = batch->B; a.nf = batch->nf; a.omega = batch->omega; a.fidx = batch->fidx;
  a.stencil = false; a.in = src; a.ident = nullptr; a.out = out; a.T = T; a.Ghat = Ghat; a.tw = tw;
  a.in_scale = sc.scale; a.out_scale = sc.inv;
  return run_operator(a, s);
}

extern "C" int ls_apply(const dbi_model *model, const dbi_batch *batch, const void *Ghat,
                        const void *u, void *out, int precision, void *work, size_t work_bytes,
                        dbi_stream stream) {
  clear_error();
  if (!model) { set_error("model is NULL"); return DBI_ERR_ARG; }
  const dbi_grid *g = &model->grid;
  int rc = check_op(g, batch, Ghat, u, out, precision, work, work_bytes, DBI_OP_APPLY);
  if (rc || batch->B == 0) return rc;
  if (!model->m) { set_error("model->m is NULL"); return DBI_ERR_ARG; }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  Arena ar(work, work_bytes);
  void *tw = ar.take(bytes_twiddles(precision));
  void *T = ar.take(bytes_spectral(g, batch->B, precision));
  Scales sc = carve_scales(ar, batch->B);
  if ((rc = ar.check(__func__))) return rc;
  if ((rc = launch_twiddles(tw, precision, s))) return rc;
  if ((rc = pow2_scales(u, precision, false, batch->B, size_t(2) * g->nz * g->nx, sc.part, sc.scale, sc.inv,
                        nullptr, s)))
    return rc;
  OpArgs a{};
  a.precision = precision; a.nz = g->nz; a.nx = g->nx; a.lz = g->lz; a.lx = g->lx; a.h = g->h;
  a.B = batch->B; a.nf = batch->nf; a.omega = batch->omega; a.fidx = batch->fidx;
  a.m = model->m; reference_values(model->ref, a.ref);
  a.stencil = true; a.in = u; a.ident = u; a.out = out; a.T = T; a.Ghat = Ghat; a.tw = tw;
  a.in_scale = sc.scale; a.out_scale = sc.inv;
  return run_operator(a, s);
}
