// Device helpers of the batched Krylov solvers (BiCGSTAB in krylov.cu, GMRES in gmres.cu).
#pragma once

#include "operator.cuh"
#include "reduce.cuh"

namespace dbi {

template <typename C> struct Acc;                         // per-thread accumulation type
template <> struct Acc<float2> { using type = float; };   // sums of a thread and of a warp, then FP64
template <> struct Acc<double2> { using type = double; };

__device__ __forceinline__ double2 zdiv(double2 a, double2 b) {
  const double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C from_z(double2 z) {
  using R = typename RealOf<C>::type;
  return mk<C>(R(z.x), R(z.y));
}

// Problem of this CTA: plist[blockIdx.y] when the launch runs a compacted list of problems.
__device__ __forceinline__ int problem_at(const int *plist, int slot) { return plist ? plist[slot] : slot; }

// Grid-stride loop over the n elements of problem b (unrolled for memory parallelism).
#define DBI_PROBLEM_LOOP(sp)                                                                  \
  const size_t off = (sp).offset(b), cnt = (sp).count(b);                                     \
  _Pragma("unroll 4")                                                                         \
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < cnt; i += size_t(gridDim.x) * blockDim.x)

// Grid-stride loop over the elements of problem b calling f.template operator()<N>(o) for the N
// consecutive elements from offset o: N = 2 (a 16-byte pair of complex64 values, loaded and stored
// with one instruction by ldN / stN) when the problem's offset and count are even, else N = 1.
template <typename C, typename F>
__device__ __forceinline__ void problem_loop_pairs(const Span &sp, int b, F &&f) {
  const size_t off = sp.offset(b), cnt = sp.count(b);
  const size_t i0 = size_t(blockIdx.x) * blockDim.x + threadIdx.x, step = size_t(gridDim.x) * blockDim.x;
  if (sizeof(C) == sizeof(float2) && ((off | cnt) & 1) == 0) {
#pragma unroll 2
    for (size_t i = i0; i < cnt / 2; i += step) f.template operator()<2>(off + 2 * i);
  } else {
#pragma unroll 4
    for (size_t i = i0; i < cnt; i += step) f.template operator()<1>(off + i);
  }
}
template <int N, typename C> __device__ __forceinline__ void ldN(const C *p, C (&v)[N]) {
  if constexpr (N == 2 && sizeof(C) == sizeof(float2)) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = mk<C>(q.x, q.y);
    v[1] = mk<C>(q.z, q.w);
  } else {
#pragma unroll
    for (int n = 0; n < N; ++n) v[n] = p[n];
  }
}
template <int N, typename C> __device__ __forceinline__ void stN(C *p, const C (&v)[N]) {
  if constexpr (N == 2 && sizeof(C) == sizeof(float2)) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  } else {
#pragma unroll
    for (int n = 0; n < N; ++n) p[n] = v[n];
  }
}

// NS sums over problem b, as partials part[c kRedSlots + k], c < nchunk. Complex64: the problem's items (pairs
// of elements as in problem_loop_pairs, or single ones) are dealt to kRedBlocks chunks in turn,
// kRedThreads at a time, and a partial is the sum over a chunk: thread t of the CTA that has chunk c adds
// its items (c + kRedBlocks j) kRedThreads + t and its warp adds the threads, both in FP32, then the
// warps are added in FP64. f.template operator()<N>(o, acc) treats the N elements from offset o and adds to
// acc. CTA blockIdx.x has the chunks blockIdx.x + gridDim.x j, at most kMaxChunks: how many CTAs share
// a problem follows the batch (red_blocks), but neither how much of a sum is added in FP32 nor its bits do.
// (With one FP32 sum per warp over all of its CTA's items a warp added 512 elements of a 128^2 problem of 64,
// now 64; the solves keep their time.) Complex128: FP64 throughout, one partial per CTA (nchunk =
// gridDim.x; chunks cost 2 to 3 % of a solve, k_update_xr of 15 problems of up to 256^2 85 against 72 us).
constexpr int kMaxChunks = 16;
template <int NS, typename C, bool PAIRS = true, typename F>
__device__ __forceinline__ void problem_sums(const Span &sp, int b, int nchunk, double *part, F &&f) {
  using A = typename Acc<C>::type;
  const size_t off = sp.offset(b), cnt = sp.count(b);
  if constexpr (sizeof(C) != sizeof(float2)) {
    A acc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0;
#pragma unroll 4
    for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < cnt; i += size_t(gridDim.x) * blockDim.x)
      f.template operator()<1>(off + i, acc);
    block_sum_store<NS>(acc, part + size_t(blockIdx.x) * kRedSlots);
    return;
  }
  constexpr int kWarps = kRedThreads / 32;
  __shared__ double sh[kMaxChunks][NS][kWarps];
  const size_t step = size_t(kRedBlocks) * kRedThreads;
  const bool two = PAIRS && ((off | cnt) & 1) == 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int n = 0;
  for (int c = blockIdx.x; c < nchunk; c += gridDim.x, ++n) {
    const size_t i0 = size_t(c) * kRedThreads + threadIdx.x;
    A acc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0;
    if (two) {
      if constexpr (PAIRS) {
#pragma unroll 2
        for (size_t i = i0; i < cnt / 2; i += step) f.template operator()<2>(off + 2 * i, acc);
      }
    } else {
#pragma unroll 4
      for (size_t i = i0; i < cnt; i += step) f.template operator()<1>(off + i, acc);
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      A a = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
      if (lane == 0) sh[n][k][warp] = double(a);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * NS; i += kRedThreads) {
    double a = 0.0;
    for (int w = 0; w < kWarps; ++w) a += sh[i / NS][i % NS][w];
    part[(blockIdx.x + size_t(i / NS) * gridDim.x) * kRedSlots + i % NS] = a;
  }
  __syncthreads();
}

// 2^-e with m in [2^e, 2^(e+1)), or 1 when m = 0.
__device__ __forceinline__ double pow2_below(double m) { return m > 0.0 ? ldexp(1.0, -ilogb(m)) : 1.0; }

}  // namespace dbi
