// Contrast source and forward row FFT of complex64 problems in one pass down the rows (lengths 128
// to 512): thread x walks column x of a chunk of rows with the z-neighbours of u and of the stress in
// registers (as source_rows of op_split.cuh), and every four rows the CTA transforms the sources it
// has just formed and stores them transposed.
//
// The tile form (rows_forward_tile) reads u at eight rows and forms the stress at six for every four
// rows of output; here a chunk of 32 rows pays the two rows above and below it once: 110 M -> 79 M
// warp instructions per 128 problems of 256^2, 308 -> 262 us per 256. Bound by shared memory (74 % of its
// wavefronts) and its latency.
// LX / 2 threads: one per column (nx <= LX / 2), and T = LX / 8 per row of the transform of four rows.
#pragma once

#include "op_tiles.cuh"

namespace dbi {

template <int LX> struct StreamCfg {
  static constexpr int T = LX / 8, ROWS = 4, NT = LX / 2, W = NT + 2;
  static constexpr int PLP = row_pitch<LX, ROWS>;
  // u and sigma rows [2][W] each, the sources [4][NT], then the FFT lines
  static constexpr size_t ring = size_t(4) * W, src = size_t(ROWS) * NT;
  static constexpr size_t fft = size_t(ROWS) * PLP;
  static constexpr size_t smem = (ring + src + fft) * sizeof(cpair);
};

// Rows [zb, ze) of one problem (ze - zb a multiple of four or ze = nz).
template <int LX, int V, typename A>
__device__ __forceinline__ void rows_stream(const A &a, int zb, int ze, float4 *smem) {
  using S = StreamCfg<LX>;
  using C = float2;
  constexpr int T = S::T, NT = S::NT, W = S::W;
  const int nz = a.nz(), nx = a.nx(), x = threadIdx.x;
  const size_t plane = size_t(nz) * nx;
  const bool col = x < nx;
  const int xc = col ? x : 0;
  const float isc = a.isc(), ms = a.ms(), f = a.inv2h(), w2 = a.w2();
  const float q0 = a.ref(0), q1 = a.ref(1), q2 = a.ref(2), q3 = a.ref(3), q4 = a.ref(4);
  const C *u1p = a.in() + xc, *u3p = u1p + plane;
  const float *m0 = a.m() + xc;
  // (u1, u3) and (sigma1, sigma5) of two rows each by parity, index x + 1; the columns x = -1 and x >= nx
  // stay zero
  float4 *su = smem + 1, *sg = su + 2 * W;
  float4 *so = smem + S::ring;
  cpair *ps = reinterpret_cast<cpair *>(so + S::src);
  for (int i = threadIdx.x; i < 4 * W; i += NT) smem[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto in_d = [&](int z) { return col && unsigned(z) < unsigned(nz); };
  auto load_u = [&](int z, C &v1, C &v3) {
    const bool in = in_d(z);
    const int o = in ? z * nx : 0;
    v1 = in ? __ldg(u1p + o) : czero<C>();
    v3 = in ? __ldg(u3p + o) : czero<C>();
  };
  struct Stiff {
    float d11, d13, d33, d55;
  };
  auto load_stiff = [&](int z, Stiff &d) {
    const bool in = in_d(z);
    const float *mz = m0 + (in ? z * nx : 0);
    d.d11 = in ? __ldg(mz + 1 * plane) : q1;
    d.d13 = in ? __ldg(mz + 2 * plane) : q2;
    d.d33 = in ? __ldg(mz + 3 * plane) : q3;
    d.d55 = in ? __ldg(mz + 4 * plane) : q4;
  };
  auto load_rho = [&](int z) { return in_d(z) ? __ldg(m0 + z * nx) : q0; };
  // window: u at rows j - 1, j (scaled); sigma3, sigma5 at rows j - 2, j - 1; loads one step ahead
  C ua1, ua3, ub1, ub3, nu1, nu3;
  C s3a = czero<C>(), s5a = czero<C>(), s3b = czero<C>(), s5b = czero<C>();
  Stiff nd;
  float nrho;
  const int j0 = zb - 1;  // odd (zb is a multiple of four), so step parities are static
  load_u(j0 - 1, ua1, ua3);
  load_u(j0, ub1, ub3);
  ua1 = cscale(ua1, isc); ua3 = cscale(ua3, isc);
  ub1 = cscale(ub1, isc); ub3 = cscale(ub3, isc);
  load_u(j0 + 1, nu1, nu3);
  load_stiff(j0, nd);
  nrho = load_rho(j0 - 1);
  __syncthreads();  // the zero fill precedes every row store
  if (col) su[(j0 & 1) * W + x] = make_float4(ub1.x, ub1.y, ub3.x, ub3.y);
  __syncthreads();
  // Step j: stress of row j from u one row up and down (registers) and one column left and right (shared
  // memory), source of row j - 1 likewise from the stress; then u of row j + 1 and the stress of row
  // j are stored for the next step. P = j & 1; `o`: where the source goes, or NULL.
  auto step = [&]<int P>(int j, float4 *o) {
    const C uc1 = cscale(nu1, isc), uc3 = cscale(nu3, isc);
    const Stiff d = nd;
    const float rho = nrho;
    load_u(j + 2, nu1, nu3);  // the next step's loads
    load_stiff(j + 1, nd);
    nrho = load_rho(j);
    C s1 = czero<C>(), s3 = czero<C>(), s5 = czero<C>();
    if (in_d(j)) {
      const float4 r = su[P * W + x + 1], l = su[P * W + x - 1];
      const C e1 = cscale(mk<C>(r.x - l.x, r.y - l.y), f);
      const C e3 = cscale(csub(uc3, ua3), f);
      const C e5 = cscale(cadd(csub(uc1, ua1), mk<C>(r.z - l.z, r.w - l.w)), f);
      const float d11 = (d.d11 - q1) * ms, d13 = (d.d13 - q2) * ms, d33 = (d.d33 - q3) * ms, d55 = (d.d55 - q4) * ms;
      s1 = cadd(cscale(e1, d11), cscale(e3, d13));
      s3 = cadd(cscale(e1, d13), cscale(e3, d33));
      s5 = cscale(e5, d55);
    }
    if (o) {
      float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
      if (in_d(j - 1)) {
        const float4 r = sg[(P ^ 1) * W + x + 1], l = sg[(P ^ 1) * W + x - 1];
        const C o1 = cscale(cadd(mk<C>(r.x - l.x, r.y - l.y), csub(s5, s5a)), f);
        const C o3 = cscale(cadd(mk<C>(r.z - l.z, r.w - l.w), csub(s3, s3a)), f);
        const float wr = w2 * (rho - q0) * ms;
        const C y1 = cadd(o1, cscale(ua1, wr)), y3 = cadd(o3, cscale(ua3, wr));  // u(j - 1)
        w = make_float4(y1.x, y3.x, y1.y, y3.y);  // as a pair
      }
      o[x] = w;
    }
    if (col) {
      su[(P ^ 1) * W + x] = make_float4(uc1.x, uc1.y, uc3.x, uc3.y);
      sg[P * W + x] = make_float4(s1.x, s1.y, s5.x, s5.y);
    }
    __syncthreads();
    ua1 = ub1; ua3 = ub3; ub1 = uc1; ub3 = uc3;
    s3a = s3b; s5a = s5b; s3b = s3; s5b = s5;
  };
  step.template operator()<1>(j0, nullptr);
  step.template operator()<0>(j0 + 1, nullptr);
  const int rr = threadIdx.x / T, t = threadIdx.x - rr * T;
  const int r = threadIdx.x % 4, tq = threadIdx.x / 4;
  const TwReg<C, LX, V> tr(t, tq, a.tw());
  for (int z0 = zb; z0 < ze; z0 += 4) {
    step.template operator()<1>(z0 + 1, so);
    step.template operator()<0>(z0 + 2, so + NT);
    step.template operator()<1>(z0 + 3, so + 2 * NT);
    step.template operator()<0>(z0 + 4, so + 3 * NT);
    cpair p[1][8];
#pragma unroll
    for (int m = 0; m < 8; ++m) p[0][m] = m < kHalf ? reinterpret_cast<const cpair *>(so)[rr * NT + t + m * T] : pzero();
    cpair *const line[1] = {ps + size_t(rr) * S::PLP}, *const line2[1] = {ps + size_t(r) * S::PLP};
    RegPlan<LX, V>::template run_regrouped<cpair, 1, false, PlanInfo<LX, V>::np - 2, true>(
        p, line, t, line2, tq, tr, RowSync<T>{1 + rr}, CtaSync{});
    cpair *Tp = reinterpret_cast<cpair *>(a.T()) + z0 + r;
    if (z0 + r < nz) {
#pragma unroll
      for (int m = 0; m < 8; ++m) Tp[size_t(tq + m * T) * nz] = p[0][m];
    }
  }
}

}  // namespace dbi
