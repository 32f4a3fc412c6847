// Four-step time-axis FFT for any ell = L1 L2 = 2^a 3^b 5^c with run-time
// factors, in FP32 and FP64: the lengths and precisions that the power-of-two
// FP32 kernels of fft_four.cuh do not serve.
//
// The factorisation, the four kernels and the intermediate's layout
// [k1][t2][complex column] are those of fft_four.cuh; here L1 and L2 are
// kernel arguments.  A CTA holds the rows of 32 complex columns of G values of
// t2 (L1 rows each) or of G k1 groups (two members of L2 rows each) in shared
// memory; a warp takes one butterfly of all 32 columns at a time (lane =
// column), so every index, twiddle and branch is uniform over the warp and
// its run-time arithmetic is paid once per 32 columns.  G fills the eight
// warps where the factors are short: with one t2 of 8 rows per CTA (ell =
// 128) a pass had one butterfly, and the kernels took 9-10 us each at n 8191.
// The passes run out of place between two buffers, so that a thread holds one butterfly: in place, with all butterflies of a
// warp in registers between two barriers, the run-time radices spilled 1 to 8
// KB a thread and the kernels ran at half the speed.
//
// Why: the single mixed-radix kernel holds whole time series, 8 columns of
// ell = 1440 in 196 KB, which left 98 CTAs of 8 warps for n = 1568 (12% of the
// warps; 44 us forward, 35-59 us inverse), and the FP64 panel kernels had 64
// CTAs for n = 1024, ell = 1024, their FP64 pipe 82% busy on 64 of 152 SMs
// (75 + 52 us, with row passes of 7 and 21 us).  Here the same shapes give
// 25 x 30 (outer kernels) and 25 x 13 (middle ones), 16 x 32 and 16 x 17 CTAs.
// FP64 is bound by the FP64 pipe, FP32 by latency and issue.
//
// The kernels are launched as dependents but do not let their successors be
// scheduled early: CTAs that wait beside the last ones cost more than their
// prologues save (whole applies with the trigger / without, n 63 ... 65535 x ell
// 16 ... 4096: 1.02 on average, n 1023 x ell 512 in FP64 1.19, n 1023 x ell 500 in
// FP32 1.14, n 5000 x ell 40 0.92).
#pragma once
#include "fft_time.cuh"
#include "fft_mixed.cuh"

namespace aao {
namespace fft {
namespace {   // included by both precision units: one private copy each

constexpr int kStepT = 256, kStepW = 32, kStepWarps = kStepT / 32;
// Shorter transforms run as one kernel.
#ifndef AAO_STEPS_MIN
#define AAO_STEPS_MIN 16
#endif

// Resident CTAs per SM the kernels are compiled for.
template <typename R> struct StepOcc { static constexpr int V = sizeof(R) == 8 ? 3 : 4; };

// Twiddles.  The rounding errors of a table are the same in the forward and in
// the inverse transform, and a four-step transform applies its middle twiddles
// to whole classes of frequencies: with rounded tables on both sides their
// product acts on the low frequencies that P^{-1} amplifies with one sign for
// every input.  The refined apply lives on the product of two such errors and
// was up to three times as far off as with one kernel per direction (1.27 times
// over 287 sizes).  So the FP32 forward transform takes its twiddles and
// constants with what their rounding left out (re, im, re lo, im lo of
// e^{-2 pi i m/ell}): 0.59 times over the same sizes, no length above 1.02, for
// 1.3% of the time (5% at n 2047 x ell 1440).  The inverse with full tables in
// its place: 0.61, ell = 16 at 1.07; both: 0.54, for 2% (7%).
template <typename R, int DIR> struct StepTw {
  static constexpr bool FULL = sizeof(R) == 4 && DIR < 0;
  using T = typename std::conditional<FULL, float4, cx<R>>::type;
};
template <typename R, int DIR> using step_tw = typename StepTw<R, DIR>::T;
template <typename R, int DIR>
inline const step_tw<R, DIR> *step_table(const StepPlan &pl, const cx<R> *tw) {
  if constexpr (StepTw<R, DIR>::FULL) return pl.tw32;
  else return tw;
}

template <typename R, int DIR>
__device__ __forceinline__ cx<R> twiddle_step(cx<R> v, cx<R> w) {
  return twiddle<R, DIR>(v, w);
}
template <typename R, int DIR>
__device__ __forceinline__ cx<float> twiddle_step(cx<float> v, float4 w) {
  return twiddle_full<DIR>(v, w);
}

// ---- butterflies beyond fft_time.cuh's 2, 4, 8, 16 and fft_mixed.cuh's 3, 5
// (refined apply at ell = 200 = 8 x 25, error against one kernel per direction:
// 2.3 with rounded tables, 1.35 with full twiddles and rounded constants, 0.85)
template <typename R, int DIR> __device__ __forceinline__ R const_fma(R x, double c, R y) {
  if constexpr (StepTw<R, DIR>::FULL) {
    const float h = (float)c, l = (float)(c - (double)h);
    return __fmaf_rn(x, h, __fmaf_rn(x, l, y));
  } else {
    return fma(x, (R)c, y);
  }
}
template <typename R, int DIR> __device__ __forceinline__ R const_mul(R x, double c) {
  if constexpr (StepTw<R, DIR>::FULL) {
    const float h = (float)c, l = (float)(c - (double)h);
    return __fmaf_rn(x, h, x * l);
  } else {
    return x * (R)c;
  }
}
// times e^{DIR i th}, c = cos th, s = sin th
template <typename R, int DIR>
__device__ __forceinline__ cx<R> const_rot(cx<R> z, double c, double s) {
  if constexpr (StepTw<R, DIR>::FULL) {
    const float ch = (float)c, sh = (float)s;
    return twiddle_step<R, DIR>(z, make_float4(ch, -sh, (float)(c - (double)ch), (float)((double)sh - s)));
  } else {
    return twiddle_step<R, DIR>(z, mk((R)c, (R)-s));
  }
}

template <typename R, int DIR>
__device__ __forceinline__ void step_dft3(cx<R> *v) {
  const double h = 0.86602540378443864676;   // sin(2 pi / 3)
  const cx<R> s = v[1] + v[2], d = v[1] - v[2];
  const cx<R> m = mk(v[0].re - (R)0.5 * s.re, v[0].im - (R)0.5 * s.im);
  const cx<R> jd = rot90<R, DIR>(mk(const_mul<R, DIR>(d.re, h), const_mul<R, DIR>(d.im, h)));
  v[0] = v[0] + s;
  v[1] = m + jd;
  v[2] = m - jd;
}

template <typename R, int DIR>
__device__ __forceinline__ void step_dft5(cx<R> *v) {
  const double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;   // cos(2pi/5), cos(4pi/5)
  const double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;    // sin(2pi/5), sin(4pi/5)
  const cx<R> t1 = v[1] + v[4], t2 = v[2] + v[3], t3 = v[1] - v[4], t4 = v[2] - v[3], x0 = v[0];
  auto lin = [](cx<R> x, cx<R> p, double a, cx<R> q, double b) {   // x + a p + b q
    return mk(const_fma<R, DIR>(q.re, b, const_fma<R, DIR>(p.re, a, x.re)), const_fma<R, DIR>(q.im, b, const_fma<R, DIR>(p.im, a, x.im)));
  };
  auto lin0 = [](cx<R> p, double a, cx<R> q, double b) {           // a p + b q
    return mk(const_fma<R, DIR>(q.re, b, const_mul<R, DIR>(p.re, a)), const_fma<R, DIR>(q.im, b, const_mul<R, DIR>(p.im, a)));
  };
  const cx<R> a1 = lin(x0, t1, c1, t2, c2), a2 = lin(x0, t1, c2, t2, c1);
  const cx<R> b1 = rot90<R, DIR>(lin0(t3, s1, t4, s2)), b2 = rot90<R, DIR>(lin0(t3, s2, t4, -s1));
  v[0] = x0 + t1 + t2;
  v[1] = a1 + b1;
  v[4] = a1 - b1;
  v[2] = a2 + b2;
  v[3] = a2 - b2;
}

// 8 = 2 x 4: n = q + 2m, k = k1 + 4 k2
template <typename R, int DIR>
__device__ __forceinline__ void step_dft8(cx<R> *v) {
  const double c8 = 0.70710678118654752440;   // cos(pi / 4)
  cx<R> b[2][4];
#pragma unroll
  for (int q = 0; q < 2; q++) {
    b[q][0] = v[q]; b[q][1] = v[q + 2]; b[q][2] = v[q + 4]; b[q][3] = v[q + 6];
    dft4<R, DIR>(b[q][0], b[q][1], b[q][2], b[q][3]);
  }
  b[1][1] = const_rot<R, DIR>(b[1][1], c8, c8);
  b[1][2] = rot90<R, DIR>(b[1][2]);
  b[1][3] = const_rot<R, DIR>(b[1][3], -c8, c8);
#pragma unroll
  for (int k1 = 0; k1 < 4; k1++) {
    v[k1] = b[0][k1] + b[1][k1];
    v[k1 + 4] = b[0][k1] - b[1][k1];
  }
}

// 6 = 2 x 3 and 10 = 2 x 5 by the Good-Thomas index maps (no twiddles):
// n = n1 M + 2 n2, k = M k1 + (M + 1) k2 mod 2M for M = 3, 5 (2^-1 mod M =
// (M + 1)/2).
template <typename R, int DIR, int M>
__device__ __forceinline__ void dft_2m(cx<R> *v) {
  cx<R> a[2][M];
#pragma unroll
  for (int q = 0; q < M; q++) {
    const cx<R> x0 = v[(2 * q) % (2 * M)], x1 = v[(M + 2 * q) % (2 * M)];
    a[0][q] = x0 + x1;
    a[1][q] = x0 - x1;
  }
#pragma unroll
  for (int q = 0; q < 2; q++) {
    if constexpr (M == 3) step_dft3<R, DIR>(a[q]);
    else step_dft5<R, DIR>(a[q]);
  }
#pragma unroll
  for (int q = 0; q < M; q++) {
    v[((M + 1) * q) % (2 * M)] = a[0][q];
    v[(M + (M + 1) * q) % (2 * M)] = a[1][q];
  }
}

// 9 = 3 x 3 (Cooley-Tukey, w = exp(DIR 2 pi i / 9)).
template <typename R, int DIR>
__device__ __forceinline__ void dft9(cx<R> *v) {
  cx<R> a[3][3];
#pragma unroll
  for (int q = 0; q < 3; q++) {
    a[q][0] = v[q]; a[q][1] = v[q + 3]; a[q][2] = v[q + 6];
    step_dft3<R, DIR>(a[q]);
  }
  const double c1 = 0.76604444311897803520, s1 = 0.64278760968653932632;    // 2 pi / 9
  const double c2 = 0.17364817766693034885, s2 = 0.98480775301220805937;    // 4 pi / 9
  const double c4 = -0.93969262078590838405, s4 = 0.34202014332566873304;   // 8 pi / 9
  a[1][1] = const_rot<R, DIR>(a[1][1], c1, s1);
  a[1][2] = const_rot<R, DIR>(a[1][2], c2, s2);
  a[2][1] = const_rot<R, DIR>(a[2][1], c2, s2);
  a[2][2] = const_rot<R, DIR>(a[2][2], c4, s4);
#pragma unroll
  for (int k1 = 0; k1 < 3; k1++) {
    cx<R> b[3] = {a[0][k1], a[1][k1], a[2][k1]};
    step_dft3<R, DIR>(b);
    v[k1] = b[0]; v[k1 + 3] = b[1]; v[k1 + 6] = b[2];
  }
}

template <typename R, int DIR, int RAD>
__device__ __forceinline__ void dft_step(cx<R> *v) {
  if constexpr (RAD == 6) dft_2m<R, DIR, 3>(v);
  else if constexpr (RAD == 10) dft_2m<R, DIR, 5>(v);
  else if constexpr (RAD == 9) dft9<R, DIR>(v);
  else if constexpr (RAD == 3) step_dft3<R, DIR>(v);
  else if constexpr (RAD == 5) step_dft5<R, DIR>(v);
  else if constexpr (RAD == 8 && StepTw<R, DIR>::FULL) step_dft8<R, DIR>(v);
  else dft<R, DIR, RAD>(v);
}

// q / d for 0 <= q < 512, 1 <= d <= 128 by a multiplication (exact: the error
// of ceil(2^16 / d) is below 1, and 512 <= 2^16 / d).
struct SmallDiv {
  unsigned m;
  __device__ __forceinline__ explicit SmallDiv(int d) : m((65536u + (unsigned)d - 1u) / (unsigned)d) {}
  __device__ __forceinline__ int operator()(int q) const { return (int)(((unsigned)q * m) >> 16); }
};

// One Stockham pass of radix RAD over nmem buffers of N rows each (buffer m
// at src + m N 32), out of place.  nmem N <= 256 rows in all.
template <typename R, int DIR, int RAD>
__device__ __forceinline__ void pass_step(const cx<R> *src, cx<R> *dst, int nmem, int N, int Ns,
                                          int L, const step_tw<R, DIR> *__restrict__ tw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = N / RAD, tot = nmem * nb, tstep = L / (Ns * RAD);
  const SmallDiv by_nb(nb), by_ns(Ns);
  for (int b = warp; b < tot; b += kStepWarps) {
    const int m = by_nb(b), j = b - m * nb;
    const int jd = by_ns(j), jm = j - jd * Ns;
    const cx<R> *s = src + (m * N + j) * kStepW + lane;
    cx<R> v[RAD];
#pragma unroll
    for (int r = 0; r < RAD; r++) v[r] = s[r * nb * kStepW];
    if (jm) {
#pragma unroll
      for (int r = 1; r < RAD; r++) v[r] = twiddle_step<R, DIR>(v[r], tw[jm * tstep * r]);
    }
    dft_step<R, DIR, RAD>(v);
    cx<R> *d = dst + (m * N + jd * Ns * RAD + jm) * kStepW + lane;
#pragma unroll
    for (int r = 0; r < RAD; r++) d[r * Ns * kStepW] = v[r];
  }
}

// N-point DFTs down the rows of every column of nmem buffers, natural order
// in and out, between a (the input) and b; returns the buffer that holds the
// result.  All threads call it; a barrier before it is the caller's.
template <typename R, int DIR>
__device__ __forceinline__ cx<R> *dft_steps(cx<R> *a, cx<R> *b, int nmem, int N, int np,
                                            const int *rad, int L, const step_tw<R, DIR> *__restrict__ tw) {
  int Ns = 1;
  for (int p = 0; p < np; p++) {
    const int r = rad[p];
#define AAO_PS(RAD) case RAD: pass_step<R, DIR, RAD>(a, b, nmem, N, Ns, L, tw); break;
    switch (r) {
      AAO_PS(2) AAO_PS(3) AAO_PS(4) AAO_PS(5) AAO_PS(6) AAO_PS(8) AAO_PS(9) AAO_PS(10)
      default: break;
    }
#undef AAO_PS
    __syncthreads();
    Ns *= r;
    cx<R> *t = a; a = b; b = t;
  }
  return a;
}

constexpr int kStepB = 8;   // rows a warp keeps in flight

// Forward 1.  grid (ncx / 32, ceil(L2 / G) groups of t2); 2 G L1 x 32 complex
// of dynamic shared memory.  XT: stored input type; NEUMANN: the input is
// x - E y (load_real).
template <typename R, typename XT, bool NEUMANN, typename YT>
__global__ void __launch_bounds__(kStepT, StepOcc<R>::V)
k_steps_forward1(const XT *__restrict__ x, const YT *__restrict__ y, const R *__restrict__ sigk,
                 cx<R> *__restrict__ inter, int n, int ncx, const step_tw<R, -1> *__restrict__ tw,
                 StepPlan pl, int G) {
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<R> *S = reinterpret_cast<cx<R> *>(smraw);
  R *Sf = reinterpret_cast<R *>(smraw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int L1 = pl.L1, L2 = pl.L2, t20 = blockIdx.y * G;
  const int ng = min(G, L2 - t20), rows = ng * L1;           // t2 values here
  const int i0 = 2 * kStepW * blockIdx.x;
  const SmallDiv by_l1(L1);
  const unsigned long long pol_stream = l2_evict_first(), pol_keep = l2_evict_last();
  pdl_wait(x, y);
  for (int q0 = 0; q0 < rows; q0 += kStepB * kStepWarps) {
    if constexpr (NEUMANN) {
#pragma unroll
      for (int u = 0; u < kStepB; u++) {
        const int q = q0 + warp + u * kStepWarps, gi = by_l1(q), t1 = q - gi * L1;
        if (q < rows) {
#pragma unroll
          for (int h = 0; h < 2; h++)
            Sf[q * 2 * kStepW + h * 32 + lane] = load_real<R, 0, true, YT>(
                x, y, sigk, n, L2 * t1 + t20 + gi, i0 + h * 32 + lane, pol_stream);
        }
      }
    } else {
      XT d[kStepB][2];
#pragma unroll
      for (int u = 0; u < kStepB; u++) {
        const int q = q0 + warp + u * kStepWarps, gi = by_l1(q), t1 = q - gi * L1;
        const XT *row = x + (size_t)(L2 * t1 + t20 + gi) * n + i0 + lane;
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const bool in = q < rows && i0 + h * 32 + lane < n;
          if constexpr (sizeof(XT) == 8) d[u][h] = in ? ld_hint(row + h * 32, pol_stream) : 0.0;
          else d[u][h] = in ? __ldg(row + h * 32) : (XT)0;
        }
      }
#pragma unroll
      for (int u = 0; u < kStepB; u++) {
        const int q = q0 + warp + u * kStepWarps;
        if (q < rows) {
#pragma unroll
          for (int h = 0; h < 2; h++) Sf[q * 2 * kStepW + h * 32 + lane] = from_any<R>(d[u][h]);
        }
      }
    }
  }
  __syncthreads();
  S = dft_steps<R, -1>(S, S + rows * kStepW, ng, L1, pl.np1, pl.rad1, pl.L, tw);
#pragma unroll 4
  for (int q = warp; q < rows; q += kStepWarps) {
    const int gi = by_l1(q), k1 = q - gi * L1, t2 = t20 + gi;
    cx<R> v = S[q * kStepW + lane];
    if (t2 * k1) v = twiddle_step<R, -1>(v, tw[t2 * k1]);
    st_hint(inter + ((size_t)k1 * L2 + t2) * ncx + kStepW * blockIdx.x + lane, v, pol_keep);
  }
}

// The buffers of G consecutive k1 groups {g, L1 - g}, g <= L1/2: buffer b =
// 2 (g - g0) + member, L2 rows each; a group without a partner (k1 = 0, L1/2)
// leaves its second buffer unused.  MULTI: G > 1.
template <bool MULTI> struct StepGroups {
  int L1, L2, g0, ng;
  SmallDiv by_l2;
  __device__ __forceinline__ StepGroups(const StepPlan &pl, int G)
      : L1(pl.L1), L2(pl.L2), g0(MULTI ? blockIdx.y * G : blockIdx.y),
        ng(MULTI ? min(G, pl.L1 / 2 + 1 - (int)blockIdx.y * G) : 1), by_l2(MULTI ? pl.L2 : 1) {}
  __device__ __forceinline__ int rows() const { return 2 * ng * L2; }
  // row q: its k1 (-1: unused), k2 and the row of the mirror frequency
  // ell - k: L2 - 1 - k2 of the other member's buffer (k1 != 0; the same
  // buffer where k1 = L1/2), or (L2 - k2) mod L2 of the same (k1 = 0)
  __device__ __forceinline__ void row(int q, int &k1, int &k2, int &qm) const {
    const int b = MULTI ? by_l2(q) : (q >= L2 ? 1 : 0);
    const int g = MULTI ? g0 + (b >> 1) : g0, gb = g ? L1 - g : 0;
    k2 = q - b * L2;
    k1 = (b & 1) ? (gb != g ? gb : -1) : g;
    qm = g == 0 ? (k2 ? b * L2 + L2 - k2 : q) : (gb != g ? (b ^ 1) : b) * L2 + L2 - 1 - k2;
  }
};

// Forward 2.  grid (ncx / 32, ceil((L1/2 + 1) / G)); 4 G L2 x 32 complex of
// dynamic shared memory.
template <typename R, bool MULTI>
__global__ void __launch_bounds__(kStepT, StepOcc<R>::V)
k_steps_forward2(const cx<R> *__restrict__ inter, cx<R> *__restrict__ spec, int n, int ncx,
                 int64_t n_pad, const step_tw<R, -1> *__restrict__ tw, StepPlan pl, int G) {
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<R> *S = reinterpret_cast<cx<R> *>(smraw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const StepGroups<MULTI> gr(pl, G);
  const int rows = gr.rows(), cb = kStepW * blockIdx.x;
  const unsigned long long pol_done = l2_evict_first(), pol_keep = l2_evict_last();
  pdl_wait(inter);
  for (int q0 = 0; q0 < rows; q0 += kStepB * kStepWarps) {
    cx<R> d[kStepB];
#pragma unroll
    for (int u = 0; u < kStepB; u++) {
      const int q = q0 + warp + u * kStepWarps;
      int k1, k2, qm;
      gr.row(q, k1, k2, qm);
      d[u] = mk((R)0, (R)0);
      if (q < rows && k1 >= 0)
        d[u] = ld_hintc(inter + ((size_t)k1 * pl.L2 + k2) * ncx + cb + lane, pol_done);
    }
#pragma unroll
    for (int u = 0; u < kStepB; u++) {
      const int q = q0 + warp + u * kStepWarps;
      if (q < rows) S[q * kStepW + lane] = d[u];
    }
  }
  __syncthreads();
  S = dft_steps<R, -1>(S, S + rows * kStepW, 2 * gr.ng, pl.L2, pl.np2, pl.rad2, pl.L, tw);
  // the two packed real columns X = (Z_k + conj Z_{ell-k})/2, Y = (Z_k - conj
  // Z_{ell-k})/(2i) of k = k1 + L1 k2 <= ell/2; stored without the factor 1/2,
  // which inverse B's scale carries (exactly: a power of two)
  const int i = 2 * (cb + lane);
#pragma unroll 4
  for (int q = warp; q < rows; q += kStepWarps) {
    int k1, k2, qm;
    gr.row(q, k1, k2, qm);
    const int k = k1 + pl.L1 * k2;
    if (k1 < 0 || 2 * k > pl.L) continue;
    const cx<R> zk = S[q * kStepW + lane], zm = S[qm * kStepW + lane];
    const cx<R> X = mk(zk.re + zm.re, zk.im - zm.im);
    const cx<R> Y = mk(zk.im + zm.im, zm.re - zk.re);
    cx<R> *dst = spec + (size_t)k * n_pad + i;
    if (i + 1 < n) st_hint2(dst, X, Y, pol_keep);
    else if (i < n) st_hint(dst, X, pol_keep);
  }
}

// Inverse A.  grid and shared memory as forward 2.
template <typename R, bool MULTI>
__global__ void __launch_bounds__(kStepT, StepOcc<R>::V)
k_steps_inverseA(const cx<R> *__restrict__ spec, cx<R> *__restrict__ inter, int n, int ncx,
                 int64_t n_pad, const step_tw<R, +1> *__restrict__ tw, StepPlan pl, int G) {
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<R> *S = reinterpret_cast<cx<R> *>(smraw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const StepGroups<MULTI> gr(pl, G);
  const int rows = gr.rows(), cb = kStepW * blockIdx.x, i = 2 * (cb + lane);
  const unsigned long long pol_done = l2_evict_first(), pol_keep = l2_evict_last();
  pdl_wait(spec);
  // X_k, Y_k of the stored half spectrum become Z_k = X + iY and, mirrored,
  // Z_{ell-k} = conj X + i conj Y
  constexpr int B = sizeof(R) == 8 ? kStepB / 2 : kStepB;
  for (int q0 = 0; q0 < rows; q0 += B * kStepWarps) {
    cx<R> X[B], Y[B];
#pragma unroll
    for (int u = 0; u < B; u++) {
      const int q = q0 + warp + u * kStepWarps;
      int k1, k2, qm;
      gr.row(q, k1, k2, qm);
      const int k = k1 + pl.L1 * k2;
      X[u] = Y[u] = mk((R)0, (R)0);
      if (q < rows && k1 >= 0 && 2 * k <= pl.L) {
        const cx<R> *src = spec + (size_t)k * n_pad + i;
        if (i + 1 < n) ld_hint2(src, X[u], Y[u], pol_done);
        else if (i < n) X[u] = ld_hintc(src, pol_done);
      }
    }
#pragma unroll
    for (int u = 0; u < B; u++) {
      const int q = q0 + warp + u * kStepWarps;
      int k1, k2, qm;
      gr.row(q, k1, k2, qm);
      const int k = k1 + pl.L1 * k2;
      if (q < rows && k1 >= 0 && 2 * k <= pl.L) {
        cx<R> a = X[u], b = Y[u];
        if (k == 0 || 2 * k == pl.L) { a.im = (R)0; b.im = (R)0; }
        S[q * kStepW + lane] = mk(a.re - b.im, a.im + b.re);
        if (k > 0 && 2 * k < pl.L) S[qm * kStepW + lane] = mk(a.re + b.im, b.re - a.im);
      }
    }
  }
  __syncthreads();
  S = dft_steps<R, +1>(S, S + rows * kStepW, 2 * gr.ng, pl.L2, pl.np2, pl.rad2, pl.L, tw);
#pragma unroll 4
  for (int q = warp; q < rows; q += kStepWarps) {
    int k1, t2, qm;
    gr.row(q, k1, t2, qm);
    if (k1 < 0) continue;
    cx<R> v = S[q * kStepW + lane];
    if (t2 * k1) v = twiddle_step<R, +1>(v, tw[t2 * k1]);
    st_hint(inter + ((size_t)k1 * pl.L2 + t2) * ncx + cb + lane, v, pol_keep);
  }
}

// Inverse B.  grid and shared memory as forward 1.  With BASE (FP64 output of
// an FP32 transform only) y = base - result.  diff_f64's rare FP64 case still
// keeps that pipe 14% busy here, and next to no time: with it cut out the refined
// apply takes 0.997 of it (286 sizes), gathered behind the loop 0.999.
template <typename R, typename OT, bool BASE>
__global__ void __launch_bounds__(kStepT, StepOcc<R>::V)
k_steps_inverseB(const cx<R> *__restrict__ inter, OT *__restrict__ y, int n, int ncx,
                 const step_tw<R, +1> *__restrict__ tw, const float *__restrict__ base, StepPlan pl, int G) {
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<R> *S = reinterpret_cast<cx<R> *>(smraw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int L1 = pl.L1, L2 = pl.L2, t20 = blockIdx.y * G;
  const int ng = min(G, L2 - t20), rows = ng * L1;
  const int i0 = 2 * kStepW * blockIdx.x;
  const SmallDiv by_l1(L1);
  const unsigned long long pol_done = l2_evict_first();
  pdl_wait(inter, base);
  for (int q0 = 0; q0 < rows; q0 += kStepB * kStepWarps) {
    cx<R> d[kStepB];
#pragma unroll
    for (int u = 0; u < kStepB; u++) {
      const int q = q0 + warp + u * kStepWarps, gi = by_l1(q), k1 = q - gi * L1;
      if (q < rows)
        d[u] = ld_hintc(inter + ((size_t)k1 * L2 + t20 + gi) * ncx + kStepW * blockIdx.x + lane, pol_done);
    }
#pragma unroll
    for (int u = 0; u < kStepB; u++) {
      const int q = q0 + warp + u * kStepWarps;
      if (q < rows) S[q * kStepW + lane] = d[u];
    }
  }
  __syncthreads();
  S = dft_steps<R, +1>(S, S + rows * kStepW, ng, L1, pl.np1, pl.rad1, pl.L, tw);
  const R *Sf = reinterpret_cast<const R *>(S);
  const R scale = (R)0.5 / (R)pl.L;   // with forward 2's 1/2
  constexpr int B = 4;
  for (int q0 = 0; q0 < rows; q0 += B * kStepWarps) {
    [[maybe_unused]] float bv[B][2];
    if constexpr (BASE) {
#pragma unroll
      for (int u = 0; u < B; u++) {
        const int q = q0 + warp + u * kStepWarps, gi = by_l1(q), t1 = q - gi * L1;
        const size_t row = (size_t)(L2 * t1 + t20 + gi) * n;
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int i = i0 + h * 32 + lane;
          bv[u][h] = (q < rows && i < n) ? __ldg(&base[row + i]) : 0.f;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < B; u++) {
      const int q = q0 + warp + u * kStepWarps, gi = by_l1(q), t1 = q - gi * L1;
      const size_t row = (size_t)(L2 * t1 + t20 + gi) * n;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int i = i0 + h * 32 + lane;
        if (q < rows && i < n) {
          const R val = scale * Sf[q * 2 * kStepW + h * 32 + lane];
          if constexpr (BASE) y[row + i] = diff_f64(bv[u][h], val);
          else if constexpr (sizeof(OT) == sizeof(R)) y[row + i] = val;
          else y[row + i] = to_f64(val);
        }
      }
    }
  }
}

// ------------------------------------------------------------- host side
// Radices of an N-point transform (N = 2^a 3^b 5^c): the fewest passes, and
// among those the smallest largest radix (more butterflies to share out).
inline bool step_radices(int N, int *rad, int &np) {
  static const int kRad[] = {2, 3, 4, 5, 6, 8, 9, 10};
  if (N == 1) { np = 0; return true; }
  int best = 1 << 30;
  for (int a : kRad) {
    if (N == a && a < best) { best = a; np = 1; rad[0] = a; }
  }
  if (best < (1 << 30)) return true;
  for (int a : kRad) {
    for (int b : kRad)
      if (a * b == N && a >= b && a < best) { best = a; np = 2; rad[0] = a; rad[1] = b; }
  }
  if (best < (1 << 30)) return true;
  for (int a : kRad) {
    for (int b : kRad)
      for (int c : kRad)
        if (a * b * c == N && a >= b && b >= c && a < best) {
          best = a; np = 3; rad[0] = a; rad[1] = b; rad[2] = c;
        }
  }
  return best < (1 << 30);
}

// FP64: L1 >= L2, L1 as small as possible (a tile of 64 rows is 32 KB).
// FP32: the smallest L1 >= 8 that leaves L2 <= 64.  The inverse's last DFT
// has length L1, and the rounding of the twiddles before it reaches the
// output shared by L1 time steps, so at the low frequencies that P^{-1}
// amplifies it is about sqrt(L1) times that of a transform whose twiddles
// come last; the refined apply squares that error.
//
// Where n fills the chip with panels of 32 columns, the forms of fft_time.cuh
// (powers of two: row and panel kernels) and fft_mixed.cuh (one kernel a
// direction) can be the faster ones, which spend fewer instructions per element.
// Whole applies, steps / the other form, on both sides of each line:
//   FP32, powers of two up to 128: n ell = 480000 up to ell 32 (32: n 14000 1.00,
//     15000 1.06, 16383 1.09; 16: 16383 0.99, 32767 1.05), 10^6 above (64: 10000
//     0.98, 16383 1.06; 128: 7500 1.01, 8191 1.10).
//   FP64, powers of two: n ell = 240000 at 16 (12000 1.00, 16383 1.08), 620000 up to
//     64 (64: 8191 0.93, 10000 1.07; 32: 16383 1.00, 32767 1.06), 850000 up to 256
//     (128: 6200 0.91, 7000 1.12; 256: 3071 0.93, 4000 1.25), never at 512 ... 2048
//     (0.94 ... 1.00 up to n 65535), n = 4000 at 4096 (2500 0.94, 4000 1.01, 8191 1.02).
//   Other lengths:
//     FP32, ell <= 64 in at most three passes, n < 32767 (there 0.9 ... 1.05): n = 4000
//       up to 40 (30: 3071 1.02, 4095 1.03, 5000 1.17), 5000 above (60: 4095 1.00,
//       5000 1.04); up to 200 in no more passes than the steps take: n = 64 ell (96:
//       5000 0.94, 6200 1.00, 8191 1.05; 120: 6200 0.94, 8191 1.02; 192: 8191 1.01,
//       16383 1.06; n >= 32767 1.02 ... 1.13).
//     FP32 refined, which has no FP32 residual with these kernels: n = 5000 (40: 4095
//       0.98, 5000 1.12), 8000 (50: 6200 0.95, 8191 1.03) and 128 ell (96: 8191 0.94,
//       16383 1.04), all n < 32767 (there 0.74 ... 1.05).
//     FP64, ell <= 64 in at most three passes, none of 16 (48: 0.83 ... 0.97), n < 32767
//       (there 0.82 ... 1.0): n = 3072 up to 50 (40: 2047 0.96, 4095 1.03, 16383 1.05),
//       6000 above (60: 5000 1.00, 6143 1.04).
//     FP64, 90 <= ell <= 192: where the panels fill the second wave of 152 SMs to
//       three quarters (n = 7300 ... 9728: 1.01 ... 1.11, but 162 0.92; beside it, n 5500
//       0.78 ... 0.91, 12000 0.84 ... 1.04).
// `steps`: the passes of the four-step plan.
inline bool panels_faster(int64_t ell, int64_t n, bool fp64, bool refined, int steps) {
  const int64_t work = n * ell;
  if ((ell & (ell - 1)) == 0) {
    if (!fp64) return ell <= 128 && work >= (ell <= 32 ? 480000 : 1000000);
    if (ell > 256) return ell == 4096 && n >= 4000;
    return work >= (ell <= 16 ? 240000 : ell <= 64 ? 620000 : 850000);
  }
  const int64_t second = (n + 31) / 32 - 152;   // panels of the second wave
  if (fp64 && ell >= 90) return ell <= 192 && 4 * second > 3 * 152 && second <= 152;
  MixedPlan mp;
  if (ell > 200 || !mixed_plan((int)ell, mp)) return false;
  if (ell > 64) return !fp64 && mp.np <= steps && (refined ? n >= 128 * ell && n < 32767 : n >= 64 * ell);
  if (mp.np > 3 || n >= 32767) return false;
  if (!fp64) return n >= (ell <= 40 ? (refined ? 5000 : 4000) : (refined ? 8000 : 5000));
  for (int p = 0; p < mp.np; p++)
    if (mp.rad[p] == 16) return false;
  return n >= (ell <= 50 ? 3072 : 6000);
}

inline bool step_plan(int64_t ell, int64_t n, bool fp64, bool refined, StepPlan &pl) {
  pl = StepPlan{};
  if (ell < AAO_STEPS_MIN) return false;
  const bool wide = !fp64 && ell >= 64;
  StepPlan st{};
  for (int64_t l1 = wide ? 8 : 1; l1 <= 128 && !st.L; l1++) {
    if (ell % l1 || (wide ? ell / l1 > 64 : l1 * l1 < ell)) continue;
    st.L1 = (int)l1;
    st.L2 = (int)(ell / l1);
    if (step_radices(st.L1, st.rad1, st.np1) && step_radices(st.L2, st.rad2, st.np2)) st.L = (int)ell;
  }
  if (!st.L || panels_faster(ell, n, fp64, refined, st.np1 + st.np2)) {
    pl.split = (ell & (ell - 1)) == 0;
    return false;
  }
  pl = st;
  return true;
}
inline int64_t steps_ncx(int64_t n) { return ((n + 1) / 2 + kStepW - 1) / kStepW * kStepW; }
template <typename R> size_t steps_inter_bytes(int64_t ell, int64_t n) {
  return (size_t)ell * (size_t)steps_ncx(n) * sizeof(cx<R>);
}

template <typename... KArgs, typename... Args>
cudaError_t steps_launch(void (*kern)(KArgs...), dim3 grid, size_t smem, cudaStream_t s, Args &&...args) {
  cudaError_t e = kernel_setup((const void *)kern, kStepT, smem, nullptr, true);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kern, grid, dim3(kStepT), smem, s, std::forward<Args>(args)...);
  note_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Units (t2 values, k1 groups) of `unit` rows per CTA: as many as fit in 64
// rows, as long as two CTAs per SM remain.
inline int steps_group(int cols, int units, int unit) {
  int G = 64 / unit;
  G = G < 1 ? 1 : (G > units ? units : G);
  while (G > 1 && (int64_t)cols * ((units + G - 1) / G) < 2 * 152) G--;
  return G;
}

template <typename R, typename XT, typename YT>
cudaError_t steps_forward(const StepPlan &pl, int64_t n, int64_t n_pad, const XT *x, const YT *y, const R *sigk,
                          cx<R> *spec, const step_tw<R, -1> *tw, cudaStream_t s, void *inter) {
  const int ncx = (int)steps_ncx(n), cols = ncx / kStepW;
  cx<R> *ip = static_cast<cx<R> *>(inter);
  const size_t row = kStepW * sizeof(cx<R>);
  const int G1 = steps_group(cols, pl.L2, pl.L1), G2 = steps_group(cols, pl.L1 / 2 + 1, 2 * pl.L2);
  const dim3 g1((unsigned)cols, (unsigned)((pl.L2 + G1 - 1) / G1)), g2((unsigned)cols, (unsigned)((pl.L1 / 2 + G2) / G2));
  const size_t sm1 = 2 * (size_t)G1 * pl.L1 * row;
  cudaError_t e;
  if constexpr (sizeof(XT) == 8) {
    e = y ? steps_launch(k_steps_forward1<R, XT, true, YT>, g1, sm1, s, x, y, sigk, ip, (int)n, ncx, tw, pl, G1)
          : steps_launch(k_steps_forward1<R, XT, false, double>, g1, sm1, s, x, (const double *)nullptr, sigk, ip, (int)n, ncx, tw, pl, G1);
  } else {
    e = steps_launch(k_steps_forward1<R, XT, false, double>, g1, sm1, s, x, (const double *)nullptr, sigk, ip, (int)n, ncx, tw, pl, G1);
  }
  if (e != cudaSuccess) return e;
  return steps_launch(G2 > 1 ? k_steps_forward2<R, true> : k_steps_forward2<R, false>, g2, 4 * (size_t)G2 * pl.L2 * row, s, ip, spec, (int)n, ncx, n_pad, tw, pl, G2);
}

template <typename R, typename OT>
cudaError_t steps_inverse(const StepPlan &pl, int64_t n, int64_t n_pad, const cx<R> *spec, OT *y, const step_tw<R, +1> *tw,
                          cudaStream_t s, void *inter, const float *base) {
  const int ncx = (int)steps_ncx(n), cols = ncx / kStepW;
  cx<R> *ip = static_cast<cx<R> *>(inter);
  const size_t row = kStepW * sizeof(cx<R>);
  const int G1 = steps_group(cols, pl.L2, pl.L1), G2 = steps_group(cols, pl.L1 / 2 + 1, 2 * pl.L2);
  const dim3 g1((unsigned)cols, (unsigned)((pl.L2 + G1 - 1) / G1)), g2((unsigned)cols, (unsigned)((pl.L1 / 2 + G2) / G2));
  const cudaError_t e = steps_launch(G2 > 1 ? k_steps_inverseA<R, true> : k_steps_inverseA<R, false>, g2, 4 * (size_t)G2 * pl.L2 * row, s, spec, ip, (int)n, ncx, n_pad, tw, pl, G2);
  if (e != cudaSuccess) return e;
  auto kern = k_steps_inverseB<R, OT, false>;
  if constexpr (sizeof(OT) > sizeof(R)) {
    if (base) kern = k_steps_inverseB<R, OT, true>;
  }
  return steps_launch(kern, g1, 2 * (size_t)G1 * pl.L1 * row, s, ip, y, (int)n, ncx, tw, base, pl, G1);
}

}  // namespace
}  // namespace fft
}  // namespace aao
