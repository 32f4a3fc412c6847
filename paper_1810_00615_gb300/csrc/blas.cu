// FP64 kernels of the outer Krylov loop: the all-at-once matvec (Section 2,
// the monolithic A is never formed), the right-hand side, the Arnoldi
// multi-dot / update / norm kernels, and the adjoint-gradient reductions.
//
// On GB300 FP64 issues at 2 operations per clock per SM (about 1.2 TFLOP/s,
// 1/64 of FP32), so these kernels are bounded by the FP64 pipe rather than by
// HBM once they do more than ~0.2 FP64 operations per byte; they are written
// to minimise FP64 operations per element.  All reductions are
// deterministic: fixed per-block order, then a fixed-order pass over the
// block partials.
#include "aao_internal.cuh"
#include <type_traits>

namespace aao {

namespace {
constexpr int kThreads = 256;
constexpr int kMaxRedBlocks = 152 * 8;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-reduce NV values per thread into partials[block * NV + j].
template <int NV>
__device__ __forceinline__ void block_store(double (&acc)[NV], double *partials) {
  __shared__ double sm[kThreads / 32][NV > 0 ? NV : 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < NV; j++) {
    const double s = warp_sum(acc[j]);
    if (lane == 0) sm[wid][j] = s;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; w++) s += sm[w][threadIdx.x];
    partials[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * NV + threadIdx.x] = s;
  }
}

// out[j] = sum_b partials[b * nv + j] in a fixed order, one block of NT threads
// per output, into device memory and, straight over the host link, into
// pinned host memory: a small result costs the stream no copy (6 of them in a
// solve at n 63 x ell 64, 8 us of its 170).  Launched as a dependent of the
// kernel that writes the partials.  (Letting that kernel's last block add them
// saved this launch but cost every block a fence and an atomic: 145 -> 166 us
// for the fused-dots matvec at n 4095 x ell 4096.)
template <int NT>
__global__ void __launch_bounds__(NT)
k_finish(const double *__restrict__ partials, int nb, int nv, RedOut out) {
  __shared__ double sm[NT / 32];
  const int j = blockIdx.x;
  pdl_wait(partials);
  double v = 0.0;
#pragma unroll 8
  for (int b = threadIdx.x; b < nb; b += NT) v += partials[(size_t)b * nv + j];
  v = warp_sum(v);
  if constexpr (NT > 32) {
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.0;
    if (threadIdx.x == 0) {
#pragma unroll
      for (int w = 0; w < NT / 32; w++) v += sm[w];
    }
  }
  if (threadIdx.x == 0) {
    out.dev[j] = v;
    if (out.host) out.host[j] = v;
  }
}
cudaError_t finish(const double *partials, int nb, int nv, const RedOut &out, cudaStream_t s) {
  const cudaError_t e =
      nb <= 64 ? launch_pdl(k_finish<32>, dim3(nv), dim3(32), 0, s, partials, nb, nv, out)
      : nb <= 2048 ? launch_pdl(k_finish<256>, dim3(nv), dim3(256), 0, s, partials, nb, nv, out)
                   : launch_pdl(k_finish<1024>, dim3(nv), dim3(1024), 0, s, partials, nb, nv, out);
  note_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

struct Ptrs8 {
  const double *p[8];
};
template <typename T> struct PtrsT {
  const T *p[8];
};
struct Coef8 {
  double c[8];
};
}  // namespace

int red_blocks(int64_t N) {
  int64_t b = (N + (int64_t)kThreads * 8 - 1) / ((int64_t)kThreads * 8);
  if (b < 1) b = 1;
  if (b > kMaxRedBlocks) b = kMaxRedBlocks;
  return (int)b;
}

// ------------------------------------------------------------------ matvec
// (A x)_t = A0^t x_t + A1 x_{t-1} (+ A2 x_{t-2}), every block a symmetric
// tridiagonal tridiag(off, diag, off) (Section 2).  The transpose runs the
// same recurrence backwards in t.  FP64 issues at 2 operations per clock per
// SM here, so the kernel is written for the fewest FP64 operations: a thread
// walks down a column i over TCH consecutive time steps, keeps the centre
// value and the neighbour sum s = x_{i-1} + x_{i+1} of the previous one or
// two steps in registers, and spends 1 add + 1 mul + 3 fma per output for the
// heat equation (2 more fma for BD2); the two neighbour loads hit L1.
constexpr int kMvCols = 128;   // columns per CTA
constexpr int kMvRows = 32;    // time steps per thread

// x is FP64, or FP32 for the preconditioned basis of the mixed solver (then
// widened exactly with integer operations: no FP64 conversion instruction).
__device__ __forceinline__ double wide(double v) { return v; }
__device__ __forceinline__ double wide(float v) { return to_f64(v); }

template <int NB, bool TR, bool SUB, typename XT, bool CIRC>
__global__ void __launch_bounds__(kMvCols)
k_matvec(const XT *__restrict__ x, double *__restrict__ y, int n, int ell,
         const double *__restrict__ d0, const double *__restrict__ o0,
         double d1, double o1, double d2, double o2, const double *__restrict__ sub) {
  const int i = blockIdx.x * kMvCols + threadIdx.x;
  if (i >= n) return;
  const int c0 = blockIdx.y * kMvRows;
  const int c1 = min(ell, c0 + kMvRows);
  auto row_vals = [&](int t, double &xc, double &sn) {
    const XT *xr = x + (int64_t)t * n;
    xc = wide(xr[i]);
    const double l = (i > 0) ? wide(xr[i - 1]) : 0.0;
    const double r = (i + 1 < n) ? wide(xr[i + 1]) : 0.0;
    sn = l + r;
  };
  // registers: previous (p1) and second previous (p2) step in walk order
  double xp1 = 0.0, sp1 = 0.0, xp2 = 0.0, sp2 = 0.0;
  const int first = TR ? c1 - 1 : c0;
  const int step = TR ? -1 : 1;
  int tp1 = first - step, tp2 = first - 2 * step;
  if (CIRC) {                       // the block circulant P: lags wrap around in time
    tp1 = ((tp1 % ell) + ell) % ell;
    tp2 = ((tp2 % ell) + ell) % ell;
  }
  if (tp1 >= 0 && tp1 < ell) row_vals(tp1, xp1, sp1);
  if (NB > 2 && tp2 >= 0 && tp2 < ell) row_vals(tp2, xp2, sp2);
  for (int k = 0; k < c1 - c0; k++) {
    const int t = first + k * step;
    double xc, sn;
    row_vals(t, xc, sn);
    double acc = d1 * xp1;
    acc = fma(o1, sp1, acc);
    if (NB > 2) {
      acc = fma(d2, xp2, acc);
      acc = fma(o2, sp2, acc);
      xp2 = xp1;
      sp2 = sp1;
    }
    acc = fma(__ldg(&d0[t]), xc, acc);
    acc = fma(__ldg(&o0[t]), sn, acc);
    if (SUB) acc -= __ldg(&sub[(int64_t)t * n + i]);
    y[(int64_t)t * n + i] = acc;
    xp1 = xc;
    sp1 = sn;
  }
}

// ------------------------------------------------ fixed-point matvec
// For the standard heat equation (any steps), BD2 and BD4 every block is
// a M + b K with M = (h/6) tridiag(1,4,1), K = (1/h) tridiag(-1,2,-1)
// (Section 2).  With q_t = 4 x_t + x_{t,i-1} + x_{t,i+1} and
// s_t = 2 x_t - x_{t,i-1} - x_{t,i+1}:
//   heat  (A x)_t = (h/6)(q_t - q_{t-1})            + beta_t s_t
//   BD2   (A x)_t = (h/6)(q_t - 2 q_{t-1} + q_{t-2}) + beta   s_t
//   BD4   (A x)_t = (h/6)(2 q_t - 5 q_{t-1} + 4 q_{t-2} - q_{t-3}) + beta s_t,
//         except the two BD2 start-up rows of C_BD4 (weights 1 and 1, -2)
// (transpose: t+1, t+2, t+3 instead of t-1, t-2, t-3).  Each warp converts its tile of
// x (its 32 columns, one halo column each side, the time steps it needs) to
// 64-bit fixed point at the tile's largest exponent, forms both sums exactly
// in integers (no cancellation error however much the terms cancel), joins
// them into one integer with the ratio of their coefficients (a 64-bit
// fixed-point fraction <= 1, one high multiply), rounds that once to FP64
// and finishes with one FMA.  GB300 issues integer operations at 64 per
// clock per SM and FP64 at 2, so this replaces six of the seven FP64
// operations per element of the FP64 form with integer work.
// The largest element of a tile keeps 58 bits (FP32 input: 34 binades below
// it are exact, FP64 input: 5); anything smaller is truncated at 2^-57 of
// the tile maximum.  BD4's weights (sum of magnitudes 12) need two guard
// bits more: 56 bits, truncation at 2^-55.  x is FP64 (the solution, the public matvec) or FP32
// (the preconditioned basis of the mixed solver).
//
// GB300: the kernel is bound by the FP64 pipe where it forms dots (an FP64
// operation per element is ~30 us of that pipe at n 4095 x ell 4096) and by
// instruction issue elsewhere, so each element is converted to fixed point
// once, into a shared-memory tile with its two halo columns, and the walk
// reads a value and its neighbours from there: no shuffles, no second pass
// over x (whose tiles did not survive in L1: 29 M L2 sectors for 13 M's worth
// of data at BD2 n 8191 x ell 2048).
// (hi:lo) >> sh (0 <= sh; all bits out from 64 on), negated where neg is -1.
__device__ __forceinline__ long long fx_shift(unsigned hi, unsigned lo, int sh, int neg) {
  const unsigned s2 = (unsigned)max(sh - 32, 0);
  const unsigned l = __funnelshift_rc(__funnelshift_rc(lo, hi, (unsigned)sh), 0u, s2);
  const unsigned h = __funnelshift_rc(hi, 0u, (unsigned)sh);
  const unsigned long long m = (unsigned long long)(long long)neg;
  return (long long)(((((unsigned long long)h << 32) | l) ^ m) - m);
}
constexpr int kFastExp = 64;   // smallest tile exponent of the fast conversions

template <typename XT> struct Fx;
template <> struct Fx<float> {
  static constexpr int kNonFinite = 255;   // exponent field of inf and NaN
  __device__ static int exp(float v) {
    const int e = (int)((__float_as_uint(v) >> 23) & 0xffu);
    return e ? e : 1;                       // subnormals scale like exponent 1
  }
  // v * 2^(184 - G - emax) as an integer (|.| < 2^(58 - G)), emax >= exp(v);
  // G guard bits leave room for larger integer weights in the sums
  template <int G>
  __device__ static long long fixed(float v, int emax) {
    const unsigned b = __float_as_uint(v);
    const unsigned e = (b >> 23) & 0xffu;
    const unsigned long long mant = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
    const int sh = min(emax - (e ? (int)e : 1), 63);
    const unsigned long long u = (mant << (34 - G)) >> sh;
    return (b >> 31) ? -(long long)u : (long long)u;
  }
  template <int G>
  __device__ static int unit(int emax) { return emax - 184 + G; }   // log2 of one unit
  // the same for emax >= kFastExp: zeros and subnormals, whose missing
  // implicit bit is not looked at, are shifted out with it
  template <int G>
  __device__ static long long fixed_fast(float v, int emax) {
    const unsigned b = __float_as_uint(v);
    const unsigned m = (b & 0x7fffffu) | 0x800000u;             // 24 bits, to 58 - G
    return fx_shift(m << (2 - G), 0u, emax - (int)((b << 1) >> 24), (int)b >> 31);
  }
};
template <> struct Fx<double> {
  static constexpr int kNonFinite = 2047;
  __device__ static int exp(double v) {
    const int e = (int)(((unsigned)__double2hiint(v) >> 20) & 0x7ffu);
    return e ? e : 1;
  }
  // v * 2^(1080 - G - emax) as an integer (|.| < 2^(58 - G)), emax >= exp(v)
  template <int G>
  __device__ static long long fixed(double v, int emax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ffu);
    const unsigned long long mant = (b & 0xfffffffffffffull) | (e ? (1ull << 52) : 0ull);
    const int sh = min(emax - (e ? e : 1), 63);
    const unsigned long long u = (mant << (5 - G)) >> sh;
    return (b >> 63) ? -(long long)u : (long long)u;
  }
  template <int G>
  __device__ static int unit(int emax) { return emax - 1080 + G; }
  template <int G>
  __device__ static long long fixed_fast(double v, int emax) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned m = (hi & 0xfffffu) | 0x100000u;
    return fx_shift(__funnelshift_l(lo, m, 5 - G), lo << (5 - G), emax - (int)((hi << 1) >> 21),
                    (int)hi >> 31);
  }
};

// S * 2^unit rounded to nearest even (|S| < 2^63).  With RANGE, results
// below the FP64 normal range flush to zero and above it give infinity (FP64
// input); FP32 input keeps every result in range, so the checks are dropped.
template <bool RANGE>
__device__ __forceinline__ double fx_to_f64(long long S, int unit) {
  const unsigned long long neg = (unsigned long long)(S >> 63);
  unsigned long long u = ((unsigned long long)S ^ neg) - neg;
  const int lz = __clzll(u);
  u <<= (lz & 63);
  unsigned long long mant = u >> 11;                       // 53 bits, top one set
  mant += (((unsigned)u & 0x7ffu) + (unsigned)(mant & 1u) + 0x3ffu) >> 11;
  const int field = 1085 + unit - lz;                      // biased exponent - 1
  const unsigned long long bits = ((unsigned long long)field << 52) + mant + (neg << 63);
  if (RANGE) {
    if (!S || field < 0) return neg ? -0.0 : 0.0;
    if (field >= 2046) return neg ? -INFINITY : INFINITY;
  } else if (!S) {
    return 0.0;
  }
  return __longlong_as_double((long long)bits);
}

// The fused dots of the matvec: every lane parks its ND accumulators in shared
// memory, and the last warp of the block to arrive adds the warps' values lane
// by lane in warp order, sums the lanes and stores the block partial (the
// result does not depend on the arrival order).  Every warp calls it exactly
// once, with all 32 lanes.  The lane sums run ND values at once, each half of
// the warp passing on half of them: 6 FP64 additions for three values instead
// of 15 per warp, which at 16 steps a tile were one FP64 operation per element.
template <int ND, int NW>
__device__ __forceinline__ void dots_commit(const double (&acc)[ND], double (*s_dot)[ND][32],
                                            int *s_cnt, double *__restrict__ dpart) {
  static_assert(ND >= 1 && ND <= 3, "one to three values");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < ND; q++) s_dot[warp][q][lane] = acc[q];
  __threadfence_block();
  __syncwarp();
  int last = 0;
  if (lane == 0) last = atomicAdd(s_cnt, 1) == NW - 1;
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  __threadfence_block();
  double t[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int q = 0; q < ND; q++)
#pragma unroll
    for (int w = 0; w < NW; w++) t[q] += reinterpret_cast<volatile double *>(s_dot[w][q])[lane];
  auto cross = [](double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); };
  double v;
  if constexpr (ND == 1) {
    v = t[0] + cross(t[0], 16);
    v += cross(v, 8);
  } else if constexpr (ND == 2) {
    const bool up = lane & 16;                        // lanes 16..: value 1
    v = (up ? t[1] : t[0]) + cross(up ? t[0] : t[1], 16);
    v += cross(v, 8);
  } else {
    const bool up = lane & 16, odd = lane & 8;        // lanes 0, 8, 16..: values 0, 1, 2
    const double a = (up ? t[2] : t[0]) + cross(up ? t[0] : t[2], 16);
    const double b = (up ? t[3] : t[1]) + cross(up ? t[1] : t[3], 16);
    v = (odd ? b : a) + cross(odd ? a : b, 8);
  }
  v += cross(v, 4);
  v += cross(v, 2);
  v += cross(v, 1);
  const size_t b = ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * ND;
  constexpr int per = ND == 3 ? 8 : 16;
  if (lane % per == 0 && lane / per < ND) dpart[b + lane / per] = v;
}

// DK >= 0 (with SUB): the kernel also forms dots of its output w = A x - v,
// as block partials in dpart, in order:
//   DK = 0: v . w, w . w
//   DK = 1: v0 . w, v . w, w . w
//   DK = 2: v . w, w . w, v . v   (the first step from x0 = 0, v = b: ||b||^2)
//   DK = 3: w . w                 (the true residual)
__host__ __device__ constexpr int fx_dots(int DK) { return DK < 0 ? 0 : (DK == 3 ? 1 : (DK == 0 ? 2 : 3)); }

// Resident CTAs per SM: the walk hides its latencies by warps.
#ifndef AAO_MVFX_MINB
#define AAO_MVFX_MINB 8
#endif
#ifndef AAO_MVFX_PRE
#define AAO_MVFX_PRE 2     // steps of prefetch of the subtrahend
#endif
template <int NB, bool TR, bool SUB, typename XT, bool CIRC, int DK, int R>
__global__ void __launch_bounds__(kMvCols, AAO_MVFX_MINB)
k_matvec_fx(const XT *__restrict__ x, double *__restrict__ y, int n, int ell,
            const MvRow *__restrict__ rows, const double *__restrict__ sub,
            const double *__restrict__ dv0, double *__restrict__ dpart) {
  constexpr int IN = R + NB - 1;                // input time steps per tile
  static_assert(IN <= 32, "a lane per halo row");
  constexpr int kWarps = kMvCols / 32;
  constexpr int G = NB == 4 ? 2 : 0;            // guard bits (sums below 2^63)
  constexpr int ND = fx_dots(DK) ? fx_dots(DK) : 1;
  static_assert(DK < 0 || SUB, "the dots need the subtrahend");
  using F = Fx<XT>;
  // columns iw - 1 .. iw + 32 of the walked steps, in fixed point
  __shared__ long long s_x[kWarps][IN][34];
  __shared__ double s_dot[DK >= 0 ? kWarps : 1][ND][32];
  __shared__ int s_cnt;
  if constexpr (DK >= 0) {
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();   // before any warp can leave
  }
  double dacc[ND];
#pragma unroll
  for (int q = 0; q < ND; q++) dacc[q] = 0.0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * kMvCols + threadIdx.x;
  const int iw = i - lane;                      // first column of the warp
  if (iw >= n) {                                // whole warp past the end
    if constexpr (DK >= 0) dots_commit<ND, kWarps>(dacc, s_dot, &s_cnt, dpart);
    return;
  }
  const bool col_ok = i < n;
  // walk step k = 0..IN-1 visits time step t0 + k dir: forward from the
  // oldest lag up, transpose from the newest lead down
  constexpr int dir = TR ? -1 : 1;
  const int c0 = blockIdx.y * R;
  const int t0 = TR ? c0 + IN - 1 : c0 - (NB - 1);
  const int64_t step = (int64_t)dir * n;
  const int ic = col_ok ? i : iw;               // a valid column for every lane
  auto t_ok = [&](int t) { return (unsigned)t < (unsigned)ell; };
  // CIRC (the block circulant P): steps outside [0, ell) wrap around
  auto wrap = [&](int t) { return ((t % ell) + ell) % ell; };
  // only the first (last) tile of a column walks past the ends in time
  const int t_min = TR ? t0 - (IN - 1) : t0, t_max = TR ? t0 : t0 + IN - 1;
  const bool full = iw + 31 < n && t_min >= 0 && t_max < ell;   // the same for the warp

  // the tile's values, all loads in flight together, and its largest exponent
  XT z[IN];
  const XT *px = x + (int64_t)t0 * n + ic;      // dereferenced only on valid steps
  if (full) {
#pragma unroll
    for (int k = 0; k < IN; k++) z[k] = __ldg(px + k * step);
  } else {
#pragma unroll
    for (int k = 0; k < IN; k++) {
      const int t = t0 + k * dir;
      const bool ok = col_ok && (CIRC || t_ok(t));
      z[k] = ok ? __ldg(CIRC && !t_ok(t) ? x + (int64_t)wrap(t) * n + ic : px + k * step) : (XT)0;
    }
  }
  XT hl = (XT)0, hr = (XT)0;                    // lane k: the halo columns of walk step k
  {
    int t = t0 + lane * dir;
    if (CIRC) t = wrap(t);
    if (lane < IN && t_ok(t)) {
      if (iw > 0) hl = __ldg(&x[(int64_t)t * n + iw - 1]);
      if (iw + 32 < n) hr = __ldg(&x[(int64_t)t * n + iw + 32]);
    }
  }
  int em = max(F::exp(hl), F::exp(hr));
#pragma unroll
  for (int k = 0; k < IN; k++) em = max(em, F::exp(z[k]));
  em = (int)__reduce_max_sync(0xffffffffu, (unsigned)em);
  if (em == F::kNonFinite) {                    // an inf or NaN in the tile
    if (col_ok)
      for (int t = c0; t < min(ell, c0 + R); t++)
        y[(int64_t)t * n + i] = __longlong_as_double(0x7ff8000000000000ll);
    if constexpr (DK >= 0) {
#pragma unroll
      for (int q = 0; q < ND; q++) dacc[q] = __longlong_as_double(0x7ff8000000000000ll);
      dots_commit<ND, kWarps>(dacc, s_dot, &s_cnt, dpart);
    }
    return;
  }
  const int unit = F::template unit<G>(em);
  long long(*sx)[34] = s_x[warp];
  if (em >= kFastExp) {
#pragma unroll
    for (int k = 0; k < IN; k++) sx[k][lane + 1] = F::template fixed_fast<G>(z[k], em);
  } else {
#pragma unroll
    for (int k = 0; k < IN; k++) sx[k][lane + 1] = F::template fixed<G>(z[k], em);
  }
  if (lane < IN) {
    sx[lane][0] = F::template fixed<G>(hl, em);
    sx[lane][33] = F::template fixed<G>(hr, em);
  }
  __syncwarp();

  // walk the output steps; the subtrahend comes kPre steps ahead so that its
  // latency hides behind the integer work of the steps in between.  FULL:
  // every column of the warp and every walked step lie inside the system;
  // RNG: results below or above the FP64 normal range are possible (FP64
  // input with an extreme tile exponent); ZERO: v0 (DK = 1) or v (DK = 2) is
  // zero on the whole tile.
  constexpr int kPre = AAO_MVFX_PRE;
  static_assert(R % kPre == 0, "whole prefetch rounds");
  const int64_t first = (int64_t)(t0 + (NB - 1) * dir) * n + ic;   // output step 0
  [[maybe_unused]] int wmax = 0;   // high word of the largest |w| of a ZERO walk, NaN above inf
  auto walk = [&](auto full_c, auto rng_c, auto zero_c) {
    constexpr bool FULL = decltype(full_c)::value, RNG = decltype(rng_c)::value;
    constexpr bool ZERO = decltype(zero_c)::value;
    constexpr bool V = SUB && !(ZERO && DK == 2), D = DK == 1 && !ZERO;   // streams read
    long long q1 = 0, q2 = 0, q3 = 0;           // q of the steps before
    auto stencil = [&](int k, long long &X, long long &P) {
      X = sx[k][lane + 1];
      P = sx[k][lane] + sx[k][lane + 2];
      return 4 * X + P;
    };
#pragma unroll
    for (int k = 0; k < NB - 1; k++) {
      long long X, P;
      q3 = q2;
      q2 = q1;
      q1 = stencil(k, X, P);
    }
    double vpre[kPre], dpre[kPre];
    const double *pv = V ? sub + first : nullptr, *pd = D ? dv0 + first : nullptr;
    auto fetch = [&](int r, int u) {
      const bool in = r < R && (FULL || (col_ok && t_ok(t0 + (NB - 1 + r) * dir)));
      if (V) vpre[u] = in ? __ldg(pv) : 0.0;
      if (D) dpre[u] = in ? __ldg(pd) : 0.0;
      if (V) pv += step;
      if (D) pd += step;
    };
#pragma unroll
    for (int u = 0; u < kPre; u++) fetch(u, u);
    double *py = y + first;
#pragma unroll 1
    for (int rb = 0; rb < R; rb += kPre) {
#pragma unroll
      for (int u = 0; u < kPre; u++) {
        const int r = rb + u, t = t0 + (NB - 1 + r) * dir;
        const double vk = V ? vpre[u] : 0.0;
        [[maybe_unused]] const double dk = D ? dpre[u] : 0.0;
        fetch(r + kPre, u);
        long long X, P;
        const long long q = stencil(NB - 1 + r, X, P);
        long long sm;
        if (NB == 2) {
          sm = q - q1;
        } else if (NB == 3) {
          sm = q - 2 * q1 + q2;
        } else {
          sm = 2 * q - 5 * q1 + 4 * q2 - q3;
          if (!CIRC && t < 2) {   // the BD2 start-up rows of C_BD4 (and their columns)
            if (!TR) sm = t == 0 ? q : q - 2 * q1;
            else sm = t == 0 ? q - 2 * q1 + 4 * q2 - q3 : q - 5 * q1 + 4 * q2 - q3;
          }
        }
        q3 = q2;
        q2 = q1;
        q1 = q;
        if (FULL || (col_ok && t_ok(t))) {
          const long long sk = 2 * X - P;
          // T = S_main + frac S_other, exact up to the truncated product; one
          // rounding to FP64 and one FMA
          const MvRow rw = rows[t];
          const long long s_main = rw.main_k ? sk : sm, s_oth = rw.main_k ? sm : sk;
          // truncated towards zero: the one-sided rounding of a floor, though
          // below a unit, adds up over a smooth field (it put a bias of 1e-10
          // into the kappa gradient at n = 16383)
          const unsigned long long so_neg = (unsigned long long)(s_oth >> 63);
          const unsigned long long so_abs = ((unsigned long long)s_oth ^ so_neg) - so_neg;
          const unsigned long long pa = __umul64hi(so_abs, rw.frac);
          const long long prod = (long long)((pa ^ so_neg) - so_neg);
          const double td = fx_to_f64<RNG>(s_main + prod, unit);
          const double yv = V ? fma(rw.coef, td, -vk) : rw.coef * td;
          *py = yv;
          if constexpr (ZERO) wmax = max(wmax, __double2hiint(yv) & 0x7fffffff);
          if constexpr (DK == 1) {
            if constexpr (!ZERO) dacc[0] = fma(dk, yv, dacc[0]);
            dacc[1] = fma(vk, yv, dacc[1]);
            dacc[2] = fma(yv, yv, dacc[2]);
          } else if constexpr (DK == 3) {
            dacc[0] = fma(yv, yv, dacc[0]);
          } else if constexpr (DK >= 0) {
            if constexpr (!ZERO) dacc[0] = fma(vk, yv, dacc[0]);
            dacc[1] = fma(yv, yv, dacc[1]);
            if constexpr (DK == 2 && !ZERO) dacc[2] = fma(vk, vk, dacc[2]);
          }
        }
        py += step;
      }
    }
  };
  // |S| < 2^63, so S 2^unit stays a normal FP64 number or zero for
  // -1022 <= unit <= 960; FP32 input always does
  constexpr bool RANGE = sizeof(XT) == 8;
  const bool in_range = !RANGE || (unit >= -1022 && unit <= 960);
  if constexpr (DK == 1 || DK == 2) {
    // The right-hand side of an all-at-once system is zero past its first
    // block rows, and in a solve from x = 0 it is v0 (DK = 1) and v (DK = 2):
    // tiles where it is zero skip the products with it, one or two FP64
    // operations of the bound pipe per element.  A dense vector costs a vote
    // on the tile's first step.  The sum of the products is zero unless an output
    // is not finite (v may hold an inf or NaN, and the scale may overflow): 0 x
    // inf and 0 x NaN are NaN.  (Walking such a tile again with the products made
    // the dense case 1.6% slower, by the code around it alone.)
    if (full && in_range && unit <= 0) {
      const double *pz = (DK == 1 ? dv0 : sub) + first;
      auto nonzero = [](double a) { return (unsigned long long)__double_as_longlong(a) << 1; };
      unsigned long long any = nonzero(__ldg(pz));
      if (!__any_sync(0xffffffffu, any != 0)) {
#pragma unroll
        for (int r = 1; r < R; r++) any |= nonzero(__ldg(pz + r * step));
        if (!__any_sync(0xffffffffu, any != 0)) {
          walk(std::true_type{}, std::false_type{}, std::true_type{});
          if (wmax >= 0x7ff00000) dacc[0] = __longlong_as_double(0x7ff8000000000000ll);
          dots_commit<ND, kWarps>(dacc, s_dot, &s_cnt, dpart);
          return;
        }
      }
    }
  }
  if (full && in_range) walk(std::true_type{}, std::false_type{}, std::false_type{});
  else walk(std::false_type{}, std::integral_constant<bool, RANGE>{}, std::false_type{});
  if constexpr (DK >= 0) dots_commit<ND, kWarps>(dacc, s_dot, &s_cnt, dpart);
}

// Output time steps per warp tile: 16, or 8 where the 16-step tiles leave
// fewer than four CTAs per SM (short walks, more of them in flight).
constexpr int kFxRows = 16, kFxRowsSmall = 8;
static bool fx_small(const Ctx &c) {
  return (c.n + kMvCols - 1) / kMvCols * ((c.ell + kFxRows - 1) / kFxRows) < 4 * 152;
}
static dim3 mv_fx_grid(const Ctx &c) {
  const int R = fx_small(c) ? kFxRowsSmall : kFxRows;
  return dim3((unsigned)((c.n + kMvCols - 1) / kMvCols), (unsigned)((c.ell + R - 1) / R));
}

template <int NB, bool TR, typename XT, bool CIRC>
static void mv_sub(const Ctx &c, dim3 grid, const XT *x, double *y, const double *sub,
                   cudaStream_t s) {
  const int n = (int)c.n, ell = (int)c.ell;
  if (sub)
    k_matvec<NB, TR, true, XT, CIRC><<<grid, kMvCols, 0, s>>>(x, y, n, ell, c.mv_d0, c.mv_o0,
                                                              c.mv_d1, c.mv_o1, c.mv_d2, c.mv_o2,
                                                              sub);
  else
    k_matvec<NB, TR, false, XT, CIRC><<<grid, kMvCols, 0, s>>>(x, y, n, ell, c.mv_d0, c.mv_o0,
                                                               c.mv_d1, c.mv_o1, c.mv_d2,
                                                               c.mv_o2, nullptr);
}

template <typename XT, bool CIRC = false>
static cudaError_t matvec_any(const Ctx &c, const XT *x, double *y, int transpose,
                              cudaStream_t s, const double *sub) {
  const int n = (int)c.n, ell = (int)c.ell;
  const dim3 grid((unsigned)((n + kMvCols - 1) / kMvCols),
                  (unsigned)((ell + kMvRows - 1) / kMvRows));
  const bool bd2 = c.equation == AAO_WAVE_BD2;
  if (bd2 && transpose) mv_sub<3, true, XT, CIRC>(c, grid, x, y, sub, s);
  else if (bd2) mv_sub<3, false, XT, CIRC>(c, grid, x, y, sub, s);
  else if (transpose) mv_sub<2, true, XT, CIRC>(c, grid, x, y, sub, s);
  else mv_sub<2, false, XT, CIRC>(c, grid, x, y, sub, s);
  note_launch();
  return cudaGetLastError();
}

template <int NB, bool TR, bool SUB, typename XT, bool CIRC, int DK>
static void run_fx(const Ctx &c, const XT *x, double *y, const double *sub, const double *v0,
                   double *dpart, cudaStream_t s) {
  const int n = (int)c.n, ell = (int)c.ell;
  const MvRow *rows = CIRC ? c.mv_rows_p : c.mv_rows;
  const dim3 grid = mv_fx_grid(c);
  if (fx_small(c))
    k_matvec_fx<NB, TR, SUB, XT, CIRC, DK, kFxRowsSmall><<<grid, kMvCols, 0, s>>>(x, y, n, ell, rows, sub, v0, dpart);
  else
    k_matvec_fx<NB, TR, SUB, XT, CIRC, DK, kFxRows><<<grid, kMvCols, 0, s>>>(x, y, n, ell, rows, sub, v0, dpart);
  note_launch();
}

template <int NB, bool TR, typename XT, bool CIRC>
static void mv_fx(const Ctx &c, const XT *x, double *y, const double *sub, cudaStream_t s) {
  if (sub) run_fx<NB, TR, true, XT, CIRC, -1>(c, x, y, sub, nullptr, nullptr, s);
  else run_fx<NB, TR, false, XT, CIRC, -1>(c, x, y, nullptr, nullptr, nullptr, s);
}

// Heat, BD2 and BD4 take the fixed-point kernel; the literal heat form (whose M
// coefficients differ between A0 and A1) the FP64 stencil.  CIRC: the block
// circulant P of Section 3 (constant step, time wrapped around) instead of A.
template <typename XT, bool CIRC = false>
static cudaError_t matvec_dispatch(const Ctx &c, const XT *x, double *y, int transpose,
                                   cudaStream_t s, const double *sub) {
  if (c.equation == AAO_HEAT_LITERAL) return matvec_any<XT, CIRC>(c, x, y, transpose, s, sub);
  const bool bd2 = c.equation == AAO_WAVE_BD2, bd4 = c.equation == AAO_WAVE_BD4;
  if (bd4 && transpose) mv_fx<4, true, XT, CIRC>(c, x, y, sub, s);
  else if (bd4) mv_fx<4, false, XT, CIRC>(c, x, y, sub, s);
  else if (bd2 && transpose) mv_fx<3, true, XT, CIRC>(c, x, y, sub, s);
  else if (bd2) mv_fx<3, false, XT, CIRC>(c, x, y, sub, s);
  else if (transpose) mv_fx<2, true, XT, CIRC>(c, x, y, sub, s);
  else mv_fx<2, false, XT, CIRC>(c, x, y, sub, s);
  return cudaGetLastError();
}

size_t matvec_dot_partials(const Ctx &c) {
  const dim3 g = mv_fx_grid(c);
  return (size_t)g.x * g.y * 3;
}

// w = A x - sub with dots of w fused in: out = [v0 . w,] sub . w, w . w
// (DK = 0, 1), sub . w, w . w, sub . sub (MvDots::SELF) or w . w alone
// (MvDots::NORM).
template <typename XT>
static cudaError_t matvec_dots_dispatch(const Ctx &c, const XT *x, double *y, int transpose,
                                        cudaStream_t s, const double *sub, const double *v0,
                                        double *dpart, const RedOut &out, MvDots what) {
  if (c.equation == AAO_HEAT_LITERAL || !sub || (v0 && what != MvDots::ARNOLDI))
    return cudaErrorNotSupported;
  const int nb = c.equation == AAO_WAVE_BD4 ? 4 : (c.equation == AAO_WAVE_BD2 ? 3 : 2);
  const int dk = v0 ? 1 : (what == MvDots::SELF ? 2 : (what == MvDots::NORM ? 3 : 0));
  const int key = nb * 8 + (transpose ? 4 : 0) + dk;
#define AAO_MVD(NBV, TRV, DKV)                                                           \
  case NBV * 8 + (TRV ? 4 : 0) + DKV:                                                    \
    run_fx<NBV, TRV, true, XT, false, DKV>(c, x, y, sub, v0, dpart, s);                  \
    break;
#define AAO_MVD3(NBV, TRV) AAO_MVD(NBV, TRV, 0) AAO_MVD(NBV, TRV, 1) AAO_MVD(NBV, TRV, 2)
  switch (key) {
    AAO_MVD3(2, false) AAO_MVD3(2, true) AAO_MVD3(3, false) AAO_MVD3(3, true)
    AAO_MVD3(4, false) AAO_MVD3(4, true)
    default:
      // the true residual's norm: of an FP64 solution only
      if constexpr (sizeof(XT) == 8) {
        switch (key) {
          AAO_MVD(2, false, 3) AAO_MVD(2, true, 3) AAO_MVD(3, false, 3) AAO_MVD(3, true, 3)
          AAO_MVD(4, false, 3) AAO_MVD(4, true, 3)
          default: return cudaErrorNotSupported;
        }
        break;
      }
      return cudaErrorNotSupported;
  }
#undef AAO_MVD3
#undef AAO_MVD
  const dim3 grid = mv_fx_grid(c);
  return finish(dpart, (int)(grid.x * grid.y), fx_dots(dk), out, s);
}

cudaError_t launch_matvec_dots(const Ctx &c, const double *x, double *y, int transpose,
                               cudaStream_t s, const double *sub, const double *v0,
                               double *dpart, const RedOut &out, MvDots what) {
  return matvec_dots_dispatch(c, x, y, transpose, s, sub, v0, dpart, out, what);
}

cudaError_t launch_matvec_dots(const Ctx &c, const float *x, double *y, int transpose,
                               cudaStream_t s, const double *sub, const double *v0,
                               double *dpart, const RedOut &out, MvDots what) {
  return matvec_dots_dispatch(c, x, y, transpose, s, sub, v0, dpart, out, what);
}

// ------------------------------------------ compensated circulant residual
// r = P z - x for an FP32 z (the refined preconditioner's residual) on the
// FP32 pipe.  r is needed to FP32 relative accuracy only (it feeds the FP32
// apply of the correction), but P z and x cancel to ~1e-7 of their size, so
// the sum is compensated: every product c z is formed exactly as an FP32
// pair (FMA; c = hi + lo to 2^-48), x is split into two FP32 halves, and the
// terms are added by Sum2 (Ogita, Rump and Oishi 2005, a TwoSum per term with
// the errors accumulated): the result is within 2^-24 |r| plus about
// n^2 2^-48 of the terms' magnitudes, n <= 14 terms.  It is rounded to FP32
// (the FP32 apply of the correction reads no more) and stored widened.  No
// FP64 instruction: the kernel runs on the FP32 and integer pipes.

// x = hi + lo: hi the FP32 rounding of x (to nearest even), lo = x - hi to
// FP32, from the bits of x with integer operations only (the FP64 pipe is
// 1/64 of the FP32 one).  |x| < 2^-74 is flushed to zero (an absolute error
// below 2^-74; the block vectors the solver applies this to are scaled to
// unit norm), |x| >= 2^127 and non-finite x give an infinite or NaN hi.
__device__ __forceinline__ void split_f64(double x, float &hi, float &lo) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned w = (unsigned)(u >> 32), l = (unsigned)u;
  const unsigned e = (w >> 20) & 0x7ffu, sign = w & 0x80000000u;
  if (e - 949u > 201u) {               // outside [949, 1150]
    const bool nan = e == 2047u && ((w & 0xfffffu) | l);
    hi = __uint_as_float(sign | (e > 1150u ? (0x7f800000u | (nan ? 0x400000u : 0u)) : 0u));
    lo = 0.f;
    return;
  }
  // exponent (rebiased, mod 2^32) and top 23 mantissa bits in one funnel shift
  unsigned bits = __funnelshift_l(l, w, 3) - 0xC0000000u;
  int rem = (int)(l & 0x1fffffffu);    // the 29 bits below hi's last place
  const bool up = (unsigned)rem + (bits & 1u) > (1u << 28);   // to nearest, ties to even
  bits += up ? 1u : 0u;
  if (up) rem -= (1 << 29);
  hi = __uint_as_float(sign | bits);
  const float fl = __int2float_rn(rem) * __uint_as_float((e - 1075u + 127u) << 23);
  lo = __uint_as_float(__float_as_uint(fl) ^ sign);
}

// An FP32 value widened to FP64 with integer operations (subnormals flushed
// to zero; infinities and NaN kept).
__device__ __forceinline__ double widen_f32(float v) {
  const unsigned u = __float_as_uint(v);
  const unsigned e = (u >> 23) & 0xffu, sign = u & 0x80000000u;
  if (e == 0u) return __hiloint2double((int)sign, 0);
  const unsigned hi = sign | ((e == 255u ? 2047u : e + 896u) << 20) | ((u & 0x7fffffu) >> 3);
  return __hiloint2double((int)hi, (int)(u << 29));
}

__device__ __forceinline__ void store_r(double *p, float v) { *p = widen_f32(v); }
__device__ __forceinline__ void store_r(float *p, float v) { *p = v; }

template <int NB, bool TR, typename RT>
__global__ void __launch_bounds__(kMvCols)
k_circ_residual_df(const float *__restrict__ z, const double *__restrict__ x,
                   RT *__restrict__ r, int n, int ell, CircDF cf) {
  const int i = blockIdx.x * kMvCols + threadIdx.x;
  if (i >= n) return;                  // no barriers in this kernel
  const int c0 = blockIdx.y * kMvRows;
  const int c1 = min(ell, c0 + kMvRows);
  auto load = [&](int t, float (&v)[3]) {
    const float *zr = z + (int64_t)t * n;
    v[0] = __ldg(&zr[i]);
    v[1] = (i > 0) ? __ldg(&zr[i - 1]) : 0.f;
    v[2] = (i + 1 < n) ? __ldg(&zr[i + 1]) : 0.f;
  };
  // lag[j]: the step j behind in walk order (time wrapped around: P)
  float lag[NB][3];
  const int first = TR ? c1 - 1 : c0, stp = TR ? -1 : 1, cnt = c1 - c0;
#pragma unroll
  for (int j = 1; j < NB; j++) {
    int tj = first - j * stp;
    tj = ((tj % ell) + ell) % ell;
    load(tj, lag[j]);
  }
  float s, e;
  auto add = [&](float chi, float clo, float v) {
    const float p = __fmul_rn(chi, v);
    const float pe = __fmaf_rn(chi, v, -p);              // chi v = p + pe exactly
    const float s1 = __fadd_rn(s, p);                    // TwoSum(s, p)
    const float bb = __fsub_rn(s1, s);
    const float er = __fadd_rn(__fsub_rn(s, __fsub_rn(s1, bb)), __fsub_rn(p, bb));
    s = s1;
    e = __fadd_rn(e, __fadd_rn(er, __fmaf_rn(clo, v, pe)));
  };
  // the next step's values are requested before this step's arithmetic
  float cur[3];
  double xc;
  load(first, cur);
  xc = __ldg(&x[(int64_t)first * n + i]);
  for (int k = 0; k < cnt; k++) {
    const int t = first + k * stp;
    float nxt[3] = {0.f, 0.f, 0.f};
    double xn = 0.0;
    if (k + 1 < cnt) {
      load(t + stp, nxt);
      xn = __ldg(&x[(int64_t)(t + stp) * n + i]);
    }
    lag[0][0] = cur[0];
    lag[0][1] = cur[1];
    lag[0][2] = cur[2];
    float xh, xl;
    split_f64(xc, xh, xl);
    s = -xh;
    e = -xl;
#pragma unroll
    for (int j = 0; j < NB; j++) {
      add(cf.hi[j][0], cf.lo[j][0], lag[j][0]);
      add(cf.hi[j][1], cf.lo[j][1], lag[j][1]);
      add(cf.hi[j][1], cf.lo[j][1], lag[j][2]);
    }
    store_r(r + (int64_t)t * n + i, __fadd_rn(s, e));   // r to FP32: all the apply reads
#pragma unroll
    for (int j = NB - 1; j >= 1; j--) {
      lag[j][0] = lag[j - 1][0];
      lag[j][1] = lag[j - 1][1];
      lag[j][2] = lag[j - 1][2];
    }
    cur[0] = nxt[0];
    cur[1] = nxt[1];
    cur[2] = nxt[2];
    xc = xn;
  }
}

// The same residual from the stencil sums of each row: per row t the pairs
// q_t = z_{i-1} + 4 z_i + z_{i+1} and k_t = 2 z_i - z_{i-1} - z_{i+1} (exact
// up to 2^-48 of their terms: two TwoSums), kept for the NB - 1 rows behind;
// S = sum_j a_j q_{t-j} with the integer time weights (exact multiples by
// 1, 2, 4; -5 q = -4 q - q), and r = mh S + bp k_t - x with two pair
// products and two TwoSums.  Each row's stencil is formed once instead of
// once per lag.  The kernel was bound by instruction issue (77%), so a thread
// takes two columns kMvCols apart and forms both at once in packed FP32 pairs:
// one f32x2 instruction for two additions or FMAs, with the roundings of one at
// a time, so the same bits.  Per launch at n 4095 x ell 4096: 71 us with one
// column a thread, 59 with two (268 MB: 4.6 TB/s, 40 us at the copy rate; the
// load latency is what is left); n 16383 x ell 1024 transposed 74 -> 59, n 1568
// x ell 1440 18 -> 11.  A walk has 8 steps: 16 or 32 leave the last wave emptier
// than their fewer halo rows save (59.6 and 67.5 us, n 1568 x ell 1440 13), 12
// differ by under 1%.  Where 8 leave fewer than two CTAs per SM a walk has 2:
// it is a chain of loads then, and 8 steps of two columns were slower than 8 of
// one (refined apply n 5000 x ell 8 58.8 us against 56.2).
constexpr int kResRows = 8, kResRowsSmall = 2;
template <int NB> __device__ __forceinline__ constexpr int qweight(int j) {
  return NB == 2 ? (j == 0 ? 1 : -1)
                 : (NB == 3 ? (j == 1 ? -2 : 1) : (j == 0 ? 2 : (j == 1 ? -5 : (j == 2 ? 4 : -1))));
}

__device__ __forceinline__ void two_sum2(f2x a, f2x b, f2x &s, f2x &e) {
  s = add2(a, b);
  const f2x bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

template <int NB, bool TR, typename RT, int ROWS>
__global__ void __launch_bounds__(kMvCols)
k_circ_residual_q(const float *__restrict__ z, const double *__restrict__ x,
                  RT *__restrict__ r, int n, int ell, CircDF cf) {
  const int i = blockIdx.x * (2 * kMvCols) + threadIdx.x, i2 = i + kMvCols;
  if (i >= n) return;                  // no barriers in this kernel
  const bool two = i2 < n;
  const int c0 = blockIdx.y * ROWS;
  const int c1 = min(ell, c0 + ROWS);
  auto load = [&](int t, f2x (&v)[3]) {
    const float *zr = z + (int64_t)t * n;
    v[0] = pack2(__ldg(&zr[i]), two ? __ldg(&zr[i2]) : 0.f);
    v[1] = pack2((i > 0) ? __ldg(&zr[i - 1]) : 0.f, two ? __ldg(&zr[i2 - 1]) : 0.f);
    v[2] = pack2((i + 1 < n) ? __ldg(&zr[i + 1]) : 0.f, (i2 + 1 < n) ? __ldg(&zr[i2 + 1]) : 0.f);
  };
  auto loadx = [&](int t, double (&v)[2]) {
    const double *xr = x + (int64_t)t * n;
    v[0] = __ldg(&xr[i]);
    v[1] = two ? __ldg(&xr[i2]) : 0.0;
  };
  const f2x zero = dup2(0.f), mhh = dup2(cf.mh_hi), mhl = dup2(cf.mh_lo), bph = dup2(cf.bp_hi),
            bpl = dup2(cf.bp_lo);
  // q (and k) of a row as pairs: zl + zr first, then + 4 z (- for k, with 2 z)
  auto qk = [&](const f2x (&v)[3], f2x &qh, f2x &ql, f2x &kh, f2x &kl) {
    f2x ah, ae, e;
    two_sum2(v[1], v[2], ah, ae);
    two_sum2(ah, mul2(dup2(4.f), v[0]), qh, e);
    ql = add2(e, ae);
    two_sum2(mul2(dup2(2.f), v[0]), sub2(zero, ah), kh, e);
    kl = sub2(e, ae);
  };
  f2x qh[NB], ql[NB];                  // [j]: the row j behind in walk order
  const int first = TR ? c1 - 1 : c0, stp = TR ? -1 : 1, cnt = c1 - c0;
#pragma unroll
  for (int j = 1; j < NB; j++) {
    int tj = first - j * stp;
    tj = ((tj % ell) + ell) % ell;     // time wrapped around: P
    f2x v[3], kh, kl;
    load(tj, v);
    qk(v, qh[j], ql[j], kh, kl);
  }
  // the next row is requested right after the current one's stencil sums
  f2x zq[3];
  double xq[2];
  load(first, zq);
  loadx(first, xq);
  for (int k = 0; k < cnt; k++) {
    const int t = first + k * stp;
    f2x kh, kl;
    qk(zq, qh[0], ql[0], kh, kl);
    const double xc[2] = {xq[0], xq[1]};
    if (k + 1 < cnt) {
      load(t + stp, zq);
      loadx(t + stp, xq);
    }
    // S = sum_j a_j q_{t-j} as a pair
    f2x sh = qh[0], sl = ql[0], e;
    if (qweight<NB>(0) != 1) {
      sh = mul2(dup2((float)qweight<NB>(0)), qh[0]);
      sl = mul2(dup2((float)qweight<NB>(0)), ql[0]);
    }
#pragma unroll
    for (int j = 1; j < NB; j++) {
      const int w = qweight<NB>(j);
      if (w == -5) {                   // -5 q = -4 q - q, each exact
        two_sum2(sh, mul2(dup2(-4.f), qh[j]), sh, e);
        sl = add2(sl, e);
        two_sum2(sh, sub2(zero, qh[j]), sh, e);
        sl = add2(sl, sub2(e, mul2(dup2(5.f), ql[j])));
      } else {
        two_sum2(sh, w == 1 ? qh[j] : mul2(dup2((float)w), qh[j]), sh, e);
        sl = add2(sl, fma2(dup2((float)w), ql[j], e));   // one rounding, as w q is exact
      }
    }
    // mh S and bp k as pairs (exact high products by FMA)
    const f2x p1 = mul2(mhh, sh);
    f2x e1 = fma2(mhh, sh, sub2(zero, p1));
    e1 = fma2(mhh, sl, e1);
    e1 = fma2(mhl, sh, e1);
    const f2x p2 = mul2(bph, kh);
    f2x e2 = fma2(bph, kh, sub2(zero, p2));
    e2 = fma2(bph, kl, e2);
    e2 = fma2(bpl, kh, e2);
    float xh[2], xl[2];
#pragma unroll
    for (int u = 0; u < 2; u++) split_f64(xc[u], xh[u], xl[u]);
    f2x sum, er1, er2;
    two_sum2(pack2(-xh[0], -xh[1]), p1, sum, er1);
    two_sum2(sum, p2, sum, er2);
    const f2x lo = add2(add2(sub2(e1, pack2(xl[0], xl[1])), e2), add2(er1, er2));
    float ra, rb;
    unpack2(add2(sum, lo), ra, rb);    // r to FP32: all the apply reads
    RT *rr = r + (int64_t)t * n;
    store_r(rr + i, ra);
    if (two) store_r(rr + i2, rb);
#pragma unroll
    for (int j = NB - 1; j >= 1; j--) {
      qh[j] = qh[j - 1];
      ql[j] = ql[j - 1];
    }
  }
}

template <int NB, bool TR, typename RT>
static void run_circ_q(const Ctx &c, const float *z, const double *x, RT *r, cudaStream_t s) {
  const unsigned gx = (unsigned)((c.n + 2 * kMvCols - 1) / (2 * kMvCols));
  const int n = (int)c.n, ell = (int)c.ell;
  auto gy = [&](int rows) { return (unsigned)((ell + rows - 1) / rows); };
  if ((int64_t)gx * gy(kResRows) >= 2 * 152)
    k_circ_residual_q<NB, TR, RT, kResRows><<<dim3(gx, gy(kResRows)), kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df);
  else
    k_circ_residual_q<NB, TR, RT, kResRowsSmall><<<dim3(gx, gy(kResRowsSmall)), kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df);
}

template <typename RT>
static cudaError_t circ_residual_df_any(const Ctx &c, const float *z, const double *x, RT *r,
                                        int transpose, cudaStream_t s) {
  const dim3 grid((unsigned)((c.n + kMvCols - 1) / kMvCols),
                  (unsigned)((c.ell + kMvRows - 1) / kMvRows));
  const int n = (int)c.n, ell = (int)c.ell;
  if (c.circ_df.int_weights) {
    switch (c.circ_df.taps * 2 + (transpose ? 1 : 0)) {
      case 4: run_circ_q<2, false, RT>(c, z, x, r, s); break;
      case 5: run_circ_q<2, true, RT>(c, z, x, r, s); break;
      case 6: run_circ_q<3, false, RT>(c, z, x, r, s); break;
      case 7: run_circ_q<3, true, RT>(c, z, x, r, s); break;
      case 8: run_circ_q<4, false, RT>(c, z, x, r, s); break;
      case 9: run_circ_q<4, true, RT>(c, z, x, r, s); break;
      default: return cudaErrorInvalidValue;
    }
    note_launch();
    return cudaGetLastError();
  }
  switch (c.circ_df.taps * 2 + (transpose ? 1 : 0)) {
    case 4: k_circ_residual_df<2, false, RT><<<grid, kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df); break;
    case 5: k_circ_residual_df<2, true, RT><<<grid, kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df); break;
    case 6: k_circ_residual_df<3, false, RT><<<grid, kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df); break;
    case 7: k_circ_residual_df<3, true, RT><<<grid, kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df); break;
    case 8: k_circ_residual_df<4, false, RT><<<grid, kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df); break;
    case 9: k_circ_residual_df<4, true, RT><<<grid, kMvCols, 0, s>>>(z, x, r, n, ell, c.circ_df); break;
    default: return cudaErrorInvalidValue;
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_circ_residual_df(const Ctx &c, const float *z, const double *x, double *r,
                                    int transpose, cudaStream_t s) {
  return circ_residual_df_any(c, z, x, r, transpose, s);
}

cudaError_t launch_circ_residual_df(const Ctx &c, const float *z, const double *x, float *r,
                                    int transpose, cudaStream_t s) {
  return circ_residual_df_any(c, z, x, r, transpose, s);
}

cudaError_t launch_circ_residual(const Ctx &c, const float *z, double *y, int transpose,
                                 cudaStream_t s, const double *sub) {
  return matvec_dispatch<float, true>(c, z, y, transpose, s, sub);
}

// u = x - E y with (E y)_t = sigk_t (2 y_i - y_{i-1} - y_{i+1}), sigk_t =
// (tau_t - tau) kappa / h (Section 2): the right-hand side of a Neumann term,
// formed in FP64 for the refined FP32 preconditioner.
__global__ void __launch_bounds__(kThreads)
k_neumann_rhs(const double *__restrict__ x, const double *__restrict__ y,
              const double *__restrict__ sigk, double *__restrict__ u, int n, int ell) {
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i >= n) return;
  for (int t = blockIdx.y; t < ell; t += gridDim.y) {
    const int64_t g = (int64_t)t * n + i;
    const double yc = y[g];
    const double s = ((i > 0) ? y[g - 1] : 0.0) + ((i + 1 < n) ? y[g + 1] : 0.0);
    u[g] = fma(-__ldg(&sigk[t]), fma(2.0, yc, -s), x[g]);
  }
}

// Grid of the kernels that walk a block vector with a thread per column and
// the time steps dealt out over blockIdx.y: one element per thread at least,
// about `want` blocks at most (no 64-bit division per element).
static dim3 column_grid(int64_t n, int64_t ell, int64_t want) {
  const int64_t gx = (n + kThreads - 1) / kThreads;
  int64_t gy = want / gx;
  gy = gy < 1 ? 1 : (gy > ell ? ell : gy);
  return dim3((unsigned)gx, (unsigned)gy);
}

cudaError_t launch_neumann_rhs(const Ctx &c, const double *x, const double *y, double *u,
                               cudaStream_t s) {
  k_neumann_rhs<<<column_grid(c.n, c.ell, 152 * 16), kThreads, 0, s>>>(x, y, c.sigk, u, (int)c.n,
                                                                       (int)c.ell);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_matvec(const Ctx &c, const double *x, double *y, int transpose,
                          cudaStream_t s, const double *sub) {
  return matvec_dispatch(c, x, y, transpose, s, sub);
}

cudaError_t launch_matvec(const Ctx &c, const float *x, double *y, int transpose,
                          cudaStream_t s, const double *sub) {
  return matvec_dispatch(c, x, y, transpose, s, sub);
}

// --------------------------------------------------------------------- rhs
// Heat: b_0 = M u0.  BD2: b_0 = A0 (u0 + tau v0) = M w + tau^2 K w,
// b_1 = -M u0.  BD4: b_0 = B (u0 + tau v0) (B = M + tau^2 K, the BD2
// block), b_1 = -M u0, b_2 = M u0.  Literal heat: b_0 = M u0.  Other
// blocks zero.  wave: 0 heat, 2 BD2, 3 BD4 (the number of start-up rows).
__global__ void k_rhs(const double *__restrict__ u0, const double *__restrict__ v0,
                      double *__restrict__ b, int n, int ell, int wave, double tau,
                      double mh, double kh) {
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i >= n) return;
  for (int t = blockIdx.y; t < ell; t += gridDim.y) {
    double out = 0.0;
    if (t <= 2) {
      auto at = [&](const double *v, int j) { return (j >= 0 && j < n) ? v[j] : 0.0; };
      auto w = [&](int j) {
        double r = at(u0, j);
        if (wave && v0 && t == 0) r = fma(tau, at(v0, j), r);
        return r;
      };
      const double wc = w(i), wl = w(i - 1), wr = w(i + 1);
      const double m = mh * fma(4.0, wc, wl + wr);
      if (t == 0) {
        out = m;
        if (wave) out = fma(tau * tau * kh, (wc - wl) - (wr - wc), out);
      } else if (t < wave) {
        // w = u0 on these rows: -M u0 (second row), +M u0 (third, BD4)
        out = t == 1 ? -m : m;
      }
    }
    b[(int64_t)t * n + i] = out;
  }
}

cudaError_t launch_rhs(const Ctx &c, const double *u0, const double *v0, double *b,
                       cudaStream_t s) {
  k_rhs<<<column_grid(c.n, c.ell, 152 * 16), kThreads, 0, s>>>(u0, v0, b, (int)c.n, (int)c.ell,
                                              c.equation == AAO_WAVE_BD2   ? 2
                                              : c.equation == AAO_WAVE_BD4 ? 3
                                                                           : 0,
                                              c.tau, c.h / 6.0,
                                              1.0 / c.h); note_launch();
  return cudaGetLastError();
}

// ------------------------------------------------------------ multi-dot
template <int NV, bool NORM>
__global__ void __launch_bounds__(kThreads)
k_multidot(Ptrs8 V, const double *__restrict__ w, int64_t N, double *__restrict__ partials) {
  constexpr int NO = NV + (NORM ? 1 : 0);
  double acc[NO];
#pragma unroll
  for (int j = 0; j < NO; j++) acc[j] = 0.0;
  for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < N;
       g += (int64_t)gridDim.x * kThreads) {
    const double wv = w[g];
#pragma unroll
    for (int j = 0; j < NV; j++) acc[j] = fma(__ldg(&V.p[j][g]), wv, acc[j]);
    if (NORM) acc[NO - 1] = fma(wv, wv, acc[NO - 1]);
  }
  block_store<NO>(acc, partials);
}

template <int NV, bool NORM>
static void run_multidot(const Ptrs8 &P, const double *w, int64_t N, int nb, double *partials,
                         cudaStream_t s) {
  k_multidot<NV, NORM><<<nb, kThreads, 0, s>>>(P, w, N, partials); note_launch();
}

// out[0] = <a, a>, out[1] = <b, b> in one pass over both vectors.
__global__ void __launch_bounds__(kThreads)
k_norms2(const double *__restrict__ a, const double *__restrict__ b, int64_t N,
         double *__restrict__ partials) {
  double acc[2] = {0.0, 0.0};
  for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < N;
       g += (int64_t)gridDim.x * kThreads) {
    const double av = a[g], bv = b[g];
    acc[0] = fma(av, av, acc[0]);
    acc[1] = fma(bv, bv, acc[1]);
  }
  block_store<2>(acc, partials);
}

cudaError_t launch_norms2(const double *a, const double *b, int64_t N, double *partials,
                          const RedOut &out, cudaStream_t s) {
  const int nb = red_blocks(N);
  k_norms2<<<nb, kThreads, 0, s>>>(a, b, N, partials); note_launch();
  return finish(partials, nb, 2, out, s);
}

cudaError_t launch_multidot(const double *const *V, int nv, const double *w, int64_t N,
                            bool with_norm, double *partials, const RedOut &out,
                            cudaStream_t s) {
  const int nb = red_blocks(N);
  int done = 0;
  if (nv == 0 && with_norm) {
    Ptrs8 P{};
    run_multidot<0, true>(P, w, N, nb, partials, s);
    return finish(partials, nb, 1, out, s);
  }
  while (done < nv) {
    const int g = (nv - done) > 8 ? 8 : (nv - done);
    const bool norm = with_norm && (done + g == nv);
    Ptrs8 P{};
    for (int j = 0; j < g; j++) P.p[j] = V[done + j];
#define AAO_MD(G)                                                         \
  case G:                                                                 \
    if (norm) run_multidot<G, true>(P, w, N, nb, partials, s);            \
    else run_multidot<G, false>(P, w, N, nb, partials, s);                \
    break;
    switch (g) {
      AAO_MD(1) AAO_MD(2) AAO_MD(3) AAO_MD(4) AAO_MD(5) AAO_MD(6) AAO_MD(7) AAO_MD(8)
    }
#undef AAO_MD
    const int no = g + (norm ? 1 : 0);
    const cudaError_t e = finish(partials, nb, no, out.at(done), s);
    if (e != cudaSuccess) return e;
    done += g;
  }
  return cudaSuccess;
}

// --------------------------------------------- update (+ dots + norm) pass
// w -= sum_j h_j V_j, its squared norm and, where they will be needed, the
// dots V_j . w of the result: a second Gram-Schmidt pass follows where the
// norm falls below half its value (the DGKS criterion), and for a nearly
// orthonormal basis that fall is known from the first pass's dots, ||w||^2 -
// sum_j h_j d_j.  AHEAD: the kernel forms that prediction from the device's own
// numbers (before = ||w||^2 at *before; 0.55 leaves room for rounding) and adds
// the dots only then, one FP64 operation per vector instead of another pass
// over w and V (52 us at n 4095 x ell 4096).  out: the NV dots (zero if not
// formed), the norm, 1 or 0 for formed or not; without AHEAD the norm alone.
// A warp of a single vector whose 32 values are all zero (the right-hand side
// of an all-at-once system past its first block rows) leaves w as it is.
template <int NV, bool AHEAD>
__global__ void __launch_bounds__(kThreads)
k_update(Ptrs8 V, const double *__restrict__ h, Coef8 f, double *__restrict__ w, int64_t N,
         double *__restrict__ partials, const double *__restrict__ div0,
         const double *__restrict__ before, RedOut flag) {
  constexpr int NO = AHEAD ? NV + 1 : 1;
  double hv[NV];
#pragma unroll
  for (int j = 0; j < NV; j++) hv[j] = h[j] * f.c[j];
  if (div0) hv[0] /= *div0;   // the first vector's squared norm, known only on the device
  bool dots = false;
  if (AHEAD) {
    const double b = *before;
    double left = b;
#pragma unroll
    for (int j = 0; j < NV; j++) left = fma(-hv[j], h[j], left);
    dots = left < 0.55 * b;
  }
  double acc[NO];
#pragma unroll
  for (int j = 0; j < NO; j++) acc[j] = 0.0;
  // U elements a thread at a time, all their loads first
  constexpr int U = NV <= 2 ? 4 : (NV <= 4 ? 2 : 1);
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  auto pass = [&](auto dots_c) {
    constexpr bool DOTS = decltype(dots_c)::value;
    for (int64_t g0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; g0 < N; g0 += U * stride) {
      double wv[U], v[U][NV];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int64_t g = g0 + u * stride;
        wv[u] = g < N ? w[g] : 0.0;
#pragma unroll
        for (int j = 0; j < NV; j++) v[u][j] = g < N ? __ldg(&V.p[j][g]) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int64_t g = g0 + u * stride;
        bool some = true;
        if (NV == 1) {
          const unsigned z = ((unsigned)__double2hiint(v[u][0]) << 1) | (unsigned)__double2loint(v[u][0]);
          const unsigned e = (unsigned)__double2hiint(wv[u]) & 0x7ff00000u;   // inf, NaN: 0 x is a NaN
          some = __any_sync(__activemask(), z != 0u || e == 0x7ff00000u);
        }
        if (some) {
#pragma unroll
          for (int j = 0; j < NV; j++) wv[u] = fma(-hv[j], v[u][j], wv[u]);
          if (g < N) w[g] = wv[u];
          if constexpr (DOTS) {
#pragma unroll
            for (int j = 0; j < NV; j++) acc[j] = fma(v[u][j], wv[u], acc[j]);
          }
        }
        acc[NO - 1] = fma(wv[u], wv[u], acc[NO - 1]);
      }
    }
  };
  if constexpr (AHEAD) {
    if (dots) pass(std::true_type{});
    else pass(std::false_type{});
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      flag.dev[0] = dots ? 1.0 : 0.0;
      if (flag.host) flag.host[0] = dots ? 1.0 : 0.0;
    }
  } else {
    pass(std::false_type{});
  }
  block_store<NO>(acc, partials);
}

cudaError_t launch_update(const double *const *V, int nv, const double *h, double *w, int64_t N,
                          double *partials, const RedOut &out, cudaStream_t s, const double *hf,
                          const double *div0, const double *before) {
  // groups of 8 vectors; the dots ahead are formed for at most 8
  const int nb = red_blocks(N);
  if (before && nv > 8) return cudaErrorInvalidValue;
  for (int done = 0; done < nv;) {
    const int g = (nv - done) > 8 ? 8 : (nv - done);
    Ptrs8 P{};
    Coef8 F{};
    for (int j = 0; j < g; j++) {
      P.p[j] = V[done + j];
      F.c[j] = hf ? hf[done + j] : 1.0;
    }
    const double *d0 = done == 0 ? div0 : nullptr;
    switch (g) {
#define AAO_UP(G)                                                                                \
  case G:                                                                                        \
    if (before) k_update<G, true><<<nb, kThreads, 0, s>>>(P, h + done, F, w, N, partials, d0, before, out.at(nv + 1)); \
    else k_update<G, false><<<nb, kThreads, 0, s>>>(P, h + done, F, w, N, partials, d0, nullptr, out);               \
    note_launch();                                                                               \
    break;
      AAO_UP(1) AAO_UP(2) AAO_UP(3) AAO_UP(4) AAO_UP(5) AAO_UP(6) AAO_UP(7) AAO_UP(8)
#undef AAO_UP
    }
    done += g;
  }
  return finish(partials, nb, before ? nv + 1 : 1, out, s);
}

// ------------------------------------------------------------ x += Z y
template <int NV, typename ZT>
__global__ void __launch_bounds__(kThreads)
k_combine(PtrsT<ZT> Z, Coef8 yv, double *__restrict__ x, int64_t N, int assign) {
  // Two elements a thread at a time, all their loads first, from three vectors
  // on: 128 against 135-144 us for four FP32 vectors at n 4095 x ell 4096 (123 us
  // is four passes' worth of FP64 FMAs); one or two vectors stream at 5.5 TB/s
  // either way (73 against 74 us for two FP64 vectors).
  constexpr int U = NV <= 2 ? 1 : 2;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t g0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; g0 < N; g0 += U * stride) {
    double a[U];
    ZT z[U][NV];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int64_t g = g0 + u * stride;
      a[u] = (assign || g >= N) ? 0.0 : x[g];   // assign: x = Z y (x not read)
#pragma unroll
      for (int j = 0; j < NV; j++) z[u][j] = g < N ? __ldg(&Z.p[j][g]) : (ZT)0;
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
#pragma unroll
      for (int j = 0; j < NV; j++) a[u] = fma(yv.c[j], wide(z[u][j]), a[u]);
      if (g0 + u * stride < N) x[g0 + u * stride] = a[u];
    }
  }
}

template <typename ZT>
static cudaError_t combine_any(const ZT *const *Z, int nv, const double *y, double *x, int64_t N,
                               cudaStream_t s, bool assign) {
  int64_t blocks = (N + kThreads - 1) / kThreads;
  if (blocks > 152 * 16) blocks = 152 * 16;
  int done = 0;
  while (done < nv) {
    const int g = (nv - done) > 8 ? 8 : (nv - done);
    PtrsT<ZT> P{};
    Coef8 Y{};
    for (int j = 0; j < g; j++) {
      P.p[j] = Z[done + j];
      Y.c[j] = y[done + j];
    }
    switch (g) {
#define AAO_CB(G) case G: k_combine<G, ZT><<<(unsigned)blocks, kThreads, 0, s>>>(P, Y, x, N, (assign && done == 0) ? 1 : 0); note_launch(); break;
      AAO_CB(1) AAO_CB(2) AAO_CB(3) AAO_CB(4) AAO_CB(5) AAO_CB(6) AAO_CB(7) AAO_CB(8)
#undef AAO_CB
    }
    done += g;
  }
  return cudaGetLastError();
}

cudaError_t launch_combine(const double *const *Z, int nv, const double *y, double *x,
                           int64_t N, cudaStream_t s, bool assign) {
  return combine_any(Z, nv, y, x, N, s, assign);
}

cudaError_t launch_combine(const float *const *Z, int nv, const double *y, double *x,
                           int64_t N, cudaStream_t s, bool assign) {
  return combine_any(Z, nv, y, x, N, s, assign);
}

// ------------------------------------------------------------ misc
// y = a * x with a = *ap (or 1/sqrt(*ap) when invert: a norm^2 on device),
// negated when negate != 0
__global__ void k_scale(const double *__restrict__ x, double *__restrict__ y,
                        const double *__restrict__ ap, int64_t N, int invert, int negate) {
  double a = *ap;
  if (invert) a = 1.0 / sqrt(a);
  if (negate) a = -a;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < N;
       g += (int64_t)gridDim.x * blockDim.x)
    y[g] = a * x[g];
}

cudaError_t launch_scale(const double *x, double *y, const double *a, int64_t N, bool invert,
                         cudaStream_t s, bool negate) {
  int64_t blocks = (N + kThreads - 1) / kThreads;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_scale<<<(unsigned)blocks, kThreads, 0, s>>>(x, y, a, N, invert ? 1 : 0, negate ? 1 : 0);
  note_launch();
  return cudaGetLastError();
}

// ------------------------------------------------------- adjoint gradients
// g_u0 = M lam_1; sum_t tau_t lam_t^T K u_t (reduced; the caller negates).
__global__ void k_grad_u0(const double *__restrict__ lam, double *__restrict__ g, int n,
                          double mh) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double c = lam[i], l = (i > 0) ? lam[i - 1] : 0.0, r = (i + 1 < n) ? lam[i + 1] : 0.0;
    g[i] = mh * fma(4.0, c, l + r);
  }
}

// sum_t tau_t lam_t^T K u_t (times kappa, from tauk = tau_t kappa / h) by its
// edges: lam^T (h K) u = sum_i (lam_{i+1} - lam_i)(u_{i+1} - u_i), i = 0 .. n
// with zero ends, two subtractions and an FMA per element where the stencil
// form took five FP64 operations (that pipe bounds the kernel: 167 us at n
// 16383 x ell 1024), and no cancellation of second differences.  A row's sum
// is scaled by tauk once per thread and row with variable steps, once per
// thread with uniform ones.
template <bool UNIFORM>
__global__ void __launch_bounds__(kThreads)
k_grad_kappa(const double *__restrict__ lam, const double *__restrict__ U, int n, int ell,
             const double *__restrict__ tauk, double *__restrict__ partials) {
  double acc[1] = {0.0};
  const int i = blockIdx.x * kThreads + threadIdx.x;   // edge between columns i - 1 and i
  if (i <= n) {
    const bool l = i > 0, r = i < n;
#pragma unroll 4
    for (int t = blockIdx.y; t < ell; t += gridDim.y) {
      const int64_t g = (int64_t)t * n + i;
      const double du = (r ? __ldg(&U[g]) : 0.0) - (l ? __ldg(&U[g - 1]) : 0.0);
      const double dl = (r ? __ldg(&lam[g]) : 0.0) - (l ? __ldg(&lam[g - 1]) : 0.0);
      acc[0] = fma(UNIFORM ? dl : __ldg(&tauk[t]) * dl, du, acc[0]);
    }
    if (UNIFORM) acc[0] *= __ldg(&tauk[0]);
  }
  block_store<1>(acc, partials);
}

cudaError_t launch_adjoint_grads(const Ctx &c, const double *lam, const double *U,
                                 double *g_u0, double *partials, const RedOut &out,
                                 cudaStream_t s) {
  const int n = (int)c.n;
  k_grad_u0<<<(n + kThreads - 1) / kThreads, kThreads, 0, s>>>(lam, g_u0, n, c.h / 6.0); note_launch();
  // beta_t = tau_t kappa / h, so tau_t lam^T K u = (beta_t / kappa) lam^T (h K) u / h ... use
  // tau_t / h directly: the matvec's beta divided by kappa.
  const dim3 grid = column_grid(c.n + 1, c.ell, kMaxRedBlocks);
  if (c.variable_steps)
    k_grad_kappa<false><<<grid, kThreads, 0, s>>>(lam, U, n, (int)c.ell, c.beta, partials);
  else
    k_grad_kappa<true><<<grid, kThreads, 0, s>>>(lam, U, n, (int)c.ell, c.beta, partials);
  note_launch();
  return finish(partials, (int)(grid.x * grid.y), 1, out, s);
}

// The library's integer-built conversions next to CUDA's own, element by
// element, for the conversion self-test.
__global__ void __launch_bounds__(kThreads)
k_convert_check(const double *__restrict__ x64, int64_t n64, float *__restrict__ lib32,
                float *__restrict__ ref32, const float *__restrict__ x32, int64_t n32,
                double *__restrict__ lib64, double *__restrict__ ref64) {
  const int64_t m = n64 > n32 ? n64 : n32;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * kThreads) {
    if (i < n64) {
      const double v = x64[i];
      lib32[i] = to_f32(v);
      ref32[i] = __double2float_rn(v);
    }
    if (i < n32) {
      const float f = x32[i];
      lib64[i] = to_f64(f);
      ref64[i] = (double)f;
    }
  }
}

cudaError_t launch_convert_check(const double *x64, int64_t n64, float *lib32, float *ref32,
                                 const float *x32, int64_t n32, double *lib64, double *ref64,
                                 cudaStream_t s) {
  const int64_t m = n64 > n32 ? n64 : n32;
  if (m <= 0) return cudaSuccess;
  const int64_t nb = (m + kThreads - 1) / kThreads;
  k_convert_check<<<(unsigned)(nb < 1024 ? nb : 1024), kThreads, 0, s>>>(x64, n64, lib32, ref32,
                                                                          x32, n32, lib64, ref64);
  note_launch();
  return cudaGetLastError();
}

}  // namespace aao
