// Tables of the recursive tridiagonal solve (RecLev in aao_internal.cuh), built
// on the device from the frequency blocks' symbols.
//
// Level l is the system (sigma, e) with last-row excess sigma_L and virtual
// right coupling o_L; with a = -e and b = -o_L its diagonal is sigma + 2a, its
// last diagonal sigma_L + a + b.  D_i is the determinant of i regular rows and
// R_i = D_i + delta D_{i-1} that of i rows with the last one, delta = (sigma_L -
// sigma) + (b - a); H_i and S_i = H_i + delta H_{i-1} + (sigma_L - sigma)
// a^{i-1} are their excess parts:
//   H_{i+1} = sigma D_i + a H_i,   D_{i+1} = a D_i + H_{i+1} + a^{i+1},
// from D_0 = 1, H_0 = 0.  Every table entry is a quotient of these (c = CH - 1
// unknowns in a regular chunk, cl in the last),
//   1/p_i = D_i / D_{i+1}, last row D_{cl-1} / R_cl;   e/p_i = -a / p_i;
//   -e g_i = a^{i+1} D_{c-1-i} / D_c,   -e gl_i = a^{i+1} R_{cl-1-i} / R_cl,
// g and gl the chunks' T^{-1} e_1, and so is the next level:
//   sigma' = sigma + 2a H_c/D_c,  sigma_L' = sigma + a H_c/D_c + a S_cl/R_cl,
//   a' = a^{c+1} / D_c,           b' = a^cl b / R_cl.
// No excess comes from a difference of diagonals, however nearly singular the
// block is, and the chain has two quotients a level.  Pairs can afford such
// differences and take the shorter recurrence D_{i+1} = (sigma + 2a) D_i - a^2
// D_{i-1}, H_i = D_i - a D_{i-1} - a^i, off by some 2^-100 of a, which no solution
// in FP64 can tell.
//
// The FP64 tables are formed in pairs of FP64 numbers and rounded once.  Their
// errors are the same for every chunk of a row, so they add up: with tables
// formed in FP64 the FP64 apply was 1.10 times as far off (95 sizes against
// extended precision) as before the recursion served every row, 0.88 with
// these.  Plain FP64 is enough for the FP32 tables.
//
// The host forms sigma and e per frequency, scaled by a power of two to
// elements of order 1 so that no product overflows or vanishes on the way
// (tau may be 1e-180); pivots scale with it, everything else is free of it.
//
// The kernel is bound by the FP64 pipe, which takes a warp 16 clocks and more
// an instruction.  So a block takes one level, and walks the levels below it
// for itself, and one of two roles: what belongs to the regular chunks, or to
// the last one.
// aao_set_kappa and a synchronise, FP32 modes / FP64 mode (the host building all
// tables; the host before the recursion served every row): n 63 x ell 64 70 / 152 us
// (131; 243), n 74 x ell 64 71 / 176 (135; 145), n 1000 x ell 900 98 / 237 (959;
// 701), n 4095 x ell 4096 168 / 386 (4222; 10467), n 16383 x ell 64 87 / 340 (186;
// 352): few frequencies are all latency, which the pairs' chains lengthen.  With
// one lane a number n 63 x ell 64 and n 1000 x ell 900 took 175 and 310 in FP64
// mode, with all levels of a role in one thread besides 268 and 463.
#include "aao_internal.cuh"

namespace aao {
namespace {

// A complex number is held by two lanes, the even one its real and the odd one
// its imaginary part: half the instructions for a warp to issue.  All lanes take
// part in every operation.
template <typename E> struct zc {
  E v;
};
__device__ __forceinline__ bool imag() { return threadIdx.x & 1; }
__device__ __forceinline__ double other(double a) { return __shfl_xor_sync(0xffffffffu, a, 1); }
__device__ __forceinline__ double lead(double a) { return a; }
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ double dot(double a, double b, double x, double y) { return fma(a, b, x * y); }
__device__ __forceinline__ double dot(double a, double b, double x, double y, double c) { return fma(a, b, fma(x, y, c)); }
__device__ __forceinline__ double recip(double a) { return 1.0 / a; }

// Pairs: unevaluated sums h + l of two FP64 numbers, |l| at most half a unit of
// h (Dekker; products split by FMA).  Rounded operations throughout: a
// contracted product would undo the splitting.  A chain of them costs its
// latency here, so products are added up before the sum is put in order once.
struct pair {
  double h, l;
  __device__ __forceinline__ pair() {}
  __device__ __forceinline__ explicit pair(double a) : h(a), l(0.0) {}
  __device__ __forceinline__ pair(double a, double b) : h(a), l(b) {}
};
__device__ __forceinline__ pair other(pair a) { return {other(a.h), other(a.l)}; }
__device__ __forceinline__ double lead(pair a) { return a.h; }
__device__ __forceinline__ pair neg(pair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ pair tidy(pair a) {                                  // |h| >= |l|
  const double s = __dadd_rn(a.h, a.l);
  return {s, __dsub_rn(a.l, __dsub_rn(s, a.h))};
}
__device__ __forceinline__ pair loose(pair a, pair b) {                         // a + b, not tidy
  const double s = __dadd_rn(a.h, b.h), t = __dsub_rn(s, a.h);
  const double e = __dadd_rn(__dsub_rn(a.h, __dsub_rn(s, t)), __dsub_rn(b.h, t));
  return {s, __dadd_rn(__dadd_rn(a.l, b.l), e)};
}
__device__ __forceinline__ pair prod(pair a, pair b) {                          // a b, not tidy
  const double p = __dmul_rn(a.h, b.h);
  return {p, __dadd_rn(__fma_rn(a.h, b.h, -p), __fma_rn(a.l, b.h, __dmul_rn(a.h, b.l)))};
}
__device__ __forceinline__ pair add(pair a, pair b) { return tidy(loose(a, b)); }
__device__ __forceinline__ pair mul(pair a, pair b) { return tidy(prod(a, b)); }
__device__ __forceinline__ pair dot(pair a, pair b, pair x, pair y) {           // a b + x y
  return tidy(loose(prod(a, b), prod(x, y)));
}
__device__ __forceinline__ pair dot(pair a, pair b, pair x, pair y, pair c) {   // a b + x y + c
  return tidy(loose(loose(prod(a, b), prod(x, y)), c));
}
__device__ __forceinline__ pair recip(pair a) {
  const double r = 1.0 / a.h;
  return tidy({r, __dmul_rn(r, __fma_rn(-a.l, r, __fma_rn(-a.h, r, 1.0)))});
}

template <typename E> __device__ __forceinline__ zc<E> real_z(double a) { return {E(imag() ? 0.0 : a)}; }
template <typename E> __device__ __forceinline__ zc<E> zadd(zc<E> a, zc<E> b) { return {add(a.v, b.v)}; }
template <typename E> __device__ __forceinline__ zc<E> zneg(zc<E> a) { return {neg(a.v)}; }
template <typename E> __device__ __forceinline__ zc<E> zsub(zc<E> a, zc<E> b) { return zadd(a, zneg(b)); }
// a b (+ c): (re re) - (im im) in the even lane, (im re) + (re im) in the odd one
template <typename E> __device__ __forceinline__ zc<E> zmul(zc<E> a, zc<E> b) {
  const E ap = other(a.v);
  return {dot(imag() ? ap : a.v, b.v, imag() ? a.v : neg(ap), other(b.v))};
}
template <typename E> __device__ __forceinline__ zc<E> zfma(zc<E> a, zc<E> b, zc<E> c) {
  const E ap = other(a.v);
  return {dot(imag() ? ap : a.v, b.v, imag() ? a.v : neg(ap), other(b.v), c.v)};
}
template <typename E> __device__ __forceinline__ zc<E> zrecip(zc<E> a) {
  const E p = other(a.v), r = mul(a.v, recip(dot(a.v, a.v, p, p)));
  return {imag() ? neg(r) : r};
}

// Where one frequency's entries of a level go; nowhere past the last frequency.
template <typename R, int CH> struct Sink {
  RecLev<R, CH> *V;
  float4 *ft;   // the fused four-step apply's copy of level 0 (aao_internal.cuh), or NULL
  int ell;
  bool live;
  // z times the power of two f, rounded to R; element i of the run that starts
  // at pair `first` of the copy (-1: not in it)
  template <typename E>
  __device__ __forceinline__ void put(cx<R> *p, const zc<E> &z, double f, int first = -1, int i = 0) const {
    if (!live) return;
    const R v = (R)(lead(z.v) * f);
    reinterpret_cast<R *>(p)[imag()] = v;
    if (ft && first >= 0)
      reinterpret_cast<float *>(ft + (size_t)(first + i / 2) * ell)[2 * (i & 1) + imag()] = (float)v;
  }
};

// What role 0 (regular chunks) or 1 (last chunk) writes of level `level`.
template <typename R, int CH, typename E>
__device__ void entries(int role, int level, const BlockSymbol &sy, const Sink<R, CH> &out, int levels,
                        const int *lsz, bool ragged) {
  using Z = zc<E>;
  constexpr int c = CH - 1;
  constexpr bool PAIRS = sizeof(E) == 16;
  const Z one = real_z<E>(1.0), nil = real_z<E>(0.0);
  Z sig{E(imag() ? sy.sig_im : sy.sig_re)}, a{E(imag() ? -sy.e_im : -sy.e_re)};
  Z sig_l = sig, b = a;
  for (int l = 0;; l++) {
    const int cl = lsz[l] - (l + 1 < levels ? lsz[l + 1] : 0) * CH;
    const int N = role && cl == CH ? CH : c;
    Z D[CH + 1], A[CH + 1], Hs[PAIRS ? 1 : CH + 1];   // A_i = a^i
    D[0] = A[0] = one;
    if constexpr (PAIRS) {
      const Z d = zadd(sig, zadd(a, a)), q = zneg(zmul(a, a));
      D[1] = d;
      A[1] = a;
#pragma unroll 1
      for (int i = 1; i < N; i++) {
        A[i + 1] = zmul(a, A[i]);
        D[i + 1] = zfma(d, D[i], zmul(q, D[i - 1]));
      }
    } else {
      Hs[0] = nil;
#pragma unroll 1
      for (int i = 0; i < N; i++) {
        Hs[i + 1] = zfma(sig, D[i], zmul(a, Hs[i]));
        A[i + 1] = zmul(a, A[i]);
        D[i + 1] = zfma(a, D[i], zadd(Hs[i + 1], A[i + 1]));
      }
    }
    auto excess = [&](int i) {   // H_i
      if constexpr (PAIRS) return i ? zsub(zfma(zneg(a), D[i - 1], D[i]), A[i]) : nil;
      else return Hs[i];
    };
    const Z x = zsub(sig_l, sig), delta = zadd(x, zsub(b, a));
    auto det_l = [&](int i) { return i ? zfma(delta, D[i - 1], D[i]) : one; };   // R_i
    const Z inv = zrecip(role && l == level ? det_l(cl) : D[c]);
    if (l < level) {
      const Z h = zmul(zmul(a, excess(c)), inv);
      if (role) {
        const Z invl = zrecip(det_l(cl));
        const Z S = zfma(x, A[cl - 1], zfma(delta, excess(cl - 1), excess(cl)));
        sig_l = zadd(sig, zfma(zmul(a, S), invl, h));
        b = zmul(zmul(A[cl], b), invl);
      }
      sig = zadd(sig, zadd(h, h));
      a = zmul(zmul(a, A[c]), inv);
      continue;
    }
    RecLev<R, CH> &V = *out.V;
    const int tinv = ragged ? kFuseTailInv : -1, tgreen = ragged ? kFuseTailGreen : -1;
    if (role == 0) {
#pragma unroll 1
      for (int i = 0; i < c; i++) {
        const Z p = zmul(D[i], zrecip(D[i + 1]));
        out.put(&V.invp[i], p, sy.scale, 0, i);
        if (i < cl - 1) out.put(&V.invt[i], p, sy.scale, tinv, i);
        out.put(&V.bp[i], zneg(zmul(a, p)), 1.0, i < c - 1 ? 8 : 15, i < c - 1 ? i : c);
        out.put(&V.fc[i], zmul(zmul(A[i + 1], D[c - 1 - i]), inv), 1.0, 15, i);
      }
      out.put(&V.e, zneg(a), 1.0 / sy.scale, 0, c);
      out.put(&V.invp[c], nil, 1.0);
      out.put(&V.bp[c], nil, 1.0);
      out.put(&V.fc[c], nil, 1.0);
      out.put(&V.pad, nil, 1.0);
    } else {
#pragma unroll 1
      for (int i = 0; i < CH; i++) {
        out.put(&V.fl[i], i < cl ? zmul(zmul(A[i + 1], det_l(cl - 1 - i)), inv) : nil, 1.0, tgreen, i);
        if (i >= cl - 1)
          out.put(&V.invt[i], i == cl - 1 ? zmul(D[i], inv) : nil, i == cl - 1 ? sy.scale : 1.0, tinv, i);
      }
    }
    return;
  }
}

// grid (frequencies / 16, role + 2 level)
template <typename R, int CH, typename E>
__global__ void __launch_bounds__(32)
k_tables(const BlockSymbol *__restrict__ sym, int nk, RecLev<R, CH> *__restrict__ tabs, int levels,
         int4 lsz_lo, int2 lsz_hi, float4 *__restrict__ fuse, int ell, int L1, int ragged) {
  const int q = blockIdx.x * 16 + threadIdx.x / 2, k = min(q, nk - 1);
  const int role = blockIdx.y & 1, level = blockIdx.y >> 1;
  const int lsz[kRecLevels] = {lsz_lo.x, lsz_lo.y, lsz_lo.z, lsz_lo.w, lsz_hi.x, lsz_hi.y};
  float4 *ft = fuse && level == 0 ? fuse + (size_t)(k % L1) * (ell / L1) + k / L1 : nullptr;
  const Sink<R, CH> out{tabs + (size_t)k * levels + level, ft, ell, q < nk};
  entries<R, CH, E>(role, level, sym[k], out, levels, lsz, ragged != 0);
}

template <typename R, int CH, typename E>
cudaError_t run_tables(const Ctx &c, void *tab, int levels, const int *lsz, void *fuse, cudaStream_t s) {
  k_tables<R, CH, E><<<dim3((unsigned)((c.nk + 15) / 16), 2 * levels), 32, 0, s>>>(
      static_cast<const BlockSymbol *>(c.symbols), (int)c.nk, static_cast<RecLev<R, CH> *>(tab), levels,
      make_int4(lsz[0], lsz[1], lsz[2], lsz[3]), make_int2(lsz[4], lsz[5]), static_cast<float4 *>(fuse),
      (int)c.ell, four_l1(c.ell), (c.n + 1) % 16 != 0 ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace

size_t rec_table_bytes(const Ctx &c, bool fp64) {
  if (!fp64) return (size_t)c.nk * c.lev32 * sizeof(RecLev<float, 16>);
  return (size_t)c.nk * c.lev64 * (c.ch64 == 8 ? sizeof(RecLev<double, 8>) : sizeof(RecLev<double, 16>));
}

cudaError_t launch_build_tables(const Ctx &c, bool fp64, cudaStream_t s) {
  if (!fp64) return run_tables<float, 16, double>(c, c.rec32, c.lev32, c.lsz32, c.fuse32, s);
  return c.ch64 == 8 ? run_tables<double, 8, pair>(c, c.rec64, c.lev64, c.lsz64, nullptr, s)
                     : run_tables<double, 16, pair>(c, c.rec64, c.lev64, c.lsz64, nullptr, s);
}

}  // namespace aao
