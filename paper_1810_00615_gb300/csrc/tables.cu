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
// block is, and the chain has two quotients a level.
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
// aao_set_kappa with its copies, against the host building the tables, and the
// host before the recursion served every row: n 63 x ell 64 153 us (124, 229), n
// 5000 x ell 300 279 (395, 300), n 1000 x ell 900 238 (934, 679), n 12345 x ell 4096
// 726 (6867, 3535).  With a lane a frequency it was 175, 371, 310 and 678; with all
// levels of a role in one thread besides 268, 542, 463 and 890.
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
__device__ __forceinline__ double fmadd(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double recip(double a) { return 1.0 / a; }

// Pairs: unevaluated sums h + l of two FP64 numbers, |l| at most half a unit of
// h (Dekker; products split by FMA).  Rounded operations throughout: a
// contracted product would undo the splitting.
struct pair {
  double h, l;
  __device__ __forceinline__ pair() {}
  __device__ __forceinline__ explicit pair(double a) : h(a), l(0.0) {}
  __device__ __forceinline__ pair(double a, double b) : h(a), l(b) {}
};
__device__ __forceinline__ pair other(pair a) { return {other(a.h), other(a.l)}; }
__device__ __forceinline__ double lead(pair a) { return a.h; }
__device__ __forceinline__ pair neg(pair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ pair tidy(double h, double l) {           // |h| >= |l|
  const double s = __dadd_rn(h, l);
  return {s, __dsub_rn(l, __dsub_rn(s, h))};
}
__device__ __forceinline__ pair add(pair a, pair b) {
  const double s = __dadd_rn(a.h, b.h), t = __dsub_rn(s, a.h);
  const double e = __dadd_rn(__dsub_rn(a.h, __dsub_rn(s, t)), __dsub_rn(b.h, t));
  return tidy(s, __dadd_rn(a.l, __dadd_rn(e, b.l)));
}
__device__ __forceinline__ pair mul(pair a, pair b) {
  const double p = __dmul_rn(a.h, b.h);
  return tidy(p, __fma_rn(a.l, b.h, __fma_rn(a.h, b.l, __fma_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ pair fmadd(pair a, pair b, pair c) { return add(mul(a, b), c); }
__device__ __forceinline__ pair recip(pair a) {
  const double r = 1.0 / a.h;
  return tidy(r, __dmul_rn(r, __fma_rn(-a.l, r, __fma_rn(-a.h, r, 1.0))));
}

template <typename E> __device__ __forceinline__ zc<E> real_z(double a) { return {E(imag() ? 0.0 : a)}; }
template <typename E> __device__ __forceinline__ zc<E> zadd(zc<E> a, zc<E> b) { return {add(a.v, b.v)}; }
template <typename E> __device__ __forceinline__ zc<E> zneg(zc<E> a) { return {neg(a.v)}; }
template <typename E> __device__ __forceinline__ zc<E> zsub(zc<E> a, zc<E> b) { return zadd(a, zneg(b)); }
// a b (+ c): (re re) - (im im) in the even lane, (re im) + (im re) in the odd one
template <typename E> __device__ __forceinline__ zc<E> zmul(zc<E> a, zc<E> b) {
  const E ap = other(a.v);
  return {fmadd(imag() ? ap : a.v, b.v, mul(imag() ? a.v : neg(ap), other(b.v)))};
}
template <typename E> __device__ __forceinline__ zc<E> zfma(zc<E> a, zc<E> b, zc<E> c) {
  const E ap = other(a.v);
  return {fmadd(imag() ? ap : a.v, b.v, fmadd(imag() ? a.v : neg(ap), other(b.v), c.v))};
}
template <typename E> __device__ __forceinline__ zc<E> zrecip(zc<E> a) {
  const E p = other(a.v), r = mul(a.v, recip(fmadd(a.v, a.v, mul(p, p))));
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
  const Z one = real_z<E>(1.0), nil = real_z<E>(0.0);
  Z sig{E(imag() ? sy.sig_im : sy.sig_re)}, a{E(imag() ? -sy.e_im : -sy.e_re)};
  Z sig_l = sig, b = a;
  for (int l = 0;; l++) {
    const int cl = lsz[l] - (l + 1 < levels ? lsz[l + 1] : 0) * CH;
    const int N = role && cl == CH ? CH : c;
    Z D[CH + 1], H[CH + 1], A[CH + 1];   // A_i = a^i
    D[0] = A[0] = one;
    H[0] = nil;
#pragma unroll 1
    for (int i = 0; i < N; i++) {
      H[i + 1] = zfma(sig, D[i], zmul(a, H[i]));
      A[i + 1] = zmul(a, A[i]);
      D[i + 1] = zfma(a, D[i], zadd(H[i + 1], A[i + 1]));
    }
    const Z x = zsub(sig_l, sig), delta = zadd(x, zsub(b, a));
    auto det_l = [&](int i) { return i ? zfma(delta, D[i - 1], D[i]) : one; };   // R_i
    const Z inv = zrecip(role && l == level ? det_l(cl) : D[c]);
    if (l < level) {
      const Z h = zmul(a, zmul(H[c], inv));
      if (role) {
        const Z invl = zrecip(det_l(cl));
        const Z S = zfma(x, A[cl - 1], zfma(delta, H[cl - 1], H[cl]));
        sig_l = zadd(sig, zfma(a, zmul(S, invl), h));
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

// grid (frequencies / 16, role + 2 level, FP64 or FP32 tables)
template <int CH64>
__global__ void __launch_bounds__(32)
k_tables(const BlockSymbol *__restrict__ sym, int nk, RecLev<float, 16> *__restrict__ tab32,
         int lev32, int4 lo32, int2 hi32, float4 *__restrict__ fuse, int ell, int L1, int ragged,
         RecLev<double, CH64> *__restrict__ tab64, int lev64, int4 lo64, int2 hi64) {
  const int q = blockIdx.x * 16 + threadIdx.x / 2, k = min(q, nk - 1);
  const int role = blockIdx.y & 1, level = blockIdx.y >> 1;
  if (blockIdx.z == 0) {
    if (level >= lev64) return;
    const int lsz[kRecLevels] = {lo64.x, lo64.y, lo64.z, lo64.w, hi64.x, hi64.y};
    const Sink<double, CH64> out{tab64 + (size_t)k * lev64 + level, nullptr, ell, q < nk};
    entries<double, CH64, pair>(role, level, sym[k], out, lev64, lsz, false);
  } else {
    if (level >= lev32) return;
    const int lsz[kRecLevels] = {lo32.x, lo32.y, lo32.z, lo32.w, hi32.x, hi32.y};
    float4 *ft = fuse && level == 0 ? fuse + (size_t)(k % L1) * (ell / L1) + k / L1 : nullptr;
    const Sink<float, 16> out{tab32 + (size_t)k * lev32 + level, ft, ell, q < nk};
    entries<float, 16, double>(role, level, sym[k], out, lev32, lsz, ragged != 0);
  }
}

template <int CH64>
cudaError_t run_tables(const Ctx &c, cudaStream_t s) {
  auto lo = [](const int *v) { return make_int4(v[0], v[1], v[2], v[3]); };
  auto hi = [](const int *v) { return make_int2(v[4], v[5]); };
  const int levels = c.lev64 > c.lev32 ? c.lev64 : c.lev32;
  k_tables<CH64><<<dim3((unsigned)((c.nk + 15) / 16), 2 * levels, 2), 32, 0, s>>>(
      static_cast<const BlockSymbol *>(c.symbols), (int)c.nk, static_cast<RecLev<float, 16> *>(c.rec32),
      c.lev32, lo(c.lsz32), hi(c.lsz32), static_cast<float4 *>(c.fuse32), (int)c.ell,
      four_l1(c.ell), (c.n + 1) % 16 != 0 ? 1 : 0, static_cast<RecLev<double, CH64> *>(c.rec64),
      c.lev64, lo(c.lsz64), hi(c.lsz64));
  return cudaGetLastError();
}

}  // namespace

size_t rec_table_bytes(const Ctx &c, bool fp64) {
  if (!fp64) return (size_t)c.nk * c.lev32 * sizeof(RecLev<float, 16>);
  return (size_t)c.nk * c.lev64 * (c.ch64 == 8 ? sizeof(RecLev<double, 8>) : sizeof(RecLev<double, 16>));
}

cudaError_t launch_build_tables(const Ctx &c, cudaStream_t s) {
  return c.ch64 == 8 ? run_tables<8>(c, s) : run_tables<16>(c, s);
}

}  // namespace aao
