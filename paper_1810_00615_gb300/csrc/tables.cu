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
// aao_set_kappa, the one allocation and the copies around it included: n 63 x
// ell 64 175 us (with all levels of a role in one thread 268; tables built and
// copied by the host 121, by the host before the recursion served every row
// 229), n 5000 x ell 300 371 (542, 406, 307), n 1000 x ell 900 310 (463, 944,
// 698), n 12345 x ell 4096 678 (890, 7089, 3599).
#include "aao_internal.cuh"

namespace aao {
namespace {

template <typename E> struct zc {
  E re, im;
};
using zd = zc<double>;
__device__ __forceinline__ double lead(double a) { return a; }
__device__ __forceinline__ zd zadd(zd a, zd b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ zd zsub(zd a, zd b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ zd zneg(zd a) { return {-a.re, -a.im}; }
__device__ __forceinline__ zd zmul(zd a, zd b) {
  return {fma(a.re, b.re, -a.im * b.im), fma(a.re, b.im, a.im * b.re)};
}
__device__ __forceinline__ zd zfma(zd a, zd b, zd c) {   // a b + c
  return {fma(-a.im, b.im, fma(a.re, b.re, c.re)), fma(a.im, b.re, fma(a.re, b.im, c.im))};
}
__device__ __forceinline__ zd zrecip(zd a) {
  const double d = fma(a.re, a.re, a.im * a.im);
  return {a.re / d, -a.im / d};
}

// Pairs: unevaluated sums h + l of two FP64 numbers, |l| at most half a unit of
// h (Dekker; products split by FMA).  Rounded operations throughout: a
// contracted product would undo the splitting.
struct pair {
  double h, l;
  __device__ __forceinline__ pair() {}
  __device__ __forceinline__ explicit pair(double a) : h(a), l(0.0) {}
  __device__ __forceinline__ pair(double a, double b) : h(a), l(b) {}
};
using zp = zc<pair>;
__device__ __forceinline__ double lead(pair a) { return a.h; }
__device__ __forceinline__ pair neg(pair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ pair tidy(pair a) {                      // |h| >= |l|
  const double s = __dadd_rn(a.h, a.l);
  return {s, __dsub_rn(a.l, __dsub_rn(s, a.h))};
}
// a + (b, c) and a + x y, left untidy
__device__ __forceinline__ pair plus(pair a, double b, double c) {
  const double s = __dadd_rn(a.h, b), t = __dsub_rn(s, a.h);
  const double e = __dadd_rn(__dsub_rn(a.h, __dsub_rn(s, t)), __dsub_rn(b, t));
  return {s, __dadd_rn(a.l, __dadd_rn(e, c))};
}
__device__ __forceinline__ pair plus(pair a, pair x, pair y) {
  const double p = __dmul_rn(x.h, y.h);
  return plus(a, p, __fma_rn(x.l, y.h, __fma_rn(x.h, y.l, __fma_rn(x.h, y.h, -p))));
}
__device__ __forceinline__ pair mul(pair x, pair y) {
  const double p = __dmul_rn(x.h, y.h);
  return {p, __fma_rn(x.l, y.h, __fma_rn(x.h, y.l, __fma_rn(x.h, y.h, -p)))};
}
__device__ __forceinline__ zp zadd(zp a, zp b) {
  return {tidy(plus(a.re, b.re.h, b.re.l)), tidy(plus(a.im, b.im.h, b.im.l))};
}
__device__ __forceinline__ zp zneg(zp a) { return {neg(a.re), neg(a.im)}; }
__device__ __forceinline__ zp zsub(zp a, zp b) { return zadd(a, zneg(b)); }
__device__ __forceinline__ zp zmul(zp a, zp b) {
  return {tidy(plus(mul(a.re, b.re), neg(a.im), b.im)), tidy(plus(mul(a.re, b.im), a.im, b.re))};
}
__device__ __forceinline__ zp zfma(zp a, zp b, zp c) {
  return {tidy(plus(plus(c.re, a.re, b.re), neg(a.im), b.im)),
          tidy(plus(plus(c.im, a.re, b.im), a.im, b.re))};
}
__device__ __forceinline__ zp zrecip(zp a) {
  const pair d = tidy(plus(mul(a.re, a.re), a.im, a.im));
  const double r = 1.0 / d.h;
  const pair inv = tidy({r, __dmul_rn(r, __fma_rn(-d.l, r, __fma_rn(-d.h, r, 1.0)))});
  return {tidy(mul(a.re, inv)), tidy(neg(mul(a.im, inv)))};
}

// a times the power of two f, rounded to R
template <typename R, typename E>
__device__ __forceinline__ cx<R> rounded(const zc<E> &a, double f) {
  return mk((R)(lead(a.re) * f), (R)(lead(a.im) * f));
}

// An element of the fused four-step apply's copy of level 0 (aao_internal.cuh):
// element i of the run that starts at pair `first`; NULL: none.
__device__ __forceinline__ void fuse_put(float4 *ft, int ell, int first, int i, cx<float> v) {
  if (ft)
    reinterpret_cast<float2 *>(ft + (size_t)(first + i / 2) * ell)[i & 1] = make_float2(v.re, v.im);
}
__device__ __forceinline__ void fuse_put(float4 *, int, int, int, cx<double>) {}

// What role 0 (regular chunks) or 1 (last chunk) writes of level `level`.
template <typename R, int CH, typename E>
__device__ void entries(int role, int level, const BlockSymbol &sy, RecLev<R, CH> &V, int levels,
                        const int *lsz, float4 *fuse, int ell, bool ragged) {
  using Z = zc<E>;
  constexpr int c = CH - 1;
  const cx<R> nil = mk((R)0, (R)0);
  Z sig{E(sy.sig_re), E(sy.sig_im)}, a{E(-sy.e_re), E(-sy.e_im)};
  Z sig_l = sig, b = a;
  for (int l = 0;; l++) {
    const int cl = lsz[l] - (l + 1 < levels ? lsz[l + 1] : 0) * CH;
    const int N = role && cl == CH ? CH : c;
    Z D[CH + 1], H[CH + 1], A[CH + 1];   // A_i = a^i
    D[0] = A[0] = {E(1.0), E(0.0)};
    H[0] = {E(0.0), E(0.0)};
#pragma unroll 1
    for (int i = 0; i < N; i++) {
      H[i + 1] = zfma(sig, D[i], zmul(a, H[i]));
      A[i + 1] = zmul(a, A[i]);
      D[i + 1] = zfma(a, D[i], zadd(H[i + 1], A[i + 1]));
    }
    const Z x = zsub(sig_l, sig), delta = zadd(x, zsub(b, a));
    auto det_l = [&](int i) { return i ? zfma(delta, D[i - 1], D[i]) : D[0]; };   // R_i
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
    float4 *ft = l == 0 ? fuse : nullptr;
    if (role == 0) {
#pragma unroll 1
      for (int i = 0; i < c; i++) {
        const Z p = zmul(D[i], zrecip(D[i + 1]));
        const cx<R> ip = rounded<R>(p, sy.scale), bp = rounded<R>(zneg(zmul(a, p)), 1.0);
        const cx<R> fc = rounded<R>(zmul(zmul(A[i + 1], D[c - 1 - i]), inv), 1.0);
        V.invp[i] = ip;
        V.bp[i] = bp;
        V.fc[i] = fc;
        fuse_put(ft, ell, 0, i, ip);
        if (i < c - 1) fuse_put(ft, ell, 8, i, bp);
        else fuse_put(ft, ell, 15, c, bp);
        fuse_put(ft, ell, 15, i, fc);
        if (i < cl - 1) {
          V.invt[i] = ip;
          if (ragged) fuse_put(ft, ell, kFuseTailInv, i, ip);
        }
      }
      const cx<R> e = rounded<R>(zneg(a), 1.0 / sy.scale);
      V.e = e;
      fuse_put(ft, ell, 0, c, e);
      V.invp[c] = V.bp[c] = V.fc[c] = V.pad = nil;
    } else {
#pragma unroll 1
      for (int i = 0; i < CH; i++) {
        const cx<R> fl =
            i < cl ? rounded<R>(zmul(zmul(A[i + 1], det_l(cl - 1 - i)), inv), 1.0) : nil;
        V.fl[i] = fl;
        if (ragged) fuse_put(ft, ell, kFuseTailGreen, i, fl);
        if (i < cl - 1) continue;
        const cx<R> last = i == cl - 1 ? rounded<R>(zmul(D[i], inv), sy.scale) : nil;
        V.invt[i] = last;
        if (ragged) fuse_put(ft, ell, kFuseTailInv, i, last);
      }
    }
    return;
  }
}

// grid (frequencies / 32, role + 2 level, FP64 or FP32 tables)
template <int CH64>
__global__ void __launch_bounds__(32)
k_tables(const BlockSymbol *__restrict__ sym, int nk, RecLev<float, 16> *__restrict__ tab32,
         int lev32, int4 lo32, int2 hi32, float4 *__restrict__ fuse, int ell, int L1, int ragged,
         RecLev<double, CH64> *__restrict__ tab64, int lev64, int4 lo64, int2 hi64) {
  const int k = blockIdx.x * 32 + threadIdx.x, role = blockIdx.y & 1, level = blockIdx.y >> 1;
  if (k >= nk) return;
  if (blockIdx.z == 0) {
    if (level >= lev64) return;
    const int lsz[kRecLevels] = {lo64.x, lo64.y, lo64.z, lo64.w, hi64.x, hi64.y};
    entries<double, CH64, pair>(role, level, sym[k], tab64[(size_t)k * lev64 + level], lev64, lsz, nullptr, ell, false);
  } else {
    if (level >= lev32) return;
    const int lsz[kRecLevels] = {lo32.x, lo32.y, lo32.z, lo32.w, hi32.x, hi32.y};
    float4 *ft = fuse ? fuse + (size_t)(k % L1) * (ell / L1) + k / L1 : nullptr;
    entries<float, 16, double>(role, level, sym[k], tab32[(size_t)k * lev32 + level], lev32, lsz, ft, ell, ragged);
  }
}

template <int CH64>
cudaError_t run_tables(const Ctx &c, cudaStream_t s) {
  auto lo = [](const int *v) { return make_int4(v[0], v[1], v[2], v[3]); };
  auto hi = [](const int *v) { return make_int2(v[4], v[5]); };
  const int levels = c.lev64 > c.lev32 ? c.lev64 : c.lev32;
  k_tables<CH64><<<dim3((unsigned)((c.nk + 31) / 32), 2 * levels, 2), 32, 0, s>>>(
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
