// Per-frequency complex tridiagonal solves (Section 3: after the Fourier
// diagonalisation, I (x) A0 + Lambda (x) A1 is block diagonal and each block
// A0 + w_k A1 (+ w_k^2 A2) is tridiagonal; the paper assigns one block per
// process and applies the Thomas algorithm).
//
// GB300 design: one CTA per frequency k, one thread per chunk of CH-1
// unknowns plus the separator unknown that follows it.  The row is read and
// written exactly once, through a shared-memory staging buffer.
//   1. Local Dirichlet solve of each chunk with the chunk LU, whose pivots are
//      shared by all chunks of a row (constant coefficients) and precomputed.
//   2. The separators satisfy a tridiagonal Schur-complement system (one row
//      per separator) whose coefficients follow from the chunk Green's
//      functions (precomputed); it has the same form again and is solved by
//      the same substructuring one level up, down to a single chunk.  The
//      tables come from the "row excess" form (sigma = a + b + c instead of
//      the diagonal), which is how the smooth, nearly singular low
//      frequencies (k = 0 is tau*kappa*K, the Laplacian) keep their accuracy
//      in FP32.
//   3. Each chunk is corrected with the two separator values around it.
// Any n is served: a level whose size does not divide into whole chunks has
// a last chunk of its own (RecLev's invt, fl).  This recursion replaced
// parallel cyclic reduction for those n: log2(n/CH) rounds of two complex
// divisions each, 88 us per FP64 solve at n = 1024, ell = 1024.
#include <cooperative_groups.h>

#include "aao_internal.cuh"

namespace cg = cooperative_groups;

namespace aao {

// Row staging: the row is moved between global and shared memory in 16-byte
// chunks by consecutive threads (coalesced), and stored with the 16-byte
// chunk index XOR-ed with (line & 7) inside each 128-byte line, so that the
// per-thread reads of one whole line (thread p owns line p) hit all 32 banks.
__device__ __forceinline__ int swz(int chunk) { return chunk ^ ((chunk >> 3) & 7); }

// Level buffers of the recursive form: one padding slot per CH values so
// that the chunk-strided accesses of the threads fall in distinct banks.
template <int CH>
__host__ __device__ __forceinline__ int rpos(int e) { return e + e / CH; }
// Values of the buffer of level l: whole chunks, the tail past lsz[l] zeroed
// by the caller, so that no chunk loop has to know the last chunk's length.
template <int CH>
__host__ __device__ __forceinline__ int level_size(const int *lsz, int levels, int l) {
  return ((l + 1 < levels ? lsz[l + 1] : 0) + 1) * CH;
}
// Lay the buffers of levels 1 .. levels-1 out from `base` (B[l], NULL for a
// size alone) and return the values they take.
template <typename R, int CH>
__host__ __device__ __forceinline__ size_t level_buffers(const int *lsz, int levels, cx<R> *base,
                                                         cx<R> **B) {
  size_t off = 0;
  for (int l = 1; l < levels; l++) {
    if (B) B[l] = base + off;
    off += (size_t)rpos<CH>(level_size<CH>(lsz, levels, l)) + 1;
  }
  return off;
}
// Zero the tails of the level buffers (nthr threads, thread p).
template <typename R, int CH>
__device__ __forceinline__ void zero_tails(cx<R> *const *B, const int *lsz, int levels, int p,
                                           int nthr) {
  for (int l = 1; l < levels; l++)
    for (int e = lsz[l] + p; e < level_size<CH>(lsz, levels, l); e += nthr)
      B[l][rpos<CH>(e)] = mk((R)0, (R)0);
}

// Copy the levels in use of a frequency's table into shared memory,
// conjugated for the transposed symbols; nthr threads, thread p.
template <typename R, int CH>
__device__ __forceinline__ void load_levels(RecLev<R, CH> *dst, const RecLev<R, CH> *__restrict__ tab,
                                            int levels, int conj, int p, int nthr) {
  constexpr int NV = (int)(sizeof(RecLev<R, CH>) / sizeof(cx<R>));
  const cx<R> *src = reinterpret_cast<const cx<R> *>(tab);
  cx<R> *d = reinterpret_cast<cx<R> *>(dst);
  for (int i = p; i < levels * NV; i += nthr) {
    cx<R> z = src[i];
    if (conj) z.im = -z.im;
    d[i] = z;
  }
}

// Dirichlet solve of one chunk in registers with the pivots inv (invp, or
// invt for the last chunk): entries whose 1/pivot is zero come out zero.  Only
// a last chunk of CH unknowns (all) has one in the separator's place; the others
// leave v[CH - 1] alone, a ninth of an FP64 chunk's arithmetic and two links
// of its chain (whole FP64 apply n 4095 x ell 4096: 1871 -> 1857 us, n 16383 x
// ell 16: 107.4 -> 105.2 with the upper levels).
template <typename R, int CH>
__device__ __forceinline__ void chunk_solve(cx<R> *v, const cx<R> *inv, const cx<R> *bp, cx<R> e,
                                            bool all) {
  v[0] = v[0] * inv[0];
#pragma unroll
  for (int i = 1; i < CH - 1; i++) v[i] = cfnms(v[i], e, v[i - 1]) * inv[i];
  if (all) {
    if constexpr (sizeof(R) == 8) asm volatile("");   // a branch: one warp of the row takes it
    v[CH - 1] = cfnms(v[CH - 1], e, v[CH - 2]) * inv[CH - 1];
    v[CH - 2] = cfnms(v[CH - 2], bp[CH - 2], v[CH - 1]);
  }
#pragma unroll
  for (int i = CH - 3; i >= 0; i--) v[i] = cfnms(v[i], bp[i], v[i + 1]);
}

// Levels 1 .. levels-1 of the recursive form on shared-memory buffers:
// B[1] holds the level-1 right-hand sides on entry and the level-1 solution
// (the level-0 separator values) on exit.  Called by all threads of one CTA.
template <typename R, int CH>
__device__ __forceinline__ void rec_upper(cx<R> *const *B, const int *lsz, int levels,
                                          const RecLev<R, CH> *T, int p) {
  const int nthr = (int)blockDim.x;
  const cx<R> zero = mk((R)0, (R)0);
  for (int l = 1; l < levels; l++) {
    const int Ml = l + 1 < levels ? lsz[l + 1] : 0, Pl = Ml + 1;
    cx<R> *Bl = B[l];
    const cx<R> el = T[l].e;
    for (int q = p; q < Pl; q += nthr) {
      const bool last = q == Ml;
      cx<R> w[CH];
#pragma unroll
      for (int i = 0; i < CH; i++) w[i] = Bl[rpos<CH>(q * CH + i)];
      // FP32 takes every chunk for a full one (w[CH - 1] comes out zero): the
      // branch costs more than it saves, n 65535 x ell 512 397 -> 402 us
      chunk_solve<R, CH>(w, last ? T[l].invt : T[l].invp, T[l].bp, el,
                         sizeof(R) == 4 || (last && lsz[l] == Pl * CH));
#pragma unroll
      for (int i = 0; i < CH - 1; i++) Bl[rpos<CH>(q * CH + i)] = w[i];
      if (last) Bl[rpos<CH>(q * CH + CH - 1)] = w[CH - 1];
    }
    __syncthreads();
    for (int q = p; q < Ml; q += nthr) {
      const cx<R> sep = Bl[rpos<CH>(q * CH + CH - 1)];
      const cx<R> lastl = Bl[rpos<CH>(q * CH + CH - 2)];
      const cx<R> firstr = Bl[rpos<CH>((q + 1) * CH)];
      B[l + 1][rpos<CH>(q)] = cfnms(sep, el, lastl + firstr);
    }
    if (Ml > 0) __syncthreads();
  }
  for (int l = levels - 2; l >= 1; l--) {
    const int Ml = lsz[l + 1], Pl = Ml + 1;
    cx<R> *Bl = B[l];
    const cx<R> *Bu = B[l + 1];
    for (int q = p; q < Pl; q += nthr) {
      const bool last = q == Ml;
      const cx<R> sl = (q > 0) ? Bu[rpos<CH>(q - 1)] : zero;
      const cx<R> sr = last ? zero : Bu[rpos<CH>(q)];
      const cx<R> *fl = last ? T[l].fl : T[l].fc;
#pragma unroll
      for (int i = 0; i < CH - 1; i++) {
        const int pos = rpos<CH>(q * CH + i);
        Bl[pos] = cfma(cfma(Bl[pos], sl, fl[i]), sr, T[l].fc[CH - 2 - i]);
      }
      const int pe = rpos<CH>(q * CH + CH - 1);
      Bl[pe] = last ? cfma(Bl[pe], sl, fl[CH - 1]) : sr;
    }
    __syncthreads();
  }
}

// One CTA per frequency row, level 0 in registers, the higher levels in
// shared memory.  SMALL: at most 256 threads (rows up to 4096), compiled for
// AAO_TRI_MINB resident CTAs per SM so that the ell/2 + 1 frequencies take
// fewer waves.  STAGE: the row fits in shared memory and moves through it;
// otherwise (FP64 rows beyond 11264, 200 KB) each thread reads its chunk directly.
#ifndef AAO_TRI_MINB
#define AAO_TRI_MINB 3
#endif
template <typename R, int CH, bool SMALL, bool STAGE>
__global__ void __launch_bounds__(SMALL ? 256 : 1024, SMALL ? AAO_TRI_MINB : 1)
k_tridiag_rec(cx<R> *__restrict__ spec, int n, int64_t n_pad,
              const RecLev<R, CH> *__restrict__ tabs, int conj_sym, int levels, int4 lsz_lo,
              int2 lsz_hi) {
  const int k = blockIdx.x;
  const int p = threadIdx.x;
  const int P = blockDim.x;
  const int M = P - 1;
  const int lsz[kRecLevels] = {lsz_lo.x, lsz_lo.y, lsz_lo.z, lsz_lo.w, lsz_hi.x, lsz_hi.y};
  __shared__ RecLev<R, CH> T[kRecLevels];
  extern __shared__ __align__(16) unsigned char smraw[];
  // level buffers B_1..B_{levels-1}, then the staged row
  cx<R> *B[kRecLevels];
  size_t off = level_buffers<R, CH>(lsz, levels, reinterpret_cast<cx<R> *>(smraw), B);
  cx<R> *s_first = reinterpret_cast<cx<R> *>(smraw) + off;   // [P]
  off += (size_t)P;
  float4 *s_row = reinterpret_cast<float4 *>(smraw + ((off * sizeof(cx<R>) + 15) & ~(size_t)15));
  constexpr int EPC = 16 / sizeof(cx<R>);
  load_levels<R, CH>(T, tabs + (size_t)k * levels, levels, conj_sym, p, P);
  zero_tails<R, CH>(B, lsz, levels, p, P);

  cx<R> *row = spec + (size_t)k * n_pad;
  const int base = p * CH;
  const unsigned long long pol_keep = l2_evict_last();
  cx<R> v[CH];
  if constexpr (STAGE) {
    const float4 *g = reinterpret_cast<const float4 *>(row);
    // P CH / EPC 16-byte chunks (n_pad >= P CH): every thread copies CH / EPC,
    // all loads issued before the first store
    float4 ch[CH / EPC];
#pragma unroll
    for (int j = 0; j < CH / EPC; j++) ch[j] = ld_hint4(&g[p + j * P], pol_keep);
#pragma unroll
    for (int j = 0; j < CH / EPC; j++) s_row[swz(p + j * P)] = ch[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < CH / EPC; j++) {
      const float4 f = s_row[swz(p * (CH / EPC) + j)];
      const cx<R> *z = reinterpret_cast<const cx<R> *>(&f);
#pragma unroll
      for (int u = 0; u < EPC; u++) v[j * EPC + u] = (base + j * EPC + u < n) ? z[u] : mk((R)0, (R)0);
    }
  } else {
#pragma unroll
    for (int i = 0; i < CH; i++) v[i] = (base + i < n) ? row[base + i] : mk((R)0, (R)0);
  }
  __syncthreads();

  // level 0: local Dirichlet solve of the chunk, its separator value aside
  const bool last = p == M;
  const cx<R> e0 = T[0].e, sep = v[CH - 1];
  chunk_solve<R, CH>(v, last ? T[0].invt : T[0].invp, T[0].bp, e0, last && n == P * CH);
  if (levels > 1) {
    // separator right-hand sides of level 1: needs the first local value of
    // the next chunk
    s_first[p] = v[0];
    __syncthreads();
    if (p < M) B[1][rpos<CH>(p)] = cfnms(sep, e0, v[CH - 2] + s_first[p + 1]);
    __syncthreads();
    rec_upper<R, CH>(B, lsz, levels, T, p);
    // level 0 correction
    const cx<R> sl = (p > 0) ? B[1][rpos<CH>(p - 1)] : mk((R)0, (R)0);
    const cx<R> sr = last ? mk((R)0, (R)0) : B[1][rpos<CH>(p)];
    const cx<R> *fl = last ? T[0].fl : T[0].fc;
#pragma unroll
    for (int i = 0; i < CH - 1; i++) v[i] = cfma(cfma(v[i], sl, fl[i]), sr, T[0].fc[CH - 2 - i]);
    v[CH - 1] = last ? cfma(v[CH - 1], sl, fl[CH - 1]) : sr;
  }

  if constexpr (STAGE) {
    // write back through the staging buffer
#pragma unroll
    for (int j = 0; j < CH / EPC; j++) {
      float4 f;
      cx<R> *z = reinterpret_cast<cx<R> *>(&f);
#pragma unroll
      for (int u = 0; u < EPC; u++) z[u] = v[j * EPC + u];
      s_row[swz(p * (CH / EPC) + j)] = f;
    }
    __syncthreads();
    float4 *g = reinterpret_cast<float4 *>(row);
    const int nlive = (n + EPC - 1) / EPC;
    for (int q = p; q < nlive; q += P) {
      if ((q + 1) * EPC <= n) {
        st_hint4(&g[q], s_row[swz(q)], pol_keep);
      } else {
        const float4 f = s_row[swz(q)];
        const cx<R> *z = reinterpret_cast<const cx<R> *>(&f);
        for (int u = 0; q * EPC + u < n; u++) row[q * EPC + u] = z[u];
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < CH; i++)
      if (base + i < n) row[base + i] = v[i];
  }
}

// Rows longer than one CTA can hold (n up to 65535 in FP32): a cluster of S
// CTAs shares one frequency; each CTA owns blockDim.x consecutive level-0
// chunks.  The level-1 right-hand sides are gathered into the shared memory
// of rank 0 through distributed shared memory, rank 0 solves levels >= 1,
// and every CTA reads its two separators back from rank 0.
template <typename R, int CH>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 1024 : 512)
k_tridiag_cluster(cx<R> *__restrict__ spec, int n, int64_t n_pad,
                  const RecLev<R, CH> *__restrict__ tabs, int conj_sym, int levels, int4 lsz_lo,
                  int2 lsz_hi) {
  cg::cluster_group cluster = cg::this_cluster();
  const int S = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int k = blockIdx.x / S;
  const int p = threadIdx.x, T = blockDim.x;
  const int g = rank * T + p;            // chunk index within the row
  const int P = S * T, M = P - 1;
  const int lsz[kRecLevels] = {lsz_lo.x, lsz_lo.y, lsz_lo.z, lsz_lo.w, lsz_hi.x, lsz_hi.y};
  __shared__ RecLev<R, CH> T0[kRecLevels];
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<R> *B[kRecLevels];
  size_t off = level_buffers<R, CH>(lsz, levels, reinterpret_cast<cx<R> *>(smraw), B);
  cx<R> *s_first = reinterpret_cast<cx<R> *>(smraw) + off;   // [T]
  off += (size_t)T;
  float4 *s_row = reinterpret_cast<float4 *>(smraw + ((off * sizeof(cx<R>) + 15) & ~(size_t)15));
  constexpr int EPC = 16 / sizeof(cx<R>);
  const int nchunks = (T * CH) / EPC;

  load_levels<R, CH>(T0, tabs + (size_t)k * levels, levels, conj_sym, p, T);
  zero_tails<R, CH>(B, lsz, levels, p, T);

  cx<R> *row = spec + (size_t)k * n_pad + (size_t)rank * T * CH;   // this CTA's segment
  const int nseg = n - rank * T * CH;                                 // unknowns left from here
  const unsigned long long pol_keep = l2_evict_last();
  cx<R> v[CH];
  {
    const float4 *gsrc = reinterpret_cast<const float4 *>(row);
    for (int q = p; q < nchunks; q += T) s_row[swz(q)] = ld_hint4(&gsrc[q], pol_keep);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < CH / EPC; j++) {
      const float4 f = s_row[swz(p * (CH / EPC) + j)];
      const cx<R> *z = reinterpret_cast<const cx<R> *>(&f);
#pragma unroll
      for (int u = 0; u < EPC; u++)
        v[j * EPC + u] = (p * CH + j * EPC + u < nseg) ? z[u] : mk((R)0, (R)0);
    }
  }
  const cx<R> e0 = T0[0].e, sep = v[CH - 1];
  chunk_solve<R, CH>(v, T0[0].invp, T0[0].bp, e0, false);   // n + 1 = P CH
  s_first[p] = v[0];
  cluster.sync();
  cx<R> *B1root = cluster.map_shared_rank(B[1], 0);
  if (g < M) {
    cx<R> nxt;
    if (p + 1 < T) nxt = s_first[p + 1];
    else nxt = *cluster.map_shared_rank(s_first, rank + 1);
    B1root[rpos<CH>(g)] = cfnms(sep, e0, v[CH - 2] + nxt);
  }
  cluster.sync();
  if (rank == 0) rec_upper<R, CH>(B, lsz, levels, T0, p);
  cluster.sync();
  const cx<R> sl = (g > 0) ? B1root[rpos<CH>(g - 1)] : mk((R)0, (R)0);
  const cx<R> sr = (g < M) ? B1root[rpos<CH>(g)] : mk((R)0, (R)0);
#pragma unroll
  for (int i = 0; i < CH - 1; i++) v[i] = cfma(cfma(v[i], sl, T0[0].fc[i]), sr, T0[0].fc[CH - 2 - i]);
  v[CH - 1] = sr;
  cluster.sync();   // rank 0's shared memory is no longer read by others

#pragma unroll
  for (int j = 0; j < CH / EPC; j++) {
    float4 f;
    cx<R> *z = reinterpret_cast<cx<R> *>(&f);
#pragma unroll
    for (int u = 0; u < EPC; u++) z[u] = v[j * EPC + u];
    s_row[swz(p * (CH / EPC) + j)] = f;
  }
  __syncthreads();
  float4 *gdst = reinterpret_cast<float4 *>(row);
  const int nlive = (nseg < T * CH) ? (nseg + EPC - 1) / EPC : nchunks;
  for (int q = p; q < nlive; q += T) {
    if ((q + 1) * EPC <= nseg) {
      st_hint4(&gdst[q], s_row[swz(q)], pol_keep);
    } else {
      const float4 f = s_row[swz(q)];
      const cx<R> *z = reinterpret_cast<const cx<R> *>(&f);
      for (int u = 0; q * EPC + u < nseg; u++) row[q * EPC + u] = z[u];
    }
  }
}

// The separator system of the fused four-step apply (fft_four_fused.cuh):
// one CTA per frequency k, a thread per level-1 chunk up to 256 (a warp per
// frequency left one warp on an SM at n = 65535, ell = 512: 8 chunks a lane
// in turn, 30 us).  The forward kernel left, for each chunk p of row k, its
// first local value v_0 and its separator's partial right-hand side
// x_sep - e v_14 in sepbuf[k P + p]; the level-1 right-hand side of separator
// p is that partial value minus e times the first local value of chunk p + 1.
// Levels 1 .. levels-1 of the recursive form are solved as in k_tridiag_rec
// and the separator values go to sep[k sstride + p].
template <int CH>
__global__ void __launch_bounds__(256)
k_tridiag_reduced(const float4 *__restrict__ sepbuf, cx<float> *__restrict__ sep,
                  int64_t sstride, const RecLev<float, CH> *__restrict__ tabs, int conj_sym,
                  int levels, int4 lsz_lo, int2 lsz_hi) {
  const int k = blockIdx.x, p = threadIdx.x, T = blockDim.x;
  const int lsz[kRecLevels] = {lsz_lo.x, lsz_lo.y, lsz_lo.z, lsz_lo.w, lsz_hi.x, lsz_hi.y};
  extern __shared__ __align__(16) unsigned char smraw[];
  RecLev<float, CH> *st = reinterpret_cast<RecLev<float, CH> *>(smraw);
  load_levels<float, CH>(st, tabs + (size_t)k * levels, levels, conj_sym, p, T);
  cx<float> *B[kRecLevels];
  level_buffers<float, CH>(lsz, levels, reinterpret_cast<cx<float> *>(st + levels), B);
  zero_tails<float, CH>(B, lsz, levels, p, T);
  __syncthreads();
  pdl_wait(sepbuf);   // the previous kernel's output
  const float4 *row = sepbuf + (size_t)k * sstride;
  const cx<float> e0 = st[0].e;
  const int M = lsz[1];
  for (int q0 = 0; q0 < M; q0 += 8 * T) {
    float4 a[8];
    float2 b[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int q = q0 + p + T * u;
      if (q < M) {
        a[u] = row[q];                                         // (v0_q, partial_q)
        b[u] = *reinterpret_cast<const float2 *>(row + q + 1);  // v0_{q+1}
      }
    }
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int q = q0 + p + T * u;
      if (q < M) B[1][rpos<CH>(q)] = cfnms(mk(a[u].z, a[u].w), e0, mk(b[u].x, b[u].y));
    }
  }
  pdl_trigger();
  __syncthreads();
  rec_upper<float, CH>(B, lsz, levels, st, p);
  cx<float> *out = sep + (size_t)k * sstride;
  for (int q = p; q < M; q += T) out[q] = B[1][rpos<CH>(q)];
}

// The same separator system when the recursive form has at most three
// levels, so at most 17 level-1 chunks (n up to 4368), in registers: lane L
// of the warp of frequency k owns level-1 chunk L (separators 16L .. 16L+15),
// forms their right-hand sides from sepbuf, solves the chunk (level-1
// pivots), hands the level-2 right-hand side of its separator to lane 0
// through shared memory, lane 0 solves level 2 (at most 16 unknowns) in one
// sweep, and every lane corrects its chunk with the two level-2 values
// around it.  No level buffer round trips: the chain of dependent steps is
// two Thomas sweeps.
// It does not let its successor be scheduled early: the correction kernel's CTAs
// then wait beside it, and what a wait costs at the end is more than the prologue
// they save (FP32 apply, with / without: n 255 x ell 4096 31.2 / 24.2 us, 127 x
// 4096 29.7 / 20.6, 511 x 4096 39.4 / 34.2, 1023 x 1024 22.1 / 19.6; before this
// kernel served two levels 28.7, 24.6, 40.2, 21.6).
template <int CH>
__global__ void __launch_bounds__(256)
k_tridiag_reduced3(const float4 *__restrict__ sepbuf, cx<float> *__restrict__ sep,
                   int64_t sstride, const RecLev<float, CH> *__restrict__ tabs, int conj_sym,
                   int M1, int M2, int levels, int nk) {
  constexpr int WPB = 8;
  using Lev = RecLev<float, CH>;
  static_assert(sizeof(Lev) % 16 == 0, "whole float4 copies");
  constexpr int NV = (int)(2 * sizeof(Lev) / 16);   // float4 of levels 1 and 2
  constexpr int UV = (NV + 31) / 32;
  __shared__ __align__(16) Lev s_tab[WPB][2];        // per warp, conjugated if transposed
  __shared__ cx<float> s2[WPB][CH + 1];              // level-2 right-hand sides / solution
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k = blockIdx.x * WPB + w;
  if (k >= nk) return;   // whole warps only; nothing below synchronises the CTA
  const int q0 = CH * lane;               // first level-1 unknown of this lane's chunk
  const bool own = lane <= M2;            // M2 + 1 level-1 chunks
  // every global load of the warp first: its frequency's tables and the
  // chunk's sepbuf entries (P = M1 + 1 per frequency)
  float4 tv[UV];
  const Lev *tab = tabs + (size_t)k * levels;
  const float4 *src = reinterpret_cast<const float4 *>(tab + 1);
  const int nv = (levels - 1) * (NV / 2);            // level 2 exists with three levels
#pragma unroll
  for (int u = 0; u < UV; u++)
    if (lane + 32 * u < nv) tv[u] = __ldg(src + lane + 32 * u);
  cx<float> e0 = tab->e;
  pdl_wait(sepbuf);   // the previous kernel's output
  const float4 *row = sepbuf + (size_t)k * sstride;
  float4 a[CH];
  float2 nxt = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < CH; j++) {
    a[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (own && q0 + j <= M1) a[j] = row[q0 + j];
  }
  if (own && q0 + CH <= M1) nxt = *reinterpret_cast<const float2 *>(row + q0 + CH);
  {
    const float sg = conj_sym ? -1.f : 1.f;   // every entry is complex: (re, im) pairs
    float4 *dst = reinterpret_cast<float4 *>(&s_tab[w][0]);
#pragma unroll
    for (int u = 0; u < UV; u++)
      if (lane + 32 * u < nv) dst[lane + 32 * u] = make_float4(tv[u].x, sg * tv[u].y, tv[u].z, sg * tv[u].w);
    e0.im *= sg;
  }
  __syncwarp();
  const Lev &T1 = s_tab[w][0], &T2 = s_tab[w][1];
  const cx<float> e1 = T1.e;
  cx<float> wv[CH];
  // level-1 right-hand sides: partial_q - e0 first_{q+1}
#pragma unroll
  for (int j = 0; j < CH; j++) {
    const cx<float> first_next = (j + 1 < CH) ? mk(a[j + 1].x, a[j + 1].y) : mk(nxt.x, nxt.y);
    wv[j] = (q0 + j < M1) ? cfnms(mk(a[j].z, a[j].w), e0, first_next) : mk(0.f, 0.f);
  }
  // level 1: the chunk's unknowns, its separator value aside
  const cx<float> sep1 = wv[CH - 1];
  chunk_solve<float, CH>(wv, lane == M2 ? T1.invt : T1.invp, T1.bp, e1, lane == M2);
  // level-2 right-hand side of separator L: sep - e1 (last of chunk L + first of chunk L+1)
  const cx<float> firstr = mk(__shfl_down_sync(0xffffffffu, wv[0].re, 1),
                              __shfl_down_sync(0xffffffffu, wv[0].im, 1));
  if (lane < M2) s2[w][lane] = cfnms(sep1, e1, wv[CH - 2] + firstr);
  __syncwarp();
  if (lane == 0 && M2 > 0) {
    cx<float> z[CH];
#pragma unroll
    for (int i = 0; i < CH; i++) z[i] = (i < M2) ? s2[w][i] : mk(0.f, 0.f);
    chunk_solve<float, CH>(z, T2.invt, T2.bp, T2.e, true);
#pragma unroll
    for (int i = 0; i < CH; i++)
      if (i < M2) s2[w][i] = z[i];
  }
  __syncwarp();
  if (!own) return;
  const cx<float> sl = lane > 0 ? s2[w][lane - 1] : mk(0.f, 0.f);
  const cx<float> sr = lane < M2 ? s2[w][lane] : mk(0.f, 0.f);
  const cx<float> *fl = lane < M2 ? T1.fc : T1.fl;
  cx<float> *out = sep + (size_t)k * sstride + q0;
#pragma unroll
  for (int i = 0; i < CH - 1; i++) {
    const cx<float> val = cfma(cfma(wv[i], sl, fl[i]), sr, T1.fc[CH - 2 - i]);
    if (q0 + i < M1) out[i] = val;
  }
  if (q0 + CH - 1 < M1) out[CH - 1] = lane < M2 ? sr : cfma(wv[CH - 1], sl, fl[CH - 1]);
}

cudaError_t launch_tridiag_reduced(const Ctx &c, const void *sepbuf, void *sep, int transpose,
                                   cudaStream_t s) {
  if (c.lev32 < 2 || c.ch32 != 16) return cudaErrorNotSupported;
  constexpr int CH = 16;
  const int levels = c.lev32;
  const int *lsz = c.lsz32;
  if (levels <= 3) {
    constexpr int WPB = 8;   // warps (frequencies) per CTA, as in the kernel
    const cudaError_t e = launch_pdl(k_tridiag_reduced3<CH>, dim3((unsigned)((c.nk + WPB - 1) / WPB)),
                                     dim3(32 * WPB), 0, s, static_cast<const float4 *>(sepbuf),
                                     static_cast<cx<float> *>(sep), (int64_t)c.P32,
                                     static_cast<const RecLev<float, CH> *>(c.rec32), transpose,
                                     lsz[1], levels > 2 ? lsz[2] : 0, levels, (int)c.nk);
    note_launch();
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  const size_t off = level_buffers<float, CH>(lsz, levels, nullptr, nullptr);
  const size_t smem = levels * sizeof(RecLev<float, CH>) + off * sizeof(cx<float>);
  if (smem > 200 * 1024) return cudaErrorNotSupported;
  const int chunks = lsz[2] + 1;                        // of level 1 (levels >= 4 here)
  const int T = chunks >= 256 ? 256 : (chunks + 31) / 32 * 32;
  cudaError_t e = kernel_setup((const void *)k_tridiag_reduced<CH>, T, smem);
  if (e != cudaSuccess) { cudaGetLastError(); return e; }
  const int4 lo = make_int4(lsz[0], lsz[1], lsz[2], lsz[3]);
  const int2 hi = make_int2(lsz[4], lsz[5]);
  e = launch_pdl(k_tridiag_reduced<CH>, dim3((unsigned)c.nk), dim3(T), smem, s,
                 static_cast<const float4 *>(sepbuf), static_cast<cx<float> *>(sep),
                 (int64_t)c.P32, static_cast<const RecLev<float, CH> *>(c.rec32), transpose,
                 levels, lo, hi);
  note_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename R, int CH>
static cudaError_t run_tridiag_cluster(const Ctx &c, void *spec, const void *tab, int T, int S,
                                       int conj, int levels, const int *lsz, cudaStream_t s) {
  const size_t off = level_buffers<R, CH>(lsz, levels, nullptr, nullptr) + (size_t)T;
  const size_t smem = ((off * sizeof(cx<R>) + 15) & ~(size_t)15) + (size_t)T * CH * sizeof(cx<R>);
  auto kern = k_tridiag_cluster<R, CH>;
  cudaError_t e = kernel_setup((const void *)kern, T, smem);
  if (e != cudaSuccess) { cudaGetLastError(); return e; }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(c.nk * S), 1, 1);
  cfg.blockDim = dim3((unsigned)T, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int4 lo = make_int4(lsz[0], lsz[1], lsz[2], lsz[3]);
  const int2 hi = make_int2(lsz[4], lsz[5]);
  e = cudaLaunchKernelEx(&cfg, kern, static_cast<cx<R> *>(spec), (int)c.n, c.n_pad,
                         static_cast<const RecLev<R, CH> *>(tab), conj, levels, lo, hi);
  note_launch();
  if (e != cudaSuccess) { cudaGetLastError(); return e; }
  return cudaGetLastError();
}

template <typename R, int CH>
static cudaError_t run_tridiag_rec(const Ctx &c, void *spec, const void *tab, int P, int conj,
                                   int levels, const int *lsz, cudaStream_t s) {
  const size_t off = level_buffers<R, CH>(lsz, levels, nullptr, nullptr) + (size_t)P;
  const size_t upper = (off * sizeof(cx<R>) + 15) & ~(size_t)15;
  const size_t staged = upper + (size_t)P * CH * sizeof(cx<R>);
  const bool stage = staged <= 200 * 1024;
  const size_t smem = stage ? staged : upper;
  auto kern = k_tridiag_rec<R, CH, false, true>;
  if constexpr (sizeof(R) == 8 && CH == 16) {   // n > 8191: 512 chunks and more
    if (!stage) kern = k_tridiag_rec<R, CH, false, false>;
  } else {                                      // at most 169 KB a row
    if (P <= 256) kern = k_tridiag_rec<R, CH, true, true>;
  }
  cudaError_t e = kernel_setup((const void *)kern, P, smem);
  if (e != cudaSuccess) { cudaGetLastError(); return e; }
  const int4 lo = make_int4(lsz[0], lsz[1], lsz[2], lsz[3]);
  const int2 hi = make_int2(lsz[4], lsz[5]);
  kern<<<(unsigned)c.nk, P, smem, s>>>(static_cast<cx<R> *>(spec), (int)c.n, c.n_pad,
                                       static_cast<const RecLev<R, CH> *>(tab), conj, levels,
                                       lo, hi);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_tridiag(const Ctx &c, void *spec, int prec, int transpose, cudaStream_t s) {
  if (c.space == AAO_SPACE_DST) return launch_dst_solve(c, spec, prec, transpose, s);
  if (prec == AAO_PREC_FP32 && c.clu32 > 1)
    return run_tridiag_cluster<float, 16>(c, spec, c.rec32, c.cta32, c.clu32, transpose, c.lev32,
                                          c.lsz32, s);
  if (prec == AAO_PREC_FP64 && c.clu64 > 1)
    return run_tridiag_cluster<double, 16>(c, spec, c.rec64, c.cta64, c.clu64, transpose,
                                           c.lev64, c.lsz64, s);
  if (prec == AAO_PREC_FP32)
    return run_tridiag_rec<float, 16>(c, spec, c.rec32, c.P32, transpose, c.lev32, c.lsz32, s);
  if (c.ch64 == 8)
    return run_tridiag_rec<double, 8>(c, spec, c.rec64, c.P64, transpose, c.lev64, c.lsz64, s);
  return run_tridiag_rec<double, 16>(c, spec, c.rec64, c.P64, transpose, c.lev64, c.lsz64, s);
}

}  // namespace aao
