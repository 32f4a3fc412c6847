// Instantiation and dispatch of the time-axis FFT kernels for one real type.
#pragma once
#include <type_traits>
#include "fft_time.cuh"
#include "fft_mixed.cuh"
#include "fft_four.cuh"
#include "fft_four_fused.cuh"
#include "fft_steps.cuh"

namespace aao {
namespace fft {

// Persistent grid: as many CTAs as fit on the device at once, capped by the
// panel count (the dynamic shared-memory opt-in happens in the same cached
// setup).  Returns 0 when the kernel cannot be set up.
template <class K>
static int persistent_grid(K kern, int threads, size_t smem, int npanels) {
  int g = 0;
  if (kernel_setup((const void *)kern, threads, smem, &g) != cudaSuccess) return 0;
  return g < npanels ? g : npanels;
}

#ifndef AAO_FFT_FOUR
#define AAO_FFT_FOUR 1
#endif
// With scratch for the intermediate: FP32, ell = 256 ... 4096 a power of two
// takes the four-step kernels compiled for it, every other length from
// AAO_STEPS_MIN on (and FP64) what step_plan says: mostly the run-time
// four-step kernels.  Shorter transforms, and calls without scratch, one
// kernel per direction.
template <typename R>
inline bool use_four(int64_t ell) {
  return AAO_FFT_FOUR && std::is_same<R, float>::value && ell >= 256 && ell <= 4096 &&
         (ell & (ell - 1)) == 0;
}

// The row and panel kernels serve the powers of two that step_plan may leave
// to them (large n).
template <typename R, int L>
constexpr bool kSplitUsed = Split<R, L>::OK && (sizeof(R) == 4 ? L <= 128 : L <= 256 || L == 4096);

// Bytes of their panel-major intermediate.
template <typename R, int L>
static size_t split_bytes(int64_t n) {
  if constexpr (kSplitUsed<R, L>) {
    const int W = 2 * Shape<R, L>::C;
    return (size_t)((n + W - 1) / W) * Split<R, L>::PANEL;
  }
  return 0;
}

template <typename R, int L, typename YT>
static cudaError_t run_forward(const StepPlan &pl, int64_t n, int64_t n_pad, const double *x, const YT *y,
                               const R *sigk, cx<R> *spec, const cx<R> *tw, cudaStream_t s, void *inter) {
  using S = Shape<R, L>;
  const int W = 2 * S::C;
  const int np = (int)((n + W - 1) / W);
  if constexpr (kSplitUsed<R, L>) {
    if (inter && pl.split) {
      const int ncx = np * S::C;
      const dim3 g1((unsigned)((ncx + kRowThreads - 1) / kRowThreads), (unsigned)Split<R, L>::LR);
      cx<R> *ip = static_cast<cx<R> *>(inter);
      if (y) k_fft_forward_rows<R, L, true, YT><<<g1, kRowThreads, 0, s>>>(x, y, sigk, ip, (int)n, ncx);
      else k_fft_forward_rows<R, L, false, double><<<g1, kRowThreads, 0, s>>>(x, nullptr, sigk, ip, (int)n, ncx);
      note_launch();
      auto kern = k_fft_forward_panels<R, L>;
      const int g = persistent_grid(kern, S::T, S::SMEM, np);
      if (g <= 0) return cudaErrorInvalidConfiguration;
      kern<<<g, S::T, S::SMEM, s>>>(ip, spec, (int)n, n_pad, tw, np);
      note_launch();
      return cudaGetLastError();
    }
  }
  if (y) {
    auto kern = k_fft_forward<R, L, true, YT>;
    const int g = persistent_grid(kern, S::T, S::SMEM, np);
    if (g <= 0) return cudaErrorInvalidConfiguration;
    kern<<<g, S::T, S::SMEM, s>>>(x, y, sigk, spec, (int)n, n_pad, tw, np);
  } else {
    auto kern = k_fft_forward<R, L, false, double>;   // no iterate: one instantiation
    const int g = persistent_grid(kern, S::T, S::SMEM, np);
    if (g <= 0) return cudaErrorInvalidConfiguration;
    kern<<<g, S::T, S::SMEM, s>>>(x, nullptr, nullptr, spec, (int)n, n_pad, tw, np);
  }
  note_launch();
  return cudaGetLastError();
}

template <typename R, int L, typename OT>
static cudaError_t run_inverse(const StepPlan &pl, int64_t n, int64_t n_pad, const cx<R> *spec, OT *y,
                               const cx<R> *tw, cudaStream_t s, void *inter, const float *base) {
  using S = Shape<R, L>;
  const int W = 2 * S::C;
  const int np = (int)((n + W - 1) / W);
  if constexpr (kSplitUsed<R, L>) {
    if (inter && pl.split) {
      cx<R> *ip = static_cast<cx<R> *>(inter);
      auto kern = k_fft_inverse_panels<R, L>;
      const int g = persistent_grid(kern, S::T, S::SMEM, np);
      if (g <= 0) return cudaErrorInvalidConfiguration;
      kern<<<g, S::T, S::SMEM, s>>>(spec, ip, (int)n, n_pad, tw, np);
      note_launch();
      const int ncx = np * S::C;
      const dim3 g2((unsigned)((ncx + kRowThreads - 1) / kRowThreads), (unsigned)(L / 16));
      k_fft_inverse_rows<R, L, OT><<<g2, kRowThreads, 0, s>>>(ip, y, (int)n, ncx, tw, base);
      note_launch();
      return cudaGetLastError();
    }
  }
  auto kern = k_fft_inverse<R, L, OT>;
  const int g = persistent_grid(kern, S::T, S::SMEM, np);
  if (g <= 0) return cudaErrorInvalidConfiguration;
  kern<<<g, S::T, S::SMEM, s>>>(spec, y, (int)n, n_pad, tw, np, base);
  note_launch();
  return cudaGetLastError();
}

// The four-step lengths, X(L) each.
#define AAO_FOUR_CASES(X) X(256) X(512) X(1024) X(2048) X(4096)
#define AAO_FFT_CASES(X) \
  X(1) X(2) X(4) X(8) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096)

template <typename R, typename YT>
cudaError_t forward_any(int64_t ell, const StepPlan &pl, int64_t n, int64_t n_pad, const double *x, const YT *y,
                        const R *sigk, cx<R> *spec, const cx<R> *tw, cudaStream_t s,
                        void *inter) {
  if (inter && use_four<R>(ell)) {
    if constexpr (std::is_same<R, float>::value) {
      switch (ell) {
#define AAO_F(L) case L: return four_forward<L>(n, n_pad, x, y, sigk, spec, tw, pl.tw32, s, inter);
        AAO_FOUR_CASES(AAO_F)
#undef AAO_F
      }
    }
  }
  if (inter && pl.L) return steps_forward<R>(pl, n, n_pad, x, y, sigk, spec, step_table<R, -1>(pl, tw), s, inter);
  switch (ell) {
#define AAO_F(L) case L: return run_forward<R, L, YT>(pl, n, n_pad, x, y, sigk, spec, tw, s, inter);
    AAO_FFT_CASES(AAO_F)
#undef AAO_F
    default: return run_forward_mixed<R, YT>(ell, n, n_pad, x, y, sigk, spec, tw, s);
  }
}

// The forward transform of an FP32 block vector (FP32 spectrum) by the
// four-step kernels; cudaErrorNotSupported where neither form serves ell.
inline cudaError_t forward_four_f32_input(int64_t ell, const StepPlan &pl, int64_t n, int64_t n_pad, const float *x,
                                          cx<float> *spec, const cx<float> *tw, cudaStream_t s,
                                          void *inter) {
  if (!inter) return cudaErrorNotSupported;
  const float *none = nullptr;
  if (use_four<float>(ell)) {
    switch (ell) {
#define AAO_F(L) case L: return four_forward<L>(n, n_pad, x, none, none, spec, tw, pl.tw32, s, inter);
      AAO_FOUR_CASES(AAO_F)
#undef AAO_F
    }
  }
  if (!pl.L) return cudaErrorNotSupported;
  return steps_forward<float>(pl, n, n_pad, x, none, none, spec, step_table<float, -1>(pl, tw), s, inter);
}

// Bytes of the four-step intermediate (0 where a single kernel serves).
template <typename R>
size_t inter_bytes_any(int64_t ell, const StepPlan &pl, int64_t n) {
  if (use_four<R>(ell)) return four_inter_bytes(ell, n);
  if (!pl.split) return pl.L ? steps_inter_bytes<R>(ell, n) : 0;
  switch (ell) {
#define AAO_B(L) case L: return split_bytes<R, L>(n);
    AAO_FFT_CASES(AAO_B)
#undef AAO_B
    default: return 0;
  }
}

template <typename R, typename OT>
cudaError_t inverse_any(int64_t ell, const StepPlan &pl, int64_t n, int64_t n_pad, const cx<R> *spec, OT *y,
                        const cx<R> *tw, cudaStream_t s, void *inter,
                        const float *base = nullptr) {
  if (inter && use_four<R>(ell)) {
    if constexpr (std::is_same<R, float>::value) {
      switch (ell) {
#define AAO_I(L) case L: return four_inverse<L, OT>(n, n_pad, spec, y, tw, s, inter, base);
        AAO_FOUR_CASES(AAO_I)
#undef AAO_I
      }
    }
  }
  if (inter && pl.L) return steps_inverse<R, OT>(pl, n, n_pad, spec, y, step_table<R, +1>(pl, tw), s, inter, base);
  switch (ell) {
#define AAO_I(L) case L: return run_inverse<R, L, OT>(pl, n, n_pad, spec, y, tw, s, inter, base);
    AAO_FFT_CASES(AAO_I)
#undef AAO_I
    default: return run_inverse_mixed<R, OT>(ell, n, n_pad, spec, y, tw, s, base);
  }
}

}  // namespace fft
}  // namespace aao
