// Complex length-M DFT in 64-bit fixed point (integer pipes) for the FP64
// coefficient recovery (Section "Previous results on SFTs": one length-M 1D
// FFT of the lattice samples).  Values are longlong2 (re, im) in units of
// 2^-kFxFrac or 2^-kFxInvFrac (fxc.cuh).
#pragma once

#include "ss_internal.cuh"

namespace ss {

constexpr int kFxFrac = 58, kFxInvFrac = 60;   // units 2^-58 (forward), 2^-60 (inverse)
constexpr int kDfFftMaxL = 4096;     // longest factor transformed in one block
constexpr int kDfFftMaxPasses = 16;

struct DfRadices {
  int n = 0;
  int r[kDfFftMaxPasses] = {};
};

// M = L1 L2 with L1, L2 <= kDfFftMaxL and every prime factor in {2, 3, 5, 7}.
// sh1, sh2: right shifts after the passes of the forward transform (their sum
// is `shift`); the last pass keeps its sums.
struct FxFftPlan {
  int64_t M = 0;
  int L1 = 1, L2 = 1;
  DfRadices rad1, rad2;
  int sh1[kDfFftMaxPasses] = {}, sh2[kDfFftMaxPasses] = {}, shift = 0;
};

// Radices of a self-sorting transform of length L (odd radices first, then
// 8, 4, 2); n = -1 when L has a prime factor above 7.
DfRadices df_radices(int L);

// False when M has a prime factor above 7 or no factor pair fits.
bool fx_fft_plan(int64_t M, FxFftPlan* out);

// tab[r] = exp(2 pi i r / M), r < M, as Q62 balanced limbs (fxc.cuh's TW), then
// the L1-th and L2-th roots: M + L1 + L2 entries.
ss_status fx_fft_table(const FxFftPlan& F, int4* tab, cudaStream_t st);

// What the bins of a class (b mod L1, then b mod L2: L1 + L2 of them) hold: the
// largest exponent field of |re| + |im| and the number of bins (0, 0: none).
// Their moduli add up to less than 2^(x - 1022 + fx_log2(y)).
__device__ __forceinline__ int fx_log2(int n) { return 32 - __clz(n - 1); }   // ceil, n >= 1
// Left shift of a column of the inverse transform: its moduli stay below 2^62 units.
__device__ __forceinline__ int fx_column_lift(const int2 k) {
  return k.x ? min(59, max(0, 1024 - k.x - fx_log2(k.y))) : 0;
}
// Left shift of a row of the forward transform: what it holds, and the rounding
// of the samples and of launch A (below 2^16 units: a sample adds up L2 <= 4096
// values of three units at most and the later passes'), stay below 1.25 2^59
// units (2^59.5 is the passes' bound).
__device__ __forceinline__ int fx_row_lift(const int2 k) {
  const int top = k.x ? k.x - (1022 - kFxFrac) + fx_log2(k.y) : 0;   // bits of the class
  return max(0, 59 - max(top, 18));
}

// Inverse and forward transform, two launches each on st; tmp holds M values,
// classes describes the bins (a device array, L1 + L2 entries).
//   fx_inverse: out[j] = sum_b in[b] exp(2 pi i j b / M) in units of 2^-kFxInvFrac;
//     the moduli of in add up to less than 4 (two real sums of l1 norm below 2).
//     out may be in's memory.
//   fx_forward: out[b] = 2^(fx_row_lift(classes[b mod L1]) - F.shift)
//     sum_j in[j] exp(-2 pi i j b / M) in units of 2^-kFxFrac, in: the inverse
//     transform's result.
ss_status fx_inverse(const FxFftPlan& F, const int4* tab, const double2* in, const int2* classes, longlong2* tmp,
                     longlong2* out, cudaStream_t st);
ss_status fx_forward(const FxFftPlan& F, const int4* tab, const longlong2* in, const int2* classes, longlong2* tmp,
                     longlong2* out, cudaStream_t st);

}  // namespace ss
