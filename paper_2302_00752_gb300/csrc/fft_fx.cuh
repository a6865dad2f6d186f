// Complex length-M DFT in 64-bit fixed point (integer pipes) for the FP64
// coefficient recovery (Section "Previous results on SFTs": one length-M 1D
// FFT of the lattice samples).  Values are longlong2 (re, im) in units of
// 2^-kFxFrac (fxc.cuh).
#pragma once

#include "ss_internal.cuh"

namespace ss {

constexpr int kFxFrac = 58;          // unit 2^-58
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

// out[k] = 2^-s sum_j in[j] exp(sign 2 pi i j k / M), s = 0 for sign = +1 and
// F.shift for sign = -1.  Bounds: for sign = +1 the moduli of the inputs sum to
// less than 4 (2^60 units), for sign = -1 every input is below 2^59.5 units in
// modulus (2 sqrt 2: two real sums of l1 norm below 2).
// tmp holds M values; out may alias in.  Two launches on st.
ss_status fx_fft(const FxFftPlan& F, const int4* tab, const longlong2* in, longlong2* tmp, longlong2* out, int sign,
                 cudaStream_t st);

}  // namespace ss
