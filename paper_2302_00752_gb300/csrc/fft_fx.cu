// Fixed-point complex FFT of a 7-smooth length M on the integer pipes.
//
// Four-step split M = L1 L2 (j = j1 L2 + j2, k = k1 + L1 k2):
//   X[k1 + L1 k2] = sum_{j2} w_{L2}^{j2 k2} w_M^{j2 k1} sum_{j1} w_{L1}^{j1 k1} x[j1 L2 + j2],
// w_n = exp(sign 2 pi i / n).  Launch A transforms the columns j2 (length L1,
// stride L2), twists by w_M^{j2 k1} and writes T[k1 L2 + j2]; launch B the rows
// k1 (length L2, contiguous in T) to X[k1 + L1 k2].  A block takes C = 2
// neighbouring columns (rows) where their number is even, so that the strided
// side moves whole 32-byte sectors, else one.  Inside a block the length-L
// transform is a self-sorting (Stockham) sequence of radix-R passes in shared
// memory (two buffers): with Ns the product of the radices already applied,
// butterfly j < L/R takes in[j + r L/R], turns input r by w_{Ns R}^{(j mod Ns) r},
// applies the R-point DFT and writes output r to out[(j / Ns) Ns R + j mod Ns + r Ns]
// (the Stockham autosort formulation, e.g. Govindaraju et al., SC 2008).
//
// Range.  An inverse transform (sign +1, units of 2^-60) sums inputs whose
// moduli add up to less than 2^62: no partial sum exceeds that (limb products:
// see mul).  Launch A's
// columns are classes of bins (mod L2), mostly with a small part of the sum or
// none: a column counts in units finer by its own power of two (fx_column_lift)
// and is brought to the common unit as it leaves, where its rounding averages
// over the L1 values of the column instead of standing in one bin.  The
// forward transform (units of 2^-58, the samples rounded to them) divides by a power of two at or above the radix after every pass
// (the plan keeps the running growth at most 1), so values enter a pass below
// 2^59.5, a product's operands stay below 2^61 and a radix-8 or radix-10 sum
// below 2^63.  The last pass keeps its sums undivided: its rounding is then the
// average of its inputs' (0.2 units where a final division would leave 0.7).
// Launch B's rows hold the classes of bins mod L1, each lifted by its own power
// of two (fx_row_lift).  So a bin carries a unit averaged over L1 or L2 values,
// and a unit of what its own row and column hold (all in the common unit: 6 to
// 20 times as much at M = 10^5 to 4 10^6, and more than in double-float, whose
// rounding follows the values).
//
// On this part an FP64 instruction issues at 1/64 of the FP32 rate, which puts
// the FP64 library transform of length 10^6 at 205 us; a double-float
// addition takes eight to eleven FP32 instructions against two integer ones
// here, and rounds at 2^-47 where this transform rounds at about 2^-56 of the
// data's l1 norm.  Bound: latency, of global loads first (12 warps an SM, issue
// slots 21 to 35 % busy).  M = 10^6, one complex transform: 65 us, 70 with 840
// terms (double-float: 82 us).
#include <cmath>

#include "fft_fx.cuh"
#include "fxc.cuh"

namespace ss {
namespace {

using namespace fxc;

struct FxPasses {
  int n;
  int r[kDfFftMaxPasses], sh[kDfFftMaxPasses];
};

// The strided side of a launch in global memory: element i of column (row) c.
template <bool ROWS>
__device__ __forceinline__ int at(int col, int i, int stride) {   // M <= 2^24: 32-bit indices
  return ROWS ? col * stride + i : i * stride + col;
}

// What a block works on.
struct FxBlock {
  const longlong2* in;
  longlong2* out;
  const int4* tab;     // exp(2 pi i r / M)
  longlong2* a;        // [L C] (element i of column c at i C + c)
  longlong2* b;        // second buffer, or a itself (in place)
  const int4* tw;      // exp(2 pi i m / L), m < L, in shared memory
  int M, col0;         // col0: first column
  int L, L1, L2;
  int lift[2];         // left shifts of the block's columns (inverse A) or rows (forward B)
};

// The double x in units of 2^-(kFxInvFrac + lift).
__device__ __forceinline__ i64 to_fixed(i64 bits, int lift) {
  return bits ? __double2ll_rn(__longlong_as_double(bits) * __hiloint2double((1023 + kFxInvFrac + lift) << 20, 0)) : 0;
}

// One pass: from global memory when `first`, to it (with the twist in launch
// A) when `last`.  In place (INPL) every thread has at most one butterfly and
// the block meets between reads and writes.  j / Ns is umulhi(j, ceil(2^32 /
// Ns)), exact for j, Ns < 2^16.
template <int R, int SIGN, bool SECOND, int C, bool INPL>
__device__ __forceinline__ void pass(const FxBlock& B, int Ns, int sh, bool first, bool last) {
  constexpr int NC = R == 8 ? 1 : (R == 10 ? 2 : (R - 1) / 2);
  constexpr int RR = R == 10 ? 5 : R;
  const int L = B.L, nb = L / R;
  TW cs[NC > 0 ? NC : 1];
#pragma unroll
  for (int m = 0; m < NC; ++m) cs[m] = ld_tw(__ldg(B.tab + (B.M / RR) * (m + 1)));
  const int tstride = L / (Ns * R);
  const unsigned nsm = Ns > 1 ? 0xffffffffu / (unsigned)Ns + 1u : 0u;
  for (int u = threadIdx.x; INPL ? u == (int)threadIdx.x : u < nb * C; u += blockDim.x) {
    const int c = u % C, j = u / C;
    const bool on = u < nb * C;
    const int jq = Ns > 1 ? (int)__umulhi((unsigned)j, nsm) : j;
    const int k = j - jq * Ns;
    CX v[R];
    if (on) {
      if (first) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          v[r] = ld(__ldcg(B.in + at<SECOND>(B.col0 + c, j + r * nb, B.L2)));
        const int up = c ? B.lift[1] : B.lift[0];
        if (SIGN > 0 && !SECOND) {
#pragma unroll
          for (int r = 0; r < R; ++r) v[r] = CX{to_fixed(v[r].re, up), to_fixed(v[r].im, up)};
        } else if (SIGN < 0 && SECOND) {
#pragma unroll
          for (int r = 0; r < R; ++r) v[r] = CX{v[r].re << up, v[r].im << up};
        } else if (SIGN < 0) {   // samples
#pragma unroll
          for (int r = 0; r < R; ++r) v[r] = scale_down(v[r], kFxInvFrac - kFxFrac);
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = ld(B.a[(j + r * nb) * C + c]);
      }
    }
    if (INPL && !first) __syncthreads();
    if (on) {
      if (Ns > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = mul_t<SIGN>(v[r], ld_tw(B.tw[tstride * (k * r)]));
      }
      dft<R, SIGN>(v, cs);
      const int base = jq * Ns * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = base + r * Ns;
        const bool twist = last && !SECOND;
        // a twist that divides by four rounds once, at a finer unit
        CX y = SIGN > 0 ? v[r] : scale_down(v[r], twist && sh >= 2 ? sh - 2 : sh);
        if (!last) {
          B.b[i * C + c] = st(y);
        } else if (SECOND) {
          B.out[B.col0 + c + B.L1 * i] = st(y);
        } else {   // twist by w_M^{j2 k1} (j2 k1 < M)
          const TW w = ld_tw(__ldg(B.tab + (B.col0 + c) * i));
          if (SIGN > 0) y = scale_down(mul(y, w), c ? B.lift[1] : B.lift[0]);
          else y = sh >= 2 ? mulq(y, conj(w)) : mul(y, conj(w));
          B.out[at<false>(B.col0 + c, i, B.L2)] = st(y);
        }
      }
    }
  }
}

template <int SIGN, bool SECOND, int C, bool INPL, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_fft_fx(const longlong2* __restrict__ in, longlong2* __restrict__ out,
                                                const int4* __restrict__ tab, const int4* __restrict__ roots,
                                                const int2* __restrict__ classes, int64_t M, int L1, int L2,
                                                FxPasses rad) {
  extern __shared__ __align__(16) longlong2 sbuf[];
  FxBlock B;
  B.L = SECOND ? L2 : L1;
  B.in = in;
  B.out = out;
  B.tab = tab;
  B.a = sbuf;
  B.b = INPL ? sbuf : sbuf + (size_t)C * B.L;
  int4* tw = reinterpret_cast<int4*>(B.b + (size_t)C * B.L);
  B.tw = tw;
  B.M = (int)M;
  B.col0 = (int)blockIdx.x * C;
  B.L1 = L1;
  B.L2 = L2;
  if constexpr (SIGN > 0 ? !SECOND : SECOND) {
    bool any = false;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int2 k = __ldg(classes + B.col0 + c);
      any |= k.x != 0;
      B.lift[c] = SECOND ? fx_row_lift(k) : fx_column_lift(k);
    }
    if (SIGN > 0 && !any) {   // columns without a bin
      for (int u = threadIdx.x; u < B.L * C; u += blockDim.x)
        out[at<false>(B.col0 + u % C, u / C, L2)] = make_longlong2(0, 0);
      return;
    }
  }
  for (int i = threadIdx.x; i < B.L; i += blockDim.x) tw[i] = __ldg(roots + i);   // read from the second pass on
  int Ns = 1;
  for (int p = 0; p < rad.n; ++p) {
    const int R = rad.r[p], sh = rad.sh[p];
    const bool first = p == 0, last = p + 1 == rad.n;
    switch (R) {
      case 10: pass<10, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      case 8: pass<8, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      case 4: pass<4, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      case 2: pass<2, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      case 5: pass<5, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      case 3: pass<3, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      case 7: pass<7, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;
      default: pass<1, SIGN, SECOND, C, INPL>(B, Ns, sh, first, last); break;   // L = 1
    }
    __syncthreads();
    if (!INPL) {
      longlong2* t = B.a;
      B.a = B.b;
      B.b = t;
    }
    Ns *= R;
  }
}

// exp(2 pi i r / M) for r < M, then the L1-th and the L2-th roots: r = r1 L2 +
// r0 turns by exp(2 pi i r1 / L1) and exp(2 pi i r0 / M), each to a unit.
__global__ void k_fx_roots(int64_t M, int L1, int L2, int4* part) {   // L1, then L2 entries
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < L1) part[i] = st_tw(exact_root(i, L1));
  else if (i < L1 + L2) part[i] = st_tw(exact_root(i - L1, M));
}
__global__ void k_fx_table(int64_t M, int L1, int L2, const int4* __restrict__ part, int4* tab) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M + L1 + L2) return;
  const int64_t r = i < M ? i : (i < M + L1 ? (i - M) * L2 : (i - M - L1) * L1);
  const TW u = ld_tw(__ldg(part + r / L2));
  const CX w = mul(CX{((i64)u.rh << 32) + u.rl, ((i64)u.ih << 32) + u.il}, ld_tw(__ldg(part + L1 + r % L2)));
  tab[i] = st_tw(to_tw(w.re, w.im));
}

template <int SIGN, bool SECOND, int C>
ss_status launch_c(const FxFftPlan& F, const int4* tab, const longlong2* in, longlong2* out, const int2* classes,
                   cudaStream_t st) {
  const int L = SECOND ? F.L2 : F.L1;
  const DfRadices& rad = SECOND ? F.rad2 : F.rad1;
  FxPasses ps;
  ps.n = rad.n;
  int rmin = 16;
  for (int p = 0; p < rad.n; ++p) {
    ps.r[p] = rad.r[p];
    ps.sh[p] = SECOND ? F.sh2[p] : F.sh1[p];
    rmin = rad.r[p] < rmin ? rad.r[p] : rmin;
  }
  // in place (a third less shared memory: four blocks an SM at L = 1000) when
  // every pass has a thread per butterfly
  const int most = (C * L / rmin + 31) / 32 * 32;
  const bool inpl = most <= 512;
  const int threads = most < 64 ? 64 : (most > 512 ? 512 : most);
  const size_t sm = ((inpl ? 1 : 2) * (size_t)C + 1) * L * sizeof(longlong2);
  auto kern = !inpl ? k_fft_fx<SIGN, SECOND, C, false, 512, 1>
                    : (threads <= 256 ? k_fft_fx<SIGN, SECOND, C, true, 256, 2> : k_fft_fx<SIGN, SECOND, C, true, 512, 1>);
  if (sm > 48 * 1024) SS_TRY(allow_smem(kern));
  ProfScope prof_("k_fft_fx", st, true);
  kern<<<(SECOND ? F.L1 : F.L2) / C, threads, sm, st>>>(in, out, tab, tab + F.M + (SECOND ? F.L1 : 0),
                                                        classes, F.M, F.L1, F.L2, ps);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

template <int SIGN, bool SECOND>
ss_status launch(const FxFftPlan& F, const int4* tab, const longlong2* in, longlong2* out, const int2* classes,
                 cudaStream_t st) {
  // two columns a block where their number is even and five buffers of L values fit
  const int L = SECOND ? F.L2 : F.L1, cols = SECOND ? F.L1 : F.L2;
  if (cols % 2 == 0 && L <= 2048) return launch_c<SIGN, SECOND, 2>(F, tab, in, out, classes, st);
  return launch_c<SIGN, SECOND, 1>(F, tab, in, out, classes, st);
}

// Radices of the fixed-point passes: 10 while both 2 and 5 divide L (a pass and
// a round of twiddles fewer than 5 and 2), odd ones, then 8, 4, 2.
DfRadices fx_radices(int L) {
  DfRadices d;
  if (L == 1) {   // one pass has to carry the data over
    d.r[d.n++] = 1;
    return d;
  }
  for (int R : {10, 7, 5, 3, 8, 4, 2})
    while (L > 1 && L % R == 0 && d.n < kDfFftMaxPasses) {
      d.r[d.n++] = R;
      L /= R;
    }
  if (L != 1) d.n = -1;
  return d;
}

}  // namespace

DfRadices df_radices(int L) {
  DfRadices d;
  // odd radices first: the first pass (Ns = 1) writes at stride R, free of
  // shared-memory bank conflicts for odd R
  for (int R : {7, 5, 3, 8, 4, 2})
    while (L > 1 && L % R == 0 && d.n < kDfFftMaxPasses) {
      d.r[d.n++] = R;
      L /= R;
    }
  if (L != 1) d.n = -1;
  return d;
}

bool fx_fft_plan(int64_t M, FxFftPlan* out) {
  if (M < 1) return false;
  int64_t best = -1;
  for (int64_t l1 = 1; l1 <= kDfFftMaxL && l1 <= M; ++l1) {
    if (M % l1 || M / l1 > kDfFftMaxL) continue;
    const int64_t l2 = M / l1;
    if (best < 0 || (l1 > l2 ? l1 - l2 : l2 - l1) < (best > M / best ? best - M / best : M / best - best)) best = l1;
  }
  if (best < 0) return false;
  FxFftPlan F;
  F.M = M;
  F.L1 = (int)best;
  F.L2 = (int)(M / best);
  F.rad1 = fx_radices(F.L1);
  F.rad2 = fx_radices(F.L2);
  if (F.rad1.n < 0 || F.rad2.n < 0) return false;
  // shifts of the forward passes: the growth not yet divided out (log2 of the
  // product of the radices, minus the shifts) stays at most 0; none after the
  // last pass
  double g = 0.0;
  auto plan = [&](const DfRadices& rad, int* sh, bool last) {
    for (int p = 0; p < rad.n; ++p) {
      g += std::log2((double)rad.r[p]);
      const int s = last && p + 1 == rad.n ? 0 : (g > 0.0 ? (int)std::ceil(g) : 0);
      sh[p] = s;
      F.shift += s;
      g -= s;
    }
  };
  plan(F.rad1, F.sh1, false);
  plan(F.rad2, F.sh2, true);
  *out = F;
  return true;
}

ss_status fx_fft_table(const FxFftPlan& F, int4* tab, cudaStream_t st) {
  DevBuf<int4> part;
  SS_TRY(part.alloc_tmp(F.L1 + F.L2, st));
  k_fx_roots<<<(F.L1 + F.L2 + 63) / 64, 64, 0, st>>>(F.M, F.L1, F.L2, part.get());
  k_fx_table<<<(unsigned)((F.M + F.L1 + F.L2 + 255) / 256), 256, 0, st>>>(F.M, F.L1, F.L2, part.get(), tab);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

ss_status fx_inverse(const FxFftPlan& F, const int4* tab, const double2* in, const int2* classes, longlong2* tmp,
                     longlong2* out, cudaStream_t st) {
  SS_TRY((launch<1, false>(F, tab, reinterpret_cast<const longlong2*>(in), tmp, classes + F.L1, st)));
  return launch<1, true>(F, tab, tmp, out, nullptr, st);
}

ss_status fx_forward(const FxFftPlan& F, const int4* tab, const longlong2* in, const int2* classes, longlong2* tmp,
                     longlong2* out, cudaStream_t st) {
  SS_TRY((launch<-1, false>(F, tab, in, tmp, nullptr, st)));
  return launch<-1, true>(F, tab, tmp, out, classes, st);
}

}  // namespace ss
