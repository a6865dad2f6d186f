// Pruned DFTs of a 7-smooth length M (the split, the index maps and the cost
// are stated in fft_pruned.cuh): in 64-bit fixed point (the FP64 recovery of
// two sums), in double-float (FP64 real samples) or in FP32 (the FP32 recovery).
//
// Inside a block a tile holds W columns of length P in shared memory, column c
// at c (P + 1) (one element of padding: threads that share a row offset and
// differ in the column hit distinct banks).  The length-P transforms run as
// self-sorting (Stockham) radix passes over all W columns at once, thread u
// taking column u mod W, butterfly u / W, with the P-th roots staged in
// shared memory.  The arithmetic is a policy (ArFX: fixed point, longlong2, the
// butterflies of fxc.cuh; ArDF: complex double-float values as float4, those of
// dfc.cuh; ArF32: float2).  All sums run in a fixed order, so results are
// bit-reproducible.
//
// Fixed point against double-float, M = 2^26, d = 100 (142 entries, 282 bins):
// evaluation 654 us, 757; forward 621 us, 774.  An addition takes 2
// instructions against 8 to 20, a product 14 to 26 against 50, and the rounding
// of a sample is 2^-55 of the l1 norm instead of 2^-47 of the values.  Bound:
// issue and latency at 16 warps an SM, the most that the registers of a radix-16
// butterfly leave (24 warps spill: 665, 684).
#include <algorithm>
#include <cmath>

#include "dfc.cuh"
#include "fxc.cuh"
#include "fft_pruned.cuh"

namespace ss {
namespace {

using namespace dfc;

constexpr int kPrTile = 2048;      // complex values of one tile (W columns x P rows), forward transform
constexpr int kPrEvalTile = 2048;  // the same for the evaluation
constexpr int kPrEvalStage = 1024; // step powers (entries x W) staged in shared memory up to this count
constexpr int kPrThreads = 256;
constexpr int kPrChunk = 256;      // entries staged in shared memory per round of the evaluation
constexpr int kPrMaxOut = 1024;    // outputs per forward launch (accumulators in shared memory)
constexpr int kPrMaxP = 1024;

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

__device__ __forceinline__ C4 conj4(const C4 a) { return C4{a.re, df_neg(a.im)}; }
__device__ __forceinline__ C4 zero4() { return C4{DF{0.f, 0.f}, DF{0.f, 0.f}}; }

// exp(sign 2 pi i r / M), r < M, from the two-level double-float table
template <int SIGN>
__device__ __forceinline__ C4 tw2(const float4* __restrict__ t0, const float4* __restrict__ t1, int b, uint64_t r) {
  const C4 w = cmul(ld(__ldg(t1 + (r >> b))), ld(__ldg(t0 + (r & ((1ull << b) - 1)))));
  return SIGN > 0 ? w : conj4(w);
}

// ------------------------------------------------------------ FP32 complex

__device__ __forceinline__ float2 fadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 fsub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 fmul(float2 a, float2 w) {
  return make_float2(fmaf(a.x, w.x, -a.y * w.y), fmaf(a.x, w.y, a.y * w.x));
}
__device__ __forceinline__ float2 fconj(float2 a) { return make_float2(a.x, -a.y); }
template <int SIGN>
__device__ __forceinline__ float2 fmul_si(float2 a) {   // a * (sign i)
  return SIGN > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <int SIGN>
__device__ __forceinline__ void fdft4(float2& v0, float2& v1, float2& v2, float2& v3) {
  const float2 t0 = fadd(v0, v2), t1 = fsub(v0, v2), t2 = fadd(v1, v3), t3 = fmul_si<SIGN>(fsub(v1, v3));
  v0 = fadd(t0, t2);
  v2 = fsub(t0, t2);
  v1 = fadd(t1, t3);
  v3 = fsub(t1, t3);
}

// R-point DFT in place, the same forms as dfc.cuh's: cs[m - 1] =
// exp(2 pi i m / R), m <= (R - 1) / 2; for R = 8, cs[0] = exp(2 pi i / 8).
template <int R, int SIGN>
__device__ __forceinline__ void fdft(float2 (&v)[R], const float2* cs) {
  if constexpr (R == 2) {
    const float2 a = v[0];
    v[0] = fadd(a, v[1]);
    v[1] = fsub(a, v[1]);
  } else if constexpr (R == 4) {
    fdft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    fdft4<SIGN>(e0, e1, e2, e3);
    fdft4<SIGN>(o0, o1, o2, o3);
    const float c = cs[0].x;   // cos(pi / 4)
    const float sg1 = SIGN > 0 ? o1.x : -o1.x, sh1 = SIGN > 0 ? o1.y : -o1.y;
    o1 = make_float2(c * (o1.x - sh1), c * (o1.y + sg1));
    o2 = fmul_si<SIGN>(o2);
    const float sg3 = SIGN > 0 ? o3.x : -o3.x, sh3 = SIGN > 0 ? o3.y : -o3.y;
    o3 = make_float2(-c * (o3.x + sh3), c * (sg3 - o3.y));
    v[0] = fadd(e0, o0);
    v[4] = fsub(e0, o0);
    v[1] = fadd(e1, o1);
    v[5] = fsub(e1, o1);
    v[2] = fadd(e2, o2);
    v[6] = fsub(e2, o2);
    v[3] = fadd(e3, o3);
    v[7] = fsub(e3, o3);
  } else {
    constexpr int H = (R - 1) / 2;
    float2 a[H], b[H];
#pragma unroll
    for (int r = 1; r <= H; ++r) {
      a[r - 1] = fadd(v[r], v[R - r]);
      b[r - 1] = fsub(v[r], v[R - r]);
    }
    const float2 v0 = v[0];
    float2 y0 = v0;
#pragma unroll
    for (int r = 0; r < H; ++r) y0 = fadd(y0, a[r]);
#pragma unroll
    for (int s = 1; s <= H; ++s) {
      float2 A = v0, Bv = make_float2(0.f, 0.f);
#pragma unroll
      for (int r = 1; r <= H; ++r) {
        const int m = (r * s) % R;
        const int mm = m <= H ? m : R - m;
        const float cm = cs[mm - 1].x;
        const float sm = m <= H ? cs[mm - 1].y : -cs[mm - 1].y;
        A.x = fmaf(cm, a[r - 1].x, A.x);
        A.y = fmaf(cm, a[r - 1].y, A.y);
        Bv.x = fmaf(sm, b[r - 1].x, Bv.x);
        Bv.y = fmaf(sm, b[r - 1].y, Bv.y);
      }
      const float2 iB = fmul_si<SIGN>(Bv);
      v[s] = fadd(A, iB);
      v[R - s] = fsub(A, iB);
    }
    v[0] = y0;
  }
}

// 16-point DFT as dft16 below, on FP32 complex values; output X[k1 + 4 k2]
// at v[4 k1 + k2].
template <int SIGN>
__device__ __forceinline__ void fdft16(float2 (&v)[16], const float2 w1, const float2 w2, const float2 w3) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) fdft4<SIGN>(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
  auto tw = [](const float2 a, const float2 w) { return fmul(a, SIGN > 0 ? w : fconj(w)); };
  v[5] = tw(v[5], w1);
  v[9] = tw(v[9], w2);
  v[13] = tw(v[13], w3);
  v[6] = tw(v[6], w2);
  v[10] = fmul_si<SIGN>(v[10]);
  v[14] = fmul_si<SIGN>(tw(v[14], w2));
  v[7] = tw(v[7], w3);
  v[11] = fmul_si<SIGN>(tw(v[11], w2));
  {
    const float2 t = tw(v[15], w1);
    v[15] = make_float2(-t.x, -t.y);
  }
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) fdft4<SIGN>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
}

// 16-point DFT in place (SIGN: exponent sign), natural input order; the
// output X[k1 + 4 k2] ends at v[4 k1 + k2].  w1, w2, w3 = exp(2 pi i j / 16).
// Four 4-point transforms (stride 4), the twiddles w16^(n2 k1), four more.
template <int SIGN>
__device__ __forceinline__ void dft16(C4 (&v)[16], const C4 w1, const C4 w2, const C4 w3) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4<SIGN>(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
  auto tw = [](const C4 a, const C4 w) { return cmul(a, SIGN > 0 ? w : conj4(w)); };
  v[5] = tw(v[5], w1);
  v[9] = tw(v[9], w2);
  v[13] = tw(v[13], w3);
  v[6] = tw(v[6], w2);
  v[10] = mul_si<SIGN>(v[10]);
  v[14] = mul_si<SIGN>(tw(v[14], w2));   // w16^6 = i w16^2
  v[7] = tw(v[7], w3);
  v[11] = mul_si<SIGN>(tw(v[11], w2));
  {
    const C4 t = tw(v[15], w1);   // w16^9 = -w16^1
    v[15] = C4{df_neg(t.re), df_neg(t.im)};
  }
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4<SIGN>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
}

// ------------------------------------------------------- arithmetic policies

// Double-float complex values stored as float4 (re.hi, re.lo, im.hi, im.lo).
struct ArDF {
  using V = float4;
  using C = C4;
  using TV = float4;   // roots, stored and as operands
  using T = C4;
  using AccV = float4; // the outputs' sums over the tiles
  using Acc = C4;
  static constexpr bool kFixed = false;
  static constexpr int kMinBlocks16 = 2;   // resident blocks per SM of the 4096-value-tile kernels
  static __device__ __forceinline__ C ld(const V v) { return dfc::ld(v); }
  static __device__ __forceinline__ V st(const C c) { return st4(c); }
  static __device__ __forceinline__ C add(const C a, const C b) { return cadd(a, b); }
  static __device__ __forceinline__ C mul(const C a, const C b) { return cmul(a, b); }
  static __device__ __forceinline__ C zero() { return zero4(); }
  static __device__ __forceinline__ C down(const C a, int) { return a; }
  static __device__ __forceinline__ C mulq(const C a, const T w) { return mul(a, w); }
  static __device__ __forceinline__ C bias(const C a, int) { return a; }
  static __device__ __forceinline__ C shr(const C a, int) { return a; }
  static __device__ __forceinline__ T ldt(const TV v) { return dfc::ld(v); }
  static __device__ __forceinline__ TV stt(const T c) { return st4(c); }
  static __device__ __forceinline__ T conjt(const T a) { return conj4(a); }
  // an entry's value, a step's root (16 bytes each, written by k_pr_entries and k_pr_steps)
  static __device__ __forceinline__ C entry(const float4 v) { return dfc::ld(v); }
  static __device__ __forceinline__ T step(const float4 v) { return dfc::ld(v); }
  static __device__ __forceinline__ AccV acc_zero() { return st4(zero4()); }
  static __device__ __forceinline__ AccV acc_add(const AccV a, const C b) { return st4(cadd(dfc::ld(a), b)); }
  template <int SIGN>
  static __device__ __forceinline__ T root(const float4* t0, const float4* t1, int b, uint64_t r) {
    return tw2<SIGN>(t0, t1, b, r);
  }
  template <int R, int SIGN>
  static __device__ __forceinline__ void dft(C (&v)[R], const T* cs) {
    dfc::dft<R, SIGN>(v, cs);
  }
  template <int SIGN>
  static __device__ __forceinline__ void dft16(C (&v)[16], const T w1, const T w2, const T w3) {
    ss::dft16<SIGN>(v, w1, w2, w3);
  }
  static __device__ __forceinline__ double2 to_double2(const AccV v) {
    return make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
  }
  using Real = double;   // real samples: FP64
  static __device__ __forceinline__ C from_real(const double x) { return C4{df_split(x), DF{0.f, 0.f}}; }
  static __device__ __forceinline__ double real_out(const V v) { return (double)v.x + (double)v.y; }
};

// FP32 complex values (the high words of the double-float tables and entries).
struct ArF32 {
  using V = float2;
  using C = float2;
  using TV = float2;
  using T = float2;
  using AccV = float2;
  static constexpr bool kFixed = false;
  static constexpr int kMinBlocks16 = 3;
  static __device__ __forceinline__ C ld(const V v) { return v; }
  static __device__ __forceinline__ V st(const C c) { return c; }
  static __device__ __forceinline__ C add(const C a, const C b) { return fadd(a, b); }
  static __device__ __forceinline__ C mul(const C a, const C b) { return fmul(a, b); }
  static __device__ __forceinline__ C zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ C down(const C a, int) { return a; }
  static __device__ __forceinline__ C mulq(const C a, const T w) { return mul(a, w); }
  static __device__ __forceinline__ C bias(const C a, int) { return a; }
  static __device__ __forceinline__ C shr(const C a, int) { return a; }
  static __device__ __forceinline__ T ldt(const TV v) { return v; }
  static __device__ __forceinline__ TV stt(const T c) { return c; }
  static __device__ __forceinline__ T conjt(const T a) { return fconj(a); }
  static __device__ __forceinline__ C entry(const float4 v) { return make_float2(v.x, v.z); }
  static __device__ __forceinline__ T step(const float4 v) { return make_float2(v.x, v.z); }
  static __device__ __forceinline__ AccV acc_zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ AccV acc_add(const AccV a, const C b) { return fadd(a, b); }
  template <int SIGN>
  static __device__ __forceinline__ T root(const float4* t0, const float4* t1, int b, uint64_t r) {
    const float4 u = __ldg(t1 + (r >> b)), l = __ldg(t0 + (r & ((1ull << b) - 1)));
    const float2 w = fmul(make_float2(u.x, u.z), make_float2(l.x, l.z));
    return SIGN > 0 ? w : fconj(w);
  }
  template <int R, int SIGN>
  static __device__ __forceinline__ void dft(C (&v)[R], const C* cs) {
    fdft<R, SIGN>(v, cs);
  }
  template <int SIGN>
  static __device__ __forceinline__ void dft16(C (&v)[16], const C w1, const C w2, const C w3) {
    fdft16<SIGN>(v, w1, w2, w3);
  }
  static __device__ __forceinline__ double2 to_double2(const V v) { return make_double2(v.x, v.y); }
  using Real = float;    // real samples: FP32
  static __device__ __forceinline__ C from_real(const float x) { return make_float2(x, 0.f); }
  static __device__ __forceinline__ float real_out(const V v) { return v.x; }
};

// Fixed-point complex values.  An entry counts units of 2^-61.  Each sum's scale
// is the power of two at or below its l1 norm: its entries' moduli add up to less
// than 2, both sums' to less than 4.  A residue of 0 or M/2 takes the whole real
// coefficient, below 2 (the constant 1 of a, for instance), the others half of
// theirs, below 1.  So an entry is one component below 2^62, or two of modulus
// below 2^61, and the products with the tile's and the column's root divide by
// four each (mulq): the middle products of the first are below 2^62 (one
// component) or 2^61.5 + 2^60.5 (two), the second's arguments below 2^60, a
// column's sum below 2^59.  The evaluation's second pass (or its end) divides by
// four as well: samples count units of 2^-55 and stay below 2^56.5.  A sample's rounding
// (a few units) is averaged over the M samples of a bin.  Forward, 4096-value
// tiles: 2^60.5 after the first pass, divided by four by the second's roots,
// 2^62.5 (P = 256) or 2^61.5 after it, divided by 2^6: Horner's sums over the
// 16 or 32 columns stay below 2^60.5.  Forward, other tiles: fwd_shifts.  (A
// column transform may be the same for every column, where its rounding does
// not average: it stays at 2^-52 of the scale or below.)  The sums over tiles
// and blocks run in FP64.  Roots: two-level table of Q62 limbs.
constexpr int kPrEntryFrac = 61, kPrSampleFrac = 55, kPrStoreShift = 6;
struct ArFX {
  using V = longlong2;
  using C = fxc::CX;
  using TV = int4;
  using T = fxc::TW;
  using AccV = double2;
  static constexpr bool kFixed = true;
  static constexpr int kMinBlocks16 = 2;
  static __device__ __forceinline__ C ld(const V v) { return fxc::ld(v); }
  static __device__ __forceinline__ V st(const C c) { return fxc::st(c); }
  static __device__ __forceinline__ C add(const C a, const C b) { return fxc::add(a, b); }
  static __device__ __forceinline__ C mul(const C a, const T w) { return fxc::mul(a, w); }
  static __device__ __forceinline__ C zero() { return C{0, 0}; }
  static __device__ __forceinline__ C mulq(const C a, const T w) { return fxc::mulq(a, w); }   // a w / 4
  // a / 2^s rounded; the same for all outputs of a transform: bias its input 0
  // (an impulse adds to every output), then shift
  static __device__ __forceinline__ C down(const C a, int s) { return fxc::scale_down(a, s); }
  static __device__ __forceinline__ C bias(const C a, int s) {
    const long long h = 1ll << (s - 1);
    return C{a.re + h, a.im + h};
  }
  static __device__ __forceinline__ C shr(const C a, int s) { return C{a.re >> s, a.im >> s}; }
  static __device__ __forceinline__ C shfl(const C a, int m) {
    return C{__shfl_xor_sync(0xffffffffu, a.re, m), __shfl_xor_sync(0xffffffffu, a.im, m)};
  }
  static __device__ __forceinline__ T ldt(const TV v) { return fxc::ld_tw(v); }
  static __device__ __forceinline__ TV stt(const T w) { return fxc::st_tw(w); }
  static __device__ __forceinline__ T conjt(const T w) { return fxc::conj(w); }
  static __device__ __forceinline__ int4 bits(const float4 v) {
    return make_int4(__float_as_int(v.x), __float_as_int(v.y), __float_as_int(v.z), __float_as_int(v.w));
  }
  static __device__ __forceinline__ float4 unbits(const int4 v) {
    return make_float4(__int_as_float(v.x), __int_as_float(v.y), __int_as_float(v.z), __int_as_float(v.w));
  }
  static __device__ __forceinline__ C entry(const float4 v) {
    const int4 i = bits(v);
    return C{(long long)(((unsigned long long)(unsigned)i.y << 32) | (unsigned)i.x),
             (long long)(((unsigned long long)(unsigned)i.w << 32) | (unsigned)i.z)};
  }
  static __device__ __forceinline__ float4 entry_bits(long long x, long long y) {
    return unbits(make_int4((int)x, (int)(x >> 32), (int)y, (int)(y >> 32)));
  }
  static __device__ __forceinline__ T step(const float4 v) { return fxc::ld_tw(bits(v)); }
  static __device__ __forceinline__ AccV acc_zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ AccV acc_add(const AccV a, const C b) {
    return make_double2(a.x + (double)b.re, a.y + (double)b.im);
  }
  template <int SIGN>
  static __device__ __forceinline__ T root(const float4* t0, const float4* t1, int b, uint64_t r) {
    const T u = step(__ldg(t1 + (r >> b))), l = step(__ldg(t0 + (r & ((1ull << b) - 1))));
    // the value of balanced limbs is h 2^32 + l
    const C w = fxc::mul(C{((long long)u.rh << 32) + u.rl, ((long long)u.ih << 32) + u.il}, l);
    const T t = fxc::to_tw(w.re, w.im);
    return SIGN > 0 ? t : fxc::conj(t);
  }
  template <int R, int SIGN>
  static __device__ __forceinline__ void dft(C (&v)[R], const T* cs) {
    fxc::dft<R, SIGN>(v, cs);
  }
  template <int SIGN>
  static __device__ __forceinline__ void dft16(C (&v)[16], const T w1, const T w2, const T w3) {
    fxc::dft16<SIGN>(v, w1, w2, w3);
  }
  static __device__ __forceinline__ double2 to_double2(const AccV v) { return v; }
  using Real = double;   // no real format
  static __device__ __forceinline__ C from_real(const double) { return zero(); }
  static __device__ __forceinline__ double real_out(const V) { return 0.0; }
};

// Shifts of the general forward transform after pass p.
struct PrShifts {
  int pass[kDfFftMaxPasses] = {};
};

__global__ void k_tl_table_fx(int64_t M, int b, int64_t n1, float4* t0, float4* t1) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < (1ll << b)) t0[i] = ArFX::unbits(fxc::st_tw(fxc::exact_root(i, M)));
  if (i < n1) t1[i] = ArFX::unbits(fxc::st_tw(fxc::exact_root(i << b, M)));
}

__global__ void k_tl_table(int64_t M, int b, int64_t n1, float4* t0, float4* t1) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double s, c;
  if (i < (1ll << b)) {
    sincospi(2.0 * (double)i / (double)M, &s, &c);
    const DF cc = df_split(c), sn = df_split(s);
    t0[i] = make_float4(cc.hi, cc.lo, sn.hi, sn.lo);
  }
  if (i < n1) {
    sincospi(2.0 * (double)(i << b) / (double)M, &s, &c);
    const DF cc = df_split(c), sn = df_split(s);
    t1[i] = make_float4(cc.hi, cc.lo, sn.hi, sn.lo);
  }
}

// One radix-R Stockham pass over the W = 2^wsh columns (length P, column
// stride CS).  j / Ns is formed as umulhi(j, ceil(2^32 / Ns)), exact for
// j, Ns < 2^16.
template <class A, int R, int SIGN>
__device__ __forceinline__ void mpass(const typename A::V* __restrict__ a, typename A::V* __restrict__ b, int P,
                                      int wsh, int CS, int Ns, const typename A::TV* __restrict__ tw, int sh) {
  using C = typename A::C;
  constexpr int NC = R == 8 ? 1 : (R - 1) / 2;
  using T = typename A::T;
  T cs[NC > 0 ? NC : 1];
#pragma unroll
  for (int m = 0; m < NC; ++m) cs[m] = A::ldt(tw[(P / R) * (m + 1)]);
  const int nb = P / R;
  const int tstride = P / (Ns * R);
  const int total = nb << wsh;
  const unsigned wmask = (1u << wsh) - 1u;
  const unsigned nsm = Ns > 1 ? 0xffffffffu / (unsigned)Ns + 1u : 0u;
  for (int u = threadIdx.x; u < total; u += blockDim.x) {
    const int c = (int)((unsigned)u & wmask), j = u >> wsh;
    const typename A::V* ac = a + c * CS;
    typename A::V* bc = b + c * CS;
    const int jq = Ns > 1 ? (int)__umulhi((unsigned)j, nsm) : j;   // j / Ns
    const int k = j - jq * Ns;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = A::ld(ac[j + r * nb]);
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const T w = A::ldt(tw[tstride * (k * r)]);
        v[r] = A::mul(v[r], SIGN > 0 ? w : A::conjt(w));
      }
    }
    A::template dft<R, SIGN>(v, cs);
    const int base = jq * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) bc[base + r * Ns] = A::st(SIGN < 0 && sh ? A::down(v[r], sh) : v[r]);
  }
}

// Length-P transforms of the W columns in `a` (b: the other buffer); returns
// the buffer that holds the result.  Ends with a block barrier.
template <class A, int SIGN>
__device__ typename A::V* columns_dft(typename A::V* a, typename A::V* b, int P, int wsh, int CS,
                                      const DfRadices& rad, const PrShifts& shifts,
                                      const typename A::TV* __restrict__ tw) {
  int Ns = 1;
  for (int p = 0; p < rad.n; ++p) {
    const int R = rad.r[p], sh = shifts.pass[p];
    switch (R) {
      case 8: mpass<A, 8, SIGN>(a, b, P, wsh, CS, Ns, tw, sh); break;
      case 4: mpass<A, 4, SIGN>(a, b, P, wsh, CS, Ns, tw, sh); break;
      case 2: mpass<A, 2, SIGN>(a, b, P, wsh, CS, Ns, tw, sh); break;
      case 5: mpass<A, 5, SIGN>(a, b, P, wsh, CS, Ns, tw, sh); break;
      case 3: mpass<A, 3, SIGN>(a, b, P, wsh, CS, Ns, tw, sh); break;
      default: mpass<A, 7, SIGN>(a, b, P, wsh, CS, Ns, tw, sh); break;
    }
    __syncthreads();
    typename A::V* t = a;
    a = b;
    b = t;
    Ns *= R;
  }
  return a;
}

// Entries of the spectrum Z = S_a / scale[0] + i S_f / scale[1] (S_a, S_f the
// Hermitian spectra of the two real sums: a term (r, c) puts c / 2 at r and
// conj(c) / 2 at M - r, or Re c at r when r = 0 or 2 r = M), bucketed by
// r mod P in term order (a's terms, then f's; r before M - r).  One block;
// boff[k] = first entry of bucket k, boff[P] = the number of entries.
// kq: scratch of 2 (na + nf) int32 (the two buckets of every term).
template <bool FX>
__global__ void k_pr_entries(const int64_t* __restrict__ qa, const double2* __restrict__ ca,
                             const int64_t* __restrict__ na_dev, const int64_t* __restrict__ qf,
                             const double2* __restrict__ cf, const int64_t* __restrict__ nf_dev,
                             const double* __restrict__ scale, int64_t M, int P, int32_t* kq_g, int64_t* er,
                             float4* ev, int32_t* boff, int kq_smem) {
  extern __shared__ int32_t cnt[];   // P + 1, then the buckets of the entries when 2 n <= kq_smem
  const int64_t na = *na_dev, nf = nf_dev ? *nf_dev : 0, n = na + nf;
  int32_t* kq = 2 * n <= kq_smem ? cnt + P + 1 : kq_g;
  auto res = [&](int64_t u) { return u < na ? qa[u] : qf[u - na]; };
  for (int k = threadIdx.x; k <= P; k += blockDim.x) cnt[k] = 0;
  __syncthreads();
  for (int64_t u = threadIdx.x; u < n; u += blockDim.x) {
    const int64_t r = res(u);
    const bool one = r == 0 || 2 * r == M;
    const int32_t k0 = (int32_t)(r % P), k1 = one ? -1 : (int32_t)((M - r) % P);
    kq[2 * u] = k0;
    kq[2 * u + 1] = k1;
    atomicAdd(cnt + k0, 1);
    if (k1 >= 0) atomicAdd(cnt + k1, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int k = 0; k < P; ++k) {
      const int c = cnt[k];
      cnt[k] = s;
      s += c;
    }
    cnt[P] = s;
  }
  __syncthreads();
  for (int k = threadIdx.x; k <= P; k += blockDim.x) boff[k] = cnt[k];
  const double ia = scale ? 1.0 / scale[0] : 1.0, jf = scale ? 1.0 / scale[1] : 1.0;   // exact: powers of two
  // stable placement: entry v goes after the earlier entries of its bucket
  for (int64_t v = threadIdx.x; v < 2 * n; v += blockDim.x) {
    const int32_t k = kq[v];
    if (k < 0) continue;
    int pos = cnt[k];
    for (int64_t w = 0; w < v; ++w) pos += kq[w] == k;
    const int64_t u = v >> 1;
    const bool neg = v & 1;
    const int64_t r = res(u);
    const bool one = r == 0 || 2 * r == M;
    double x, y;
    if (u < na) {
      const double2 c = ca[u];
      if (one) {
        x = c.x * ia;
        y = 0.0;
      } else {
        x = 0.5 * c.x * ia;
        y = (neg ? -0.5 : 0.5) * c.y * ia;
      }
    } else {
      const double2 c = cf[u - na];
      if (one) {
        x = 0.0;
        y = c.x * jf;
      } else {
        x = (neg ? 0.5 : -0.5) * c.y * jf;
        y = 0.5 * c.x * jf;
      }
    }
    er[pos] = neg ? M - r : r;
    if (FX) {
      const double un = ldexp(1.0, kPrEntryFrac);
      ev[pos] = ArFX::entry_bits(__double2ll_rn(x * un), __double2ll_rn(y * un));
    } else {
      const DF dx = df_split(x), dy = df_split(y);
      ev[pos] = make_float4(dx.hi, dx.lo, dy.hi, dy.lo);
    }
  }
}

// tab[e][i] = exp(sign 2 pi i (i r_e mod M) / M) for e < n (device count n_dev
// when given, else n_host), i < W.
template <int SIGN, bool FX>
__global__ void k_pr_steps(const int64_t* __restrict__ r, const int32_t* __restrict__ n_dev, int64_t n_host, int W,
                           int64_t M, const float4* __restrict__ t0, const float4* __restrict__ t1, int b,
                           float4* tab) {
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = n_dev ? *n_dev : n_host;
  const int64_t e = id / W;
  const int i = (int)(id % W);
  if (e >= n) return;
  const uint64_t idx = ((uint64_t)i * (uint64_t)r[e]) % (uint64_t)M;
  if (FX) tab[id] = ArFX::unbits(fxc::st_tw(ArFX::root<SIGN>(t0, t1, b, idx)));
  else tab[id] = st4(tw2<SIGN>(t0, t1, b, idx));
}

// Output bins: bucket b mod P of every output.
__global__ void k_pr_kout(const int64_t* __restrict__ bins, int64_t n, int P, int32_t* kout) {
  const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (o < n) kout[o] = (int32_t)(bins[o] % P);
}

// Evaluation: s[q + Q p] for every tile of W columns (grid-stride over tiles).
// Fixed point: 80 registers and three blocks an SM (M = 3^16, 300 terms: 1.69 ms,
// 102 registers and two blocks: 1.89).
template <class A, bool OUT_REAL>
__global__ void __launch_bounds__(kPrThreads, A::kFixed ? 3 : 0)
    k_pr_eval(int64_t M, int P, int64_t Q, int wsh, DfRadices rad, const float4* __restrict__ t0,
              const float4* __restrict__ t1, int b, const int64_t* __restrict__ er, const float4* __restrict__ ev,
              const int32_t* __restrict__ boff_g, const float4* __restrict__ estep, int n_stage, int64_t n_tiles,
              void* __restrict__ out) {
  using V = typename A::V;
  using C = typename A::C;
  using TV = typename A::TV;
  using T = typename A::T;
  extern __shared__ __align__(16) float4 sm4[];
  const int CS = P + 1, W = 1 << wsh;
  const unsigned wmask = (unsigned)W - 1u;
  V* Av = reinterpret_cast<V*>(sm4);
  V* Bf = Av + W * CS;
  TV* tw = reinterpret_cast<TV*>(Bf + W * CS);
  V* base = reinterpret_cast<V*>(tw + P);
  TV* es = reinterpret_cast<TV*>(base + kPrChunk);   // staged step powers (n_stage > 0)
  int32_t* boff = reinterpret_cast<int32_t*>(es + n_stage);
  const uint64_t Mu = (uint64_t)M, inv = ~0ull / Mu;
  for (int m = threadIdx.x; m < P; m += blockDim.x)
    tw[m] = A::stt(A::template root<1>(t0, t1, b, (uint64_t)m * (uint64_t)Q));
  for (int k = threadIdx.x; k <= P; k += blockDim.x) boff[k] = boff_g[k];
  __syncthreads();
  const int ne = boff[P];
  // the step powers exp(2 pi i i r_e / M) are the same for every tile
  if (n_stage > 0) {
    for (int x = threadIdx.x; x < ne * W; x += blockDim.x) es[x] = A::stt(A::step(__ldg(estep + x)));
    __syncthreads();
  }
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t q0 = tile * W;
    // C[k][i] = sum_{e in bucket k} v_e w^{(q0 + i) r_e}, in chunks of entries
    int e0 = 0;
    do {
      const int e1 = min(ne, e0 + kPrChunk);
      for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x)
        base[e - e0] = A::st(A::mulq(A::entry(__ldg(ev + e)),
                                    A::template root<1>(t0, t1, b, mulmod((uint64_t)q0, (uint64_t)er[e], Mu, inv))));
      __syncthreads();
#pragma unroll 4
      for (int u = threadIdx.x; u < P * W; u += blockDim.x) {
        const int i = (int)((unsigned)u & wmask), k = u >> wsh;
        const int lo = max(boff[k], e0), hi = min(boff[k + 1], e1);
        C s = e0 == 0 ? A::zero() : A::ld(Av[i * CS + k]);
        if (n_stage > 0) {
          for (int e = lo; e < hi; ++e) s = A::add(s, A::mulq(A::ld(base[e - e0]), A::ldt(es[e * W + i])));
        } else {
          for (int e = lo; e < hi; ++e)
            s = A::add(s, A::mulq(A::ld(base[e - e0]), A::step(__ldg(estep + (int64_t)e * W + i))));
        }
        Av[i * CS + k] = A::st(s);
      }
      __syncthreads();
      e0 += kPrChunk;
    } while (e0 < ne);
    // s[q0 + i + Q p] = sum_k w_P^{p k} C[k][i]
    const V* res = columns_dft<A, 1>(Av, Bf, P, wsh, CS, rad, PrShifts{}, tw);
    for (int u = threadIdx.x; u < P * W; u += blockDim.x) {
      const int i = (int)((unsigned)u & wmask), p = u >> wsh;
      const int64_t q = q0 + i;
      if (q >= Q) continue;
      if (OUT_REAL)
        static_cast<typename A::Real*>(out)[q + Q * p] = A::real_out(res[i * CS + p]);
      else
        static_cast<V*>(out)[q + Q * p] = A::st(A::down(A::ld(res[i * CS + p]), 2));
    }
    __syncthreads();
  }
}

// FP32 evaluation with P = 16 or 32: a thread holds a whole column in registers,
// so the length-P transform (radix 8, then P / 8) needs neither shared memory
// nor index arithmetic, and writes its P samples (a warp: 32 neighbours of each
// p).  The tiles of W columns, their entries and every operation are
// k_pr_eval's, in its order: the same samples bit for bit.  256 / W tiles per
// block at once, the base values of kPrColRounds rounds of them together (their
// table reads overlap).
// M = 2^26, 42 entries, P = 32: 370 us by k_pr_eval (integer and shared-memory
// issue: 130 instructions a sample), 216 us so (latency of the entry loops at 16
// warps an SM; 24 warps spill); the 537 MB of samples take 79.
constexpr int kPrColEntries = 128;   // step powers in shared memory (64 KB at W = 64)
constexpr int kPrColRounds = 4;

__host__ __device__ constexpr bool pr_col_supported(int P) { return P == 16 || P == 32; }

template <int P, bool OUT_REAL>
__global__ void __launch_bounds__(kPrThreads, 2) k_pr_eval_col(int64_t M, int64_t Q, const float4* __restrict__ t0,
                                                               const float4* __restrict__ t1, int b,
                                                               const int64_t* __restrict__ er,
                                                               const float4* __restrict__ ev,
                                                               const int32_t* __restrict__ boff_g,
                                                               const float4* __restrict__ estep, int n_stage,
                                                               int64_t n_tiles, void* __restrict__ out) {
  using A = ArF32;
  constexpr int W = kPrEvalTile / P, SUB = kPrThreads / W, R2 = P / 8;
  static_assert(W <= kPrThreads, "a tile within a block");
  extern __shared__ __align__(16) float4 sm4[];
  float2* tw = reinterpret_cast<float2*>(sm4);
  float2* es = tw + P;                              // [ne][W]
  float2* base = es + n_stage;                      // [kPrColRounds][SUB][ne]
  __shared__ int32_t boff[P + 1];
  const uint64_t Mu = (uint64_t)M, inv = ~0ull / Mu;
  for (int m = threadIdx.x; m < P; m += blockDim.x) tw[m] = A::root<1>(t0, t1, b, (uint64_t)m * (uint64_t)Q);
  for (int k = threadIdx.x; k <= P; k += blockDim.x) boff[k] = boff_g[k];
  __syncthreads();
  const int ne = boff[P];
  for (int x = threadIdx.x; x < ne * W; x += blockDim.x) es[x] = A::step(__ldg(estep + x));
  const float2 cs[1] = {tw[P / 8]};
  const int sub = threadIdx.x / W, i = threadIdx.x % W;
  // the block's tiles: SUB neighbours a round, the rounds gridDim.x SUB tiles apart
  const int64_t stride = (int64_t)gridDim.x * SUB;
  for (int64_t first = (int64_t)blockIdx.x * SUB; first < n_tiles; first += kPrColRounds * stride) {
    __syncthreads();   // the last rounds' values are read
#pragma unroll 4
    for (int x = threadIdx.x; x < kPrColRounds * SUB * ne; x += blockDim.x) {
      const int t = x / ne, e = x - t * ne;   // tile t % SUB of round t / SUB
      const uint64_t q0 = (uint64_t)min(first + (t / SUB) * stride + t % SUB, n_tiles - 1) * W;
      base[x] = A::mul(A::entry(__ldg(ev + e)), A::root<1>(t0, t1, b, mulmod(q0, (uint64_t)er[e], Mu, inv)));
    }
    __syncthreads();
#pragma unroll 1
    for (int rnd = 0; rnd < kPrColRounds && first + rnd * stride < n_tiles; ++rnd) {
      const int64_t tile0 = first + rnd * stride;
      const float2* bs = base + (rnd * SUB + sub) * ne;
      const float2* ei = es + i;
      // every bucket's first entry without a branch (its reads overlap), the others after it
      float2 c[P];
#pragma unroll
      for (int k = 0; k < P; ++k) {
        const int lo = boff[k], e = max(0, min(lo, ne - 1));
        const float2 x = A::add(A::zero(), A::mul(bs[e], ei[e * W]));
        c[k] = lo < boff[k + 1] ? x : A::zero();
      }
#pragma unroll
      for (int k = 0; k < P; ++k) {
        const int hi = boff[k + 1];
        for (int e = boff[k] + 1; e < hi; ++e) c[k] = A::add(c[k], A::mul(bs[e], ei[e * W]));
      }
      // radix 8: butterfly j takes j + r P / 8, output r goes to 8 j + r
#pragma unroll
      for (int j = 0; j < R2; ++j) {
        float2 v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = c[j + r * R2];
        A::dft<8, 1>(v, cs);
#pragma unroll
        for (int r = 0; r < 8; ++r) c[j + r * R2] = v[r];   // position 8 j + r
      }
      // radix P / 8: butterfly k takes k + 8 r (butterfly r's output k), output r is the sample k + 8 r
      const int64_t q = (tile0 + sub) * W + i;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        float2 v[R2];
#pragma unroll
        for (int r = 0; r < R2; ++r) v[r] = r && k ? A::mul(c[r + k * R2], tw[k * r]) : c[r + k * R2];
        A::dft<R2, 1>(v, nullptr);
        if (q >= Q) continue;
#pragma unroll
        for (int r = 0; r < R2; ++r) {
          if (OUT_REAL) static_cast<float*>(out)[q + Q * (k + 8 * r)] = A::real_out(v[r]);
          else static_cast<float2*>(out)[q + Q * (k + 8 * r)] = v[r];
        }
      }
    }
  }
}

// Pruned forward transform: per tile the length-P transforms of the W
// columns, then every output o accumulates
//   w^{-q0 b_o} sum_i Y[b_o mod P][q0 + i] z_o^i,   z_o = w^{-b_o},
// the sum over the tile's columns by Horner's scheme (thread o mod blockDim
// owns output o for the whole launch).  FEW (fixed point, at most a thread per
// output): lanes share the columns of an output and three blocks an SM hide what
// is left of the chains; with more outputs the work is in them and two blocks
// with all registers take less (M = 2^26, 2400 bins: 3.52 ms against 3.77).
// M = 2^26, 4 bins: 805 us (one lane: 2164), 84 bins: 967 (1143).
template <class A, bool IN_REAL, bool FEW>
__global__ void __launch_bounds__(kPrThreads, FEW ? 3 : 0)
    k_pr_fwd(int64_t M, int P, int64_t Q, int wsh, DfRadices rad, PrShifts shifts, const float4* __restrict__ t0,
             const float4* __restrict__ t1, int b, const void* __restrict__ in, const int64_t* __restrict__ ob,
             const int32_t* __restrict__ kout, int n_out, const float4* __restrict__ oz, int64_t n_tiles,
             typename A::AccV* __restrict__ partial) {
  using V = typename A::V;
  using C = typename A::C;
  using TV = typename A::TV;
  using T = typename A::T;
  using AccV = typename A::AccV;
  extern __shared__ __align__(16) float4 sm4[];
  const int CS = P + 1, W = 1 << wsh;
  const unsigned wmask = (unsigned)W - 1u;
  V* Av = reinterpret_cast<V*>(sm4);
  V* Bf = Av + W * CS;
  TV* tw = reinterpret_cast<TV*>(Bf + W * CS);
  AccV* acc = reinterpret_cast<AccV*>(tw + P);
  const uint64_t Mu = (uint64_t)M, inv = ~0ull / Mu;
  int G = 1;   // lanes per output
  while (2 * G * n_out <= kPrThreads && G < 32 && 2 * G <= W) G *= 2;
  for (int m = threadIdx.x; m < P; m += blockDim.x)
    tw[m] = A::stt(A::template root<1>(t0, t1, b, (uint64_t)m * (uint64_t)Q));
  for (int o = threadIdx.x; o < n_out; o += blockDim.x) acc[o] = A::acc_zero();
  __syncthreads();
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t q0 = tile * W;
    for (int u = threadIdx.x; u < P * W; u += blockDim.x) {
      const int i = (int)((unsigned)u & wmask), p = u >> wsh;
      const int64_t q = q0 + i;
      C v = A::zero();
      if (q < Q) {
        if (IN_REAL) v = A::from_real(__ldg(static_cast<const typename A::Real*>(in) + q + Q * p));
        else v = A::ld(__ldg(static_cast<const V*>(in) + q + Q * p));
      }
      Av[i * CS + p] = A::st(v);
    }
    __syncthreads();
    const V* res = columns_dft<A, -1>(Av, Bf, P, wsh, CS, rad, shifts, tw);
    const int wl = Q - q0 < (int64_t)W ? (int)(Q - q0) : W;
    if constexpr (FEW) {
      // G lanes an output, each with its W / G columns (zero beyond Q): Horner's
      // chain of fixed-point products is long where the outputs are few
      const int cols = W / G, g = threadIdx.x & (G - 1);
      for (int o0 = 0; o0 < n_out; o0 += kPrThreads / G) {
        const int o = o0 + threadIdx.x / G;
        C s = A::zero();
        if (o < n_out) {
          const uint64_t q = (uint64_t)(q0 + g * cols);
          const T w = A::template root<-1>(t0, t1, b, mulmod(q, (uint64_t)ob[o], Mu, inv));
          const T z = A::step(__ldg(oz + 2 * o));
          const V* r = res + (g * cols) * CS + kout[o];
          s = A::ld(r[(cols - 1) * CS]);
          for (int i = cols - 2; i >= 0; --i) s = A::add(A::mul(s, z), A::ld(r[i * CS]));
          s = A::mul(s, w);
        }
        for (int m = G / 2; m > 0; m >>= 1) s = A::add(s, A::shfl(s, m));
        if (g == 0 && o < n_out) acc[o] = A::acc_add(acc[o], s);
      }
      __syncthreads();
      continue;
    }
    for (int o = threadIdx.x; o < n_out; o += blockDim.x) {
      const int k = kout[o];
      const T w = A::template root<-1>(t0, t1, b, mulmod((uint64_t)q0, (uint64_t)ob[o], Mu, inv));
      const T z = A::step(__ldg(oz + 2 * o));   // oz: stride 2 (the step table of width 2, entry 1)
      C s = A::ld(res[(wl - 1) * CS + k]);
      for (int i = wl - 2; i >= 0; --i) s = A::add(A::mul(s, z), A::ld(res[i * CS + k]));
      acc[o] = A::acc_add(acc[o], A::mul(s, w));
    }
    __syncthreads();
  }
  for (int o = threadIdx.x; o < n_out; o += blockDim.x) partial[(int64_t)blockIdx.x * n_out + o] = acc[o];
}

// ------------------------------------------- 4096-value tiles, radix 16
//
// Double-float transforms with P = 128 or 256: tiles of W = 4096 / P columns,
// the column transforms as two in-place Stockham passes, a radix-16 one and
// one of radix P / 16.  Every thread holds one radix-16 butterfly (or two
// radix-8 ones) in registers between a read phase and a write phase, so one
// shared buffer serves both passes (two barriers per pass).  The forward
// kernel's first pass reads the samples straight from global memory and the
// evaluation's second pass writes them straight there.
constexpr int kPr16Tile = 4096;
constexpr int kPr16Threads = 256;   // butterflies of a radix-16 pass over a tile

__host__ __device__ constexpr bool pr16_supported(int P) { return P == 128 || P == 256; }

// Second pass (Ns = 16) of one column in place: butterflies k (and k + 8 when
// the radix is 8) read k + 16 r, take the twiddles w_P^(SIGN k r) and write
// output r at k + 16 r.  out(p, value) receives the outputs (position p in the
// column); with IN_PLACE the block synchronises between reads and writes.
template <class A, int P, int SIGN, bool IN_PLACE, class Out>
__device__ __forceinline__ void pr16_pass2(const typename A::V* col, int k, const typename A::TV* tw,
                                           const typename A::T w1, const typename A::T w2, const typename A::T w3,
                                           Out out) {
  using C = typename A::C;
  using T = typename A::T;
  if constexpr (P == 256) {
    C v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = A::ld(col[k + 16 * r]);
    if (IN_PLACE) __syncthreads();
#pragma unroll
    for (int r = 1; r < 16; ++r) {
      const T w = A::ldt(tw[k * r]);
      v[r] = A::mulq(v[r], SIGN > 0 ? w : A::conjt(w));
    }
    v[0] = A::down(v[0], 2);
    if (SIGN < 0) v[0] = A::bias(v[0], kPrStoreShift);
    A::template dft16<SIGN>(v, w1, w2, w3);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) out(k + 16 * (k1 + 4 * k2), v[4 * k1 + k2]);
  } else {   // P = 128: radix 8, butterflies k and k + 8
    C v[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < 8; ++r) v[h][r] = A::ld(col[k + 8 * h + 16 * r]);
    if (IN_PLACE) __syncthreads();
    const T cs[1] = {w2};   // exp(2 pi i / 8)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int kk = k + 8 * h;
#pragma unroll
      for (int r = 1; r < 8; ++r) {
        const T w = A::ldt(tw[kk * r]);
        v[h][r] = A::mulq(v[h][r], SIGN > 0 ? w : A::conjt(w));
      }
      v[h][0] = A::down(v[h][0], 2);
      if (SIGN < 0) v[h][0] = A::bias(v[h][0], kPrStoreShift);
      A::template dft<8, SIGN>(v[h], cs);
#pragma unroll
      for (int r = 0; r < 8; ++r) out(kk + 16 * r, v[h][r]);
    }
  }
}

// Evaluation with 4096-value tiles (see above); the bucket phase as k_pr_eval.
template <class A, int P, bool OUT_REAL>
__global__ void __launch_bounds__(kPr16Threads, A::kMinBlocks16) k_pr_eval16(int64_t M, int64_t Q, const float4* __restrict__ t0,
                                                               const float4* __restrict__ t1, int b,
                                                               const int64_t* __restrict__ er,
                                                               const float4* __restrict__ ev,
                                                               const int32_t* __restrict__ boff_g,
                                                               const float4* __restrict__ estep, int n_stage,
                                                               int64_t n_tiles, void* __restrict__ out) {
  using V = typename A::V;
  using C = typename A::C;
  using TV = typename A::TV;
  using T = typename A::T;
  constexpr int W = kPr16Tile / P, CS = P + 1, R2 = P / 16;
  extern __shared__ __align__(16) float4 sm4[];
  V* tl = reinterpret_cast<V*>(sm4);
  TV* tw = reinterpret_cast<TV*>(tl + W * CS);
  V* base = reinterpret_cast<V*>(tw + P);
  TV* es = reinterpret_cast<TV*>(base + kPrChunk);
  int32_t* boff = reinterpret_cast<int32_t*>(es + n_stage);
  const uint64_t Mu = (uint64_t)M, inv = ~0ull / Mu;
  for (int m = threadIdx.x; m < P; m += blockDim.x)
    tw[m] = A::stt(A::template root<1>(t0, t1, b, (uint64_t)m * (uint64_t)Q));
  for (int k = threadIdx.x; k <= P; k += blockDim.x) boff[k] = boff_g[k];
  __syncthreads();
  const int ne = boff[P];
  if (n_stage > 0) {
    for (int x = threadIdx.x; x < ne * W; x += blockDim.x) es[x] = A::stt(A::step(__ldg(estep + x)));
    __syncthreads();
  }
  const T w1 = A::ldt(tw[P / 16]), w2 = A::ldt(tw[2 * P / 16]), w3 = A::ldt(tw[3 * P / 16]);
  const int u = threadIdx.x;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t q0 = tile * W;
    // C[k][i] = sum_{e in bucket k} v_e w^{(q0 + i) r_e}, in chunks of entries
    int e0 = 0;
    do {
      const int e1 = min(ne, e0 + kPrChunk);
      for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x)
        base[e - e0] = A::st(A::mulq(A::entry(__ldg(ev + e)),
                                    A::template root<1>(t0, t1, b, mulmod((uint64_t)q0, (uint64_t)er[e], Mu, inv))));
      __syncthreads();
      for (int x = threadIdx.x; x < P * W; x += blockDim.x) {
        const int i = x % W, k = x / W;
        const int lo = max(boff[k], e0), hi = min(boff[k + 1], e1);
        C sum = e0 == 0 ? A::zero() : A::ld(tl[i * CS + k]);
        for (int e = lo; e < hi; ++e) {
          const T st = n_stage > 0 ? A::ldt(es[e * W + i]) : A::step(__ldg(estep + (int64_t)e * W + i));
          sum = A::add(sum, A::mulq(A::ld(base[e - e0]), st));
        }
        tl[i * CS + k] = A::st(sum);
      }
      __syncthreads();
      e0 += kPrChunk;
    } while (e0 < ne);
    // pass 1 (radix 16, Ns = 1): butterfly j of column c reads j + R2 r, writes 16 j + r
    {
      const int c = u % W, j = u / W;
      V* col = tl + c * CS;
      C v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = A::ld(col[j + R2 * r]);
      __syncthreads();
      A::template dft16<1>(v, w1, w2, w3);
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) col[16 * j + k1 + 4 * k2] = A::st(v[4 * k1 + k2]);
    }
    __syncthreads();
    // pass 2 straight to the samples s[q0 + c + Q p]
    {
      const int c = u % W, k = u / W;
      const int64_t q = q0 + c;
      pr16_pass2<A, P, 1, false>(tl + c * CS, k, tw, w1, w2, w3, [&](int p, const C val) {
        if (q >= Q) return;
        if (OUT_REAL)
          static_cast<typename A::Real*>(out)[q + Q * p] = A::real_out(A::st(val));
        else
          static_cast<V*>(out)[q + Q * p] = A::st(val);
      });
    }
    __syncthreads();
  }
}

// Pruned forward transform with 4096-value tiles (see above); the Horner
// phase as k_pr_fwd.
template <class A, int P, bool IN_REAL>
__global__ void __launch_bounds__(kPr16Threads, A::kMinBlocks16) k_pr_fwd16(int64_t M, int64_t Q, const float4* __restrict__ t0,
                                                              const float4* __restrict__ t1, int b,
                                                              const void* __restrict__ in,
                                                              const int64_t* __restrict__ ob,
                                                              const int32_t* __restrict__ kout, int n_out,
                                                              const float4* __restrict__ oz, int64_t n_tiles,
                                                              typename A::AccV* __restrict__ partial) {
  using V = typename A::V;
  using C = typename A::C;
  using TV = typename A::TV;
  using T = typename A::T;
  using AccV = typename A::AccV;
  constexpr int W = kPr16Tile / P, CS = P + 1, R2 = P / 16;
  extern __shared__ __align__(16) float4 sm4[];
  V* tl = reinterpret_cast<V*>(sm4);
  TV* tw = reinterpret_cast<TV*>(tl + W * CS);
  AccV* acc = reinterpret_cast<AccV*>(tw + P);
  const uint64_t Mu = (uint64_t)M, inv = ~0ull / Mu;
  for (int m = threadIdx.x; m < P; m += blockDim.x)
    tw[m] = A::stt(A::template root<1>(t0, t1, b, (uint64_t)m * (uint64_t)Q));
  for (int o = threadIdx.x; o < n_out; o += blockDim.x) acc[o] = A::acc_zero();
  __syncthreads();
  const T w1 = A::ldt(tw[P / 16]), w2 = A::ldt(tw[2 * P / 16]), w3 = A::ldt(tw[3 * P / 16]);
  const int u = threadIdx.x;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t q0 = tile * W;
    // pass 1 (radix 16, Ns = 1) from the samples: butterfly j of column c
    // reads p = j + R2 r, writes 16 j + r
    {
      const int c = u % W, j = u / W;
      const int64_t q = q0 + c;
      C v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int64_t p = j + R2 * r;
        if (q >= Q) v[r] = A::zero();
        else if (IN_REAL) v[r] = A::from_real(__ldg(static_cast<const typename A::Real*>(in) + q + Q * p));
        else v[r] = A::ld(__ldg(static_cast<const V*>(in) + q + Q * p));
      }
      A::template dft16<-1>(v, w1, w2, w3);
      V* col = tl + c * CS;
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) col[16 * j + k1 + 4 * k2] = A::st(v[4 * k1 + k2]);
    }
    __syncthreads();
    {
      const int c = u % W, k = u / W;
      V* col = tl + c * CS;
      pr16_pass2<A, P, -1, true>(col, k, tw, w1, w2, w3, [&](int p, const C val) {
        col[p] = A::st(A::shr(val, kPrStoreShift));
      });
    }
    __syncthreads();
    const int wl = Q - q0 < (int64_t)W ? (int)(Q - q0) : W;
    for (int o = threadIdx.x; o < n_out; o += blockDim.x) {
      const int k = kout[o];
      const T w = A::template root<-1>(t0, t1, b, mulmod((uint64_t)q0, (uint64_t)ob[o], Mu, inv));
      const T z = A::step(__ldg(oz + 2 * o));
      C sum = A::ld(tl[(wl - 1) * CS + k]);
      for (int i = wl - 2; i >= 0; --i) sum = A::add(A::mul(sum, z), A::ld(tl[i * CS + k]));
      acc[o] = A::acc_add(acc[o], A::mul(sum, w));
    }
    __syncthreads();
  }
  for (int o = threadIdx.x; o < n_out; o += blockDim.x) partial[(int64_t)blockIdx.x * n_out + o] = acc[o];
}

// X[o] = sum over blocks of partial[blk][o] in FP64: one warp per output,
// lanes in a fixed stride, then a fixed butterfly; times unit.
template <class A>
__global__ void k_pr_reduce(const typename A::AccV* __restrict__ partial, int nb, int n_out, double unit,
                            double2* __restrict__ X) {
  const int64_t o = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (o >= n_out) return;   // warp-uniform
  double sr = 0.0, si = 0.0;
  for (int blk = lane; blk < nb; blk += 32) {
    const double2 v = A::to_double2(partial[(int64_t)blk * n_out + o]);
    sr += v.x;
    si += v.y;
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, m);
    si += __shfl_xor_sync(0xffffffffu, si, m);
  }
  if (lane == 0) X[o] = make_double2(sr * unit, si * unit);
}

template <class A>
const float4* table0(const TwoLevelTable& T) { return A::kFixed ? T.x0.get() : T.t0.get(); }
template <class A>
const float4* table1(const TwoLevelTable& T) { return A::kFixed ? T.x1.get() : T.t1.get(); }

template <class A>
size_t eval_smem(const PrunedSplit& S, int64_t n_stage) {
  return (size_t)(2 * S.W * (S.P + 1) + S.P + kPrChunk + n_stage) * sizeof(typename A::V) +
         (size_t)(S.P + 1) * sizeof(int32_t);
}

template <class A>
size_t fwd_smem(const PrunedSplit& S, int n_out) {
  return (size_t)(2 * S.W * (S.P + 1) + S.P + n_out) * sizeof(typename A::V);
}

template <typename K>
ss_status grid_for(K kernel, size_t smem, int64_t n_tiles, int* grid) {
  SS_TRY(allow_smem(kernel));
  int per_sm = 0;
  SS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPrThreads, smem));
  if (per_sm < 1) SS_FAIL(SS_ERR_CUDA, "pruned transform: a block of %zu bytes of shared memory does not fit", smem);
  *grid = (int)std::max<int64_t>(1, std::min<int64_t>(n_tiles, (int64_t)per_sm * sm_count()));
  return SS_OK;
}

template <class A, bool OUT_REAL>
ss_status launch_eval(const TwoLevelTable& T, const PrunedSplit& S, int wsh, const int64_t* er, const float4* ev,
                      const int32_t* boff, const float4* estep, int64_t n_stage, void* out, cudaStream_t st) {
  const int64_t n_tiles = (S.Q + S.W - 1) / S.W;
  const size_t smem = eval_smem<A>(S, n_stage);
  int grid = 0;
  SS_TRY(grid_for(k_pr_eval<A, OUT_REAL>, smem, n_tiles, &grid));
  k_pr_eval<A, OUT_REAL><<<grid, kPrThreads, smem, st>>>(T.M, S.P, S.Q, wsh, S.rad, table0<A>(T), table1<A>(T), T.b, er,
                                                         ev, boff, estep, (int)n_stage, n_tiles, out);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

template <class A, int P, bool OUT_REAL>
ss_status launch_eval16(const TwoLevelTable& T, const PrunedSplit& S, const int64_t* er, const float4* ev,
                        const int32_t* boff, const float4* estep, int64_t n_stage, void* out, cudaStream_t st) {
  constexpr int W = kPr16Tile / P;
  const int64_t n_tiles = (S.Q + W - 1) / W;
  const size_t smem =
      (size_t)(W * (P + 1) + P + kPrChunk + n_stage) * sizeof(typename A::V) + (P + 1) * sizeof(int32_t);
  int grid = 0;
  SS_TRY(grid_for(k_pr_eval16<A, P, OUT_REAL>, smem, n_tiles, &grid));
  k_pr_eval16<A, P, OUT_REAL><<<grid, kPr16Threads, smem, st>>>(T.M, S.Q, table0<A>(T), table1<A>(T), T.b, er, ev, boff,
                                                                 estep, (int)n_stage, n_tiles, out);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

template <class A, bool OUT_REAL>
ss_status launch_eval16_p(const TwoLevelTable& T, const PrunedSplit& S, const int64_t* er, const float4* ev,
                          const int32_t* boff, const float4* estep, int64_t n_stage, void* out, cudaStream_t st) {
  if (S.P == 256) return launch_eval16<A, 256, OUT_REAL>(T, S, er, ev, boff, estep, n_stage, out, st);
  return launch_eval16<A, 128, OUT_REAL>(T, S, er, ev, boff, estep, n_stage, out, st);
}

template <int P, bool OUT_REAL>
ss_status launch_eval_col(const TwoLevelTable& T, const PrunedSplit& S, int64_t ne_max, const int64_t* er,
                          const float4* ev, const int32_t* boff, const float4* estep, void* out, cudaStream_t st) {
  constexpr int W = kPrEvalTile / P, SUB = kPrThreads / W;
  const int64_t n_tiles = (S.Q + W - 1) / W;
  const size_t smem = (size_t)(P + ne_max * W + kPrColRounds * SUB * ne_max) * sizeof(float2);
  int grid = 0;
  SS_TRY(grid_for(k_pr_eval_col<P, OUT_REAL>, smem, (n_tiles + SUB - 1) / SUB, &grid));
  k_pr_eval_col<P, OUT_REAL><<<grid, kPrThreads, smem, st>>>(T.M, S.Q, T.t0.get(), T.t1.get(), T.b, er, ev, boff, estep,
                                                            (int)(ne_max * W), n_tiles, out);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

template <class A, int P, bool IN_REAL>
ss_status launch_fwd16(const TwoLevelTable& T, const PrunedSplit& S, const void* in, const int64_t* ob,
                       const int32_t* kout, int nc, const float4* oz, double unit, double2* X, cudaStream_t st) {
  constexpr int W = kPr16Tile / P;
  const int64_t n_tiles = (S.Q + W - 1) / W;
  const size_t smem = (size_t)(W * (P + 1) + P + nc) * sizeof(typename A::V);
  int grid = 0;
  SS_TRY(grid_for(k_pr_fwd16<A, P, IN_REAL>, smem, n_tiles, &grid));
  DevBuf<typename A::AccV> partial;
  SS_TRY(partial.alloc_tmp((size_t)grid * nc, st));
  {
    ProfScope prof_("k_pr_fwd", st, true);
    k_pr_fwd16<A, P, IN_REAL><<<grid, kPr16Threads, smem, st>>>(T.M, S.Q, table0<A>(T), table1<A>(T), T.b, in, ob, kout,
                                                                 nc, oz, n_tiles, partial.get());
    SS_LAUNCH_CHECK();
  }
  k_pr_reduce<A><<<nblk((int64_t)nc * 32), 256, 0, st>>>(partial.get(), grid, nc, unit, X);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

template <class A, bool IN_REAL>
ss_status launch_fwd16_p(const TwoLevelTable& T, const PrunedSplit& S, const void* in, const int64_t* ob,
                         const int32_t* kout, int nc, const float4* oz, double unit, double2* X, cudaStream_t st) {
  if (S.P == 256) return launch_fwd16<A, 256, IN_REAL>(T, S, in, ob, kout, nc, oz, unit, X, st);
  return launch_fwd16<A, 128, IN_REAL>(T, S, in, ob, kout, nc, oz, unit, X, st);
}

template <class A, bool IN_REAL>
ss_status launch_fwd(const TwoLevelTable& T, const PrunedSplit& S, int wsh, const PrShifts& shifts, const void* in,
                     const int64_t* ob,
                     const int32_t* kout, int nc, const float4* oz, double unit, double2* X, cudaStream_t st) {
  const int64_t n_tiles = (S.Q + S.W - 1) / S.W;
  const size_t smem = fwd_smem<A>(S, nc);
  int grid = 0;
  auto kern = k_pr_fwd<A, IN_REAL, false>;
  if constexpr (A::kFixed) {
    if (nc <= kPrThreads) kern = k_pr_fwd<A, IN_REAL, true>;
  }
  SS_TRY(grid_for(kern, smem, n_tiles, &grid));
  DevBuf<typename A::AccV> partial;
  SS_TRY(partial.alloc_tmp((size_t)grid * nc, st));
  {
    ProfScope prof_("k_pr_fwd", st, true);
    kern<<<grid, kPrThreads, smem, st>>>(T.M, S.P, S.Q, wsh, S.rad, shifts, table0<A>(T), table1<A>(T), T.b, in,
                                                         ob, kout, nc, oz, n_tiles, partial.get());
    SS_LAUNCH_CHECK();
  }
  k_pr_reduce<A><<<nblk((int64_t)nc * 32), 256, 0, st>>>(partial.get(), grid, nc, unit, X);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

// Samples stay below 2^56.5; a value enters a pass below 2^59.5 (a radix-8 sum
// then stays below 2^62.5), and 2^wsh columns add up to less than 2^60.5: the
// last pass divides for them, once per value.  Returns the sum of the shifts.
int fwd_shifts(const PrunedSplit& S, int wsh, PrShifts* out) {
  double g = -3.0;   // log2 of a value, less 59.5
  int sum = 0;
  for (int p = 0; p < S.rad.n; ++p) {
    g += std::log2((double)S.rad.r[p]);
    if (p + 1 == S.rad.n) g += wsh - 1.0;
    const int sh = g > 0.0 ? (int)std::ceil(g) : 0;
    out->pass[p] = sh;
    sum += sh;
    g -= sh;
  }
  return sum;
}

}  // namespace

ss_status two_level_table(int64_t M, bool fx, TwoLevelTable* T, cudaStream_t st) {
  int bits = 0;
  while ((1ll << bits) < M) ++bits;
  T->M = M;
  T->b = (bits + 1) / 2;
  const int64_t n0 = 1ll << T->b, n1 = (M + n0 - 1) >> T->b;
  SS_TRY(T->t0.alloc(n0, st));
  SS_TRY(T->t1.alloc(n1, st));
  k_tl_table<<<nblk(std::max(n0, n1)), 256, 0, st>>>(M, T->b, n1, T->t0.get(), T->t1.get());
  if (fx) {
    SS_TRY(T->x0.alloc(n0, st));
    SS_TRY(T->x1.alloc(n1, st));
    k_tl_table_fx<<<nblk(std::max(n0, n1)), 256, 0, st>>>(M, T->b, n1, T->x0.get(), T->x1.get());
  }
  SS_LAUNCH_CHECK();
  return SS_OK;
}

bool pruned_split(int64_t M, int64_t n, PrunedSplit* out, int tile) {
  // cost per point ~ log2 P (the transform) + n / P (the sparse side)
  double best = 1e300;
  PrunedSplit S;
  for (int P = 8; P <= kPrMaxP; ++P) {
    if (M % P || M / P < 2) continue;
    const DfRadices r = df_radices(P);
    if (r.n < 0) continue;
    const double c = std::log2((double)P) + (double)std::max<int64_t>(n, 1) / P;
    if (c < best) {
      best = c;
      S.P = P;
      S.Q = M / P;
      S.W = 1;
      while (2 * S.W * P <= tile) S.W *= 2;   // W: a power of two, W P <= tile
      S.rad = r;
    }
  }
  if (S.P == 0) return false;
  *out = S;
  return true;
}

bool pruned_supported(int64_t M) {
  int64_t m = M;
  for (int64_t p : {2, 3, 5, 7})
    while (m % p == 0) m /= p;
  PrunedSplit S;
  return m == 1 && M < (1ll << 31) && pruned_split(M, 2, &S) && S.P >= 8;
}

ss_status pruned_eval_pair(const TwoLevelTable& T, const int64_t* qa, const double2* ca, const int64_t* na_dev,
                           int64_t na_max, const int64_t* qf, const double2* cf, const int64_t* nf_dev,
                           int64_t nf_max, const double* scale, void* out, PrunedFormat fmt, cudaStream_t st) {
  const int64_t M = T.M;
  if (!qf) nf_max = 0;
  const int64_t ne_max = std::max<int64_t>(1, 2 * (na_max + nf_max));
  if (ne_max > (1ll << 30)) SS_FAIL(SS_ERR_INVALID, "pruned evaluation: too many terms");
  PrunedSplit S;
  if (!pruned_split(M, ne_max, &S, kPrEvalTile))
    SS_FAIL(SS_ERR_INVALID, "pruned evaluation: M = %lld has no split", (long long)M);
  // P = 128 or 256: 4096-value tiles (k_pr_eval16)
  const bool t16 = pr16_supported(S.P);
  const int Wt = t16 ? kPr16Tile / S.P : S.W;
  DevBuf<int64_t> er;
  DevBuf<float4> ev, estep;
  DevBuf<int32_t> boff, kq;
  SS_TRY(er.alloc_tmp(ne_max, st));
  SS_TRY(ev.alloc_tmp(ne_max, st));
  SS_TRY(boff.alloc_tmp(S.P + 1, st));
  SS_TRY(kq.alloc_tmp(ne_max, st));
  SS_TRY(estep.alloc_tmp((size_t)ne_max * Wt, st));
  {
    ProfScope prof_setup("pr_setup", st);
    const int eb = std::min(1024, (S.P + 31) / 32 * 32);
    // the entries' buckets in shared memory when they fit (48 KB with the counts)
    const int kq_smem = (int)std::min<int64_t>(ne_max, 12288 - (S.P + 1));
    const bool fx = fmt == PrunedFormat::kFxComplex;
    const auto entries = fx ? k_pr_entries<true> : k_pr_entries<false>;
    entries<<<1, eb, (S.P + 1 + kq_smem) * sizeof(int32_t), st>>>(qa, ca, na_dev, qf, cf, qf ? nf_dev : nullptr, scale,
                                                                  M, S.P, kq.get(), er.get(), ev.get(), boff.get(),
                                                                  kq_smem);
    SS_LAUNCH_CHECK();
    const auto steps = fx ? k_pr_steps<1, true> : k_pr_steps<1, false>;
    steps<<<nblk(ne_max * Wt), 256, 0, st>>>(er.get(), boff.get() + S.P, 0, Wt, M, fx ? T.x0.get() : T.t0.get(),
                                             fx ? T.x1.get() : T.t1.get(), T.b, estep.get());
    SS_LAUNCH_CHECK();
  }
  int wsh = 0;
  while ((1 << wsh) < S.W) ++wsh;
  // the entries' step powers go to shared memory once per block when they fit
  const int64_t n_stage = ne_max * Wt <= kPrEvalStage ? ne_max * Wt : 0;
  ProfScope prof_("k_pr_eval", st, true);
  if (t16) {
    switch (fmt) {
      case PrunedFormat::kFxComplex:
        return launch_eval16_p<ArFX, false>(T, S, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
      case PrunedFormat::kF64Real:
        return launch_eval16_p<ArDF, true>(T, S, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
      case PrunedFormat::kF32Complex:
        return launch_eval16_p<ArF32, false>(T, S, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
      default:
        return launch_eval16_p<ArF32, true>(T, S, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
    }
  }
  // FP32, P = 16 or 32, the step powers within shared memory: a column per
  // thread.  (FP64: a column of double-floats does not fit the registers.)
  const bool f32 = fmt == PrunedFormat::kF32Complex || fmt == PrunedFormat::kF32Real;
  if (f32 && pr_col_supported(S.P) && ne_max <= kPrColEntries && S.W == kPrEvalTile / S.P) {
    const bool real = fmt == PrunedFormat::kF32Real;
    auto go = [&](auto launch) { return launch(T, S, ne_max, er.get(), ev.get(), boff.get(), estep.get(), out, st); };
    if (S.P == 16) return real ? go(launch_eval_col<16, true>) : go(launch_eval_col<16, false>);
    return real ? go(launch_eval_col<32, true>) : go(launch_eval_col<32, false>);
  }
  switch (fmt) {
    case PrunedFormat::kFxComplex:
      return launch_eval<ArFX, false>(T, S, wsh, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
    case PrunedFormat::kF64Real:
      return launch_eval<ArDF, true>(T, S, wsh, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
    case PrunedFormat::kF32Complex:
      return launch_eval<ArF32, false>(T, S, wsh, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
    default:
      return launch_eval<ArF32, true>(T, S, wsh, er.get(), ev.get(), boff.get(), estep.get(), n_stage, out, st);
  }
}

ss_status pruned_forward(const TwoLevelTable& T, const void* s, PrunedFormat fmt, const int64_t* bins, int64_t n_out,
                         double2* X, cudaStream_t st) {
  const int64_t M = T.M;
  if (n_out < 1) return SS_OK;
  PrunedSplit S;
  if (!pruned_split(M, n_out, &S)) SS_FAIL(SS_ERR_INVALID, "pruned transform: M = %lld has no split", (long long)M);
  int wsh = 0;
  while ((1 << wsh) < S.W) ++wsh;
  const bool fx = fmt == PrunedFormat::kFxComplex, t16 = pr16_supported(S.P);   // 4096-value tiles
  double unit = 1.0;
  PrShifts shifts;
  if (fx) {   // what the passes and Horner's sums divide out
    const int sh = t16 ? 2 + kPrStoreShift : fwd_shifts(S, wsh, &shifts);
    unit = std::ldexp(1.0, sh - kPrSampleFrac);
  }
  for (int64_t o0 = 0; o0 < n_out; o0 += kPrMaxOut) {
    const int nc = (int)std::min<int64_t>(kPrMaxOut, n_out - o0);
    DevBuf<int32_t> kout;
    DevBuf<float4> oz;
    SS_TRY(kout.alloc_tmp(nc, st));
    SS_TRY(oz.alloc_tmp((size_t)nc * 2, st));
    k_pr_kout<<<nblk(nc), 256, 0, st>>>(bins + o0, nc, S.P, kout.get());
    // oz[2 o + 1] = exp(-2 pi i b_o / M): the Horner root of output o
    const auto steps = fx ? k_pr_steps<-1, true> : k_pr_steps<-1, false>;
    steps<<<nblk((int64_t)nc * 2), 256, 0, st>>>(bins + o0, nullptr, nc, 2, M, fx ? T.x0.get() : T.t0.get(),
                                                 fx ? T.x1.get() : T.t1.get(), T.b, oz.get());
    SS_LAUNCH_CHECK();
    const float4* z = oz.get() + 1;
    switch (fmt) {
      case PrunedFormat::kFxComplex:
        if (t16) SS_TRY((launch_fwd16_p<ArFX, false>(T, S, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        else SS_TRY((launch_fwd<ArFX, false>(T, S, wsh, shifts, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        break;
      case PrunedFormat::kF64Real:
        if (t16) SS_TRY((launch_fwd16_p<ArDF, true>(T, S, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        else SS_TRY((launch_fwd<ArDF, true>(T, S, wsh, shifts, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        break;
      case PrunedFormat::kF32Complex:
        if (t16) SS_TRY((launch_fwd16_p<ArF32, false>(T, S, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        else SS_TRY((launch_fwd<ArF32, false>(T, S, wsh, shifts, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        break;
      default:
        if (t16) SS_TRY((launch_fwd16_p<ArF32, true>(T, S, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        else SS_TRY((launch_fwd<ArF32, true>(T, S, wsh, shifts, s, bins + o0, kout.get(), nc, z, unit, X + o0, st)));
        break;
    }
  }
  return SS_OK;
}

}  // namespace ss
