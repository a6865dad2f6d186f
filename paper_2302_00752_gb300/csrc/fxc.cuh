// Complex fixed-point values and the small DFT kernels of the fixed-point
// transforms (fft_fx.cu: full length-M transform; fft_pruned.cu: sparse-input
// evaluation and pruned-output transform).
//
// A real part is a 64-bit integer counting units of a power of two that the
// transform fixes once, so an addition is one 64-bit addition (two integer
// instructions; a double-float addition takes eight to eleven) and rounds
// nothing: only products and scalings round, each by at most two units.  The
// transforms keep |value| <= 2^62 by construction (the bounds stand with each
// transform), which puts a unit at 2^-57 or less of the data's l1 norm: below
// the rounding of the same transform in FP64, and 2^-10 of it in double-float.
//
// Roots of unity are Q62 integers split into balanced 32-bit limbs, w = rh 2^32
// + rl with rl signed; a product keeps three of the four limb products (the low
// one is below one unit): x w / 2^62 = 4 xh wh + ((xh wl + xl wh + 2^29) >> 30),
// where each limb product is one 32 x 32 + 64 bit multiply-add.
#pragma once

#include "df.cuh"

namespace ss {
namespace fxc {

using i64 = long long;

struct CX {
  i64 re, im;
};

// Q62 root, balanced limbs.
struct TW {
  int rl, rh, il, ih;
};

__device__ __forceinline__ i64 mad(int a, int b, i64 c) {
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ i64 mulw(int a, int b) {
  i64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}

// Balanced limbs of x: x = h 2^32 + l, l signed.
__device__ __forceinline__ void split(i64 x, int& h, int& l) {
  l = (int)x;
  h = (int)((unsigned long long)(x + 0x80000000ll) >> 32);
}

// (a low limb of -2^31 has no negative: such a root moves by one unit of 2^-62,
// so that limbs of roots may be negated freely; limbs of values are not)
__device__ __forceinline__ TW to_tw(i64 re, i64 im) {
  TW w;
  split((unsigned)re == 0x80000000u ? re + 1 : re, w.rh, w.rl);
  split((unsigned)im == 0x80000000u ? im + 1 : im, w.ih, w.il);
  return w;
}
__device__ __forceinline__ TW ld_tw(const int4 v) { return TW{v.x, v.y, v.z, v.w}; }
__device__ __forceinline__ int4 st_tw(const TW w) { return make_int4(w.rl, w.rh, w.il, w.ih); }
__device__ __forceinline__ TW conj(const TW w) { return TW{w.rl, w.rh, -w.il, -w.ih}; }

__device__ __forceinline__ CX ld(const longlong2 v) { return CX{v.x, v.y}; }
__device__ __forceinline__ longlong2 st(const CX c) { return make_longlong2(c.re, c.im); }
__device__ __forceinline__ CX add(const CX a, const CX b) { return CX{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ CX sub(const CX a, const CX b) { return CX{a.re - b.re, a.im - b.im}; }
template <int SIGN>
__device__ __forceinline__ CX mul_si(const CX a) {   // a * (sign i)
  return SIGN > 0 ? CX{-a.im, a.re} : CX{a.im, -a.re};
}

constexpr i64 kHalf = 1ll << 29;   // rounds the middle limbs' shift to nearest

// x c, c real Q62 (limbs ch, cl)
__device__ __forceinline__ i64 rmul(i64 x, int ch, int cl) {
  int h, l;
  split(x, h, l);
  const i64 m = mad(h, cl, mad(l, ch, kHalf));
  return (mulw(h, ch) << 2) + (m >> 30);
}

// a w.  |a| <= 2^62: the high products stay below 2^60 (2^62 shifted), the middle
// ones add up to sqrt 2 (2^31 2^30 + 2^30 2^31) < 2^63.
__device__ __forceinline__ CX mul(const CX a, const TW w) {
  int ah, al, bh, bl;
  split(a.re, ah, al);
  split(a.im, bh, bl);
  const int nh = -w.ih, nl = -w.il;
  const i64 hr = mad(bh, nh, mulw(ah, w.rh)), hi = mad(bh, w.rh, mulw(ah, w.ih));
  const i64 mr = mad(bl, nh, mad(bh, nl, mad(al, w.rh, mad(ah, w.rl, kHalf))));
  const i64 mi = mad(bl, w.rh, mad(bh, w.rl, mad(al, w.ih, mad(ah, w.il, kHalf))));
  return CX{(hr << 2) + (mr >> 30), (hi << 2) + (mi >> 30)};
}

// a w / 4, where the caller has the range to spare: the middle products' high
// words are added as they are (14 integer instructions less per product).
__device__ __forceinline__ CX mulq(const CX a, const TW w) {
  constexpr i64 half = 1ll << 31;
  int ah, al, bh, bl;
  split(a.re, ah, al);
  split(a.im, bh, bl);
  const int nh = -w.ih, nl = -w.il;
  const i64 hr = mad(bh, nh, mulw(ah, w.rh)), hi = mad(bh, w.rh, mulw(ah, w.ih));
  const i64 mr = mad(bl, nh, mad(bh, nl, mad(al, w.rh, mad(ah, w.rl, half))));
  const i64 mi = mad(bl, w.rh, mad(bh, w.rl, mad(al, w.ih, mad(ah, w.il, half))));
  return CX{mad((int)(mr >> 32), 1, hr), mad((int)(mi >> 32), 1, hi)};
}

template <int SIGN>
__device__ __forceinline__ CX mul_t(const CX a, const TW w) {   // a w or a conj(w)
  return mul(a, SIGN > 0 ? w : conj(w));
}

template <int SIGN>
__device__ __forceinline__ void dft4(CX& v0, CX& v1, CX& v2, CX& v3) {
  const CX t0 = add(v0, v2), t1 = sub(v0, v2), t2 = add(v1, v3), t3 = mul_si<SIGN>(sub(v1, v3));
  v0 = add(t0, t2);
  v2 = sub(t0, t2);
  v1 = add(t1, t3);
  v3 = sub(t1, t3);
}

// a exp(sign i pi / 4) and a exp(sign 3 i pi / 4), w8 = exp(2 pi i / 8)
template <int SIGN>
__device__ __forceinline__ CX mul_w8(const CX a, const TW w8) {
  const i64 x = SIGN > 0 ? a.re - a.im : a.re + a.im, y = SIGN > 0 ? a.im + a.re : a.im - a.re;
  return CX{rmul(x, w8.rh, w8.rl), rmul(y, w8.rh, w8.rl)};
}

// 16-point DFT in place; the output X[k1 + 4 k2] ends at v[4 k1 + k2].  w1, w2,
// w3 = exp(2 pi i j / 16).
template <int SIGN>
__device__ __forceinline__ void dft16(CX (&v)[16], const TW w1, const TW w2, const TW w3) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4<SIGN>(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
  v[5] = mul_t<SIGN>(v[5], w1);
  v[9] = mul_w8<SIGN>(v[9], w2);
  v[13] = mul_t<SIGN>(v[13], w3);
  v[6] = mul_w8<SIGN>(v[6], w2);
  v[10] = mul_si<SIGN>(v[10]);
  v[14] = mul_si<SIGN>(mul_w8<SIGN>(v[14], w2));   // w16^6 = i w16^2
  v[7] = mul_t<SIGN>(v[7], w3);
  v[11] = mul_si<SIGN>(mul_w8<SIGN>(v[11], w2));
  {
    const CX t = mul_t<SIGN>(v[15], w1);   // w16^9 = -w16^1
    v[15] = CX{-t.re, -t.im};
  }
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4<SIGN>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
}

// p = s1 x + s2 y, q = s2 x - s1 y with the sines of w1 and w2 (radix 5)
__device__ __forceinline__ void rot5(i64 x, i64 y, const TW w1, const TW w2, i64& p, i64& q) {
  int xh, xl, yh, yl;
  split(x, xh, xl);
  split(y, yh, yl);
  const i64 mp = mad(yl, w2.ih, mad(yh, w2.il, mad(xl, w1.ih, mad(xh, w1.il, kHalf))));
  p = (mad(yh, w2.ih, mulw(xh, w1.ih)) << 2) + (mp >> 30);
  const int nh = -w1.ih, nl = -w1.il;
  const i64 mq = mad(yl, nh, mad(yh, nl, mad(xl, w2.ih, mad(xh, w2.il, kHalf))));
  q = (mad(yh, nh, mulw(xh, w2.ih)) << 2) + (mq >> 30);
}

// R-point DFT in place; cs[m - 1] = exp(2 pi i m / R) (unconjugated), m <= (R - 1) / 2,
// and for R = 8 cs[0] = exp(2 pi i / 8).  Odd R: the symmetric form
// y_s = v_0 + sum_r cos(2 pi r s / R) (v_r + v_{R-r}) + sign i sin(2 pi r s / R) (v_r - v_{R-r}).
template <int R, int SIGN>
__device__ __forceinline__ void dft(CX (&v)[R], const TW* cs) {
  if constexpr (R == 1) {
  } else if constexpr (R == 2) {
    const CX a = v[0];
    v[0] = add(a, v[1]);
    v[1] = sub(a, v[1]);
  } else if constexpr (R == 4) {
    dft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    CX e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<SIGN>(e0, e1, e2, e3);
    dft4<SIGN>(o0, o1, o2, o3);
    o1 = mul_w8<SIGN>(o1, cs[0]);
    o2 = mul_si<SIGN>(o2);
    o3 = mul_si<SIGN>(mul_w8<SIGN>(o3, cs[0]));   // w8^3 = i w8
    v[0] = add(e0, o0);
    v[4] = sub(e0, o0);
    v[1] = add(e1, o1);
    v[5] = sub(e1, o1);
    v[2] = add(e2, o2);
    v[6] = sub(e2, o2);
    v[3] = add(e3, o3);
    v[7] = sub(e3, o3);
  } else if constexpr (R == 3) {
    // cos 120 = -1/2: halves to even (a one-sided rounding would add up in the
    // bins that all butterflies feed alike), one product per part
    const CX t = add(v[1], v[2]), d = sub(v[1], v[2]);
    auto half = [](i64 x) { return (x + ((x >> 1) & 1)) >> 1; };
    const CX m = CX{v[0].re - half(t.re), v[0].im - half(t.im)};
    const CX b = mul_si<SIGN>(CX{rmul(d.re, cs[0].ih, cs[0].il), rmul(d.im, cs[0].ih, cs[0].il)});
    v[0] = add(v[0], t);
    v[1] = add(m, b);
    v[2] = sub(m, b);
  } else if constexpr (R == 5) {
    // cos and sin of 72 and 144 degrees; (cos72 + cos144) / 2 = -1/4 exactly, so
    // the real parts need one product, by (cos72 - cos144) / 2 = sqrt 5 / 4
    constexpr i64 kC = 0x23C6EF372FE94F82ll;   // round(2^62 sqrt 5 / 4)
    const int ch = (int)((kC + 0x80000000ll) >> 32), cl = (int)kC;
    const TW w1 = cs[0], w2 = cs[1];
    const CX a1 = add(v[1], v[4]), b1 = sub(v[1], v[4]), a2 = add(v[2], v[3]), b2 = sub(v[2], v[3]);
    const CX t = add(a1, a2), u = sub(a1, a2);
    const CX m1 = CX{v[0].re - (t.re >> 2), v[0].im - (t.im >> 2)};
    const CX m2 = CX{rmul(u.re, ch, cl), rmul(u.im, ch, cl)};
    v[0] = add(v[0], t);
    const CX A1 = add(m1, m2), A2 = sub(m1, m2);
    CX B1, B2;
    rot5(b1.re, b2.re, w1, w2, B1.re, B2.re);
    rot5(b1.im, b2.im, w1, w2, B1.im, B2.im);
    const CX i1 = mul_si<SIGN>(B1), i2 = mul_si<SIGN>(B2);
    v[1] = add(A1, i1);
    v[4] = sub(A1, i1);
    v[2] = add(A2, i2);
    v[3] = sub(A2, i2);
  } else if constexpr (R == 10) {
    // coprime factors 2 and 5 (no twiddles): n = 5 a + 2 b, and k mod 2, k mod 5
    // pick X[k] = sum_b w5^(b k) sum_a (-1)^(a k) x[5 a + 2 b]; cs: as for R = 5
    CX e[5], o[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) {
      e[b] = add(v[2 * b], v[(2 * b + 5) % 10]);
      o[b] = sub(v[2 * b], v[(2 * b + 5) % 10]);
    }
    dft<5, SIGN>(e, cs);
    dft<5, SIGN>(o, cs);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      v[(6 * k) % 10] = e[k];
      v[(6 * k + 5) % 10] = o[k];
    }
  } else {
    constexpr int H = (R - 1) / 2;
    CX a[H], b[H];
#pragma unroll
    for (int r = 1; r <= H; ++r) {
      a[r - 1] = add(v[r], v[R - r]);
      b[r - 1] = sub(v[r], v[R - r]);
    }
    const CX v0 = v[0];
    // limbs of a and b once; products with the H cosines and sines
    int ah[H][2], al[H][2], bh[H][2], bl[H][2];
#pragma unroll
    for (int r = 0; r < H; ++r) {
      split(a[r].re, ah[r][0], al[r][0]);
      split(a[r].im, ah[r][1], al[r][1]);
      split(b[r].re, bh[r][0], bl[r][0]);
      split(b[r].im, bh[r][1], bl[r][1]);
      v[0] = add(v[0], a[r]);
    }
#pragma unroll
    for (int s = 1; s <= H; ++s) {
      CX A, B;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        i64 hc = 0, mc = kHalf, hs = 0, ms = kHalf;
#pragma unroll
        for (int r = 1; r <= H; ++r) {
          const int m = (r * s) % R;
          const int mm = m <= H ? m : R - m;
          const TW w = cs[mm - 1];
          const int sh = m <= H ? w.ih : -w.ih, sl = m <= H ? w.il : -w.il;
          hc = mad(ah[r - 1][p], w.rh, hc);
          mc = mad(ah[r - 1][p], w.rl, mad(al[r - 1][p], w.rh, mc));
          hs = mad(bh[r - 1][p], sh, hs);
          ms = mad(bh[r - 1][p], sl, mad(bl[r - 1][p], sh, ms));
        }
        (p ? A.im : A.re) = (p ? v0.im : v0.re) + (hc << 2) + (mc >> 30);
        (p ? B.im : B.re) = (hs << 2) + (ms >> 30);
      }
      const CX iB = mul_si<SIGN>(B);
      v[s] = add(A, iB);
      v[R - s] = sub(A, iB);
    }
  }
}

// a / 2^s, rounded to nearest
__device__ __forceinline__ CX scale_down(const CX a, int s) {
  const i64 h = s > 0 ? 1ll << (s - 1) : 0;
  return CX{(a.re + h) >> s, (a.im + h) >> s};
}

// exp(2 pi i r / M) in units of 2^-62, to about one unit (FP64's 2^-54 would
// stand above the transforms' own rounding): the angle reduced to [0, pi/4] by
// integers, the series in pairs of doubles.
struct D2 {
  double h, l;
};
__device__ __forceinline__ D2 d2_norm(double h, double l) {
  const double s = h + l;
  return D2{s, l - (s - h)};
}
__device__ __forceinline__ D2 d2_mul(const D2 a, const D2 b) {
  const double p = a.h * b.h;
  return d2_norm(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ D2 d2_div(const D2 a, double n) {
  const double q = a.h / n;
  return d2_norm(q, (fma(-q, n, a.h) + a.l) / n);
}
__device__ __forceinline__ D2 d2_one_minus(const D2 a) {
  const double s = 1.0 - a.h;   // |a| < 1
  return d2_norm(s, (1.0 - s) - a.h - a.l);
}
__device__ inline long long d2_q62(const D2 a) {
  const double x = a.h * 0x1p62, y = rint(x);
  return (long long)y + __double2ll_rn((x - y) + a.l * 0x1p62);
}
__device__ inline TW exact_root(int64_t r, int64_t M) {
  const int64_t q = 8 * r / M, rem = 8 * r - q * M, y = q & 1 ? M - rem : rem;
  const double t = (double)y / (double)M, m = (double)M;
  const D2 x = d2_mul(D2{0.78539816339744830962, 3.0616169978683830e-17}, D2{t, fma(-t, m, (double)y) / m});
  const D2 x2 = d2_mul(x, x);
  D2 c{1.0, 0.0}, sn{1.0, 0.0};
  for (int k = 12; k > 0; --k) {   // x^26 / 26! < 2^-95
    c = d2_one_minus(d2_div(d2_mul(x2, c), (double)((2 * k - 1) * (2 * k))));
    sn = d2_one_minus(d2_div(d2_mul(x2, sn), (double)((2 * k) * (2 * k + 1))));
  }
  sn = d2_mul(x, sn);
  long long a = d2_q62(c), b = d2_q62(sn);   // octant 0
  if ((q + 1) & 2) {                         // octants 1, 2, 5, 6: nearer to the imaginary axis
    const long long v = a;
    a = b;
    b = v;
  }
  if (q >= 2 && q <= 5) a = -a;
  if (q >= 4) b = -b;
  return to_tw(a, b);
}

}  // namespace fxc
}  // namespace ss
