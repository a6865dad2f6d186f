// Monte Carlo form of the proxy error (Lemma ProxyError; Section "Code and
// testing overview"): r(x) = f(x) - f^{s,N}(x) at uniform random points of
// T^d, with f^{s,N} = L[a_hat] u^{s,N} known through its coefficients on
// S^{N+1} (Proposition LExpansion).  The work is a dense trigonometric sum of
// |terms| x |points| cosines.
//
// Points lie on the grid (2^-32 Z)^d, so the phase k.x mod 1 of every term is
// the exact integer (k.X mod 2^32) / 2^32, formed with wrapping 32-bit
// multiply-adds.  A term is Re(c exp(2 pi i k.x)) = |c| cos(2 pi (k.x + phi)):
// the argument phi of c joins the phase (32 bits as an integer, the rest as a
// float), so that no complex product is left.  On a symmetric set the terms k
// and -k are one, with c_k + conj(c_-k): half the terms.
//
// The cosine comes from one table entry h (2^13 of them on half a turn, cos and
// sin as double-floats, 128 KB of shared memory; the phase's top bit is the
// sign) and the rest delta, |delta| <= pi / 2^14 = 1.9e-4:
//   cos(h + delta) = cos h (1 - delta^2/2) - sin h (delta - delta^3/6)
// (next terms: 6e-17, 2e-21).  The bracket's excess over 1 is below 1.9e-8, so
// FP32 holds it to 1e-15; the sine is a double-float product.  The sum is a
// double-float, renormalised every other term.
//
// Bound: instruction issue (about 55 per term and point) beside the table's
// gathers (random 16-byte reads, about 10 shared-memory cycles per warp) and
// their latency.  d = 10, 330,000 frequencies, 1000 points: 308 us; three
// table entries and double-float complex products per term, without the
// pairing: 3.7 ms.  The error against 64 bits is two thirds of that one's.
#include <algorithm>

#include "df.cuh"
#include "keys.cuh"
#include "ss_internal.cuh"

namespace ss {
namespace {

constexpr int kMcThreads = 512;
// Points per thread, which share the term's loads: as many as the registers
// hold beside their coordinates (d = 10, 330,000 frequencies, 1000 points, the whole call: 393 us with
// four, 451 with two).
__host__ __device__ constexpr int mc_pts(int d) { return d <= 10 ? 4 : 2; }
constexpr int kTabBits = 13;
constexpr int kTab = 1 << kTabBits;      // (cos, sin)(pi h / 2^13)
constexpr int kRest = 31 - kTabBits;     // bits of the phase below the table's
constexpr size_t kTabBytes = kTab * sizeof(float4);
constexpr int kMcRegDims = 16;           // coordinates of a point kept in registers
constexpr double kTurn = 6.283185307179586 / 4294967296.0;   // radians per unit of the phase

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

__global__ void k_mc_tables(float4* tab) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kTab) return;
  double s, c;
  sincospi((double)i / kTab, &s, &c);      // the quotient is exact
  const DF cc = df_split(c), ss_ = df_split(s);
  tab[i] = make_float4(cc.hi, cc.lo, ss_.hi, ss_.lo);
}

// Head of a term's record: |c| as a double-float, arg c / 2 pi in units of
// 2^-32 (plus half a table step, so that the table index rounds), and the rest
// of arg c in radians.  The argument is the table's nearest angle plus a small
// one, tan = im / re after the turn back; what that does not cover (zero,
// floats out of range, not finite) goes through atan2 and hypot.
__device__ int4 term_head(double2 c, const float4* __restrict__ tab) {
  const int h = (int)rintf(atan2f((float)c.y, (float)c.x) * (float)(kTab / 3.141592653589793)) & (2 * kTab - 1);
  const float4 e = tab[h & (kTab - 1)];
  const double sg = h < kTab ? 1.0 : -1.0, er = sg * ((double)e.x + (double)e.y), ei = sg * ((double)e.z + (double)e.w);
  const double re = c.x * er + c.y * ei, im = c.y * er - c.x * ei;
  const double t = im / re, t2 = t * t;
  double mag, turn;   // turn: in units of 2^-32
  if (re > 0.0 && t2 < 1e-6) {
    mag = re * (1.0 + t2 * (0.5 + t2 * -0.125));
    turn = (double)((int64_t)h << kRest) + t * (1.0 + t2 * (-1.0 / 3.0 + t2 * 0.2)) / kTurn;
  } else {
    mag = hypot(c.x, c.y);
    turn = atan2(c.y, c.x) / kTurn;
    if (!isfinite(turn)) turn = 0.0;
  }
  const double n = rint(turn);
  const DF m = df_split(mag);
  return make_int4(__float_as_int(m.hi), __float_as_int(m.lo),
                   (int)(uint32_t)((int64_t)n + (1ll << (kRest - 1))), __float_as_int((float)((turn - n) * kTurn)));
}

// Records of f's terms: head, then the d coordinates, zero padded to w int4s.
__global__ void k_mc_recs_f(const int32_t* __restrict__ freq, const double2* __restrict__ coef, int64_t n, int d, int w,
                            const float4* __restrict__ tab, int4* __restrict__ rec) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  int4* o = rec + t * w;
  o[0] = term_head(coef[t], tab);
  auto k = [&](int c) { return c < d ? freq[t * d + c] : 0; };
  for (int c = 0; c + 1 < w; ++c) o[c + 1] = make_int4(k(4 * c), k(4 * c + 1), k(4 * c + 2), k(4 * c + 3));
}

// Records of -f^{s,N} from its coefficients y on S: row t, or (plus, mirror:
// the set is symmetric) the row plus[t] together with its mirror image.
__global__ void k_mc_recs_g(KeyParams P, const uint64_t* __restrict__ keys, const double2* __restrict__ y, int64_t n,
                            const int32_t* __restrict__ plus, const int64_t* __restrict__ mirror, int w,
                            const float4* __restrict__ tab, int4* __restrict__ rec) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int64_t g = plus ? plus[t] : t;
  double2 c = y[g];
  if (plus) {
    const double2 m = y[mirror[g]];
    c = make_double2(c.x + m.x, c.y - m.y);
  }
  int4* o = rec + t * w;
  o[0] = term_head(make_double2(-c.x, -c.y), tab);
  const uint64_t* key = keys + g * P.WT;
  auto k = [&](int c) { return c < P.d ? unpack_coord(key, P, c) : 0; };
  for (int c = 0; c + 1 < w; ++c) o[c + 1] = make_int4(k(4 * c), k(4 * c + 1), k(4 * c + 2), k(4 * c + 3));
}

// Points [Q][d] -> [(d + 3) / 4][Q] of four coordinates, zero padded (more
// coordinates than the registers hold: read along q).
__global__ void k_mc_points(const uint32_t* __restrict__ X, int64_t Q, int d, int w, uint4* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Q * w) return;
  const int64_t q = i % Q;
  const int c = 4 * (int)(i / Q);
  auto x = [&](int j) { return j < d ? X[q * d + j] : 0u; };
  out[i] = make_uint4(x(c), x(c + 1), x(c + 2), x(c + 3));
}

// acc += |c| cos(2 pi ph / 2^32 + rest); ph includes half a table step.
__device__ __forceinline__ void add_term(DF& acc, const int4 head, uint32_t ph, const float4* __restrict__ s_tab) {
  const float4 e = s_tab[(ph >> kRest) & (kTab - 1)];
  const uint32_t sign = ph & 0x80000000u;
  const float mh = __int_as_float(head.x ^ (int)sign), ml = __int_as_float(head.y ^ (int)sign);
  // the low bits as a float: put into the mantissa of 2^23, which is taken off again
  const float r = __fsub_rn(__int_as_float(0x4b000000 | (int)(ph & ((1u << kRest) - 1))),
                            8388608.f + (float)(1 << (kRest - 1)));
  constexpr float kh = (float)kTurn, kl = (float)(kTurn - (double)kh);
  const float dh = __fmul_rn(r, kh);
  const float dl = __fadd_rn(__fmaf_rn(r, kh, -dh), __fmaf_rn(r, kl, __int_as_float(head.w)));
  const float d2 = __fmul_rn(dh, dh);
  const float sl = __fmaf_rn(dh, __fmul_rn(d2, -1.f / 6.f), dl);              // sin(delta) = dh + sl
  const float cm = __fmul_rn(dh, __fmaf_rn(dh, -0.5f, -dl));                  // cos(delta) - 1
  const float v = __fmul_rn(e.z, dh);
  float ve = __fmaf_rn(e.z, dh, -v);
  ve = __fmaf_rn(e.z, sl, ve);
  ve = __fmaf_rn(e.w, dh, ve);
  // |cos h| is 0 or at least 3.8e-4 > |v|: FastTwoSum (Dekker)
  const float s = __fsub_rn(e.x, v);
  float lo = __fsub_rn(__fsub_rn(e.x, s), v);
  lo = __fadd_rn(__fsub_rn(lo, ve), __fmaf_rn(cm, e.x, e.y));
  const float p = __fmul_rn(mh, s);
  float pe = __fmaf_rn(mh, s, -p);
  pe = __fmaf_rn(mh, lo, pe);
  pe = __fmaf_rn(ml, s, pe);
  const float a = __fadd_rn(acc.hi, p);
  const float bb = __fsub_rn(a, acc.hi);
  const float t = __fadd_rn(__fsub_rn(acc.hi, __fsub_rn(a, bb)), __fsub_rn(p, bb));
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t, pe));
  acc.hi = a;
}

__device__ __forceinline__ void renorm(DF& a) {
  const float h = __fadd_rn(a.hi, a.lo);
  a.lo = __fsub_rn(a.lo, __fsub_rn(h, a.hi));
  a.hi = h;
}

struct McWork {
  const int4* rec;          // n records of w int4s, f's n_f first
  int64_t n_f, n;
  int w, d;
  const uint32_t* X;        // [Q][d]
  const uint4* Xt;          // [w - 1][Q] (d > kMcRegDims)
  int64_t Q;
  const float4* tab;
  // Units: tiles of mc_pts(d) qt points times chunks of L terms (f's chunks first);
  // the threads of a block are `groups` rows of qt, each row with its share of
  // the chunk's terms.
  int qt, groups;
  int64_t tiles, L, chunks_f, chunks;
  double* part;             // [chunks * groups][Q]
};

// D: coordinates read, rounded up to an even number; 0: any number, points in Xt.
template <int D>
__global__ void __launch_bounds__(kMcThreads, 1) k_mc_terms(const McWork W) {
  extern __shared__ float4 s_tab[];
  for (int i = threadIdx.x; i < kTab; i += kMcThreads) s_tab[i] = __ldg(W.tab + i);
  __syncthreads();
  const int row = threadIdx.x / W.qt, col = threadIdx.x % W.qt;
  if (row >= W.groups) return;
  constexpr int NK = D ? (D + 3) / 4 : 1, kMcPts = mc_pts(D ? D : kMcRegDims + 1);
  for (int64_t u = blockIdx.x; u < W.tiles * W.chunks; u += gridDim.x) {
    const int64_t chunk = u / W.tiles, q0 = (u % W.tiles) * kMcPts * W.qt + col;
    const bool g = chunk >= W.chunks_f;
    const int64_t b0 = (g ? W.n_f : 0) + (chunk - (g ? W.chunks_f : 0)) * W.L;
    const int64_t b1 = min(b0 + W.L, g ? W.n : W.n_f), share = (b1 - b0 + W.groups - 1) / W.groups;
    const int64_t t0 = min(b0 + row * share, b1), t1 = min(t0 + share, b1);
    int64_t q[kMcPts];
    uint32_t x[kMcPts][D ? D : 1];
    DF acc[kMcPts];
#pragma unroll
    for (int j = 0; j < kMcPts; ++j) {
      q[j] = q0 + j * W.qt;
      acc[j] = DF{0.f, 0.f};
      if (D) {
#pragma unroll
        for (int c = 0; c < (D ? D : 1); ++c) x[j][c] = q[j] < W.Q && c < W.d ? __ldg(W.X + q[j] * W.d + c) : 0u;
      }
    }
    // the next record is on its way while a term is worked on
    const int4* rec = W.rec + t0 * W.w;
    int4 cur[NK + 1], nxt[NK + 1];
    auto fetch = [&](int4* v, bool go) {
      if (!go) return;
#pragma unroll
      for (int c = 0; c < (D ? NK + 1 : 1); ++c) v[c] = __ldg(rec + c);
      rec += W.w;
    };
    auto term = [&](const int4* v, const int4* k0) {
      uint32_t ph[kMcPts];
#pragma unroll
      for (int j = 0; j < kMcPts; ++j) ph[j] = (uint32_t)v[0].z;
      if (D) {
#pragma unroll
        for (int c = 0; c < NK; ++c) {
          const int kk[4] = {v[c + 1].x, v[c + 1].y, v[c + 1].z, v[c + 1].w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (4 * c + e < D) {
#pragma unroll
              for (int j = 0; j < kMcPts; ++j) ph[j] += (uint32_t)kk[e] * x[j][(D ? 4 * c + e : 0) % (D ? D : 1)];
            }
        }
      } else {
        for (int c = 0; c + 1 < W.w; ++c) {
          const int4 k = __ldg(k0 + c);
          if ((k.x | k.y | k.z | k.w) == 0) continue;   // long frequencies have few nonzeros
#pragma unroll
          for (int j = 0; j < kMcPts; ++j) {
            const uint4 p = __ldg(W.Xt + c * W.Q + min(q[j], W.Q - 1));
            ph[j] += (uint32_t)k.x * p.x + (uint32_t)k.y * p.y + (uint32_t)k.z * p.z + (uint32_t)k.w * p.w;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kMcPts; ++j) add_term(acc[j], v[0], ph[j], s_tab);
    };
    fetch(cur, t0 < t1);
    for (int64_t t = t0; t < t1; t += 2) {
      fetch(nxt, t + 1 < t1);
      term(cur, W.rec + t * W.w + 1);
      if (t + 1 < t1) {
        fetch(cur, t + 2 < t1);
        term(nxt, W.rec + (t + 1) * W.w + 1);
      }
#pragma unroll
      for (int j = 0; j < kMcPts; ++j) renorm(acc[j]);
    }
#pragma unroll
    for (int j = 0; j < kMcPts; ++j)
      if (q[j] < W.Q) W.part[(chunk * W.groups + row) * W.Q + q[j]] = (double)acc[j].hi + (double)acc[j].lo;
  }
}

// f[q] = sum of the first n_f rows of part, r[q] = f[q] + the others (which
// hold -f^{s,N}).  32 points a block, their rows dealt out to the warps, as many
// as there are rows (the whole call at 300,000 points and 6 frequencies: 381 us
// with 32 warps always, 280 so);
// the order of the additions depends on the sizes alone.
constexpr int kFinWarps = 32;
__global__ void __launch_bounds__(32 * kFinWarps) k_mc_finish(const double* __restrict__ part, int64_t n_f, int64_t n,
                                                              int64_t Q, double* __restrict__ r,
                                                              double* __restrict__ f) {
  __shared__ double sf[kFinWarps][32], sg[kFinWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t q = (int64_t)blockIdx.x * 32 + lane;
  double a = 0.0, b = 0.0;
  if (q < Q) {
    for (int64_t c = w; c < n_f; c += nw) a += part[c * Q + q];
#pragma unroll 4
    for (int64_t c = n_f + w; c < n; c += nw) b += part[c * Q + q];
  }
  sf[w][lane] = a;
  sg[w][lane] = b;
  __syncthreads();
  if (w || q >= Q) return;
  for (int i = 1; i < nw; ++i) a += sf[i][lane], b += sg[i][lane];
  f[q] = a;
  r[q] = a + b;
}

using McKernel = void (*)(McWork);

McKernel mc_kernel(int d) {
  switch (d > kMcRegDims ? 0 : (d + 1) / 2) {
    case 1: return k_mc_terms<2>;
    case 2: return k_mc_terms<4>;
    case 3: return k_mc_terms<6>;
    case 4: return k_mc_terms<8>;
    case 5: return k_mc_terms<10>;
    case 6: return k_mc_terms<12>;
    case 7: return k_mc_terms<14>;
    case 8: return k_mc_terms<16>;
  }
  return k_mc_terms<0>;
}

// The tiles and chunks: every block (one per SM, the table fills its shared
// memory) gets the same number of equal units where there are few tiles, about
// eight units each where there are many.  Fewer than kMcMinTerms terms do not
// pay for a row of threads of their own, unless that leaves fewer units than SMs
// (few terms at many points): then the tiles take fewer points and the rows few
// terms (the whole call at 56 frequencies, 3000 points, d = 10: 169 -> 129 us).
constexpr int64_t kMcMinTerms = 32;
void mc_split(McWork* W) {
  const int64_t sm = sm_count(), n_g = W->n - W->n_f, pts = mc_pts(W->d);
  W->qt = (int)std::min<int64_t>(kMcThreads, (((W->Q + pts - 1) / pts + 31) / 32) * 32);
  W->groups = kMcThreads / W->qt;
  W->tiles = (W->Q + pts * W->qt - 1) / (pts * W->qt);
  const int64_t want = W->tiles <= sm / 8 ? sm / W->tiles : (8 * sm + W->tiles - 1) / W->tiles;
  W->L = std::max<int64_t>((W->n + want - 1) / want, kMcMinTerms * W->groups);
  const bool few = W->L > (W->n + want - 1) / want;
  auto chunks = [&](int64_t n) { return (n + W->L - 1) / W->L; };
  while (chunks(W->n_f) + chunks(n_g) > std::max<int64_t>(want, 2)) W->L += W->L / 64 + 1;
  W->chunks_f = chunks(W->n_f);
  W->chunks = W->chunks_f + chunks(n_g);
  if (few && W->tiles * W->chunks < sm) {
    const int64_t tiles = (sm + W->chunks - 1) / W->chunks, qt = (W->Q + tiles * pts - 1) / (tiles * pts);
    W->qt = (int)std::min<int64_t>(W->qt, std::max<int64_t>(32, (qt + 31) / 32 * 32));
    W->groups = kMcThreads / W->qt;
    W->tiles = (W->Q + pts * W->qt - 1) / (pts * W->qt);
  }
}

}  // namespace
}  // namespace ss

using namespace ss;

extern "C" ss_status proxy_mc(ss_stamp s, const double* u_prefix, int64_t n_u, const ss_trig* f, const uint32_t* X,
                              int64_t Q, double* r_out, double* f_out, void* stream) {
  if (!s || !f || (n_u > 0 && !u_prefix) || (Q > 0 && (!X || !r_out || !f_out)))
    SS_FAIL(SS_ERR_INVALID, "proxy_mc: null argument");
  if (f->d != s->d) SS_FAIL(SS_ERR_INVALID, "proxy_mc: dimension %d != %d", f->d, s->d);
  if (n_u < 0 || n_u > s->size) SS_FAIL(SS_ERR_INVALID, "proxy_mc: n_u = %lld outside [0, |S|]", (long long)n_u);
  if (Q < 0 || f->n_terms < 0 || (f->n_terms > 0 && (!f->freq || !f->coef)))
    SS_FAIL(SS_ERR_INVALID, "proxy_mc: bad sizes");
  if (Q == 0) return SS_OK;
  const McKernel kern = mc_kernel(s->d);
  SS_TRY(allow_smem(kern));
  cudaStream_t st = as_stream(stream);
  DevBuf<float4> tab;
  DevBuf<int4> rec;
  DevBuf<uint4> Xt;
  DevBuf<double2> y;
  DevBuf<double> part;
  SS_TRY(tab.alloc(kTab, st));
  k_mc_tables<<<nblk(kTab), 256, 0, st>>>(tab.get());
  SS_LAUNCH_CHECK();
  // f^{s,N} on S: L applied to u (prefix).  A symmetric set (the half system
  // stands, its error words read) gives one term per pair +-k; k = 0 has the
  // coefficient 0 there (below).
  const bool fold = s->half_ok && !s->check_pending;
  const int64_t n_g = fold ? s->n_plus : s->size;
  McWork W{};
  W.n_f = f->n_terms;
  W.n = f->n_terms + n_g;
  W.w = 1 + (s->d + 3) / 4;
  W.d = s->d;
  W.X = X;
  W.Q = Q;
  W.tab = tab.get();
  if (s->d > kMcRegDims) {
    SS_TRY(Xt.alloc((size_t)Q * (W.w - 1), st));
    k_mc_points<<<nblk(Q * (W.w - 1)), 256, 0, st>>>(X, Q, s->d, W.w - 1, Xt.get());
    SS_LAUNCH_CHECK();
    W.Xt = Xt.get();
  }
  SS_TRY(rec.alloc((size_t)std::max<int64_t>(W.n, 1) * W.w, st));
  W.rec = rec.get();
  if (W.n_f > 0) {
    k_mc_recs_f<<<nblk(W.n_f), 256, 0, st>>>(f->freq, reinterpret_cast<const double2*>(f->coef), W.n_f, s->d, W.w,
                                             tab.get(), rec.get());
    SS_LAUNCH_CHECK();
  }
  if (n_g > 0) {
    SS_TRY(y.alloc(s->size, st));
    SS_TRY(launch_apply64(s, reinterpret_cast<const double2*>(u_prefix), n_u, y.get(), st));
    // (L u)_0 = 0 exactly for the diffusion operator (the factor k.l); its
    // stored identity row is for the solve
    if (identity_row(s) >= 0) SS_CUDA(cudaMemsetAsync(y.get() + identity_row(s), 0, sizeof(double2), st));
    k_mc_recs_g<<<nblk(n_g), 256, 0, st>>>(make_key_params(s->key), s->keys.get(), y.get(), n_g,
                                           fold ? s->plus_rows.get() : nullptr, fold ? s->mirror.get() : nullptr, W.w,
                                           tab.get(), rec.get() + W.n_f * W.w);
    SS_LAUNCH_CHECK();
  }
  if (W.n > 0) {
    mc_split(&W);
    SS_TRY(part.alloc((size_t)(W.chunks * W.groups) * Q, st));
    W.part = part.get();
    kern<<<(unsigned)std::min<int64_t>(sm_count(), W.tiles * W.chunks), kMcThreads, kTabBytes, st>>>(W);
    SS_LAUNCH_CHECK();
  }
  const int64_t rows_f = W.chunks_f * W.groups, rows = W.chunks * W.groups;
  const int fw = (int)std::max<int64_t>(1, std::min<int64_t>(kFinWarps, std::max(rows_f, rows - rows_f)));
  k_mc_finish<<<nblk(Q, 32), 32 * fw, 0, st>>>(part.get(), rows_f, rows, Q, r_out, f_out);
  SS_LAUNCH_CHECK();
  return SS_OK;
}
