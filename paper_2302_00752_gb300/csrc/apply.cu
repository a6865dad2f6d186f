// galerkin_apply: y = L_{N,s} u on the stamping set (eq. FiniteGalerkinOperator).
// One thread per row, one warp per 32-row slice of the sliced-ELL table: the
// index stream is read coalesced (column-major inside a slice) and u_l is
// gathered straight from the caller's array.  FP64: beside the stored entry
// coefficients.  FP32: the coefficient is formed from the stamp's norm words.
//
// FP64, 334,440 rows: 18 to 19 us (two or eight entries in flight: 22.0, 18.4);
// with the values copied into a record array first 23 us.  Bound: the gathers'
// L2 sectors (32 bytes for 16).
#include <algorithm>

#include "apply.cuh"

namespace ss {
namespace {

constexpr int kApply64Unroll = 4;   // entries in flight per thread

// u: n values, zero after.
template <bool REAL>
__global__ void __launch_bounds__(256) k_apply64(OpView op, int64_t size, int64_t rows_pad,
                                                 const double2* __restrict__ u, int64_t n, int64_t zero_idx,
                                                 double2* __restrict__ y) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows_pad) return;
  const int64_t s = row / kSlice;
  const int lane = (int)(row % kSlice);
  double2 acc = row_apply64_direct<REAL, kApply64Unroll>(op, s, lane, n, u);
  if (row == zero_idx) acc = row < n ? u[row] : make_double2(0.0, 0.0);
  if (row < size) y[row] = acc;
}

// One row per thread; 40 registers (six 256-thread blocks per SM) keep four
// index words and eight gathers in flight per thread.
template <bool WIDE>
__global__ void __launch_bounds__(256, 6) k_apply32(OpView op, int64_t size, int64_t rows_pad,
                                                    const int32_t* __restrict__ nw, const float2* __restrict__ u,
                                                    const float2* __restrict__ ca, const int32_t* __restrict__ pn,
                                                    int64_t zero_idx, float2* __restrict__ y) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows_pad) return;
  const int64_t s = row / kSlice;
  const int lane = (int)(row % kSlice);
  float2 acc = row_apply32_direct<WIDE, 4>(op, s, lane, __ldg(nw + row), size, u, nw, ca, pn);
  if (row < size) y[row] = row == zero_idx ? u[row] : acc;
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

constexpr int kNormThreads = 256;

// Per block: sum |f - y|^2 and |f|^2 over a fixed row range, fixed tree.
__global__ void k_resid_partials(const double2* __restrict__ f, const double2* __restrict__ y, int64_t n,
                                 int64_t rows_per_block, double2* part) {
  __shared__ double2 sh[kNormThreads];
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
  const int64_t r1 = min(n, r0 + rows_per_block);
  double num = 0.0, den = 0.0;
  for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
    const double2 a = f[i], b = y[i];
    const double ex = a.x - b.x, ey = a.y - b.y;
    num += ex * ex + ey * ey;
    den += a.x * a.x + a.y * a.y;
  }
  sh[threadIdx.x] = make_double2(num, den);
  __syncthreads();
  for (int o = kNormThreads / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[threadIdx.x].x += sh[threadIdx.x + o].x;
      sh[threadIdx.x].y += sh[threadIdx.x + o].y;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_sum_partials(const double2* __restrict__ part, int n, double2* out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double2 s = make_double2(0.0, 0.0);
  for (int i = 0; i < n; ++i) {
    s.x += part[i].x;
    s.y += part[i].y;
  }
  *out = s;
}

__global__ void k_ecoef_df(const double2* __restrict__ in, int64_t n, bool real, float4* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 c = real ? make_double2(reinterpret_cast<const double*>(in)[i], 0.0) : in[i];
  out[i] = cdf(df_split(c.x), df_split(c.y));
}

}  // namespace

ss_status ensure_ecoefdf(ss_stamp_s* s, cudaStream_t st) {
  if (s->ecoefdf.get()) return SS_OK;
  const int64_t n = s->n_ent + 1;
  SS_TRY(s->ecoefdf.alloc(n, st));
  k_ecoef_df<<<nblk(n), 256, 0, st>>>(s->ecoef64.get(), n, s->a_real, s->ecoefdf.get());
  SS_LAUNCH_CHECK();
  SS_CUDA(cudaStreamSynchronize(st));
  s->ecoefdf.settle();
  return SS_OK;
}

ss_status ensure_ecoefdf_half(ss_stamp_s* s, cudaStream_t st) {
  if (s->ecoefdf_h.get()) return SS_OK;
  const int64_t n = s->ecoef_h.n;
  SS_TRY(s->ecoefdf_h.alloc(n, st));
  k_ecoef_df<<<nblk(n), 256, 0, st>>>(s->ecoef_h.get(), n, s->a_real, s->ecoefdf_h.get());
  SS_LAUNCH_CHECK();
  SS_CUDA(cudaStreamSynchronize(st));
  s->ecoefdf_h.settle();
  return SS_OK;
}

// FP32 copies of the entry coefficients (the refined solve); the entries in
// use are counted on the device (woff[n_slices] rows of 32), so nothing is
// read back.
__global__ void k_ecoef_f32(const double* __restrict__ in, const int32_t* __restrict__ rows, int per_entry,
                            const int32_t* __restrict__ err, float* __restrict__ out) {
  if (__ldg(err) != 0) return;   // a failed build: the offsets are incomplete
  const int64_t n2 = (int64_t)__ldg(rows) * kSlice * per_entry / 2;   // pairs (32 rows: always whole)
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(in) + i);
    reinterpret_cast<float2*>(out)[i] = make_float2((float)v.x, (float)v.y);
  }
}

ss_status ensure_ecoef32(ss_stamp_s* s, bool half, cudaStream_t st) {
  DevBuf<float>& dst = half ? s->ecoef32_h : s->ecoef32;
  if (dst.get()) return SS_OK;
  const int per = s->a_real ? 1 : 2;
  const int64_t cap = half ? (int64_t)s->ecoef_h.n : s->n_ent + 1;
  SS_TRY(dst.alloc((size_t)cap * per, st));
  const int32_t* rows = half ? s->woff_h.get() + s->n_slices_h : s->slice_off.get() + s->n_slices;
  k_ecoef_f32<<<4 * sm_count(), 256, 0, st>>>(
      reinterpret_cast<const double*>(half ? s->ecoef_h.get() : s->ecoef64.get()), rows, per, s->err_dev.get(), dst.get());
  SS_LAUNCH_CHECK();
  return SS_OK;
}

OpView op_view(const ss_stamp_s* s) {
  OpView op;
  op.woff = s->slice_off.get();
  op.ent = s->ent.get();
  op.ecoef = s->ecoef64.get();
  op.ecoefdf = s->ecoefdf.get();
  op.colbits = colbits_of(s->jbits);
  op.colmask = colmask_of(s->jbits);
  op.realc = s->a_real;
  return op;
}

ss_status launch_apply64(const ss_stamp_s* s, const double2* u, int64_t n_u, double2* y, cudaStream_t st) {
  if (y < u + n_u && u < y + s->size) {   // in place: the rows read u while others write y
    SS_CUDA(cudaMemcpyAsync(s->rec64.get(), u, n_u * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    u = s->rec64.get();
  }
  ProfScope prof_("k_apply64", st, true);
  const auto kern = s->a_real ? k_apply64<true> : k_apply64<false>;
  kern<<<nblk(s->rows_pad), 256, 0, st>>>(op_view(s), s->size, s->rows_pad, u, n_u, identity_row(s), y);
  SS_LAUNCH_CHECK();
  return SS_OK;
}

ss_status launch_apply32(const ss_stamp_s* s, const float2* u, float2* y, cudaStream_t st) {
  if (s->adr) SS_FAIL(SS_ERR_INVALID, "the FP32 operator is not available for ADR stamps (use SS_FP64)");
  if (s->wide)
    {
      ProfScope prof_("k_apply32", st, true);
      k_apply32<true><<<nblk(s->rows_pad), 256, 0, st>>>(op_view(s), s->size, s->rows_pad, s->nw32.get(), u,
                                                         s->ca32.get(), s->pn32.get(), s->zero_idx, y);
    }
  else
    {
      ProfScope prof_("k_apply32", st, true);
      k_apply32<false><<<nblk(s->rows_pad), 256, 0, st>>>(op_view(s), s->size, s->rows_pad, s->nw32.get(), u,
                                                          s->ca32.get(), s->pn32.get(), s->zero_idx, y);
    }
  SS_LAUNCH_CHECK();
  return SS_OK;
}

}  // namespace ss

using namespace ss;

extern "C" ss_status galerkin_apply(ss_stamp s, const void* u, void* y, ss_precision prec, void* stream) {
  if (!s || !u || !y) SS_FAIL(SS_ERR_INVALID, "galerkin_apply: null argument");
  cudaStream_t st = as_stream(stream);
  if (s->size == 0) return SS_OK;
  if (prec == SS_FP64)
    return launch_apply64(s, reinterpret_cast<const double2*>(u), s->size, reinterpret_cast<double2*>(y), st);
  if (prec == SS_FP32)
    return launch_apply32(s, reinterpret_cast<const float2*>(u), reinterpret_cast<float2*>(y), st);
  SS_FAIL(SS_ERR_INVALID, "galerkin_apply: unknown precision %d", (int)prec);
}

extern "C" ss_status proxy_residual(ss_stamp s, const double* u_prefix, int64_t n_u, const double* f_on_S,
                                    double* out2, void* stream) {
  if (!s || !f_on_S || !out2 || (n_u > 0 && !u_prefix)) SS_FAIL(SS_ERR_INVALID, "proxy_residual: null argument");
  if (n_u < 0 || n_u > s->size) SS_FAIL(SS_ERR_INVALID, "proxy_residual: n_u = %lld outside [0, |S|]", (long long)n_u);
  cudaStream_t st = as_stream(stream);
  DevBuf<double2> y, part, sum;
  const int64_t rows_per_block = 4096;
  const int nb = (int)std::max<int64_t>(1, (s->size + rows_per_block - 1) / rows_per_block);
  SS_TRY(y.alloc(s->size, st));
  SS_TRY(part.alloc(nb, st));
  SS_TRY(sum.alloc(1, st));
  SS_TRY(launch_apply64(s, reinterpret_cast<const double2*>(u_prefix), n_u, y.get(), st));
  k_resid_partials<<<nb, kNormThreads, 0, st>>>(reinterpret_cast<const double2*>(f_on_S), y.get(), s->size,
                                                rows_per_block, part.get());
  k_sum_partials<<<1, 32, 0, st>>>(part.get(), nb, sum.get());
  SS_LAUNCH_CHECK();
  double2 h;
  SS_CUDA(cudaMemcpyAsync(&h, sum.get(), sizeof(h), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  out2[0] = h.x;
  out2[1] = h.y;
  return SS_OK;
}
