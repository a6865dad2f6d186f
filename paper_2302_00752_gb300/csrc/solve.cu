// Persistent Jacobi-preconditioned CG for L_{N,s} u = f (eq.
// SparseSpectralSFTEquation), one cooperative launch per solve.
//
// Two-colour reduction.  A step of supp a_hat moves a frequency by one level
// of the stamping set (Prop. LExpansion), so the rows of the levels N, N - 2,
// ... ("black") couple to each other only through chance relations between
// the steps; rows that do are counted as red (the build's colour masks), and
// the black block of L is exactly its diagonal D_B.  The solver runs CG on the
// Schur complement of the red rows,
//   S u_R = (D_R + offdiag - C D_B^-1 C^H) u_R = f_R - C D_B^-1 f_B,
// which has the same solution, needs about half the iterations (the Jacobi
// spectrum 1 +- mu becomes 1 - mu^2), and keeps the CG vectors on the red rows
// alone - at d = 100 one row in fourteen, since the last level is black.  One
// application of S is one pass over the entries of L in two half passes:
//   v_B = -D_B^-1 (C^H u_R)  on the black rows, then  w_R = (L (u_R, v_B))_R  on the
// red ones; the black solution D_B^-1 (f_B - C^H u_R) follows once at the end.
// A set without colours (N = 0, more than 16 levels, ADR operators, or too few
// black rows to pay: colours_pay in the build) has only red rows and skips the
// black phases: plain CG.
// The CG's stopping test needs the red rows alone (S u_R = ... has that residual
// when the black rows are solved for u_R); the residual reported at the end is
// evaluated on all rows, the black ones' rounding included where it can show
// (BlackRow).
//
// The rows of one or many instances form one row space cut into 32-row slices
// (one warp each); the slices that hold rows of a colour are listed in order,
// and a phase walks the list of its colour.  One instance: chunk c of n takes
// the warps' slices in turn (c + warp n, then every (warps n)-th), so that the
// wide slices of the inner levels spread over all SMs.  Batches: contiguous
// chunks balanced by entries.  A grid-wide barrier separates phases.  Inner
// products are reduced deterministically: per chunk and instance, each lane
// adds its rows in slice order, each warp folds its lanes with a fixed
// butterfly, the block adds its warps in order into one partial slot, and
// every block that needs a scalar sums that instance's slots with the same
// fixed warp reduction.  Per-instance state that crosses phases (rho, active
// flags) is double-buffered by iteration parity and written only by the
// instance's owner block (the one holding its first red chunk), so no phase
// reads a value that is written in the same phase.
//
// Modes
//   FP64  plain CG on the FP64 operator.
//   FP32  iterative refinement: r = f - L x with the FP64 operator, then CG on
//         the FP32 operator with FP32 vectors (inner products reduced in FP64,
//         FP64 scalars) to a relative reduction inner_tol, then x += delta in
//         FP64.
//   ADR   BiCGStab on the FP64 operator of Remark ADR (not Hermitian), right
//         Jacobi preconditioning with its complex diagonal.
// The CG preconditioner is D_k = 4 pi^2 Re(a_hat_0) |k|^2 (the diagonal of L),
// 1 on the zero row and on padding rows.
#include <algorithm>
#include <mutex>
#include <cmath>
#include <type_traits>

#include "solve.cuh"

namespace ss {
namespace {

// Grid-wide barrier (all blocks are co-resident: cooperative launch), entered
// after the block's stores are ordered (a block barrier, or warp 0 alone after
// one).  The count only grows: a block adds one with release order and polls
// with acquire loads until every block of this epoch has (no sleep between
// polls: the waits are short; no generation word to read before the arrival
// and none for the last block to publish: 1.2 against 2.6 us on 152 blocks).
// A wait longer than spin_limit ns sets SS_ERR_TIMEOUT and returns false; so
// does any error already posted by another block.  A launch of one block has
// nobody to wait for.
struct GridBar {
  unsigned target;   // arrivals that complete the current epoch
  int ok;
};

struct Smem {
  double acc[kMaxWarps][kMaxInstPerChunk][kNQ];
  double ca[kMaxInstPerChunk];
  double cb[kMaxInstPerChunk];
  double cc[kMaxInstPerChunk];
  double cd[kMaxInstPerChunk];
  int32_t flag[kMaxInstPerChunk];
  GridBar bar;
};

__device__ __forceinline__ long long gtimer() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ bool grid_wait(const SolveParams& P, GridBar& gb) {
  if (gridDim.x == 1) {
    __syncthreads();
    return true;
  }
  if (threadIdx.x == 0) {
    const unsigned target = gb.target += gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(P.bar) : "memory");
    const long long t0 = gtimer();
    int ok = 1;
    for (unsigned it = 1; (int)(ld_acquire(P.bar) - target) < 0; ++it) {
      if (it == 1 || (it & 255u) == 0) {
        if (*(volatile int*)P.err) { ok = 0; break; }
        if (gtimer() - t0 > P.spin_limit) {
          atomicCAS(P.err, 0, (int)SS_ERR_TIMEOUT);
          ok = 0;
          break;
        }
      }
    }
    gb.ok = ok;   // an error posted elsewhere stops the waiters in their poll loop
  }
  __syncthreads();
  return gb.ok != 0;
}

__device__ __forceinline__ bool grid_sync(const SolveParams& P, Smem& sm) {
  __syncthreads();
  return grid_wait(P, sm.bar);
}

// Counter read by one thread and broadcast to the block (uniform control flow).
__device__ int block_counter(const SolveParams& P, int idx) {
  __shared__ int s_cnt;
  __syncthreads();
  if (threadIdx.x == 0) s_cnt = atomicAdd(P.counters + idx, 0);
  __syncthreads();
  return s_cnt;
}

// Sums of the kNQ quantities over the partial slots of instance i (colour slot
// ci: 0 red or all rows, 1 black), by one warp in a fixed order (lane-strided,
// then a fixed butterfly; lane 0's result is broadcast), so every block that
// needs them gets the same bits.  Loads of four slots per lane are issued
// before they are added.
__device__ void inst_sums(const SolveParams& P, int i, int ci, double out[kNQ]) {
  const int lane = threadIdx.x & 31;
  const SolveInst& in = P.inst[i];
  const int len = in.c_last[ci] - in.c_first[ci] + 1;
  const double2* base = reinterpret_cast<const double2*>(P.part + (int64_t)in.part_base[ci] * kNQ);
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int c = lane;
  for (; c + 96 < len; c += 128) {
    double2 x[8];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[2 * u] = __ldcg(base + 2 * (c + 32 * u));
      x[2 * u + 1] = __ldcg(base + 2 * (c + 32 * u) + 1);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a0 += x[2 * u].x;
      a1 += x[2 * u].y;
      a2 += x[2 * u + 1].x;
      a3 += x[2 * u + 1].y;
    }
  }
  for (; c < len; c += 32) {
    const double2 x0 = __ldcg(base + 2 * c), x1 = __ldcg(base + 2 * c + 1);
    a0 += x0.x;
    a1 += x0.y;
    a2 += x1.x;
    a3 += x1.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a0 += __shfl_xor_sync(0xffffffffu, a0, o);
    a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    a2 += __shfl_xor_sync(0xffffffffu, a2, o);
    a3 += __shfl_xor_sync(0xffffffffu, a3, o);
  }
  out[0] = __shfl_sync(0xffffffffu, a0, 0);
  out[1] = __shfl_sync(0xffffffffu, a1, 0);
  out[2] = __shfl_sync(0xffffffffu, a2, 0);
  out[3] = __shfl_sync(0xffffffffu, a3, 0);
}

__device__ __forceinline__ double warp_reduce(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Lane accumulators of run_phase: FP64; double-float for the DF64 CG and FP32
// for the FP32 inner solve (kept on the FP32 pipe, converted to FP64 once per
// warp fold).
__device__ __forceinline__ double acc_fold(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return (double)v;
}
__device__ __forceinline__ double acc_fold(double v) { return warp_reduce(v); }

// Rows a phase runs over.
enum Colour { kAll = 0, kRed = 1, kBlack = 2 };

// Run one phase over the block's chunks of a colour's slices.  Partial sums:
// every lane adds its rows' values in slice order, the warp folds its lanes
// once per run of slices of one instance (fixed butterfly), the block adds its
// warps in order.
//   scal(ch, k, i, owner, lane): per instance of the chunk (one warp each),
//                             fills sm.ca/cb/flag[k] and does the owner's
//                             bookkeeping;
//   row(g, s, lane, i, k, run): per row of the colour, adds its values to the
//                             lane's running sums run[q], q in qmask.
// One instance whose phase has nothing to prepare passes scal = nullptr.
template <class Acc = double, class Scal, class Row>
__device__ void run_phase(const SolveParams& P, Smem& sm, Colour col, unsigned qmask, Scal scal, Row row) {
  constexpr bool kScal = !std::is_same<Scal, std::nullptr_t>::value;
  const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ci = col == kBlack ? 1 : 0, nch = P.n_chunks[ci];
  const int32_t* list = P.list[ci];
  for (int c = blockIdx.x; c < nch; c += gridDim.x) {
    Chunk ch;
    int64_t step;
    if (P.chunk[ci]) {
      ch = P.chunk[ci][c];
      step = nw;
    } else {   // one instance: the warps of all chunks take the listed slices in turn
      ch = Chunk{c, P.n_items ? (int64_t)__ldg(P.n_items + ci) : P.n_slices, 0, 0};
      step = (int64_t)nw * nch;
    }
    const int64_t first = ch.s0 + (P.chunk[ci] ? warp : (int64_t)warp * nch);
    const int ni = ch.inst1 - ch.inst0 + 1;
    if (qmask)
      for (int t = threadIdx.x; t < nw * ni * kNQ; t += blockDim.x)
        sm.acc[t / (ni * kNQ)][t / kNQ % ni][t % kNQ] = 0.0;
    if constexpr (kScal) {
      for (int k = warp; k < ni; k += nw) {
        const int i = ch.inst0 + k;
        scal(ch, k, i, c == P.inst[i].c_first[ci], lane);
      }
    }
    if (kScal || qmask) __syncthreads();
    int cur_k = -1;
    Acc run[kNQ] = {};
    auto fold = [&]() {
#pragma unroll
      for (int q = 0; q < kNQ; ++q) {
        const double t = (qmask & (1u << q)) ? acc_fold(run[q]) : 0.0;
        if (lane == 0) sm.acc[warp][cur_k][q] += t;
        run[q] = Acc{};
      }
    };
    for (int64_t it = first; it < ch.s1; it += step) {
      const int64_t s = list ? (int64_t)__ldg(list + it) : it;
      const int i = P.slice_inst ? __ldg(P.slice_inst + s) : 0;
      const int k = i - ch.inst0;
      const int64_t g = s * kSlice + lane;
      if (qmask && k != cur_k) {   // warp-uniform
        if (cur_k >= 0) fold();
        cur_k = k;
      }
      const bool on = col == kAll || !P.black || (((__ldg(P.black + s) >> lane) & 1u) != 0) == (col == kBlack);
      if (on) row(g, s, lane, i, k, run);
      __syncwarp();
    }
    if (qmask && cur_k >= 0) fold();
    if (qmask) {
      __syncthreads();
      for (int t = threadIdx.x; t < ni * kNQ; t += blockDim.x) {
        const int k = t / kNQ, q = t % kNQ;
        if (!(qmask & (1u << q))) continue;
        double v = 0.0;
        for (int w = 0; w < nw; ++w) v += sm.acc[w][k][q];
        const SolveInst& in = P.inst[ch.inst0 + k];
        P.part[(int64_t)(in.part_base[ci] + (c - in.c_first[ci])) * kNQ + q] = v;
      }
    }
    __syncthreads();
  }
}

// Power-of-two scale of an inner (FP32) solve: the residual handed to it has
// RMS entry near 1, so that the FP32 inner products r.D^-1 r and p.Lp stay far
// from FP32 underflow however small the outer residual and however large the
// Jacobi diagonal 4 pi^2 a_0 |k|^2 get.  Exact in FP64; 1 when rr = 0.
__device__ __forceinline__ double inner_scale(double rr, int64_t rows) {
  if (!(rr > 0.0)) return 1.0;
  return ldexp(1.0, -ilogb(sqrt(rr / (double)(rows > 0 ? rows : 1))));
}

__device__ __forceinline__ double jacobi(const SolveParams& P, const SolveInst& in, int64_t g) {
  const int64_t nk = __ldg(P.norm + g);
  return nk > 0 ? in.dscale * (double)nk : 1.0;
}

__device__ __forceinline__ float jacobi32(const SolveParams& P, const SolveInst& in, int64_t g) {
  const int64_t nk = __ldg(P.norm + g);
  return nk > 0 ? (float)in.dscale * (float)nk : 1.0f;
}

__device__ __forceinline__ double2 f_at(const SolveInst& in, int64_t g) {
  const int64_t l = g - in.row0;
  return l < in.rows ? in.f[l] : make_double2(0.0, 0.0);
}

// Row g of L applied to the records; SKIP leaves out the diagonal entry (the
// black rows' half pass; the zero row is red).
template <bool SKIP = false>
__device__ __forceinline__ double2 apply64_row(const SolveParams& P, const SolveInst& in, int64_t s, int lane,
                                               int64_t g, const double2* rec) {
  if (!SKIP && g == in.zero_row) return __ldcg(rec + g);
  return row_apply64<true, SKIP>(P.op, s, lane, rec, (uint32_t)g);
}

template <bool SKIP = false>
__device__ __forceinline__ float2 apply32_row(const SolveParams& P, const SolveInst& in, int64_t s, int lane,
                                              int64_t g) {
  if (!SKIP && g == in.zero_row) {
    const float4 v = __ldcg(P.urec32 + g);
    return make_float2(v.x, v.y);
  }
  return row_apply32<true, SKIP>(P.op, s, lane, __ldg(P.norm + g), in.wide != 0, P.urec32, P.ca32 + in.coef_off,
                                 P.pn + in.coef_off, (uint32_t)g);
}

__device__ __forceinline__ void owner_done(const SolveParams& P, InstState& st, int status) {
  st.status = status;
  atomicAdd(P.counters + 0, 1);
}

// ------------------------------------------------------------ CG recurrences
//
// Every mode uses the Chronopoulos-Gear form of preconditioned CG, which needs
// one reduction per iteration; on the red rows, with S in place of L:
//   p_i = u_i + beta_i p_{i-1},  s_i = w_i + beta_i s_{i-1}   (s_i = S p_i)
//   x_{i+1} = x_i + alpha_i p_i, r_{i+1} = r_i - alpha_i s_i, u_{i+1} = D^-1 r_{i+1}
//   w_{i+1} = S u_{i+1};  gamma = <r,u>, delta = <w,u>
//   beta_{i+1} = gamma_{i+1}/gamma_i,
//   alpha_{i+1} = gamma_{i+1} / (delta_{i+1} - beta_{i+1} gamma_{i+1} / alpha_i),
// with beta_0 = 0, alpha_0 = gamma_0 / delta_0.  Phase X does the scalars and
// the vector updates, phase B the black half pass and phase Y the red one with
// the three inner products (gamma, delta, |r|^2): three grid barriers per
// iteration (two without colours).  Partial slot q3 holds |f|^2.
// r is also the residual of the whole system, up to the rounding of the black
// rows' solution.

struct Coeffs {
  double alpha, beta;
};

__device__ __forceinline__ Coeffs cg_coeffs(int it, double gam, double del, double gam_prev, double alpha_prev) {
  Coeffs c;
  if (it == 0) {
    c.beta = 0.0;
    c.alpha = gam / del;
  } else {
    c.beta = gam / gam_prev;
    c.alpha = gam / (del - c.beta * gam / alpha_prev);
  }
  return c;
}

// Black rows to eliminate (one instance: its masks may have been dropped on the
// device; a batch without any has no masks).
__device__ __forceinline__ bool has_black(const SolveParams& P) {
  return P.black && (!P.n_items || __ldg(P.n_items + 1) > 0);
}

// |f|^2 of instance i from the two colours' slots (all lanes).
__device__ __forceinline__ double sum_bb(const SolveParams& P, int i, const double t[kNQ]) {
  double b[kNQ];
  if (!has_black(P)) return t[3];
  inst_sums(P, i, 1, b);
  return t[3] + b[3];
}

// Scalars of CG iteration `it` of the FP64 and DF64 modes for instance i (one
// warp; lane 0 gets the result), and the owner's bookkeeping.
__device__ __forceinline__ Coeffs cg_scalars(const SolveParams& P, int i, int it, bool owner, int lane, double tol2,
                                             bool* go_out) {
  const int cur = it & 1, nxt = cur ^ 1;
  double t[kNQ];
  inst_sums(P, i, 0, t);
  const double bb0 = it == 0 ? sum_bb(P, i, t) : 0.0;
  Coeffs cf{0.0, 0.0};
  if (lane == 0) {
    InstState& st = P.state[i];
    const int act = it == 0 ? 1 : __ldcg(&st.act[cur]);
    const double bb = it == 0 ? bb0 : __ldcg(&st.bb);
    const bool conv = t[2] <= tol2 * bb;
    const bool cap = it >= P.max_iter;
    cf = cg_coeffs(it, t[0], t[1], it ? __ldcg(&st.rho[cur]) : 0.0, it ? __ldcg(&st.alpha[cur]) : 0.0);
    const bool go = act && !conv && !cap;
    *go_out = go;
    if (owner) {
      if (it == 0) {
        st.bb = bb;
        st.applies = 1;
        st.outer_iters = 1;
      }
      st.act[nxt] = go;
      st.rho[nxt] = t[0];
      st.alpha[nxt] = cf.alpha;
      if (act) {
        st.rr = t[2];
        st.iters = it;
        if (conv) owner_done(P, st, SS_OK);
        else if (cap) owner_done(P, st, SS_ERR_NOT_CONVERGED);
        else st.applies += 1;
      }
    }
  }
  return cf;
}

// All instances done?  One instance: every block formed the same flag in the
// phase just run; batches read the owners' count (after the grid barrier).
__device__ __forceinline__ bool one_done(const SolveParams& P, const Smem& sm) { return !P.slice_inst && !sm.flag[0]; }

// End of the FP64 modes: every instance's residual norm, both colours.
__device__ void final_rr(const SolveParams& P) {
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
  for (int i = blockIdx.x * nw + (threadIdx.x >> 5); i < P.n_inst; i += gridDim.x * nw) {
    double t[kNQ], b[kNQ] = {};
    inst_sums(P, i, 0, t);
    if (has_black(P)) inst_sums(P, i, 1, b);
    if (lane == 0) {
      P.state[i].rr = t[2] + b[2];
      P.state[i].applies += 1;
    }
  }
}

// Residual f - (L x)_g of a black row: its product with the red rows, added up
// from start() on (the solution was formed from the bare product; added to the
// diagonal's term it rounds anew, as in any evaluation of the row).  A scaled
// table's black rows hold -D^-1 C^H: there the sum is -x + D^-1 (-C^H x).  What
// the row needs beside its entries is loaded by start, ahead of the sum.  That is
// one more FP64 pass over the black rows (d = 100: 18 us, a batch of 128: 80),
// and rounding stands 2^10 times and more below a red residual above 2^-43 ||f||:
// then the black rows are not evaluated.
constexpr double kShow = 0x1p-86, kShowDf = 0x1p-72;   // squared; double-float rounds at 2^-47
struct BlackRow {
  double2 f;
  int64_t nk;
  __device__ __forceinline__ double2 start(const SolveParams& P, const SolveInst& in, int64_t g, double2 x) {
    f = f_at(in, g);
    nk = __ldg(P.norm + g);
    if (P.op.scaled) return make_double2(-x.x, -x.y);
    const double d = diag(in);
    return make_double2(d * x.x, d * x.y);
  }
  __device__ __forceinline__ double diag(const SolveInst& in) const { return nk > 0 ? in.dscale * (double)nk : 1.0; }
  __device__ __forceinline__ double norm2(const SolveParams& P, const SolveInst& in, double2 s) const {
    const double m = P.op.scaled ? diag(in) : -1.0, rx = fma(m, s.x, f.x), ry = fma(m, s.y, f.y);
    return fma(rx, rx, ry * ry);
  }
};
// The general phases' sum of them into q2 (0 where it cannot show); the state
// holds the instances' last red residuals.
__device__ void black_rr(const SolveParams& P, Smem& sm) {
  run_phase(P, sm, kBlack, 0b0100u, [&](const Chunk&, int k, int i, bool, int lane) {
    if (lane == 0) sm.flag[k] = __ldcg(&P.state[i].rr) <= kShow * __ldcg(&P.state[i].bb);
  }, [&](int64_t g, int64_t s, int lane, int i, int k, double* v) {
    if (!sm.flag[k]) return;
    const SolveInst& in = P.inst[i];
    BlackRow r;
    const double2 a = r.start(P, in, g, P.xrec[g]);
    v[2] += r.norm2(P, in, row_apply64<true, true>(P.op, s, lane, P.xrec, (uint32_t)g, a));
  });
}

// D^-1 (f - C^H x_R) of a black row from its product y with x_R (a scaled
// table's black rows hold -D^-1 C^H).
__device__ __forceinline__ double2 black_x(const SolveParams& P, const SolveInst& in, int64_t g, double2 y) {
  const double2 f = f_at(in, g);
  const double rD = P.rdiag[g];
  if (P.op.scaled) return make_double2(fma(rD, f.x, y.x), fma(rD, f.y, y.y));
  return make_double2(rD * (f.x - y.x), rD * (f.y - y.y));
}

// --------------------------------------------------------------- FP64 CG

__device__ void solve_fp64(const SolveParams& P, Smem& sm) {
  const double tol2 = P.tol * P.tol;
  const bool colours = has_black(P), scaled = P.op.scaled;
  // The residual is kept as r = D u (D the Jacobi diagonal, u = D^-1 r the
  // preconditioned residual and the gathered record): the vector phase
  // updates u = u - alpha D^-1 s directly, and the apply phase forms
  // <r, u> = sum D |u|^2 and <r, r> = sum D^2 |u|^2.  No r vector is read or
  // written (152 instead of 184 bytes per row and iteration in the vector
  // phase); P.r holds D (one double per row).
  double* dg = reinterpret_cast<double*>(P.r);
  // u_R = 0 with the black rows solved: x_B = D^-1 f_B; |f|^2
  if (colours)
    run_phase(P, sm, kBlack, 0b1000u, nullptr, [&](int64_t g, int64_t, int, int i, int, double* v) {
      const SolveInst& in = P.inst[i];
      const double2 f = f_at(in, g);
      const double rD = 1.0 / jacobi(P, in, g);
      P.rdiag[g] = rD;
      P.xrec[g] = make_double2(f.x * rD, f.y * rD);
      v[3] += f.x * f.x + f.y * f.y;
    });
  run_phase(P, sm, kRed, 0b1000u, nullptr, [&](int64_t g, int64_t, int, int i, int, double* v) {
    const SolveInst& in = P.inst[i];
    const double2 f = f_at(in, g);
    const double dk = jacobi(P, in, g), rD = 1.0 / dk;
    P.rdiag[g] = rD;
    dg[g] = dk;
    P.xrec[g] = make_double2(0.0, 0.0);
    if (!colours) P.urec64[g] = make_double2(f.x * rD, f.y * rD);
    P.pd[g] = make_double2(0.0, 0.0);
    P.sd[g] = make_double2(0.0, 0.0);
    v[3] += f.x * f.x + f.y * f.y;
  });
  if (!grid_sync(P, sm)) return;
  if (colours) {   // u = D^-1 r, r = f_R - C D_B^-1 f_B
    run_phase(P, sm, kRed, 0u, nullptr, [&](int64_t g, int64_t s, int lane, int i, int, double*) {
      const SolveInst& in = P.inst[i];
      const double2 y = apply64_row(P, in, s, lane, g, P.xrec);
      const double2 f = f_at(in, g);
      const double rD = P.rdiag[g];
      P.urec64[g] = make_double2((f.x - y.x) * rD, (f.y - y.y) * rD);
    });
    if (!grid_sync(P, sm)) return;
  }
  auto active = [&](unsigned par) {
    return [&P, &sm, par](const Chunk&, int k, int i, bool, int lane) {
      if (lane == 0) sm.flag[k] = par > 1 ? 1 : (P.slice_inst ? __ldcg(&P.state[i].act[par]) : 1);
    };
  };
  // v_B and w_R (see the file comment); par: activity parity, 2 for every instance
  auto apply = [&](unsigned par) -> bool {
    if (colours) {
      run_phase(P, sm, kBlack, 0u, active(par), [&](int64_t g, int64_t s, int lane, int i, int k, double*) {
        if (!sm.flag[k]) return;
        const double2 y = apply64_row<true>(P, P.inst[i], s, lane, g, P.urec64);
        const double m = scaled ? 1.0 : -P.rdiag[g];
        P.urec64[g] = make_double2(m * y.x, m * y.y);
      });
      if (!grid_sync(P, sm)) return false;
    }
    run_phase(P, sm, kRed, 0b0111u, active(par), [&](int64_t g, int64_t s, int lane, int i, int k, double* v) {
      if (!sm.flag[k]) return;
      const SolveInst& in = P.inst[i];
      const double2 w = apply64_row(P, in, s, lane, g, P.urec64);
      const double2 u = P.urec64[g];
      const double dk = dg[g];
      P.w64[g] = w;
      const double du = dk * fma(u.y, u.y, u.x * u.x);   // D |u|^2 = <r, u> of this row
      v[0] += du;
      v[1] = fma(w.y, u.y, fma(w.x, u.x, v[1]));
      v[2] = fma(dk, du, v[2]);                           // |r|^2 = D^2 |u|^2
    });
    return grid_sync(P, sm);
  };
  if (!apply(2)) return;
  for (int it = 0;; ++it) {
    run_phase(P, sm, kRed, 0u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      bool go = false;
      const Coeffs cf = cg_scalars(P, i, it, owner, lane, tol2, &go);
      if (lane == 0) {
        sm.flag[k] = go;
        sm.ca[k] = cf.alpha;
        sm.cb[k] = cf.beta;
      }
    }, [&](int64_t g, int64_t, int, int i, int k, double*) {
      if (!sm.flag[k]) return;
      const double a = sm.ca[k], b = sm.cb[k];
      double2 u = P.urec64[g];
      const double2 w = P.w64[g];
      double2 p = P.pd[g], sv = P.sd[g], x = P.xrec[g];
      p.x = u.x + b * p.x; p.y = u.y + b * p.y;
      sv.x = w.x + b * sv.x; sv.y = w.y + b * sv.y;
      x.x += a * p.x; x.y += a * p.y;
      const double t = a * P.rdiag[g];   // u - alpha D^-1 s = D^-1 (r - alpha s)
      u.x = fma(-t, sv.x, u.x);
      u.y = fma(-t, sv.y, u.y);
      P.pd[g] = p;
      P.sd[g] = sv;
      P.xrec[g] = x;
      P.urec64[g] = u;
    });
    if (one_done(P, sm)) {
      // without colours the next phase writes the slots that others may still read
      if (!colours && !grid_sync(P, sm)) return;
      break;
    }
    if (!grid_sync(P, sm)) return;
    if (P.slice_inst && block_counter(P, 0) >= P.n_inst) break;
    if (!apply((it & 1) ^ 1)) return;
  }
  // x_B = D^-1 (f_B - C^H x_R), the output, and the true residual f - L x in FP64
  if (colours) {
    run_phase(P, sm, kBlack, 0u, nullptr, [&](int64_t g, int64_t s, int lane, int i, int, double*) {
      const SolveInst& in = P.inst[i];
      const double2 x = black_x(P, in, g, apply64_row<true>(P, in, s, lane, g, P.xrec));
      P.xrec[g] = x;
      const int64_t l = g - in.row0;
      if (l < in.rows) in.u[l] = x;
    });
    if (!grid_sync(P, sm)) return;
    black_rr(P, sm);
  }
  run_phase(P, sm, kRed, 0b0100u, nullptr, [&](int64_t g, int64_t s, int lane, int i, int, double* v) {
    const SolveInst& in = P.inst[i];
    const double2 y = apply64_row(P, in, s, lane, g, P.xrec);
    const double2 f = f_at(in, g);
    const double2 r = make_double2(f.x - y.x, f.y - y.y);
    v[2] += r.x * r.x + r.y * r.y;
    const int64_t l = g - in.row0;
    if (l < in.rows) in.u[l] = P.xrec[g];
  });
  if (!grid_sync(P, sm)) return;
  final_rr(P);
}

// ------------------------------------------------- FP32 CG in FP64 refinement

__device__ void solve_refined(const SolveParams& P, Smem& sm) {
  const double tol2 = P.tol * P.tol, itol2 = P.inner_tol * P.inner_tol;
  const bool colours = has_black(P);
  float* rd32 = reinterpret_cast<float*>(P.dlt);   // 1 / D in FP32
  for (int ot = 0;; ++ot) {
    const int ocur = ot & 1, onxt = ocur ^ 1;
    auto running = [&](const Chunk&, int k, int i, bool, int lane) {
      if (lane == 0) sm.flag[k] = ot == 0 || !P.slice_inst ? 1 : __ldcg(&P.state[i].act[ocur]);
    };
    // the black rows solved for the current x_R (FP64): x_B = D^-1 (f_B - C^H x_R),
    // x_R = 0 at first; |f|^2
    if (colours)
      run_phase(P, sm, kBlack, ot == 0 ? 0b1000u : 0u, running,
                [&](int64_t g, int64_t s, int lane, int i, int k, double* v) {
        if (!sm.flag[k]) return;
        const SolveInst& in = P.inst[i];
        if (ot == 0) {
          const double2 f = f_at(in, g);
          const double rD = 1.0 / jacobi(P, in, g);
          P.rdiag[g] = rD;
          rd32[g] = 1.0f / jacobi32(P, in, g);
          P.xrec[g] = make_double2(rD * f.x, rD * f.y);
          v[3] += f.x * f.x + f.y * f.y;
        } else {
          P.xrec[g] = black_x(P, in, g, apply64_row<true>(P, in, s, lane, g, P.xrec));
        }
      });
    if (ot == 0)
      run_phase(P, sm, kRed, 0b1000u, nullptr, [&](int64_t g, int64_t, int, int i, int, double* v) {
        const SolveInst& in = P.inst[i];
        const double2 f = f_at(in, g);
        rd32[g] = 1.0f / jacobi32(P, in, g);
        P.xrec[g] = make_double2(0.0, 0.0);
        v[3] += f.x * f.x + f.y * f.y;
      });
    if ((colours || ot == 0) && !grid_sync(P, sm)) return;
    // rhat = f - L64 x on the red rows, |rhat|^2
    run_phase(P, sm, kRed, 0b0100u, running, [&](int64_t g, int64_t s, int lane, int i, int k, double* v) {
      if (!sm.flag[k]) return;
      const SolveInst& in = P.inst[i];
      const double2 y = apply64_row(P, in, s, lane, g, P.xrec);
      const double2 f = f_at(in, g);
      const double2 r = make_double2(f.x - y.x, f.y - y.y);
      P.rhat[g] = r;
      v[2] += r.x * r.x + r.y * r.y;
    });
    if (!grid_sync(P, sm)) return;
    // outer test; inner start (all FP32): r = rhat * scale, delta = 0, u = D^-1 r, p = s = 0
    run_phase(P, sm, kRed, 0u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      double t[kNQ];
      inst_sums(P, i, 0, t);
      const double bb0 = ot == 0 ? sum_bb(P, i, t) : 0.0;
      if (lane == 0) {
        InstState& st = P.state[i];
        const int act = ot == 0 ? 1 : __ldcg(&st.act[ocur]);
        const double bb = ot == 0 ? bb0 : __ldcg(&st.bb), rr = t[2];
        const bool conv = rr <= tol2 * bb;
        const bool cap = ot >= P.max_outer;
        const bool go = act && !conv && !cap;
        sm.flag[k] = go;
        sm.ca[k] = inner_scale(rr, P.inst[i].rows);
        if (owner) {
          if (ot == 0) st.bb = bb;
          st.act[onxt] = go;
          st.inn[0] = go;
          if (act) {
            st.rr = rr;
            st.applies += 1;
            if (conv) owner_done(P, st, SS_OK);
            else if (cap) owner_done(P, st, SS_ERR_NOT_CONVERGED);
            else {
              st.outer_iters = ot + 1;
              st.applies += 1;
              atomicAdd(P.counters + 1, 1);
            }
          }
        }
      }
    }, [&](int64_t g, int64_t, int, int i, int k, double*) {
      if (!sm.flag[k]) return;
      const double2 rh = P.rhat[g];
      const double sc = sm.ca[k];
      const float2 r = make_float2((float)(rh.x * sc), (float)(rh.y * sc));
      const float rD = rd32[g];
      P.r32[g] = r;
      P.d32[g] = make_float2(0.f, 0.f);
      P.p32[g] = make_float2(0.f, 0.f);
      P.s32[g] = make_float2(0.f, 0.f);
      reinterpret_cast<float2*>(P.urec32 + g)[0] = make_float2(r.x * rD, r.y * rD);
    });
    if (one_done(P, sm)) break;
    if (!grid_sync(P, sm)) return;
    if (P.slice_inst && block_counter(P, 0) >= P.n_inst) break;
    // inner CG on the FP32 operator with FP32 vectors (relative tolerance
    // 1e-5): the inner products are summed in FP32 per lane and in FP64 from
    // the warp fold on, scalars stay FP64
    auto apply = [&](int par) -> bool {
      auto active = [&P, &sm, par](const Chunk&, int k, int i, bool, int lane) {
        if (lane == 0) sm.flag[k] = P.slice_inst ? __ldcg(&P.state[i].inn[par]) : 1;
      };
      if (colours) {
        run_phase(P, sm, kBlack, 0u, active, [&](int64_t g, int64_t s, int lane, int i, int k, double*) {
          if (!sm.flag[k]) return;
          const float2 y = apply32_row<true>(P, P.inst[i], s, lane, g);
          const float rD = -rd32[g];
          reinterpret_cast<float2*>(P.urec32 + g)[0] = make_float2(rD * y.x, rD * y.y);
        });
        if (!grid_sync(P, sm)) return false;
      }
      run_phase<float>(P, sm, kRed, 0b0111u, active, [&](int64_t g, int64_t s, int lane, int i, int k, float* v) {
        if (!sm.flag[k]) return;
        const float2 w = apply32_row(P, P.inst[i], s, lane, g);
        const float4 u = P.urec32[g];
        const float2 r = P.r32[g];
        P.w32[g] = w;
        v[0] += r.x * u.x + r.y * u.y;
        v[1] += w.x * u.x + w.y * u.y;
        v[2] += r.x * r.x + r.y * r.y;
      });
      return grid_sync(P, sm);
    };
    if (!apply(0)) return;
    for (int it = 0;; ++it) {
      const int cur = it & 1, nxt = cur ^ 1;
      run_phase(P, sm, kRed, 0u, [&](const Chunk&, int k, int i, bool owner, int lane) {
        double t[kNQ];
        inst_sums(P, i, 0, t);
        if (lane == 0) {
          InstState& st = P.state[i];
          const int act = __ldcg(&st.inn[cur]);
          const double rr = __ldcg(&st.rr), sc = inner_scale(rr, P.inst[i].rows);
          const bool conv = t[2] <= itol2 * rr * sc * sc;     // r32 carries the scale
          const bool cap = it >= P.max_inner;
          const Coeffs cf = cg_coeffs(it, t[0], t[1], it ? __ldcg(&st.rho[cur]) : 0.0,
                                      it ? __ldcg(&st.alpha[cur]) : 0.0);
          const bool go = act && !conv && !cap;
          sm.flag[k] = go;
          sm.ca[k] = cf.alpha;
          sm.cb[k] = cf.beta;
          if (owner) {
            st.inn[nxt] = go;
            st.rho[nxt] = t[0];
            st.alpha[nxt] = cf.alpha;
            if (act) {
              if (go) {
                st.inner_iters += 1;
                st.applies += 1;
              } else {
                atomicAdd(P.counters + 2, 1);
              }
            }
          }
        }
      }, [&](int64_t g, int64_t, int, int, int k, double*) {
        if (!sm.flag[k]) return;
        const float a = (float)sm.ca[k], b = (float)sm.cb[k];
        const float4 u = P.urec32[g];
        const float2 w = P.w32[g];
        float2 p = P.p32[g], sv = P.s32[g], dl = P.d32[g], r = P.r32[g];
        p.x = fmaf(b, p.x, u.x); p.y = fmaf(b, p.y, u.y);
        sv.x = fmaf(b, sv.x, w.x); sv.y = fmaf(b, sv.y, w.y);
        dl.x = fmaf(a, p.x, dl.x); dl.y = fmaf(a, p.y, dl.y);
        r.x = fmaf(-a, sv.x, r.x); r.y = fmaf(-a, sv.y, r.y);
        const float rD = rd32[g];
        P.p32[g] = p;
        P.s32[g] = sv;
        P.d32[g] = dl;
        P.r32[g] = r;
        reinterpret_cast<float2*>(P.urec32 + g)[0] = make_float2(r.x * rD, r.y * rD);
      });
      if (one_done(P, sm)) break;
      if (!grid_sync(P, sm)) return;
      if (P.slice_inst && block_counter(P, 2) >= block_counter(P, 1)) break;
      if (!apply(nxt)) return;
    }
    // x_R += delta
    run_phase(P, sm, kRed, 0u, [&](const Chunk&, int k, int i, bool, int lane) {
      if (lane == 0) {
        sm.flag[k] = P.slice_inst ? __ldcg(&P.state[i].act[onxt]) : 1;
        sm.ca[k] = 1.0 / inner_scale(__ldcg(&P.state[i].rr), P.inst[i].rows);
      }
    }, [&](int64_t g, int64_t, int, int, int k, double*) {
      if (!sm.flag[k]) return;
      double2 x = P.xrec[g];
      const float2 dl = P.d32[g];
      const double us = sm.ca[k];
      x.x += (double)dl.x * us;
      x.y += (double)dl.y * us;
      P.xrec[g] = x;
    });
    if (!grid_sync(P, sm)) return;
  }
  if (colours) {   // the black rows' part of the residual
    black_rr(P, sm);
    if (!grid_sync(P, sm)) return;
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    for (int i = blockIdx.x * nw + (threadIdx.x >> 5); i < P.n_inst; i += gridDim.x * nw) {
      double b[kNQ];
      inst_sums(P, i, 1, b);
      if (lane == 0) P.state[i].rr += b[2];
    }
  }
  auto put = [&](int64_t g, int64_t, int, int i, int, double*) {
    const SolveInst& in = P.inst[i];
    const int64_t l = g - in.row0;
    if (l < in.rows) in.u[l] = P.xrec[g];
  };
  if (colours) run_phase(P, sm, kBlack, 0u, nullptr, put);
  run_phase(P, sm, kRed, 0u, nullptr, put);
}

// ------------------------------------------------------ one instance
//
// One instance's CG is bound by latency, not by bytes: at d = 100 the red
// vectors are 0.7 MB, and a phase of every smaller set is a chain of a few L2
// round trips, FP64 operations (a warp's FP64 instruction occupies its quarter
// of the SM for 64 clocks) and the barrier.  So, against the general phases
// (run_phase), which serve batches:
//  - every warp keeps its first units (slice, widths, colours) in shared
//    memory for the whole solve; the barrier's acquire empties the L1, so each
//    phase would otherwise start with two more dependent L2 reads;
//  - rows are split over 1, 2, 4 or 8 lanes, whichever gives a warp the fewest
//    steps (rounds of units times batches of a unit and one more for its end,
//    at the width of the last slice: the colour's largest level);
//  - entry words and gathers run ahead of the products (op_phase);
//  - four inner products are folded together (6 FP64 additions instead of 20),
//    in one warp per quantity across the blocks;
//  - the CG scalars stay in the block (every block forms the same ones), with
//    one division on the critical path;
//  - 512 threads and 128 registers: half the warps to synchronise, at the
//    same number of loads in flight.

constexpr int kMeta = 8;   // units per warp kept in shared memory

struct SmemS {
  double red[kMaxWarps][kNQ];
  double t[kNQ];             // sums of the last reduction over all blocks
  double ca, cb, ig, ia;     // alpha, beta, 1 / gamma and 1 / alpha of the previous iteration
  double bb, stop, sc, us;   // |f|^2, the squared residual to reach, FP32 scale and its inverse
  GridBar bar;
  float dfs[4];              // DF64: alpha and beta as double-float
  int go;
  int4 meta[3][kMaxWarps][kMeta];   // unit table: slice, first entry row, width, colour mask
};

// Unit tables: the red slices one warp each (vector phases), the red and the
// black rows of the operator phases in units of 32 >> split rows.
enum { kVec = 0, kOpR = 1, kOpB = 2 };

struct Units {
  int n[3], split[3];   // units; log2 of the lanes per row
};

__device__ __forceinline__ int4 load_unit(const SolveParams& P, int tab, int split, int64_t it) {
  const int ci = tab == kOpB ? 1 : 0;
  const int64_t x = it >> split;
  const int s = P.list[ci] ? __ldg(P.list[ci] + x) : (int)x;
  const int w0 = __ldg(P.op.woff + s);
  const uint32_t m = P.black ? __ldg(P.black + s) : 0u;
  return make_int4(s, w0, __ldg(P.op.woff + s + 1) - w0, (int)(ci ? m : ~m));
}

// First unit and stride of this warp: consecutive units go to different blocks.
__device__ __forceinline__ int64_t unit_first() { return blockIdx.x + (int64_t)(threadIdx.x >> 5) * gridDim.x; }
__device__ __forceinline__ int64_t unit_step() { return (int64_t)(blockDim.x >> 5) * gridDim.x; }

__device__ Units setup_units(const SolveParams& P, SmemS& sm) {
  Units U;
  const int64_t warps = unit_step();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int tab = 0; tab < 3; ++tab) {
    const int n = __ldg(P.n_items + (tab == kOpB ? 1 : 0));
    int sp = 0;
    if (tab != kVec && n > 0) {
      const int w = load_unit(P, tab, 0, n - 1).z;
      int64_t best = INT64_MAX;
      for (int q = 0; q < 4; ++q) {
        const int64_t cost = (((int64_t)n << q) + warps - 1) / warps * ((w + (4 << q) - 1) / (4 << q) + 1);
        if (cost < best) {
          best = cost;
          sp = q;
        }
      }
    }
    U.split[tab] = sp;
    U.n[tab] = n << sp;
    const int64_t it = unit_first() + lane * unit_step();
    if (lane < kMeta && it < U.n[tab]) sm.meta[tab][warp][lane] = load_unit(P, tab, sp, it);
  }
  __syncthreads();
  return U;
}

// row(g) for the rows of the warp's units (vector phases: no split).
template <class Row>
__device__ __forceinline__ void rows_phase(const SolveParams& P, const SmemS& sm, const Units& U, int tab, Row row) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int k = 0;
  // the tables of the operator phases list a slice 2^split times
  const int64_t step = unit_step();
  const int n = U.n[tab];
  for (int64_t it = unit_first(); it < n; it += step, ++k) {
    const int4 u = k < kMeta ? sm.meta[tab][warp][k] : load_unit(P, tab, U.split[tab], it);
    const int sp = U.split[tab], rows = 32 >> sp;
    const int rl = (int)(it & ((1 << sp) - 1)) * rows + (lane & (rows - 1));
    if (lane < rows && ((uint32_t)u.w >> rl & 1u)) row((int64_t)u.x * kSlice + rl);
  }
}

// Fold four values over the warp with six additions: halves keep two, quarters
// one; lane 8 q' then holds quantity q = (lane >> 4) * 2 + ((lane >> 3) & 1).
template <class T, class Add>
__device__ __forceinline__ T fold4(T a, T b, T c, T d, Add add) {
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, q = lane & 8;
  auto xchg = [](const T& v, int o) {
    T r;
    if constexpr (sizeof(T) == 4) {
      r = __shfl_xor_sync(0xffffffffu, v, o);
    } else if constexpr (std::is_same<T, DF>::value) {
      r = DF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    } else {
      r = __shfl_xor_sync(0xffffffffu, v, o);
    }
    return r;
  };
  const T k0 = h ? c : a, k1 = h ? d : b, s0 = h ? a : c, s1 = h ? b : d;
  const T x0 = add(k0, xchg(s0, 16)), x1 = add(k1, xchg(s1, 16));
  T x = add(q ? x1 : x0, xchg(q ? x0 : x1, 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x = add(x, xchg(x, o));
  return x;
}

__device__ __forceinline__ double plus_d(double a, double b) { return a + b; }
__device__ __forceinline__ double fold4d(const float* v) {
  return (double)fold4<float>(v[0], v[1], v[2], v[3], [](float a, float b) { return a + b; });
}
__device__ __forceinline__ double fold4d(const double* v) { return fold4<double>(v[0], v[1], v[2], v[3], plus_d); }
__device__ __forceinline__ double fold4d(const DF* v) {
  return df_to_double(fold4<DF>(v[0], v[1], v[2], v[3], [](DF a, DF b) { return df_add(a, b); }));
}

// Grid barrier that carries the block's four sums of `run` (warp 0 adds the
// warps' values and arrives: the block barrier before it orders every other
// thread's stores).  Two sets of slots alternate, so that a block may still
// read one reduction while another block writes the next.
template <class Acc>
__device__ bool sync_sum(const SolveParams& P, SmemS& sm, int& par, const Acc* run) {
  const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double f = fold4d(run);
  if ((lane & 7) == 0) sm.red[warp][lane >> 3] = f;
  __syncthreads();
  if (warp == 0) {
    double v[kNQ] = {};
    if (lane < nw) {
#pragma unroll
      for (int q = 0; q < kNQ; ++q) v[q] = sm.red[lane][q];
    }
    const double s = fold4d(v);
    if ((lane & 7) == 0) P.part[((int64_t)par * gridDim.x + blockIdx.x) * kNQ + (lane >> 3)] = s;
    __syncwarp();
  }
  par ^= 1;
  return grid_wait(P, sm.bar);
}

// Grid barrier after the block's stores.
__device__ __forceinline__ bool sync_all(const SolveParams& P, SmemS& sm) {
  __syncthreads();
  return grid_wait(P, sm.bar);
}

// sm.t = the sums of the last sync_sum over all blocks (par: the parity it
// left): one warp per quantity, lanes in a fixed stride, then a fixed butterfly.
__device__ void all_sums(const SolveParams& P, SmemS& sm, int par) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < kNQ) {
    const double* p = P.part + (int64_t)(par ^ 1) * gridDim.x * kNQ + warp;
    const int len = gridDim.x;
    double s = 0.0;
    for (int c = lane; c < len; c += 160) {
      double x[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) x[q] = c + 32 * q < len ? __ldcg(p + (int64_t)(c + 32 * q) * kNQ) : 0.0;
      s += ((x[0] + x[1]) + (x[2] + x[3])) + x[4];
    }
    s = warp_reduce(s);
    if (lane == 0) sm.t[warp] = s;
  }
  __syncthreads();
}

// alpha and beta of CG iteration `it` from sm.t (one warp; every lane returns
// them): beta = gamma (1 / gamma_prev), alpha = gamma / (delta - beta gamma / alpha_prev).
// 1 / gamma for the next iteration is the same division in another lane.
__device__ __forceinline__ Coeffs one_coeffs(SmemS& sm, int it) {
  const int lane = threadIdx.x & 31;
  const double gam = sm.t[0], del = sm.t[1];
  const double beta = it ? gam * sm.ig : 0.0;
  const double den = it ? fma(-beta, gam * sm.ia, del) : del;
  const double q = (lane == 0 ? gam : 1.0) / (lane == 0 ? den : gam);
  const double alpha = __shfl_sync(0xffffffffu, q, 0), ig = __shfl_sync(0xffffffffu, q, 1);
  __syncwarp();
  if (lane == 0) {
    sm.ig = ig;
    sm.ia = den * ig;
  }
  return Coeffs{alpha, beta};
}

// ---- operator phases: rows of L applied to records, split over 2^sp lanes per
// row (lane `sub` takes the entries sub, sub + 2^sp, ...).  SKIP leaves out the
// diagonal (the black half pass).  A warp's batches of NB entries per lane run
// through its units as one pipeline: the entry words of the next batch (PIPE:
// also the next batch's gathers and coefficients, and the words of the one
// after it) are in flight while a batch is multiplied, across the units' borders (the last level's rows hold one batch each,
// so without this every unit would wait for three dependent reads).

__device__ __forceinline__ double lanes_sum(double v, int sp) {
  for (int o = 32 >> sp; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float lanes_sum(float v, int sp) {
  for (int o = 32 >> sp; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ DF lanes_sum(DF v, int sp) {
  for (int o = 32 >> sp; o < 32; o <<= 1)
    v = df_add(v, DF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
  return v;
}

// Arithmetic of an operator phase: coefficients C, records V, sums A.
struct K64R {   // FP64, real coefficients
  static constexpr bool PIPE = false;   // the second set of gathers spills: 16.5 against 11.5 us on d = 100's red rows
  using C = double;
  using V = double2;
  using A = double;
  static constexpr int NB = 4;
  static __device__ __forceinline__ const C* coef(const OpView& op) { return reinterpret_cast<const double*>(op.ecoef); }
  static __device__ __forceinline__ C czero() { return 0.0; }
  static __device__ __forceinline__ V vzero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ A zero() { return 0.0; }
  static __device__ __forceinline__ V conj(V v, bool c, uint32_t e) {
    v.y = conj_if(v.y, c, e);
    return v;
  }
  static __device__ __forceinline__ void mad(A& ar, A& ai, C c, V v) {
    ar = fma(c, v.x, ar);
    ai = fma(c, v.y, ai);
  }
  static __device__ __forceinline__ V pack(A ar, A ai) { return make_double2(ar, ai); }
  static __device__ __forceinline__ void set(A& ar, A& ai, V v) {
    ar = v.x;
    ai = v.y;
  }
};
struct K64C : K64R {   // FP64, complex coefficients
  using C = double2;
  static __device__ __forceinline__ const C* coef(const OpView& op) { return op.ecoef; }
  static __device__ __forceinline__ C czero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ void mad(A& ar, A& ai, C c, V v) {
    ar = fma(c.x, v.x, ar);
    ar = fma(-c.y, v.y, ar);
    ai = fma(c.x, v.y, ai);
    ai = fma(c.y, v.x, ai);
  }
};
struct K32R {   // FP32, real coefficients
  static constexpr bool PIPE = true;
  using C = float;
  using V = float2;
  using A = float;
  static constexpr int NB = 4;
  static __device__ __forceinline__ const C* coef(const OpView& op) { return reinterpret_cast<const float*>(op.ecoef32); }
  static __device__ __forceinline__ C czero() { return 0.f; }
  static __device__ __forceinline__ V vzero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ A zero() { return 0.f; }
  static __device__ __forceinline__ V conj(V v, bool c, uint32_t e) {
    v.y = conj_if(v.y, c, e);
    return v;
  }
  static __device__ __forceinline__ void mad(A& ar, A& ai, C c, V v) {
    ar = fmaf(c, v.x, ar);
    ai = fmaf(c, v.y, ai);
  }
  static __device__ __forceinline__ V pack(A ar, A ai) { return make_float2(ar, ai); }
};
struct K32C : K32R {   // FP32, complex coefficients
  using C = float2;
  static __device__ __forceinline__ const C* coef(const OpView& op) { return op.ecoef32; }
  static __device__ __forceinline__ C czero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ void mad(A& ar, A& ai, C c, V v) {
    ar = fmaf(c.x, v.x, ar);
    ar = fmaf(-c.y, v.y, ar);
    ai = fmaf(c.x, v.y, ai);
    ai = fmaf(c.y, v.x, ai);
  }
};
struct KDF {   // double-float
  static constexpr bool PIPE = false;
  using C = float4;
  using V = float4;
  using A = DF;
  static constexpr int NB = 2;
  static __device__ __forceinline__ const C* coef(const OpView& op) { return op.ecoefdf; }
  static __device__ __forceinline__ C czero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ V vzero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ A zero() { return DF{0.f, 0.f}; }
  static __device__ __forceinline__ V conj(V v, bool c, uint32_t e) {
    v.z = conj_if(v.z, c, e);
    v.w = conj_if(v.w, c, e);
    return v;
  }
  static __device__ __forceinline__ void mad(A& ar, A& ai, C c, V v) {
    df_fma(ar, re_of(c), re_of(v));
    df_fma(ai, re_of(c), im_of(v));
    if (c.z != 0.f || c.w != 0.f) {   // complex coefficients
      df_fma(ar, df_neg(im_of(c)), im_of(v));
      df_fma(ai, im_of(c), re_of(v));
    }
  }
  static __device__ __forceinline__ V pack(A ar, A ai) { return cdf(ar, ai); }
  static __device__ __forceinline__ void set(A& ar, A& ai, V v) {
    ar = re_of(v);
    ai = im_of(v);
  }
};

// Entry words of one batch, and where its coefficients and row are.
template <int NB>
struct Words {
  uint32_t e[NB];
  int64_t at;          // first coefficient of the lane
  int32_t row;         // the lane's row
  int32_t left;        // entries of the lane's row from this batch's first on
  bool on, first, last, ok;   // row of the phase's colour; first, last batch of its unit; there is a batch
};

// row(g, y) receives every row's product, on one lane per row.  The sum starts
// at start(g, x), x the row's own record (nullptr: at zero).
template <class K, bool SKIP, class Row, class Start = std::nullptr_t>
__device__ __forceinline__ void op_phase(const SolveParams& P, const SmemS& sm, const Units& U, int tab,
                                         const typename K::V* rec, Row row, Start start = nullptr) {
  using V = typename K::V;
  using W = Words<K::NB>;
  const OpView& op = P.op;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sp = U.split[tab], rows = 32 >> sp, n = U.n[tab], ns = 1 << sp;
  const int64_t step = unit_step();
  const typename K::C* coef = K::coef(op);
  // cursor of the batch to fetch next
  int64_t it = unit_first();
  if (it >= n) return;
  const int tfirst = SKIP && op.diag0 ? 1 : 0;
  int k = 0, t = tfirst;
  int4 u = sm.meta[tab][warp][0];
  auto fetch = [&]() {
    W b;
    b.ok = it < n;
    if (!b.ok) return b;
    const int rl = (int)(it & (ns - 1)) * rows + (lane & (rows - 1));
    b.row = u.x * kSlice + rl;
    b.on = (uint32_t)u.w >> rl & 1u;
    const int t0 = t + (lane >> (5 - sp));
    b.left = (b.on && (SKIP || b.row != P.zero_row) ? u.z : 0) - t0;
    b.at = ((int64_t)u.y + t0) * kSlice + rl;
#pragma unroll
    for (int q = 0; q < K::NB; ++q)
      b.e[q] = q * ns < b.left ? __ldg(op.ent + b.at + (int64_t)q * ns * kSlice) : op.pad;
    b.first = t == tfirst;
    t += K::NB * ns;
    b.last = t >= u.z;   // warp-uniform
    if (b.last) {
      t = tfirst;
      it += step;
      if (it < n) u = ++k < kMeta ? sm.meta[tab][warp][k] : load_unit(P, tab, sp, it);
    }
    return b;
  };
  auto gather = [&](const W& b, V* v, typename K::C* c) {
#pragma unroll
    for (int q = 0; q < K::NB; ++q) {
      v[q] = __ldcg(rec + (b.e[q] & op.colmask));
      c[q] = q * ns < b.left ? __ldg(coef + b.at + (int64_t)q * ns * kSlice) : K::czero();
    }
  };
  typename K::A ar = K::zero(), ai = K::zero();
  W b0 = fetch(), b1;
  V v0[K::NB], v1[K::PIPE ? K::NB : 1];
  typename K::C c0[K::NB], c1[K::PIPE ? K::NB : 1];
  if constexpr (K::PIPE) {
    b1 = fetch();
    gather(b0, v0, c0);
  }
#pragma unroll 1
  for (;;) {
    W b2;
    if constexpr (K::PIPE) {
      if (b1.ok) gather(b1, v1, c1);
      b2 = fetch();
    } else {
      gather(b0, v0, c0);
      b1 = fetch();
    }
    if constexpr (!std::is_same<Start, std::nullptr_t>::value) {
      if (b0.first && b0.on && lane < rows) K::set(ar, ai, start((int64_t)b0.row, __ldcg(rec + b0.row)));
    }
#pragma unroll
    for (int q = 0; q < K::NB; ++q) {
      V v = K::conj(v0[q], op.conj, b0.e[q]);
      if (SKIP && !op.diag0 && (b0.e[q] & op.colmask) == (uint32_t)b0.row) v = K::vzero();
      K::mad(ar, ai, c0[q], v);
    }
    if (b0.last) {
      V y = K::pack(lanes_sum(ar, sp), lanes_sum(ai, sp));
      if (b0.on && lane < rows) {
        if (!SKIP && b0.row == P.zero_row) y = __ldcg(rec + b0.row);   // the identity row
        row((int64_t)b0.row, y);
      }
      ar = ai = K::zero();
    }
    if (!b1.ok) break;
    b0 = b1;
    if constexpr (K::PIPE) {
      b1 = b2;
#pragma unroll
      for (int q = 0; q < K::NB; ++q) {
        v0[q] = v1[q];
        c0[q] = c1[q];
      }
    }
  }
}

// Statistics of a single solve (block 0).
__device__ __forceinline__ void put_stats(const SolveParams& P, const SmemS& sm, double rr, int iters, int inner,
                                          int outer, int applies, int status) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  InstState& st = P.state[0];
  st.bb = sm.bb;
  st.rr = rr;
  st.iters = iters;
  st.inner_iters = inner;
  st.outer_iters = outer;
  st.applies = applies;
  st.status = status;
}

// The sum over the black rows into v[2].
template <class K64>
__device__ __forceinline__ void one_black_rr(const SolveParams& P, const SmemS& sm, const Units& U, double* v) {
  const SolveInst& in = P.inst[0];
  BlackRow r;
  op_phase<K64, true>(P, sm, U, kOpB, P.xrec, [&](int64_t, double2 s) { v[2] += r.norm2(P, in, s); },
                      [&](int64_t g, double2 x) { return r.start(P, in, g, x); });
}
// The residual of all rows in FP64.
template <class K64>
__device__ __forceinline__ void one_rr(const SolveParams& P, const SmemS& sm, const Units& U, bool show, double* v) {
  const SolveInst& in = P.inst[0];
  if (show) one_black_rr<K64>(P, sm, U, v);
  op_phase<K64, false>(P, sm, U, kOpR, P.xrec, [&](int64_t g, double2 y) {
    const double2 f = f_at(in, g);
    const double rx = f.x - y.x, ry = f.y - y.y;
    v[2] = fma(rx, rx, fma(ry, ry, v[2]));
  });
}

template <class K64>
__device__ __forceinline__ void one_fp64(const SolveParams& P, SmemS& sm) {
  const double tol2 = P.tol * P.tol;
  const bool colours = has_black(P), scaled = P.op.scaled;
  const SolveInst& in = P.inst[0];
  // r = D u (D the Jacobi diagonal, u = D^-1 r the gathered record): the
  // vector phase updates u directly, the apply phase forms <r, u> = sum D |u|^2
  // and <r, r> = sum D^2 |u|^2; P.r holds D.  A scaled table's black rows hold
  // -D^-1 C^H already.
  double* dg = reinterpret_cast<double*>(P.r);
  const Units U = setup_units(P, sm);
  int par = 0;
  auto black_x = [&](int64_t g, double2 y) {   // D^-1 (f - C^H x_R), y the row's product
    const double2 f = f_at(in, g);
    double2 x = scaled ? y : make_double2(-y.x, -y.y);
    if (!scaled) {
      const double rD = P.rdiag[g];
      return make_double2(rD * (f.x - y.x), rD * (f.y - y.y));
    }
    if (f.x != 0.0 || f.y != 0.0) {
      const double rD = 1.0 / jacobi(P, in, g);
      x.x = fma(rD, f.x, x.x);
      x.y = fma(rD, f.y, x.y);
    }
    return x;
  };
  // x_R = 0, x_B = D^-1 f_B; |f|^2 of both
  {
    double v[kNQ] = {};   // q2: black, q3: red
    if (colours)
      rows_phase(P, sm, U, kOpB, [&](int64_t g) {
        const double2 f = f_at(in, g);
        if (!scaled) P.rdiag[g] = 1.0 / jacobi(P, in, g);
        P.xrec[g] = black_x(g, make_double2(0.0, 0.0));
        if (f.x != 0.0 || f.y != 0.0) v[2] += f.x * f.x + f.y * f.y;
      });
    rows_phase(P, sm, U, kVec, [&](int64_t g) {
      const double2 f = f_at(in, g);
      const double dk = jacobi(P, in, g), rD = 1.0 / dk;
      P.rdiag[g] = rD;
      dg[g] = dk;
      P.xrec[g] = make_double2(0.0, 0.0);
      P.urec64[g] = make_double2(f.x * rD, f.y * rD);
      P.pd[g] = make_double2(0.0, 0.0);
      P.sd[g] = make_double2(0.0, 0.0);
      v[3] += f.x * f.x + f.y * f.y;
    });
    if (!sync_sum(P, sm, par, v)) return;
    all_sums(P, sm, par);
    if (threadIdx.x == 0) {
      sm.bb = sm.t[2] + sm.t[3];
      sm.stop = tol2 * sm.bb;
    }
  }
  if (colours && sm.t[2] != 0.0) {   // u = D^-1 r, r = f_R - C D_B^-1 f_B; nothing to add when f_B = 0
    op_phase<K64, false>(P, sm, U, kOpR, P.xrec, [&](int64_t g, double2 y) {
      const double2 f = f_at(in, g);
      const double rD = __ldcg(P.rdiag + g);
      P.urec64[g] = make_double2((f.x - y.x) * rD, (f.y - y.y) * rD);
    });
    if (!sync_all(P, sm)) return;
  }
  auto apply = [&]() -> bool {
    if (colours) {
      op_phase<K64, true>(P, sm, U, kOpB, P.urec64, [&](int64_t g, double2 y) {
        if (!scaled) {
          const double rD = __ldcg(P.rdiag + g);
          y = make_double2(-rD * y.x, -rD * y.y);
        }
        P.urec64[g] = y;
      });
      if (!sync_all(P, sm)) return false;
    }
    double v[kNQ] = {};
    op_phase<K64, false>(P, sm, U, kOpR, P.urec64, [&](int64_t g, double2 w) {
      const double2 u = __ldcg(P.urec64 + g);
      const double dk = __ldcg(dg + g);
      P.w64[g] = w;
      const double du = dk * fma(u.y, u.y, u.x * u.x);   // D |u|^2 = <r, u> of this row
      v[0] += du;
      v[1] = fma(w.y, u.y, fma(w.x, u.x, v[1]));
      v[2] = fma(dk, du, v[2]);                           // |r|^2 = D^2 |u|^2
    });
    return sync_sum(P, sm, par, v);
  };
  int it = 0, applies = 1, status = SS_OK;
  for (;; ++it) {
    if (!apply()) return;
    all_sums(P, sm, par);
    if (threadIdx.x < 32) {
      const bool conv = sm.t[2] <= sm.stop, cap = it >= P.max_iter;
      const Coeffs cf = one_coeffs(sm, it);
      if (threadIdx.x == 0) {
        sm.go = conv ? 1 : (cap ? 2 : 0);
        sm.ca = cf.alpha;
        sm.cb = cf.beta;
      }
    }
    __syncthreads();
    if (sm.go) break;
    const double a = sm.ca, b = sm.cb;
    rows_phase(P, sm, U, kVec, [&](int64_t g) {
      double2 u = __ldcg(P.urec64 + g), w = __ldcg(P.w64 + g);
      double2 p = P.pd[g], sv = P.sd[g], x = P.xrec[g];
      const double rD = P.rdiag[g];
      p.x = u.x + b * p.x; p.y = u.y + b * p.y;
      sv.x = w.x + b * sv.x; sv.y = w.y + b * sv.y;
      x.x += a * p.x; x.y += a * p.y;
      const double t = a * rD;   // u - alpha D^-1 s = D^-1 (r - alpha s)
      u.x = fma(-t, sv.x, u.x);
      u.y = fma(-t, sv.y, u.y);
      P.pd[g] = p;
      P.sd[g] = sv;
      P.xrec[g] = x;
      P.urec64[g] = u;
    });
    ++applies;
    if (!sync_all(P, sm)) return;
  }
  if (sm.go == 2) status = SS_ERR_NOT_CONVERGED;
  // x_B, the output, and the true residual f - L x in FP64
  double v[kNQ] = {};
  const bool show = sm.t[2] <= kShow * sm.bb;
  if (colours) {
    op_phase<K64, true>(P, sm, U, kOpB, P.xrec, [&](int64_t g, double2 y) {
      const double2 x = black_x(g, y);
      P.xrec[g] = x;
      const int64_t l = g - in.row0;
      if (l < in.rows) in.u[l] = x;
    });
    if (!sync_all(P, sm)) return;
    if (show) one_black_rr<K64>(P, sm, U, v);
  }
  op_phase<K64, false>(P, sm, U, kOpR, P.xrec, [&](int64_t g, double2 y) {
    const double2 f = f_at(in, g);
    const double2 r = make_double2(f.x - y.x, f.y - y.y);
    v[2] = fma(r.x, r.x, fma(r.y, r.y, v[2]));
    const int64_t l = g - in.row0;
    if (l < in.rows) in.u[l] = __ldcg(P.xrec + g);
  });
  if (!sync_sum(P, sm, par, v)) return;
  if (blockIdx.x == 0) {
    all_sums(P, sm, par);
    put_stats(P, sm, sm.t[2], it, 0, 1, applies + 1, status);
  }
}

__device__ __forceinline__ void one_df64(const SolveParams& P, SmemS& sm) {
  const double tol2 = P.tol * P.tol;
  const bool colours = has_black(P), scaled = P.op.scaled;
  const SolveInst& in = P.inst[0];
  float4* r4 = reinterpret_cast<float4*>(P.r);
  float4* w4 = reinterpret_cast<float4*>(P.w64);
  float4* p4 = reinterpret_cast<float4*>(P.pd);
  float4* s4 = reinterpret_cast<float4*>(P.sd);
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const Units U = setup_units(P, sm);
  int par = 0;
  auto rdiag = [&](int64_t g) {
    const float2 d = __ldcg(P.d32 + g);
    return DF{d.x, d.y};
  };
  auto black_x = [&](int64_t g, float4 y) {
    const double2 f = f_at(in, g);
    if (!scaled) {
      const DF rD = rdiag(g);
      return cdf(df_mul(rD, df_sub(df_split(f.x), re_of(y))), df_mul(rD, df_sub(df_split(f.y), im_of(y))));
    }
    if (f.x != 0.0 || f.y != 0.0) {
      const DF rD = df_split(1.0 / jacobi(P, in, g));
      DF a = re_of(y), b = im_of(y);
      df_fma(a, rD, df_split(f.x));
      df_fma(b, rD, df_split(f.y));
      return cdf(a, b);
    }
    return y;
  };
  {
    double v[kNQ] = {};   // q2: black, q3: red
    if (colours)
      rows_phase(P, sm, U, kOpB, [&](int64_t g) {
        const double2 f = f_at(in, g);
        if (!scaled) {
          const DF rD = df_split(1.0 / jacobi(P, in, g));
          P.d32[g] = make_float2(rD.hi, rD.lo);
        }
        P.xdf[g] = black_x(g, z4);
        if (f.x != 0.0 || f.y != 0.0) v[2] += f.x * f.x + f.y * f.y;
      });
    rows_phase(P, sm, U, kVec, [&](int64_t g) {
      const double2 f = f_at(in, g);
      const DF rD = df_split(1.0 / jacobi(P, in, g)), fr = df_split(f.x), fi = df_split(f.y);
      P.d32[g] = make_float2(rD.hi, rD.lo);
      r4[g] = cdf(fr, fi);
      P.xdf[g] = z4;
      P.udf[g] = cdf(df_mul(rD, fr), df_mul(rD, fi));
      p4[g] = z4;
      s4[g] = z4;
      v[3] += f.x * f.x + f.y * f.y;
    });
    if (!sync_sum(P, sm, par, v)) return;
    all_sums(P, sm, par);
    if (threadIdx.x == 0) {
      sm.bb = sm.t[2] + sm.t[3];
      sm.stop = tol2 * sm.bb;
    }
  }
  if (colours && sm.t[2] != 0.0) {
    op_phase<KDF, false>(P, sm, U, kOpR, P.xdf, [&](int64_t g, float4 y) {
      const float4 f = __ldcg(r4 + g);
      const DF rr = df_sub(re_of(f), re_of(y)), ri = df_sub(im_of(f), im_of(y)), rD = rdiag(g);
      r4[g] = cdf(rr, ri);
      P.udf[g] = cdf(df_mul(rD, rr), df_mul(rD, ri));
    });
    if (!sync_all(P, sm)) return;
  }
  auto apply = [&]() -> bool {
    if (colours) {
      op_phase<KDF, true>(P, sm, U, kOpB, P.udf, [&](int64_t g, float4 y) {
        if (!scaled) {
          const DF rD = df_neg(rdiag(g));
          y = cdf(df_mul(rD, re_of(y)), df_mul(rD, im_of(y)));
        }
        P.udf[g] = y;
      });
      if (!sync_all(P, sm)) return false;
    }
    const DF z{0.f, 0.f};
    DF v[kNQ] = {z, z, z, z};
    op_phase<KDF, false>(P, sm, U, kOpR, P.udf, [&](int64_t g, float4 w) {
      const float4 u = __ldcg(P.udf + g), r = __ldcg(r4 + g);
      w4[g] = w;
      df_fma(v[0], re_of(r), re_of(u));
      df_fma(v[0], im_of(r), im_of(u));
      df_fma(v[1], re_of(w), re_of(u));
      df_fma(v[1], im_of(w), im_of(u));
      df_fma(v[2], re_of(r), re_of(r));
      df_fma(v[2], im_of(r), im_of(r));
    });
    return sync_sum(P, sm, par, v);
  };
  int it = 0, applies = 1, status = SS_OK;
  for (;; ++it) {
    if (!apply()) return;
    all_sums(P, sm, par);
    if (threadIdx.x < 32) {
      const bool conv = sm.t[2] <= sm.stop, cap = it >= P.max_iter;
      const Coeffs cf = one_coeffs(sm, it);
      if (threadIdx.x == 0) {
        sm.go = conv ? 1 : (cap ? 2 : 0);
        const DF a = df_split(cf.alpha), b = df_split(cf.beta);
        sm.dfs[0] = a.hi;
        sm.dfs[1] = a.lo;
        sm.dfs[2] = b.hi;
        sm.dfs[3] = b.lo;
      }
    }
    __syncthreads();
    if (sm.go) break;
    const DF a{sm.dfs[0], sm.dfs[1]}, b{sm.dfs[2], sm.dfs[3]}, na = df_neg(a);
    rows_phase(P, sm, U, kVec, [&](int64_t g) {
      const float4 u = __ldcg(P.udf + g), w = __ldcg(w4 + g), po = p4[g], so = s4[g], xo = P.xdf[g],
                   ro = __ldcg(r4 + g);
      DF pr = re_of(u), pi = im_of(u), sr = re_of(w), si = im_of(w);
      df_fma(pr, b, re_of(po));
      df_fma(pi, b, im_of(po));
      df_fma(sr, b, re_of(so));
      df_fma(si, b, im_of(so));
      DF xr = re_of(xo), xi = im_of(xo), rr = re_of(ro), ri = im_of(ro);
      df_fma(xr, a, pr);
      df_fma(xi, a, pi);
      df_fma(rr, na, sr);
      df_fma(ri, na, si);
      const DF rD = rdiag(g);
      p4[g] = cdf(pr, pi);
      s4[g] = cdf(sr, si);
      P.xdf[g] = cdf(xr, xi);
      r4[g] = cdf(rr, ri);
      P.udf[g] = cdf(df_mul(rD, rr), df_mul(rD, ri));
    });
    ++applies;
    if (!sync_all(P, sm)) return;
  }
  if (sm.go == 2) status = SS_ERR_NOT_CONVERGED;
  const bool show = colours && sm.t[2] <= kShowDf * sm.bb;
  auto put = [&](int64_t g, float4 x4) {   // the output, and the FP64 record of the residual
    const double2 x = make_double2(df_to_double(re_of(x4)), df_to_double(im_of(x4)));
    P.xrec[g] = x;
    const int64_t l = g - in.row0;
    if (l < in.rows) in.u[l] = x;
  };
  if (colours) op_phase<KDF, true>(P, sm, U, kOpB, P.xdf, [&](int64_t g, float4 y) { put(g, black_x(g, y)); });
  rows_phase(P, sm, U, kVec, [&](int64_t g) { put(g, P.xdf[g]); });
  if (!sync_all(P, sm)) return;
  double v[kNQ] = {};
  if (P.op.realc) one_rr<K64R>(P, sm, U, show, v);
  else one_rr<K64C>(P, sm, U, show, v);
  if (!sync_sum(P, sm, par, v)) return;
  if (blockIdx.x == 0) {
    all_sums(P, sm, par);
    put_stats(P, sm, sm.t[2], it, 0, 1, applies + 1, status);
  }
}

// FP32 CG in FP64 refinement.  The FP32 operator reads FP32 copies of the
// entry coefficients and compact 8-byte records.
template <class K64, class K32>
__device__ __forceinline__ void one_refined(const SolveParams& P, SmemS& sm) {
  const double tol2 = P.tol * P.tol, itol2 = P.inner_tol * P.inner_tol;
  const bool colours = has_black(P), scaled = P.op.scaled;
  const SolveInst& in = P.inst[0];
  float* rd32 = reinterpret_cast<float*>(P.dlt);         // 1 / D in FP32
  float2* rec = reinterpret_cast<float2*>(P.urec32);     // u on the red rows, v on the black ones
  const Units U = setup_units(P, sm);
  int par = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) rec[P.op.pad] = make_float2(0.f, 0.f);
  int inner = 0, applies = 0, status = SS_OK, ot = 0;
  double rr = 0.0;
  for (;; ++ot) {
    // the black rows solved for the current x_R (FP64): x_B = D^-1 (f_B - C^H x_R)
    // (x_R = 0 at first), then rhat = f - L64 x on the red rows
    double v[kNQ] = {};
    if (colours) {
      auto put = [&](int64_t g, double2 y) {
        const double2 f = f_at(in, g);
        double2 x = y;
        if (!scaled) {
          const double rD = P.rdiag[g];
          x = make_double2(rD * (f.x - y.x), rD * (f.y - y.y));
        } else if (f.x != 0.0 || f.y != 0.0) {
          const double rD = 1.0 / jacobi(P, in, g);
          x.x = fma(rD, f.x, x.x);
          x.y = fma(rD, f.y, x.y);
        }
        P.xrec[g] = x;
      };
      if (ot == 0)
        rows_phase(P, sm, U, kOpB, [&](int64_t g) {
          if (!scaled) {
            P.rdiag[g] = 1.0 / jacobi(P, in, g);
            rd32[g] = 1.0f / jacobi32(P, in, g);
          }
          put(g, make_double2(0.0, 0.0));
          const double2 f = f_at(in, g);
          if (f.x != 0.0 || f.y != 0.0) v[2] += f.x * f.x + f.y * f.y;
        });
      else
        op_phase<K64, true>(P, sm, U, kOpB, P.xrec, put);
    }
    if (ot == 0) {
      rows_phase(P, sm, U, kVec, [&](int64_t g) {
        const double2 f = f_at(in, g);
        rd32[g] = 1.0f / jacobi32(P, in, g);
        P.xrec[g] = make_double2(0.0, 0.0);
        P.rhat[g] = f;
        v[3] += f.x * f.x + f.y * f.y;
      });
      if (!sync_sum(P, sm, par, v)) return;
      all_sums(P, sm, par);
      rr = sm.t[3];
      if (threadIdx.x == 0) sm.bb = sm.t[2] + sm.t[3];
    } else if (colours) {
      if (!sync_all(P, sm)) return;
    }
    if (ot > 0 || (colours && sm.t[2] != 0.0)) {   // at first rhat = f when f_B = 0
      double r2[kNQ] = {};
      op_phase<K64, false>(P, sm, U, kOpR, P.xrec, [&](int64_t g, double2 y) {
        const double2 f = f_at(in, g);
        const double2 r = make_double2(f.x - y.x, f.y - y.y);
        P.rhat[g] = r;
        r2[2] = fma(r.x, r.x, fma(r.y, r.y, r2[2]));
      });
      if (!sync_sum(P, sm, par, r2)) return;
      all_sums(P, sm, par);
      rr = sm.t[2];
    }
    ++applies;
    if (threadIdx.x == 0) {   // one thread: FP64 operations of a whole block would cost microseconds
      const double sc = inner_scale(rr, in.rows);
      sm.go = rr <= tol2 * sm.bb ? 1 : (ot >= P.max_outer ? 2 : 0);
      sm.sc = sc;
      sm.us = 1.0 / sc;
      sm.stop = itol2 * rr * sc * sc;   // r32 carries the scale
    }
    __syncthreads();
    if (sm.go) break;
    // inner start (all FP32): r = rhat * scale, delta = 0, u = D^-1 r, p = s = 0
    const double sc = sm.sc;
    rows_phase(P, sm, U, kVec, [&](int64_t g) {
      const double2 rh = __ldcg(P.rhat + g);
      const float2 r = make_float2((float)(rh.x * sc), (float)(rh.y * sc));
      const float rD = rd32[g];
      P.r32[g] = r;
      P.d32[g] = make_float2(0.f, 0.f);
      P.p32[g] = make_float2(0.f, 0.f);
      P.s32[g] = make_float2(0.f, 0.f);
      rec[g] = make_float2(r.x * rD, r.y * rD);
    });
    if (!sync_all(P, sm)) return;
    // inner CG to the relative tolerance 1e-5: inner products summed in FP32
    // per lane and warp, in FP64 from there on; scalars FP64
    auto apply = [&]() -> bool {
      if (colours) {
        op_phase<K32, true>(P, sm, U, kOpB, rec, [&](int64_t g, float2 y) {
          if (!scaled) {
            const float rD = -rd32[g];
            y = make_float2(rD * y.x, rD * y.y);
          }
          rec[g] = y;
        });
        if (!sync_all(P, sm)) return false;
      }
      float q[kNQ] = {};
      op_phase<K32, false>(P, sm, U, kOpR, rec, [&](int64_t g, float2 w) {
        const float2 u = __ldcg(rec + g), r = __ldcg(P.r32 + g);
        P.w32[g] = w;
        q[0] += r.x * u.x + r.y * u.y;
        q[1] += w.x * u.x + w.y * u.y;
        q[2] += r.x * r.x + r.y * r.y;
      });
      return sync_sum(P, sm, par, q);
    };
    ++applies;
    for (int it = 0;; ++it) {
      if (!apply()) return;
      all_sums(P, sm, par);
      if (threadIdx.x < 32) {
        const bool done = sm.t[2] <= sm.stop || it >= P.max_inner;
        const Coeffs cf = one_coeffs(sm, it);
        if (threadIdx.x == 0) {
          sm.go = done;
          sm.ca = cf.alpha;
          sm.cb = cf.beta;
        }
      }
      __syncthreads();
      if (sm.go) break;
      const float a = (float)sm.ca, b = (float)sm.cb;
      rows_phase(P, sm, U, kVec, [&](int64_t g) {
        const float2 u = __ldcg(rec + g), w = __ldcg(P.w32 + g);
        float2 p = P.p32[g], sv = P.s32[g], dl = P.d32[g], r = __ldcg(P.r32 + g);
        const float rD = rd32[g];
        p.x = fmaf(b, p.x, u.x); p.y = fmaf(b, p.y, u.y);
        sv.x = fmaf(b, sv.x, w.x); sv.y = fmaf(b, sv.y, w.y);
        dl.x = fmaf(a, p.x, dl.x); dl.y = fmaf(a, p.y, dl.y);
        r.x = fmaf(-a, sv.x, r.x); r.y = fmaf(-a, sv.y, r.y);
        P.p32[g] = p;
        P.s32[g] = sv;
        P.d32[g] = dl;
        P.r32[g] = r;
        rec[g] = make_float2(r.x * rD, r.y * rD);
      });
      ++inner;
      ++applies;
      if (!sync_all(P, sm)) return;
    }
    // x_R += delta
    const double us = sm.us;
    rows_phase(P, sm, U, kVec, [&](int64_t g) {
      double2 x = P.xrec[g];
      const float2 dl = P.d32[g];
      x.x += (double)dl.x * us;
      x.y += (double)dl.y * us;
      P.xrec[g] = x;
    });
    if (!sync_all(P, sm)) return;
  }
  auto put = [&](int64_t g) {
    const int64_t l = g - in.row0;
    if (l < in.rows) in.u[l] = __ldcg(P.xrec + g);
  };
  if (colours) rows_phase(P, sm, U, kOpB, put);
  rows_phase(P, sm, U, kVec, put);
  if (sm.go == 2) status = SS_ERR_NOT_CONVERGED;
  if (colours && rr <= kShow * sm.bb) {   // the black rows' part of the residual
    double v[kNQ] = {};
    one_black_rr<K64>(P, sm, U, v);
    if (!sync_sum(P, sm, par, v)) return;
    if (blockIdx.x == 0) {
      all_sums(P, sm, par);
      rr += sm.t[2];
    }
  }
  put_stats(P, sm, rr, 0, inner, ot, applies, status);
}

// ------------------------------------------------- BiCGStab (ADR operator)
//
// The operator of Remark ADR is not Hermitian.  BiCGStab (van der Vorst, 1992)
// with right Jacobi preconditioning y = D^-1 p, D = diag L (complex), and the
// shadow residual r^ = r_0 = f:
//   rho = <r^, r>, beta = (rho / rho_prev) (alpha / omega)
//   p = r + beta (p - omega v),  v = L D^-1 p
//   alpha = rho / <r^, v>,  s = r - alpha v,  x += alpha D^-1 p
//   t = L D^-1 s,  omega = <t, s> / <t, t>,  x += omega D^-1 s,  r = s - omega t
// with <a, b> = sum conj(a) b.  Five phases per iteration, each closed by a
// grid barrier; every block recomputes the scalars from the deterministic
// partial sums, and the owner keeps rho, alpha and omega by iteration parity.
// The half step stops the iteration when |s| already meets the tolerance
// (x = x + alpha y is then the answer).  A vanishing or non-finite scalar
// restarts the direction (beta = 0) or skips the step (alpha or omega = 0);
// the iteration cap then reports non-convergence.

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double n = b.x * b.x + b.y * b.y;
  if (n == 0.0) return make_double2(0.0, 0.0);
  return make_double2((a.x * b.x + a.y * b.y) / n, (a.y * b.x - a.x * b.y) / n);
}
__device__ __forceinline__ double2 finite_or_zero(double2 a) {
  return (isfinite(a.x) && isfinite(a.y)) ? a : make_double2(0.0, 0.0);
}
// conj(a) b
__device__ __forceinline__ double2 cdot(double2 a, double2 b) {
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

__device__ void solve_bicgstab(const SolveParams& P, Smem& sm) {
  const double tol2 = P.tol * P.tol;
  // x = 0, r = r^ = f, p = v = 0, dlt = D^-1;  <r^, r> = |f|^2 + 0 i (q0, q1), |r|^2 (q2), |f|^2 (q3).
  // q1 is written (as zero) too: the first iteration reads rho = (q0, q1),
  // and a slot left out would hold whatever an earlier phase or solve left there.
  run_phase(P, sm, kAll, 0b1111u, nullptr, [&](int64_t g, int64_t, int, int i, int, double* v) {
    const double2 f = f_at(P.inst[i], g);
    P.xrec[g] = make_double2(0.0, 0.0);
    P.r[g] = f;
    P.rhat[g] = f;
    P.pd[g] = make_double2(0.0, 0.0);
    P.w64[g] = make_double2(0.0, 0.0);
    P.dlt[g] = cdiv(make_double2(1.0, 0.0), __ldg(P.cdiag + g));
    const double ff = f.x * f.x + f.y * f.y;
    v[0] += ff;
    v[2] += ff;
    v[3] += ff;
  });
  if (!grid_sync(P, sm)) return;
  for (int it = 0;; ++it) {
    const int cur = it & 1, nxt = cur ^ 1;
    // A: test, beta; p = r + beta (p - omega v); y = D^-1 p (records of urec64)
    run_phase(P, sm, kAll, 0u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      double t[kNQ];
      inst_sums(P, i, 0, t);
      if (lane == 0) {
        InstState& st = P.state[i];
        // inn[par]: the instance finished at the half step of that iteration
        const int act = it == 0 ? 1 : (__ldcg(&st.act[cur]) && !__ldcg(&st.inn[cur]));
        const double bb = it == 0 ? t[3] : __ldcg(&st.bb);
        const bool conv = t[2] <= tol2 * bb;
        const bool cap = it >= P.max_iter;
        const bool go = act && !conv && !cap;
        const double2 rho = make_double2(t[0], t[1]);
        double2 beta = make_double2(0.0, 0.0), om = make_double2(0.0, 0.0);
        if (it > 0) {
          om = __ldcg(&st.zomega[cur]);
          beta = finite_or_zero(cmul(cdiv(rho, __ldcg(&st.zrho[cur])), cdiv(__ldcg(&st.zalpha[cur]), om)));
        }
        sm.flag[k] = go;
        sm.ca[k] = beta.x;
        sm.cb[k] = beta.y;
        sm.cc[k] = om.x;
        sm.cd[k] = om.y;
        if (owner) {
          if (it == 0) {
            st.bb = bb;
            st.outer_iters = 1;
          }
          st.act[nxt] = go;
          st.zrho[nxt] = rho;
          if (act) {
            st.rr = t[2];
            st.iters = it;
            if (conv) owner_done(P, st, SS_OK);
            else if (cap) owner_done(P, st, SS_ERR_NOT_CONVERGED);
          }
        }
      }
    }, [&](int64_t g, int64_t, int, int, int k, double*) {
      if (!sm.flag[k]) return;
      const double2 beta = make_double2(sm.ca[k], sm.cb[k]), om = make_double2(sm.cc[k], sm.cd[k]);
      const double2 r = P.r[g], v = P.w64[g];
      double2 p = P.pd[g];
      const double2 q = make_double2(p.x - (om.x * v.x - om.y * v.y), p.y - (om.x * v.y + om.y * v.x));
      p = make_double2(r.x + (beta.x * q.x - beta.y * q.y), r.y + (beta.x * q.y + beta.y * q.x));
      P.pd[g] = p;
      P.urec64[g] = cmul(P.dlt[g], p);
    });
    if (!grid_sync(P, sm)) return;
    if (block_counter(P, 0) >= P.n_inst) break;
    // B: v = L y;  <r^, v>
    run_phase(P, sm, kAll, 0b0011u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      if (lane == 0) {
        sm.flag[k] = __ldcg(&P.state[i].act[nxt]);
        if (owner && sm.flag[k]) P.state[i].applies += 1;
      }
    }, [&](int64_t g, int64_t s, int lane, int i, int k, double* v) {
      if (!sm.flag[k]) return;
      const double2 w = apply64_row(P, P.inst[i], s, lane, g, P.urec64);
      P.w64[g] = w;
      const double2 q = cdot(P.rhat[g], w);
      v[0] += q.x;
      v[1] += q.y;
    });
    if (!grid_sync(P, sm)) return;
    // C: alpha = rho / <r^, v>; s = r - alpha v; x += alpha y; z = D^-1 s;  |s|^2
    run_phase(P, sm, kAll, 0b0100u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      double t[kNQ];
      inst_sums(P, i, 0, t);
      if (lane == 0) {
        InstState& st = P.state[i];
        const double2 alpha = finite_or_zero(cdiv(__ldcg(&st.zrho[nxt]), make_double2(t[0], t[1])));
        sm.flag[k] = __ldcg(&st.act[nxt]);
        sm.ca[k] = alpha.x;
        sm.cb[k] = alpha.y;
        if (owner) st.zalpha[nxt] = alpha;
      }
    }, [&](int64_t g, int64_t, int, int, int k, double* vq) {
      if (!sm.flag[k]) return;
      const double2 alpha = make_double2(sm.ca[k], sm.cb[k]);
      const double2 r = P.r[g], v = P.w64[g], y = P.urec64[g];
      const double2 av = cmul(alpha, v), ay = cmul(alpha, y);
      const double2 s = make_double2(r.x - av.x, r.y - av.y);
      double2 x = P.xrec[g];
      x.x += ay.x;
      x.y += ay.y;
      P.xrec[g] = x;
      P.sd[g] = s;
      P.zrec[g] = cmul(P.dlt[g], s);
      vq[2] += s.x * s.x + s.y * s.y;
    });
    if (!grid_sync(P, sm)) return;
    // D: half-step test on |s|; t = L z;  <t, s>, <t, t>
    run_phase(P, sm, kAll, 0b0111u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      double t[kNQ];
      inst_sums(P, i, 0, t);
      if (lane == 0) {
        InstState& st = P.state[i];
        const int act = __ldcg(&st.act[nxt]);
        const bool half = act && t[2] <= tol2 * __ldcg(&st.bb);
        sm.flag[k] = act && !half;
        if (owner) {
          st.inn[nxt] = half;
          if (half) {
            st.rr = t[2];
            st.iters = it + 1;
            owner_done(P, st, SS_OK);
          } else if (act) {
            st.applies += 1;
          }
        }
      }
    }, [&](int64_t g, int64_t s, int lane, int i, int k, double* v) {
      if (!sm.flag[k]) return;
      const double2 t = apply64_row(P, P.inst[i], s, lane, g, P.zrec);
      P.tv[g] = t;
      const double2 q = cdot(t, P.sd[g]);
      v[0] += q.x;
      v[1] += q.y;
      v[2] += t.x * t.x + t.y * t.y;
    });
    if (!grid_sync(P, sm)) return;
    // E: omega = <t, s> / <t, t>; x += omega z; r = s - omega t;  <r^, r>, |r|^2
    run_phase(P, sm, kAll, 0b0111u, [&](const Chunk&, int k, int i, bool owner, int lane) {
      double t[kNQ];
      inst_sums(P, i, 0, t);
      if (lane == 0) {
        InstState& st = P.state[i];
        const double2 om =
            finite_or_zero(t[2] > 0.0 ? make_double2(t[0] / t[2], t[1] / t[2]) : make_double2(0.0, 0.0));
        sm.flag[k] = __ldcg(&st.act[nxt]) && !__ldcg(&st.inn[nxt]);
        sm.ca[k] = om.x;
        sm.cb[k] = om.y;
        if (owner) st.zomega[nxt] = om;
      }
    }, [&](int64_t g, int64_t, int, int, int k, double* v) {
      if (!sm.flag[k]) return;
      const double2 om = make_double2(sm.ca[k], sm.cb[k]);
      const double2 s = P.sd[g], t = P.tv[g], z = P.zrec[g];
      const double2 oz = cmul(om, z), ot = cmul(om, t);
      double2 x = P.xrec[g];
      x.x += oz.x;
      x.y += oz.y;
      P.xrec[g] = x;
      const double2 r = make_double2(s.x - ot.x, s.y - ot.y);
      P.r[g] = r;
      const double2 q = cdot(P.rhat[g], r);
      v[0] += q.x;
      v[1] += q.y;
      v[2] += r.x * r.x + r.y * r.y;
    });
    if (!grid_sync(P, sm)) return;
  }
  // true residual f - L x in FP64, and the output
  run_phase(P, sm, kAll, 0b0100u, nullptr, [&](int64_t g, int64_t s, int lane, int i, int, double* v) {
    const SolveInst& in = P.inst[i];
    const double2 y = apply64_row(P, in, s, lane, g, P.xrec);
    const double2 f = f_at(in, g);
    const double2 r = make_double2(f.x - y.x, f.y - y.y);
    v[2] += r.x * r.x + r.y * r.y;
    const int64_t l = g - in.row0;
    if (l < in.rows) in.u[l] = P.xrec[g];
  });
  if (!grid_sync(P, sm)) return;
  final_rr(P);
}

// The general phases (batches, the allocation-free solve, ADR, one instance on
// blocks of 1024 threads), or one instance's own (real or complex entry
// coefficients apart: half the live registers).
template <int MODE>
__global__ void __launch_bounds__(1024) k_solve(SolveParams P) {
  __shared__ Smem sm;
  if (threadIdx.x == 0) sm.bar.target = 0;   // ordered by the block barriers of the first phase
  if constexpr (MODE == 0) solve_fp64(P, sm);
  else if constexpr (MODE == 1) solve_refined(P, sm);
  else solve_bicgstab(P, sm);
}

template <int MODE, bool REAL, int MAXT>
__global__ void __launch_bounds__(MAXT) k_solve_one(SolveParams P) {
  __shared__ SmemS sm;
  if (threadIdx.x == 0) sm.bar.target = 0;   // ordered by the block barrier of setup_units
  using K64 = typename std::conditional<REAL, K64R, K64C>::type;
  using K32 = typename std::conditional<REAL, K32R, K32C>::type;
  if constexpr (MODE == 0) one_fp64<K64>(P, sm);
  else if constexpr (MODE == 1) one_refined<K64, K32>(P, sm);
  else one_df64(P, sm);
}

constexpr int kOneThreads = 512;   // largest block of the one-instance kernels at 128 registers

// Whether a mode runs the one-instance kernel on blocks of `block` threads.
bool one_kernel(int mode, bool single, int block) {
  return single && mode != 2 && (mode == 3 || block <= kOneThreads);
}

// The kernel of a mode for blocks of `block` threads.
using SolveKernel = void (*)(SolveParams);
SolveKernel solve_kernel(int mode, bool single, int block, bool real) {
  if (!one_kernel(mode, single, block)) return mode == 0 ? k_solve<0> : (mode == 1 ? k_solve<1> : k_solve<2>);
  if (mode == 0) return real ? k_solve_one<0, true, kOneThreads> : k_solve_one<0, false, kOneThreads>;
  if (mode == 1) return real ? k_solve_one<1, true, kOneThreads> : k_solve_one<1, false, kOneThreads>;
  return block <= kOneThreads ? k_solve_one<3, false, kOneThreads> : k_solve_one<3, false, 1024>;
}

__global__ void k_init_solve_records(const int64_t* __restrict__ norm, int64_t n, const int8_t* __restrict__ wide_rows,
                                     bool wide, double2* xrec, double2* prec64, float4* prec32) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n) return;
  const int64_t nr = norm[g];
  const bool wd = wide_rows ? wide_rows[g] != 0 : wide;
  xrec[g] = make_double2(0.0, 0.0);
  prec64[g] = make_double2(0.0, 0.0);
  prec32[g] = make_float4(0.f, 0.f, __int_as_float(norm_word(nr, wd)), 0.f);
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// Everything a single-instance solve writes before its kernel starts, in one
// launch of one block: the barrier, counter and error words, the instance
// state, one caller word (the half system's Hermitian flag), the instance
// descriptor and, when the plan is new, the lists of the slices that hold red
// and black rows, in slice order (from the colour masks; without colours only
// the count).  Computed here because the masks live on the device: no read-back
// between the stamp and the solve.  If the stamp's build reported an error
// (err[0]; its check may still be pending) both lists are empty and the solve
// reads no entry.
constexpr int kPlanThreads = 1024;

struct Prologue {
  unsigned* bar;
  int* counters;
  int* err;
  InstState* state;
  int32_t* extra;
  SolveInst* inst_dst;
  SolveInst inst;
  int lists;                 // write n_items and the lists
  const uint32_t* black;     // colour masks, or null
  int64_t n;                 // slices
  const int32_t* stamp_err;
  int32_t* list[2];
  int32_t* n_items;
};

__global__ void __launch_bounds__(kPlanThreads) k_solve_prologue(Prologue p) {
  const int tid = threadIdx.x;
  if (tid < 2) p.bar[tid] = 0u;
  if (tid < 4) p.counters[tid] = 0;
  if (tid == 0) {
    *p.err = 0;
    if (p.extra) *p.extra = 0;
    *p.inst_dst = p.inst;
  }
  static_assert(sizeof(InstState) % sizeof(int32_t) == 0, "InstState is zeroed in 32-bit words");
  for (int i = tid; i < (int)(sizeof(InstState) / sizeof(int32_t)); i += blockDim.x)
    reinterpret_cast<int32_t*>(p.state)[i] = 0;
  if (!p.lists) return;
  if (!p.black || __ldg(p.stamp_err) != 0) {
    if (tid == 0) {
      p.n_items[0] = __ldg(p.stamp_err) != 0 ? 0 : (int32_t)p.n;
      p.n_items[1] = 0;
    }
    return;
  }
  // thread t takes the slices [t q, (t + 1) q): count, block scan, write
  __shared__ int2 s_warp[kPlanThreads / 32];
  const int lane = tid & 31, warp = tid >> 5;
  const int64_t q = (p.n + kPlanThreads - 1) / kPlanThreads;
  const int64_t s0 = tid * q < p.n ? tid * q : p.n, s1 = s0 + q < p.n ? s0 + q : p.n;
  int red = 0, blk = 0;
  for (int64_t s = s0; s < s1; ++s) {
    const uint32_t m = __ldg(p.black + s);
    red += m != 0xffffffffu;
    blk += m != 0u;
  }
  int r = red, k = blk;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, r, o), b = __shfl_up_sync(0xffffffffu, k, o);
    if (lane >= o) {
      r += a;
      k += b;
    }
  }
  if (lane == 31) s_warp[warp] = make_int2(r, k);
  __syncthreads();
  int2 before = make_int2(0, 0), all = make_int2(0, 0);
  for (int w = 0; w < kPlanThreads / 32; ++w) {
    const int2 v = s_warp[w];
    if (w < warp) {
      before.x += v.x;
      before.y += v.y;
    }
    all.x += v.x;
    all.y += v.y;
  }
  r += before.x - red;
  k += before.y - blk;
  for (int64_t s = s0; s < s1; ++s) {
    const uint32_t m = __ldg(p.black + s);
    if (m != 0xffffffffu) p.list[0][r++] = (int32_t)s;
    if (m != 0u) p.list[1][k++] = (int32_t)s;
  }
  if (tid == 0) {
    p.n_items[0] = all.x;
    p.n_items[1] = all.y;
  }
}

}  // namespace

// ---------------------------------------------------------------- host side

// The single-instance plan: K chunks that take the colours' slices in turn (one
// partial slot per chunk and colour); the lists are written by the prologue.
static void plan_single(SolvePlan& plan, int64_t n_slices, int target, const uint32_t* black,
                        const int32_t* stamp_err) {
  const int K = (int)std::max<int64_t>(1, std::min<int64_t>(target, n_slices));
  plan.n_chunks[0] = K;
  plan.n_chunks[1] = black ? K : 0;
  plan.n_parts = 2 * K;   // both colours, or the two alternating sets of one instance's solver
  SolveInst& in = plan.inst[0];
  for (int ci = 0; ci < 2; ++ci) {
    in.c_first[ci] = 0;
    in.c_last[ci] = plan.n_chunks[ci] - 1;
    in.part_base[ci] = ci * K;
  }
  plan.single = true;
  plan.lists_pending = true;
  plan.n_slices = n_slices;
  plan.black = black;
  plan.stamp_err = stamp_err;
}

// The prologue of a single-instance plan into the given words and tables; the
// slice lists only when the plan's are not there yet.
static ss_status launch_prologue(SolvePlan& plan, unsigned* bar, int* counters, int* err, InstState* state,
                                 int32_t* extra, SolveInst* inst_dst, int32_t* lists, cudaStream_t st) {
  Prologue p{};
  p.bar = bar;
  p.counters = counters;
  p.err = err;
  p.state = state;
  p.extra = extra;
  p.inst_dst = inst_dst;
  p.inst = plan.inst[0];
  p.lists = plan.lists_pending ? 1 : 0;
  p.black = plan.black;
  p.n = plan.n_slices;
  p.stamp_err = plan.stamp_err;
  p.n_items = lists;
  p.list[0] = lists + 2;
  p.list[1] = lists + 2 + plan.n_slices;
  k_solve_prologue<<<1, kPlanThreads, 0, st>>>(p);
  SS_LAUNCH_CHECK();
  plan.lists_pending = false;
  return SS_OK;
}

ss_status plan_chunks(SolvePlan& plan, const std::vector<int32_t>& woff, const std::vector<int32_t>& slice_inst,
                      const std::vector<uint32_t>& black, int target_chunks) {
  const int64_t n_slices = (int64_t)woff.size() - 1;
  const int n_inst = (int)plan.inst.size();
  if (n_slices <= 0) SS_FAIL(SS_ERR_INVALID, "solve: empty operator");
  plan.single = false;
  plan.n_slices = n_slices;
  int32_t base = 0;
  for (int ci = 0; ci < 2; ++ci) {
    std::vector<Chunk>& chunk = plan.chunk[ci];
    std::vector<int32_t>& list = plan.list[ci];
    chunk.clear();
    list.clear();
    for (int64_t s = 0; s < n_slices; ++s) {
      const uint32_t m = black.empty() ? 0u : black[s];
      if (ci == 0 ? m != 0xffffffffu : m != 0u) list.push_back((int32_t)s);
    }
    // weight of a slice: its entries (gathers) plus the vector work of 32 rows
    // (the black rows keep no CG vectors)
    auto weight = [&](int32_t s) { return (double)(woff[s + 1] - woff[s]) + (ci == 0 ? 6.0 : 2.0); };
    double total = 0;
    for (int32_t s : list) total += weight(s);
    const double target = total / std::max(1, target_chunks);
    const int64_t n = (int64_t)list.size();
    int64_t i0 = 0;
    double acc = 0;
    for (int64_t i = 0; i < n; ++i) {
      acc += weight(list[i]);
      const bool last = i + 1 == n;
      bool cut = last || acc >= target;
      if (!last && slice_inst[list[i + 1]] - slice_inst[list[i0]] + 1 > kMaxInstPerChunk) cut = true;
      if (cut) {
        chunk.push_back(Chunk{i0, i + 1, slice_inst[list[i0]], slice_inst[list[i]]});
        i0 = i + 1;
        acc = 0;
      }
    }
    for (auto& in : plan.inst) {
      in.c_first[ci] = 0;
      in.c_last[ci] = -1;
    }
    for (int c = 0; c < (int)chunk.size(); ++c)
      for (int i = chunk[c].inst0; i <= chunk[c].inst1; ++i) {
        SolveInst& in = plan.inst[i];
        if (in.c_last[ci] < 0) in.c_first[ci] = c;
        in.c_last[ci] = c;
      }
    for (int i = 0; i < n_inst; ++i) {
      SolveInst& in = plan.inst[i];
      if (ci == 0 && in.c_last[0] < 0) SS_FAIL(SS_ERR_INVALID, "solve: instance %d has no rows", i);
      in.part_base[ci] = base;
      base += in.c_last[ci] - in.c_first[ci] + 1;
    }
    plan.n_chunks[ci] = (int)chunk.size();
  }
  plan.n_parts = base;
  return SS_OK;
}

ss_status work_alloc(SolveWork& W, int64_t rows_total, const int64_t* norm, const int8_t* wide_rows, bool wide,
                     cudaStream_t st) {
  if (W.rows_total == rows_total) return SS_OK;
  if (W.cap_rows >= rows_total) {
    // a workspace kept from an earlier stamp: new records, same buffers
    W.rows_total = rows_total;
    k_init_solve_records<<<nblk(rows_total), 256, 0, st>>>(norm, rows_total, wide_rows, wide, W.xrec.get(),
                                                           W.urec64.get(), W.urec32.get());
    SS_LAUNCH_CHECK();
    return SS_OK;
  }
  W.rows_total = rows_total;
  W.cap_rows = rows_total;
  W.df_rows = W.bi_rows = -1;
  {
    // one allocation, carved in 256-byte aligned pieces
    size_t off = 0;
    auto take = [&](auto& view, size_t count) {
      using T = typename std::remove_pointer<decltype(view.p)>::type;
      view.p = reinterpret_cast<T*>(off);   // offset for now, rebased below
      off += (count * sizeof(T) + 255) / 256 * 256;
    };
    const size_t n = (size_t)rows_total;
    take(W.xrec, n); take(W.urec64, n); take(W.urec32, n); take(W.r, n); take(W.w64, n); take(W.w32, n);
    take(W.pd, n); take(W.sd, n); take(W.rhat, n); take(W.dlt, n); take(W.r32, n); take(W.p32, n);
    take(W.s32, n); take(W.d32, n); take(W.rdiag, n); take(W.bar, 2); take(W.counters, 4); take(W.err, 1);
    take(W.list, solve_list_words(rows_total / kSlice));
    SS_TRY(W.arena.alloc(off, st));
    const uintptr_t b = reinterpret_cast<uintptr_t>(W.arena.get());
    auto rebase = [&](auto& view) {
      using T = typename std::remove_pointer<decltype(view.p)>::type;
      view.p = reinterpret_cast<T*>(b + reinterpret_cast<uintptr_t>(view.p));
    };
    rebase(W.xrec); rebase(W.urec64); rebase(W.urec32); rebase(W.r); rebase(W.w64); rebase(W.w32);
    rebase(W.pd); rebase(W.sd); rebase(W.rhat); rebase(W.dlt); rebase(W.r32); rebase(W.p32);
    rebase(W.s32); rebase(W.d32); rebase(W.rdiag); rebase(W.bar); rebase(W.counters); rebase(W.err);
    rebase(W.list);
  }
  k_init_solve_records<<<nblk(rows_total), 256, 0, st>>>(norm, rows_total, wide_rows, wide, W.xrec.get(),
                                                         W.urec64.get(), W.urec32.get());
  SS_LAUNCH_CHECK();
  // The workspace is reused by later calls, possibly on other streams: both
  // callers synchronise `st` before they return (solve when it reads the
  // statistics, batch_create right after this), which orders those calls
  // after these allocations.
  W.arena.settle();
  return SS_OK;
}

ss_status work_alloc_bicgstab(SolveWork& W, cudaStream_t st) {
  if (W.zrec.n >= (size_t)W.rows_total && W.tv.n >= (size_t)W.rows_total) {
    if (W.bi_rows != W.rows_total) {   // the dummy row of this row count must read as zero
      SS_CUDA(cudaMemsetAsync(W.zrec.get() + (W.rows_total - 1), 0, sizeof(double2), st));
      W.bi_rows = W.rows_total;
    }
    return SS_OK;
  }
  W.bi_rows = W.rows_total;
  SS_TRY(W.zrec.alloc(W.rows_total, st));
  SS_TRY(W.tv.alloc(W.rows_total, st));
  SS_CUDA(cudaMemsetAsync(W.zrec.get(), 0, W.rows_total * sizeof(double2), st));
  SS_CUDA(cudaStreamSynchronize(st));
  W.zrec.settle();
  W.tv.settle();
  return SS_OK;
}

ss_status work_alloc_df64(SolveWork& W, cudaStream_t st) {
  if (W.xdf.n >= (size_t)W.rows_total && W.udf.n >= (size_t)W.rows_total) {
    if (W.df_rows != W.rows_total) {   // the dummy record of this row count must read as zero
      SS_CUDA(cudaMemsetAsync(W.xdf.get() + (W.rows_total - 1), 0, sizeof(float4), st));
      SS_CUDA(cudaMemsetAsync(W.udf.get() + (W.rows_total - 1), 0, sizeof(float4), st));
      W.df_rows = W.rows_total;
    }
    return SS_OK;
  }
  W.df_rows = W.rows_total;
  SS_TRY(W.xdf.alloc(W.rows_total, st));
  SS_TRY(W.udf.alloc(W.rows_total, st));
  // the dummy record (last row) must read as zero
  SS_CUDA(cudaMemsetAsync(W.xdf.get(), 0, W.rows_total * sizeof(float4), st));
  SS_CUDA(cudaMemsetAsync(W.udf.get(), 0, W.rows_total * sizeof(float4), st));
  SS_CUDA(cudaStreamSynchronize(st));
  W.xdf.settle();
  W.udf.settle();
  return SS_OK;
}

ss_status work_upload(SolveWork& W, SolvePlan& plan, bool lists, cudaStream_t st) {
  const int n_inst = (int)plan.inst.size();
  if (n_inst > W.cap_inst) { SS_TRY(W.inst.alloc(n_inst, st)); SS_TRY(W.state.alloc(n_inst, st)); W.cap_inst = n_inst; }
  if (plan.n_parts > W.cap_parts) { SS_TRY(W.part.alloc(plan.n_parts * kNQ, st)); W.cap_parts = plan.n_parts; }
  if (!plan.single && plan.n_chunks[0] + plan.n_chunks[1] > W.cap_chunk) {
    W.cap_chunk = plan.n_chunks[0] + plan.n_chunks[1];
    SS_TRY(W.chunk.alloc(W.cap_chunk, st));
  }
  W.inst.settle(); W.state.settle(); W.chunk.settle(); W.part.settle();   // reused across calls (see read_stats)
  if (plan.single) return SS_OK;   // descriptor, lists and zeroed words: work_prologue
  SS_TRY(upload(st, {{W.inst.get(), plan.inst.data(), n_inst * sizeof(SolveInst)}}));
  if (!lists) return SS_OK;
  int32_t* l = W.list.get();
  return upload(st, {{W.chunk.get(), plan.chunk[0].data(), plan.chunk[0].size() * sizeof(Chunk)},
                     {W.chunk.get() + plan.n_chunks[0], plan.chunk[1].data(), plan.chunk[1].size() * sizeof(Chunk)},
                     {l + 2, plan.list[0].data(), plan.list[0].size() * sizeof(int32_t)},
                     {l + 2 + plan.n_slices, plan.list[1].data(), plan.list[1].size() * sizeof(int32_t)}});
}

// The prologue of a single-instance plan into its workspace (after
// work_upload); `extra` is one more word to zero (or null).  The solve is then
// launched with zeroed = true.
static ss_status work_prologue(SolveWork& W, SolvePlan& plan, int32_t* extra, cudaStream_t st) {
  return launch_prologue(plan, W.bar.get(), W.counters.get(), W.err.get(), W.state.get(), extra, W.inst.get(),
                         W.list.get(), st);
}

ss_status max_grid(int mode, bool single, bool real, int block, int* grid) {
  // resident blocks per SM, looked up once per device, kernel and block size
  static std::mutex mu;
  static int cache[64][16][4] = {};
  const int kid = mode + (single ? 4 : 0) + (real ? 8 : 0);
  int dev = 0;
  SS_CUDA(cudaGetDevice(&dev));
  const int bi = block == 128 ? 0 : block == 256 ? 1 : block == 512 ? 2 : 3;
  if (dev >= 0 && dev < 64 && mode >= 0 && mode < 4) {
    std::lock_guard<std::mutex> lk(mu);
    if (cache[dev][kid][bi] > 0) {
      *grid = cache[dev][kid][bi] * sm_count();
      return SS_OK;
    }
  }
  int nb = 0;
  SS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, solve_kernel(mode, single, block, real), block, 0));
  if (nb < 1) SS_FAIL(SS_ERR_CUDA, "solve: kernel does not fit on an SM with %d threads", block);
  if (dev >= 0 && dev < 64 && mode >= 0 && mode < 4) {
    std::lock_guard<std::mutex> lk(mu);
    cache[dev][kid][bi] = nb;
  }
  *grid = nb * sm_count();
  return SS_OK;
}

// The work split of a plan: its chunk tables and slice lists.
static void set_split(SolveParams& P, const SolvePlan& plan, const Chunk* chunk, const int32_t* lists) {
  P.n_slices = plan.n_slices;
  P.black = plan.black;
  P.n_items = plan.single ? lists : nullptr;
  for (int ci = 0; ci < 2; ++ci) {
    P.n_chunks[ci] = plan.n_chunks[ci];
    P.chunk[ci] = plan.single ? nullptr : chunk + ci * plan.n_chunks[0];
    P.list[ci] = plan.black ? lists + 2 + ci * plan.n_slices : nullptr;
  }
}

// Fill params and launch (capturable: no host synchronisation).
ss_status launch_solve(SolveWork& W, const SolvePlan& plan, const OpView& op, const int32_t* slice_inst,
                       const int64_t* norm, const double2* ca64, const float2* ca32, const int32_t* pn,
                       double tol, int max_iter, int mode, cudaStream_t st, cudaEvent_t ev_begin,
                       cudaEvent_t ev_end, const double2* cdiag, bool zeroed) {
  if (mode == 2 && (!cdiag || !W.zrec.get() || !W.tv.get()))
    SS_FAIL(SS_ERR_INVALID, "solve: BiCGStab needs the operator diagonal and its workspace");
  if (mode == 3 && (!op.ecoefdf || !W.xdf.get() || !W.udf.get()))
    SS_FAIL(SS_ERR_INVALID, "solve: DF64 CG needs double-float coefficients and its workspace");
  SolveParams P{};
  P.n_inst = (int)plan.inst.size();
  const bool one = one_kernel(mode, plan.single, plan.block);
  if (one && mode == 1 && !op.ecoef32) SS_FAIL(SS_ERR_INVALID, "solve: the refined solve needs FP32 coefficients");
  P.zero_row = plan.inst[0].zero_row;
  set_split(P, plan, W.chunk.get(), W.list.get());
  P.inst = W.inst.get();
  P.state = W.state.get();
  P.op = op;
  P.slice_inst = slice_inst;
  P.norm = norm;
  P.ca64 = ca64;
  P.ca32 = ca32;
  P.pn = pn;
  P.xrec = W.xrec.get();
  P.urec64 = W.urec64.get();
  P.urec32 = W.urec32.get();
  P.r = W.r.get();
  P.w64 = W.w64.get();
  P.w32 = W.w32.get();
  P.pd = W.pd.get();
  P.sd = W.sd.get();
  P.rhat = W.rhat.get();
  P.dlt = W.dlt.get();
  P.r32 = W.r32.get();
  P.p32 = W.p32.get();
  P.s32 = W.s32.get();
  P.d32 = W.d32.get();
  P.rdiag = W.rdiag.get();
  P.cdiag = cdiag;
  P.zrec = W.zrec.get();
  P.tv = W.tv.get();
  P.xdf = W.xdf.get();
  P.udf = W.udf.get();
  P.part = W.part.get();
  P.bar = W.bar.get();
  P.counters = W.counters.get();
  P.err = W.err.get();
  P.tol = tol;
  P.inner_tol = 1e-5;
  P.max_iter = max_iter;
  P.max_inner = std::max(1, std::min(max_iter, 200));
  P.max_outer = std::max(1, max_iter);
  P.spin_limit = plan.spin_limit;   // 2 s unless solve_set_wait_limit changed it
  if (!zeroed) {
    SS_TRY(fill_small(st, {{W.bar.get(), 2 * sizeof(unsigned), 0}, {W.counters.get(), 4 * sizeof(int), 0}}));
    SS_CUDA(cudaMemsetAsync(W.err.get(), 0, sizeof(int), st));
    SS_CUDA(cudaMemsetAsync(W.state.get(), 0, plan.inst.size() * sizeof(InstState), st));
  }
  // cooperative launch: all blocks co-resident (required by the grid barrier);
  // expressed as a launch attribute so that it can be captured in a graph
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.grid);
  cfg.blockDim = dim3(plan.block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (ev_begin) SS_CUDA(cudaEventRecord(ev_begin, st));
  {
    static const char* const names[4] = {"k_solve<0>", "k_solve<1>", "k_solve<2>", "k_solve<3>"};
    ProfScope prof_(names[mode & 3], st, true);
    SS_CUDA(cudaLaunchKernelEx(&cfg, solve_kernel(mode, plan.single, plan.block, op.realc), P));
  }
  if (ev_end) SS_CUDA(cudaEventRecord(ev_end, st));
  return SS_OK;
}

ss_status read_stats(SolveWork& W, int n_inst, ss_solve_stats* stats, ss_status* worst, cudaStream_t st,
                     cudaEvent_t ev_begin, cudaEvent_t ev_end) {
  std::vector<InstState> hs(n_inst);
  int herr = 0;
  SS_TRY(read_back(st, {{hs.data(), W.state.get(), n_inst * sizeof(InstState)}, {&herr, W.err.get(), sizeof(int)}}));
  float kms = 0.f;
  if (ev_begin && ev_end) cudaEventElapsedTime(&kms, ev_begin, ev_end);
  *worst = SS_OK;
  if (herr) {
    *worst = (ss_status)herr;
    set_error("solve: a device-side wait gave up (status %d)", herr);
  }
  for (int i = 0; i < n_inst; ++i) {
    const InstState& s = hs[i];
    if (stats) {
      stats[i].status = herr ? herr : s.status;
      stats[i].outer_iters = s.outer_iters;
      stats[i].inner_iters = s.inner_iters ? s.inner_iters : s.iters;
      stats[i].applies = s.applies;
      stats[i].rel_residual = s.bb > 0 ? std::sqrt(s.rr / s.bb) : 0.0;
      stats[i].kernel_ms = kms;
      stats[i].half_system = 0;
      stats[i].real_coefficients = 0;
    }
    if (*worst == SS_OK && s.status != SS_OK) {
      *worst = (ss_status)s.status;
      set_error("solve: instance %d did not converge (relative residual %.3e)", i,
                s.bb > 0 ? std::sqrt(s.rr / s.bb) : 0.0);
    }
  }
  return SS_OK;
}

}  // namespace ss

// ------------------------------------------------------- per-stamp solve state

struct ss_solve_ctx {
  ss::SolveWork work;
  ss::SolvePlan plan;
  int planned_mode = -1;
  int block = 512, blocks_per_sm = 1, chunks_per_block = 1;   // tile shape (solve_set_config)
  long long wait_ns = 2000000000ll;   // grid-barrier wait bound (solve_set_wait_limit)
  double2* f0_host = nullptr;   // pinned copy of f_hat_0, checked after the solve's own synchronisation
  // Hermitian half system (FP64 CG): its own plan and workspace, the compact
  // right-hand side and solution, and the "f is not Hermitian" flag
  bool use_half = true;
  ss_solve_ctx* half = nullptr;
  ss::DevBuf<double2> fh, uh;
  ss::DevBuf<int32_t> hflag;
  int32_t* hflag_host = nullptr;
  int32_t* chk_host = nullptr;   // pinned copy of a pending stamp's error words (stamp_build_pending)
  ~ss_solve_ctx() {
    if (f0_host) cudaFreeHost(f0_host);
    if (hflag_host) cudaFreeHost(hflag_host);
    if (chk_host) cudaFreeHost(chk_host);
    delete half;
  }
};

namespace ss {

static ss_status stamp_plan(ss_stamp_s* s, ss_solve_ctx& C, int mode, cudaStream_t st) {
  if (C.planned_mode == mode) return SS_OK;
  if (!s->slice_off.get() || s->n_slices < 1) SS_FAIL(SS_ERR_INVALID, "solve: stamp has no slice table");
  C.plan.inst.assign(1, SolveInst{});
  SolveInst& in = C.plan.inst[0];
  in.row0 = 0;
  in.rows = s->size;
  in.rows_pad = s->rows_pad;
  in.zero_row = identity_row(s);
  in.coef_off = 0;
  in.dscale = 2.0 * kTwoPiSq * s->a0;   // 4 pi^2 Re(a_hat_0)
  in.wide = s->wide ? 1 : 0;
  int grid = 0;
  C.plan.block = C.block;
  SS_TRY(max_grid(mode, mode != 2, s->a_real, C.plan.block, &grid));
  if (C.blocks_per_sm > 0) grid = std::min(grid, C.blocks_per_sm * sm_count());
  const int by_size = (int)std::max<int64_t>(1, s->n_slices / 8);   // at least 8 slices per chunk
  const int target = std::min<int64_t>((int64_t)grid * C.chunks_per_block, by_size);
  plan_single(C.plan, s->n_slices, target, s->colours && mode != 2 ? s->cmask.get() : nullptr, s->err_dev.get());
  C.plan.grid = std::min<int>(grid, C.plan.n_chunks[0]);
  SS_TRY(work_alloc(C.work, s->rows_pad + 1, s->norm.get(), nullptr, s->wide, st));
  if (mode == 2) SS_TRY(work_alloc_bicgstab(C.work, st));
  if (mode == 1) SS_TRY(ensure_ecoef32(s, false, st));
  if (mode == 3) {
    SS_TRY(ensure_ecoefdf(s, st));
    SS_TRY(work_alloc_df64(C.work, st));
  }
  C.planned_mode = mode;   // the plan goes to the device with the call's f and u (solve)
  return SS_OK;
}

// Plan and workspace of the Hermitian half system (FP64, FP32-refined and DF64 modes).
static ss_status stamp_plan_half(ss_stamp_s* s, ss_solve_ctx& H, int mode, cudaStream_t st) {
  if (H.planned_mode == mode) return SS_OK;
  if (!s->woff_h.get() || s->n_slices_h < 1) SS_FAIL(SS_ERR_INVALID, "solve: no half-system table");
  H.plan.inst.assign(1, SolveInst{});
  SolveInst& in = H.plan.inst[0];
  in.row0 = 0;
  in.rows = s->n_plus;
  in.rows_pad = s->rows_pad_h;
  in.zero_row = -1;                      // k = 0 is not a row of the half system
  in.coef_off = 0;
  in.dscale = 2.0 * kTwoPiSq * s->a0;
  in.wide = s->wide ? 1 : 0;
  int grid = 0;
  H.plan.block = H.block;
  SS_TRY(max_grid(mode, true, s->a_real, H.plan.block, &grid));
  if (H.blocks_per_sm > 0) grid = std::min(grid, H.blocks_per_sm * sm_count());
  const int by_size = (int)std::max<int64_t>(1, s->n_slices_h / 8);
  const int target = std::min<int64_t>((int64_t)grid * H.chunks_per_block, by_size);
  plan_single(H.plan, s->n_slices_h, target, s->colours ? s->cmask_h.get() : nullptr, s->err_dev.get());
  H.plan.grid = std::min<int>(grid, H.plan.n_chunks[0]);
  SS_TRY(work_alloc(H.work, s->rows_pad_h + 1, s->norm_h.get(), nullptr, s->wide, st));
  if (mode == 1) SS_TRY(ensure_ecoef32(s, true, st));
  if (mode == 3) {
    SS_TRY(ensure_ecoefdf_half(s, st));
    SS_TRY(work_alloc_df64(H.work, st));
  }
  H.planned_mode = mode;
  return SS_OK;
}

namespace {

// Compact right-hand side f_h[i] = f[k_i] (k_i > 0); flags an f that is not
// Hermitian (f_{-k} != conj(f_k) bit for bit) so the full system is solved instead.
__global__ void k_half_gather(const double2* __restrict__ f, const int32_t* __restrict__ plus_rows,
                              const int64_t* __restrict__ mirror, int64_t n_plus, double2* f_h, int32_t* flag) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_plus) return;
  const int64_t g = plus_rows[i];
  const int64_t m = mirror[g];   // -1: -k not found (the stamp's check fails): solved as the full system
  const double2 a = f[g];
  if (m < 0) {
    atomicExch(flag, 1);
  } else {
    const double2 b = f[m];
    if (!(a.x == b.x && a.y == -b.y)) atomicExch(flag, 1);
  }
  f_h[i] = a;
}

// u on S from the compact solution: u_k (k > 0), conj(u_{-k}) (k < 0), 0 (k = 0).
__global__ void k_half_scatter(const double2* __restrict__ u_h, const int32_t* __restrict__ hpos, int64_t size,
                               int64_t n_plus, double2* u) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= size) return;
  const int32_t h = hpos[g];
  // positions outside the compact rows only come from a half system whose
  // build failed (reported by the stamp's check); nothing is read there
  if (h == -1 || h >= n_plus || (h < -1 && -2 - (int64_t)h >= n_plus)) {
    u[g] = make_double2(0.0, 0.0);
  } else if (h >= 0) {
    u[g] = u_h[h];
  } else {
    const double2 v = u_h[-2 - h];
    u[g] = make_double2(v.x, -v.y);
  }
}

}  // namespace

}  // namespace ss

using namespace ss;

// The per-stamp context lives in a side table keyed by the stamp pointer so
// that the stamp layout stays independent of the solver.
#include <mutex>
#include <unordered_map>
static std::mutex g_ctx_mu;
static std::unordered_map<const ss_stamp_s*, ss_solve_ctx*> g_ctx;

namespace ss {
// Contexts of destroyed stamps are kept (a few) with their device buffers and
// given to the next stamps: a new stamp then needs no allocation for its
// solves, only new records (work_alloc re-initialises them for its rows).
static std::vector<ss_solve_ctx*> g_spare_ctx;
constexpr size_t kMaxSpareCtx = 4;

static void reset_ctx(ss_solve_ctx* C) {
  C->planned_mode = -1;
  C->work.rows_total = 0;
  C->block = 512;
  C->blocks_per_sm = 1;
  C->chunks_per_block = 1;
  C->use_half = true;
  C->wait_ns = 2000000000ll;
  if (C->half) reset_ctx(C->half);
}

void drop_solve_ctx(const ss_stamp_s* s) {
  std::lock_guard<std::mutex> lk(g_ctx_mu);
  auto it = g_ctx.find(s);
  if (it != g_ctx.end()) {
    ss_solve_ctx* C = it->second;
    g_ctx.erase(it);
    if (g_spare_ctx.size() < kMaxSpareCtx) {
      reset_ctx(C);
      g_spare_ctx.push_back(C);
    } else {
      delete C;
    }
  }
}
}  // namespace ss

static ss_solve_ctx* solve_ctx(const ss_stamp_s* s) {
  std::lock_guard<std::mutex> lk(g_ctx_mu);
  auto& slot = g_ctx[s];
  if (!slot) {
    if (!g_spare_ctx.empty()) {
      slot = g_spare_ctx.back();
      g_spare_ctx.pop_back();
    } else {
      slot = new ss_solve_ctx();
    }
  }
  return slot;
}

extern "C" ss_status solve_set_config(ss_stamp s, int32_t block, int32_t blocks_per_sm, int32_t chunks_per_block) {
  if (!s || (block != 128 && block != 256 && block != 512 && block != 1024) || blocks_per_sm < 0 ||
      chunks_per_block < 1)
    SS_FAIL(SS_ERR_INVALID, "solve_set_config: block in {128,256,512,1024}, blocks_per_sm >= 0, chunks >= 1");
  ss_solve_ctx* C = solve_ctx(s);
  C->block = block;
  C->blocks_per_sm = blocks_per_sm;
  C->chunks_per_block = chunks_per_block;
  C->planned_mode = -1;
  C->work.rows_total = 0;   // the records anew: the two solver kernels lay them out differently
  return SS_OK;
}

extern "C" ss_status solve_set_wait_limit(ss_stamp s, int64_t ns) {
  if (!s || ns < 0) SS_FAIL(SS_ERR_INVALID, "solve_set_wait_limit: null stamp or negative limit");
  solve_ctx(s)->wait_ns = ns == 0 ? -1 : (long long)ns;   // 0: give up at the first poll
  return SS_OK;
}

extern "C" ss_status solve_set_symmetry(ss_stamp s, int32_t use_half) {
  if (!s) SS_FAIL(SS_ERR_INVALID, "solve_set_symmetry: null stamp");
  solve_ctx(s)->use_half = use_half != 0;
  return SS_OK;
}

extern "C" ss_status solve(ss_stamp s, const double* f_on_S, double* u_on_S, double tol, int32_t max_iter,
                           ss_precision prec, ss_solve_stats* stats, void* stream) {
  if (!s || !f_on_S || !u_on_S) SS_FAIL(SS_ERR_INVALID, "solve: null argument");
  if (!(tol > 0.0) || max_iter < 1) SS_FAIL(SS_ERR_INVALID, "solve: need tol > 0 and max_iter >= 1");
  if (prec != SS_FP64 && prec != SS_FP32 && prec != SS_DF64) SS_FAIL(SS_ERR_INVALID, "solve: bad precision");
  cudaStream_t st = as_stream(stream);
  if (s->adr && prec != SS_FP64) SS_FAIL(SS_ERR_INVALID, "solve: ADR stamps solve in SS_FP64 (BiCGStab)");
  ss_solve_ctx* C = solve_ctx(s);
  // Host checks read back with the solve's statistics (one synchronisation
  // for all), queued behind the solve kernel so that they do not delay it:
  // f_hat_0 (must vanish) and the error words of a stamp whose build left
  // them to this synchronisation (the one-call pipeline).
  const bool pending = s->check_pending;
  const bool check_f0 = !s->adr && s->zero_idx >= 0;
  bool checks_queued = false;
  auto queue_checks = [&]() -> ss_status {
    if (checks_queued) return SS_OK;
    checks_queued = true;
    if (pending) {
      if (!C->chk_host) {
        note_alloc();
        SS_CUDA(cudaMallocHost(&C->chk_host, 4 * sizeof(int32_t)));
      }
      SS_CUDA(cudaMemcpyAsync(C->chk_host, s->err_dev.get(), 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    }
    if (check_f0) {
      if (!C->f0_host) {
        note_alloc();
        SS_CUDA(cudaMallocHost(&C->f0_host, sizeof(double2)));
      }
      SS_CUDA(cudaMemcpyAsync(C->f0_host, reinterpret_cast<const double2*>(f_on_S) + s->zero_idx, sizeof(double2),
                              cudaMemcpyDeviceToHost, st));
    }
    return SS_OK;
  };
  const int mode = s->adr ? 2 : (prec == SS_FP64 ? 0 : (prec == SS_FP32 ? 1 : 3));
  if (mode != 2 && s->half_ok && C->use_half) {
    // Real data: solve the Hermitian half system (rows k >lex 0, neighbours
    // below read as conjugates), then unfold; if f turns out not to be
    // Hermitian the full system below is solved instead.
    if (!C->half) C->half = new ss_solve_ctx();
    ss_solve_ctx* H = C->half;
    if (H->block != C->block || H->blocks_per_sm != C->blocks_per_sm || H->chunks_per_block != C->chunks_per_block) {
      H->block = C->block;
      H->blocks_per_sm = C->blocks_per_sm;
      H->chunks_per_block = C->chunks_per_block;
      H->planned_mode = -1;
      H->work.rows_total = 0;
    }
    SS_TRY(stamp_plan_half(s, *H, mode, st));
    SS_TRY(C->fh.ensure(s->rows_pad_h, st));
    SS_TRY(C->uh.ensure(s->rows_pad_h, st));
    SS_TRY(C->hflag.ensure(1, st));
    if (!C->hflag_host) {
      note_alloc();
      SS_CUDA(cudaMallocHost(&C->hflag_host, sizeof(int32_t)));
    }
    H->plan.inst[0].f = C->fh.get();
    H->plan.inst[0].u = C->uh.get();
    SS_TRY(work_upload(H->work, H->plan, false, st));
    SS_TRY(work_prologue(H->work, H->plan, C->hflag.get(), st));   // also clears the Hermitian flag
    const unsigned gb = (unsigned)((s->n_plus + 255) / 256), sb = (unsigned)((s->size + 255) / 256);
    k_half_gather<<<gb, 256, 0, st>>>(reinterpret_cast<const double2*>(f_on_S), s->plus_rows.get(), s->mirror.get(),
                                      s->n_plus, C->fh.get(), C->hflag.get());
    SS_LAUNCH_CHECK();
    OpView hop;
    hop.woff = s->woff_h.get();
    hop.ent = s->ent_h.get();
    hop.ecoef = s->ecoef_h.get();
    hop.ecoefdf = s->ecoefdf_h.get();
    hop.colbits = s->colbits_h;
    hop.colmask = (1u << s->colbits_h) - 1u;
    hop.jmask = (1u << s->jbits) - 1u;
    hop.conj = true;
    hop.realc = s->a_real;
    hop.ecoef32 = reinterpret_cast<const float2*>(s->ecoef32_h.get());
    hop.pad = (uint32_t)s->rows_pad_h;
    hop.diag0 = true;
    hop.scaled = s->colours;
    if (!H->work.ev[0]) {
      SS_CUDA(cudaEventCreate(&H->work.ev[0]));
      SS_CUDA(cudaEventCreate(&H->work.ev[1]));
    }
    H->plan.spin_limit = C->wait_ns;
    SS_TRY(launch_solve(H->work, H->plan, hop, nullptr, s->norm_h.get(), s->ca64.get(), s->ca32.get(), s->pn32.get(),
                        tol, max_iter, mode, st, H->work.ev[0], H->work.ev[1], nullptr, true));
    k_half_scatter<<<sb, 256, 0, st>>>(C->uh.get(), s->hpos.get(), s->size, s->n_plus,
                                       reinterpret_cast<double2*>(u_on_S));
    SS_LAUNCH_CHECK();
    SS_CUDA(cudaMemcpyAsync(C->hflag_host, C->hflag.get(), sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    SS_TRY(queue_checks());
    ss_status worst;
    ss_solve_stats one{};
    SS_TRY(read_stats(H->work, 1, &one, &worst, st, H->work.ev[0], H->work.ev[1]));
    C->fh.settle();
    C->uh.settle();
    C->hflag.settle();
    s->ecoef32_h.settle();
    if (pending) SS_TRY(stamp_check_pending(s, C->chk_host));   // may withdraw the half system
    if (*C->hflag_host == 0 && s->half_ok) {
      one.half_system = 1;
      one.real_coefficients = s->a_real;
      if (check_f0 && (C->f0_host->x != 0.0 || C->f0_host->y != 0.0)) {
        one.status = SS_ERR_INVALID;
        if (stats) *stats = one;
        SS_FAIL(SS_ERR_INVALID, "solve: f_hat_0 must be 0 (mean-zero forcing)");
      }
      if (stats) *stats = one;
      return worst;
    }
  }
  SS_TRY(stamp_plan(s, *C, mode, st));
  C->plan.inst[0].f = reinterpret_cast<const double2*>(f_on_S);
  C->plan.inst[0].u = reinterpret_cast<double2*>(u_on_S);
  SS_TRY(work_upload(C->work, C->plan, false, st));
  SS_TRY(work_prologue(C->work, C->plan, nullptr, st));
  OpView op;
  op.woff = s->slice_off.get();
  op.ent = s->ent.get();
  op.ecoef = s->ecoef64.get();
  op.ecoefdf = s->ecoefdf.get();
  op.colbits = colbits_of(s->jbits);
  op.colmask = colmask_of(s->jbits);
  op.realc = s->a_real;
  op.ecoef32 = reinterpret_cast<const float2*>(s->ecoef32.get());
  op.pad = (uint32_t)s->rows_pad;
  if (!C->work.ev[0]) {
    SS_CUDA(cudaEventCreate(&C->work.ev[0]));
    SS_CUDA(cudaEventCreate(&C->work.ev[1]));
  }
  C->plan.spin_limit = C->wait_ns;
  SS_TRY(launch_solve(C->work, C->plan, op, nullptr, s->norm.get(), s->ca64.get(), s->ca32.get(), s->pn32.get(), tol,
                      max_iter, mode, st, C->work.ev[0], C->work.ev[1], s->adr ? s->diag64.get() : nullptr, true));
  SS_TRY(queue_checks());
  ss_status worst;
  ss_solve_stats one{};
  SS_TRY(read_stats(C->work, 1, &one, &worst, st, C->work.ev[0], C->work.ev[1]));
  s->ecoef32.settle();
  if (pending) SS_TRY(stamp_check_pending(s, C->chk_host));
  one.real_coefficients = s->a_real;
  if (check_f0 && (C->f0_host->x != 0.0 || C->f0_host->y != 0.0)) {
    one.status = SS_ERR_INVALID;
    if (stats) *stats = one;
    SS_FAIL(SS_ERR_INVALID, "solve: f_hat_0 must be 0 (mean-zero forcing)");
  }
  if (stats) *stats = one;
  return worst;
}

// ------------------------------------------------------ allocation-free solve
//
// solve_noalloc runs the general phases (k_solve, blocks of 1024 threads) on the
// full system, never the Hermitian half system; its FP32 operator forms the entry
// coefficients as it goes.  solve() runs one instance by k_solve_one with 512
// threads and stored FP32 coefficients: the two may differ in rounding and in
// iterations.  All of the workspace is one file-scope device array.
// It serves callers that may not allocate device memory once they run:
// plug-ins inside a host application that owns all device memory, code that
// must not stall on cudaMalloc (allocation synchronises the device), or code
// that runs under a fixed device-memory budget set at start-up.  The array holds a stamping set of at
// most kNoAllocRows padded rows (stamps of up to 32,736 frequencies, a few MB
// of device memory on every GPU that loads the library, kept until exit).

namespace ss {
namespace {

constexpr int64_t kNoAllocRows = 32768;                 // padded rows of S
constexpr int64_t kNoAllocRecs = kNoAllocRows + 1;      // plus the dummy record
constexpr int kNoAllocChunks = 1024;
constexpr int64_t kNoAllocParts = 2 * kNoAllocChunks;

constexpr size_t a256(size_t x) { return (x + 255) / 256 * 256; }

// byte offsets of the workspace inside the array
constexpr size_t kOffXrec = 0;
constexpr size_t kOffU64 = kOffXrec + a256(2 * kNoAllocRecs * sizeof(double2));
constexpr size_t kOffU32 = kOffU64 + a256(2 * kNoAllocRecs * sizeof(double2));
constexpr size_t kOffR = kOffU32 + a256(kNoAllocRecs * sizeof(float4));
constexpr size_t kOffW64 = kOffR + a256(kNoAllocRecs * sizeof(double2));
constexpr size_t kOffPd = kOffW64 + a256(kNoAllocRecs * sizeof(double2));
constexpr size_t kOffSd = kOffPd + a256(kNoAllocRecs * sizeof(double2));
constexpr size_t kOffRhat = kOffSd + a256(kNoAllocRecs * sizeof(double2));
constexpr size_t kOffDlt = kOffRhat + a256(kNoAllocRecs * sizeof(double2));
constexpr size_t kOffW32 = kOffDlt + a256(kNoAllocRecs * sizeof(double2));
constexpr size_t kOffR32 = kOffW32 + a256(kNoAllocRecs * sizeof(float2));
constexpr size_t kOffP32 = kOffR32 + a256(kNoAllocRecs * sizeof(float2));
constexpr size_t kOffS32 = kOffP32 + a256(kNoAllocRecs * sizeof(float2));
constexpr size_t kOffD32 = kOffS32 + a256(kNoAllocRecs * sizeof(float2));
constexpr size_t kOffRdiag = kOffD32 + a256(kNoAllocRecs * sizeof(float2));
constexpr size_t kOffPart = kOffRdiag + a256(kNoAllocRecs * sizeof(double));
constexpr size_t kOffBar = kOffPart + a256(kNoAllocParts * kNQ * sizeof(double));
constexpr size_t kOffCnt = kOffBar + 256;
constexpr size_t kOffErr = kOffCnt + 256;
constexpr size_t kOffState = kOffErr + 256;
constexpr size_t kOffInst = kOffState + a256(sizeof(InstState));
constexpr size_t kOffList = kOffInst + a256(sizeof(SolveInst));
constexpr size_t kNoAllocBytes = kOffList + a256(solve_list_words(kNoAllocRows / kSlice) * sizeof(int32_t));

}  // namespace
}  // namespace ss

// The shared workspace (one per device; every call uses all of it).
static __device__ __align__(256) unsigned char ss_noalloc_scratch[ss::kNoAllocBytes];

namespace ss {
namespace {

std::mutex g_noalloc_mu;
unsigned char* g_noalloc_base[64] = {};

// Device address of the array for the current device, looked up once per
// device (host code cannot use the array's name as a device address).
ss_status noalloc_base(unsigned char** out) {
  int dev = 0;
  SS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) SS_FAIL(SS_ERR_INVALID, "solve_noalloc: device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_base[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, ss_noalloc_scratch);
    if (e != cudaSuccess || !p)
      SS_FAIL(SS_ERR_CUDA, "solve_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
    g_noalloc_base[dev] = static_cast<unsigned char*>(p);
  }
  *out = g_noalloc_base[dev];
  return SS_OK;
}

}  // namespace
}  // namespace ss

extern "C" ss_status solve_noalloc(ss_stamp s, const double* f_on_S, double* u_on_S, double tol, int32_t max_iter,
                                   ss_precision prec, ss_solve_stats* stats, void* stream) {
  if (!s || !f_on_S || !u_on_S) SS_FAIL(SS_ERR_INVALID, "solve_noalloc: null argument");
  if (!(tol > 0.0) || max_iter < 1) SS_FAIL(SS_ERR_INVALID, "solve_noalloc: need tol > 0 and max_iter >= 1");
  if (prec != SS_FP64 && prec != SS_FP32) SS_FAIL(SS_ERR_INVALID, "solve_noalloc: bad precision");
  if (s->adr) SS_FAIL(SS_ERR_INVALID, "solve_noalloc: ADR stamps are solved by solve (BiCGStab)");
  if (s->rows_pad > kNoAllocRows)
    SS_FAIL(SS_ERR_INVALID,
            "solve_noalloc: |S| = %lld (%lld padded rows) exceeds the allocation-free workspace of %lld rows",
            (long long)s->size, (long long)s->rows_pad, (long long)kNoAllocRows);
  cudaStream_t st = as_stream(stream);
  unsigned char* base = nullptr;
  SS_TRY(noalloc_base(&base));
  if (!s->slice_off.get() || s->n_slices < 1) SS_FAIL(SS_ERR_INVALID, "solve_noalloc: stamp has no slice table");
  // static work split, as solve() with its default tile shape: the slice lists
  // are written on the device into the workspace
  const int mode = prec == SS_FP64 ? 0 : 1;
  SolvePlan plan;
  plan.inst.assign(1, SolveInst{});
  SolveInst& in = plan.inst[0];
  in.row0 = 0;
  in.rows = s->size;
  in.rows_pad = s->rows_pad;
  in.zero_row = s->zero_idx;
  in.coef_off = 0;
  in.dscale = 2.0 * kTwoPiSq * s->a0;
  in.wide = s->wide ? 1 : 0;
  in.f = reinterpret_cast<const double2*>(f_on_S);
  in.u = reinterpret_cast<double2*>(u_on_S);
  plan.block = 1024;
  int grid = 0;
  SS_TRY(max_grid(mode, false, false, plan.block, &grid));
  grid = std::min(grid, sm_count());
  const int by_size = (int)std::max<int64_t>(1, s->n_slices / 8);
  plan_single(plan, s->n_slices, std::min(grid, by_size), s->colours ? s->cmask.get() : nullptr, s->err_dev.get());
  plan.grid = std::min<int>(grid, plan.n_chunks[0]);
  if (plan.n_chunks[0] > kNoAllocChunks || plan.n_parts > kNoAllocParts)
    SS_FAIL(SS_ERR_INVALID, "solve_noalloc: work split exceeds the workspace tables");
  // pointers into the shared workspace
  auto at = [&](size_t off) { return static_cast<void*>(base + off); };
  SolveInst* d_inst = static_cast<SolveInst*>(at(kOffInst));
  int32_t* d_list = static_cast<int32_t*>(at(kOffList));
  InstState* d_state = static_cast<InstState*>(at(kOffState));
  unsigned* d_bar = static_cast<unsigned*>(at(kOffBar));
  int* d_cnt = static_cast<int*>(at(kOffCnt));
  int* d_err = static_cast<int*>(at(kOffErr));
  // the array keeps the previous call's contents: the prologue writes the
  // descriptor and the lists and resets what must start at zero (barrier,
  // counters, error word, instance state); the records are set up below
  SS_TRY(launch_prologue(plan, d_bar, d_cnt, d_err, d_state, nullptr, d_inst, d_list, st));
  const int64_t recs = s->rows_pad + 1;
  k_init_solve_records<<<nblk(recs), 256, 0, st>>>(s->norm.get(), recs, nullptr, s->wide,
                                                  static_cast<double2*>(at(kOffXrec)),
                                                  static_cast<double2*>(at(kOffU64)), static_cast<float4*>(at(kOffU32)));
  SS_LAUNCH_CHECK();
  SolveParams P{};
  P.n_inst = 1;
  set_split(P, plan, nullptr, d_list);
  P.inst = d_inst;
  P.state = d_state;
  P.op.woff = s->slice_off.get();
  P.op.ent = s->ent.get();
  P.op.ecoef = s->ecoef64.get();
  P.op.colbits = colbits_of(s->jbits);
  P.op.colmask = colmask_of(s->jbits);
  P.op.realc = s->a_real;
  P.slice_inst = nullptr;
  P.norm = s->norm.get();
  P.ca64 = s->ca64.get();
  P.ca32 = s->ca32.get();
  P.pn = s->pn32.get();
  P.xrec = static_cast<double2*>(at(kOffXrec));
  P.urec64 = static_cast<double2*>(at(kOffU64));
  P.urec32 = static_cast<float4*>(at(kOffU32));
  P.r = static_cast<double2*>(at(kOffR));
  P.w64 = static_cast<double2*>(at(kOffW64));
  P.pd = static_cast<double2*>(at(kOffPd));
  P.sd = static_cast<double2*>(at(kOffSd));
  P.rhat = static_cast<double2*>(at(kOffRhat));
  P.dlt = static_cast<double2*>(at(kOffDlt));
  P.w32 = static_cast<float2*>(at(kOffW32));
  P.r32 = static_cast<float2*>(at(kOffR32));
  P.p32 = static_cast<float2*>(at(kOffP32));
  P.s32 = static_cast<float2*>(at(kOffS32));
  P.d32 = static_cast<float2*>(at(kOffD32));
  P.rdiag = static_cast<double*>(at(kOffRdiag));
  P.part = static_cast<double*>(at(kOffPart));
  P.bar = d_bar;
  P.counters = d_cnt;
  P.err = d_err;
  P.tol = tol;
  P.inner_tol = 1e-5;
  P.max_iter = max_iter;
  P.max_inner = std::max(1, std::min(max_iter, 200));
  P.max_outer = std::max(1, max_iter);
  P.spin_limit = 2000000000ll;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.grid);
  cfg.blockDim = dim3(plan.block);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SS_CUDA(cudaLaunchKernelEx(&cfg, solve_kernel(mode, false, plan.block, false), P));
  // statistics, error word and f_hat_0 read back with one synchronisation
  InstState hs;
  int herr = 0;
  double2 f0 = make_double2(0.0, 0.0);
  SS_CUDA(cudaMemcpyAsync(&hs, d_state, sizeof(hs), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
  if (s->zero_idx >= 0)
    SS_CUDA(cudaMemcpyAsync(&f0, reinterpret_cast<const double2*>(f_on_S) + s->zero_idx, sizeof(f0),
                            cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  const double rel = hs.bb > 0 ? std::sqrt(hs.rr / hs.bb) : 0.0;
  if (stats) {
    stats->status = herr ? herr : hs.status;
    stats->outer_iters = hs.outer_iters;
    stats->inner_iters = hs.inner_iters ? hs.inner_iters : hs.iters;
    stats->applies = hs.applies;
    stats->rel_residual = rel;
    stats->kernel_ms = 0.0;
    stats->half_system = 0;
    stats->real_coefficients = s->a_real;
  }
  if (f0.x != 0.0 || f0.y != 0.0) {
    if (stats) stats->status = SS_ERR_INVALID;
    SS_FAIL(SS_ERR_INVALID, "solve_noalloc: f_hat_0 must be 0 (mean-zero forcing)");
  }
  if (herr) SS_FAIL((ss_status)herr, "solve_noalloc: a device-side wait gave up (status %d)", herr);
  if (hs.status != SS_OK) SS_FAIL((ss_status)hs.status, "solve_noalloc: not converged (relative residual %.3e)", rel);
  return SS_OK;
}
