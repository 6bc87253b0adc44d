// Batched conjugate gradients on (outputscale K~ + noise I) X = B (Sec. 2: Krylov
// solvers that need only MVMs; App. A: at most 500 iterations).
//
// Every right-hand side c is an independent CG with its own scalars; a column that has
// converged (||r_c|| / ||b_c|| <= tol), hit max_iter or broken down (<p, Ap> <= 0) is
// frozen by a device-side flag, so extra iterations leave it unchanged.  The iterate x and
// the residual r (whose recurrences are where fp32 rounding makes CG lose orthogonality)
// carry ~48 bits as double-float pairs (hi + lo fp32, updated with error-free
// transformations: FP64 arithmetic is slow on this part); the search direction p and A p
// are fp32, the operands of the lattice MVM.  Dot products are accumulated per thread in
// double-float, per block and across blocks in fp64 in a fixed order (fixed column per
// thread, shared-memory tree), so the result does not depend on scheduling.  One iteration is captured
// in a CUDA graph and replayed; the host reads the flags every check_every iterations.
#include <algorithm>
#include <cmath>
#include <vector>

#include "sgp_internal.cuh"
#include "values.cuh"

namespace sgp {
namespace {

struct CgState {
  double* partial;  // [blocks][k] per-block column sums
  double* rho;      // <r, r> of the current residual (<r, z> when preconditioned)
  dfloat* alpha;    // as double-float pairs, the form the vector updates use
  dfloat* beta;
  double* bnorm;
  double* rr;       // <r, r> after the last iteration of the column
  int* active;
  int* iters;
  float tol;
  int max_iter;
  // optional Lanczos record (plain CG): alpha_j, beta_j of column c at [j][k], j < hcap
  double* ha;
  double* hb;
  int hcap;
  // optional residual history: ||r_c|| / ||b_c|| after iteration j of column c at [j][k]
  double* hist;
  int hist_cap;
  // optional: the preconditioner's split residual [n][64] (bf16; part p of column c < 16
  // at 16 p + c), written by the x, r update
  bf16* r3;
};

// What the totals of a kernel's column sums are used for.
enum CgEnd {
  CG_INIT = 0,  // sum = <b, b>: norms, first rho, columns that start stopped
  CG_ALPHA,     // sum = <p, A p>: step sizes
  CG_BETA,      // sum = <r, r>: convergence and the next direction's beta (plain CG)
  CG_CHECK,     // sum = <r, r>: convergence only (preconditioned)
  CG_RHO_INIT,  // sum = <r, z> at the start
  CG_BETA_PRE,  // sum = <r, z>: beta (preconditioned)
};

// What one thread holds of a column before its sum is known.
struct CgColumn {
  double rho = 0.0, bnorm = 0.0;
  int active = 0, iters = 0;
};

__device__ __forceinline__ void cg_end_column(CgEnd what, int c, int k, double sum,
                                              const CgColumn& col, const CgState& S) {
  switch (what) {
    case CG_INIT:
      S.rho[c] = sum;
      S.rr[c] = sum;
      S.bnorm[c] = sqrt(sum);
      S.iters[c] = 0;
      S.alpha[c] = S.beta[c] = {0.f, 0.f};
      S.active[c] = sum != 0.0 && 1.0 > (double)S.tol && S.max_iter > 0 ? 1 : 0;
      return;
    case CG_ALPHA: {
      double alpha = 0.0;
      if (col.active) {
        if (sum > 0.0 && isfinite(sum)) {
          alpha = col.rho / sum;
          if (S.ha && col.iters < S.hcap) S.ha[(int64_t)col.iters * k + c] = alpha;
        } else {
          S.active[c] = 0;  // breakdown: the operator is not positive definite on p
        }
      }
      S.alpha[c] = df_from_double(alpha);
      return;
    }
    case CG_BETA:
    case CG_CHECK: {
      if (!col.active) return;
      const int it = col.iters + 1;
      S.iters[c] = it;
      S.rr[c] = sum;
      if (S.hist && it <= S.hist_cap) S.hist[(int64_t)(it - 1) * k + c] = sqrt(sum) / col.bnorm;
      if (it >= S.max_iter || cg_stops(sum, col.bnorm, S.tol)) {
        S.active[c] = 0;
        return;
      }
      if (what == CG_CHECK) return;
      const double beta = sum / col.rho;
      S.beta[c] = df_from_double(beta);
      S.rho[c] = sum;
      if (S.hb && it - 1 < S.hcap) S.hb[(int64_t)(it - 1) * k + c] = beta;
      return;
    }
    case CG_RHO_INIT:
      S.rho[c] = sum;
      if (!(sum > 0.0) || !isfinite(sum)) S.active[c] = 0;
      return;
    case CG_BETA_PRE:
      if (!col.active) return;
      if (!(sum > 0.0) || !isfinite(sum)) {
        S.active[c] = 0;
        return;
      }
      S.beta[c] = df_from_double(sum / col.rho);
      S.rho[c] = sum;
      return;
    default:
      return;
  }
}

// Column c's sum over `nblk` block partials and what follows from it.  One warp per column
// (blockIdx.x = c).  The order of the additions is part of the result (a preconditioned
// solve of 100 iterations carries a last-place change of one sum to the fifth digit of its
// answer): 256 strided sums over the blocks, then a tree over them, halves first.  A lane
// holds eight of the 256 sums, all its loads are in flight together and the tree needs no
// barrier: a dependent fp64 addition takes some 100 clocks on this part, so the kernel is a
// chain of latencies (n = 50k: 4.2-5.4 us for the three of an iteration).
// Letting the last block of the producing kernel do this instead was slower: its twelve
// columns share one SM's fp64 pipe (slice and sums of n = 50k, k = 12: 27 us, apart 17 us).
__global__ void __launch_bounds__(32) k_cg_end(CgEnd what, int nblk, int k, CgState S) {
  pdl_enter();
  const int lane = (int)threadIdx.x, c = (int)blockIdx.x;
  CgColumn col;
  if (lane == 0 && what != CG_INIT) {
    col.rho = S.rho[c];
    col.bnorm = S.bnorm[c];
    col.active = S.active[c];
    col.iters = S.iters[c];
  }
  double v[8];  // sums lane, lane + 32, ..., lane + 224
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = 0.0;
#pragma unroll 4
  for (int b0 = lane; b0 < nblk; b0 += 256) {
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      x[q] = b0 + 32 * q < nblk ? S.partial[(int64_t)(b0 + 32 * q) * k + c] : 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] += x[q];
  }
#pragma unroll
  for (int half = 4; half >= 1; half /= 2)
#pragma unroll
    for (int q = 0; q < half; ++q) v[q] += v[q + half];
#pragma unroll
  for (int half = 16; half >= 1; half /= 2) v[0] += __shfl_down_sync(0xffffffffu, v[0], half);
  if (lane == 0) cg_end_column(what, c, k, v[0], col, S);
}


// VEC consecutive elements of a row: fp32 (one float4 when VEC = 4) and fp64 (two double2).
template <int VEC>
__device__ __forceinline__ void ldf(const float* p, float (&v)[VEC]) {
  if (VEC == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[VEC - 1] = t.w;
  } else {
    v[0] = *p;
  }
}
template <int VEC>
__device__ __forceinline__ void stf(float* p, const float (&v)[VEC]) {
  if (VEC == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[VEC - 1]);
  else *p = v[0];
}
// Grid-stride over rows with a fixed column group per thread: G = k / VEC threads per row,
// blockDim.x = a whole number of rows.
#define SGP_ROWS_LOOP(row)                                                                  \
  const int G = k / VEC;                                                                    \
  const int rows_per_block = blockDim.x / G;                                                \
  const int c0 = (int)(threadIdx.x % G) * VEC;                                              \
  for (int64_t row = (int64_t)blockIdx.x * rows_per_block + threadIdx.x / G; row < n;       \
       row += (int64_t)gridDim.x * rows_per_block)

// The solver's vectors live in the lattice's locality order: row p holds the caller's
// row perm[p], so the MVM's splat gathers and slice writes stay local.  B and X are the
// caller's buffers (any alignment): read and written element by element.
// The caller's B has kb <= k columns; columns kb .. k - 1 of the solver's vectors are zero
// right-hand sides (inactive from the start).
template <int VEC>
__global__ void k_cg_init(const float* B, int kb, const int32_t* __restrict__ perm,
                          float* __restrict__ xh, float* __restrict__ xl,
                          float* __restrict__ rh, float* __restrict__ rl, float* __restrict__ p,
                          int64_t n, int k, CgState S) {
  pdl_enter();
  dfloat acc[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) acc[j] = {0.f, 0.f};
  SGP_ROWS_LOOP(row) {
    const float* b = B + (int64_t)perm[row] * kb + c0;
    float bv[VEC], zero[VEC];
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      bv[j] = c0 + j < kb ? b[j] : 0.f;
      zero[j] = 0.f;
      acc[j] = df_add(acc[j], df_two_prod(bv[j], bv[j]));
    }
    const int64_t e = row * k + c0;
    stf<VEC>(xh + e, zero);
    stf<VEC>(xl + e, zero);
    stf<VEC>(rh + e, bv);
    stf<VEC>(rl + e, zero);
    stf<VEC>(p + e, bv);
  }
  double dd[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) dd[j] = df_to_double(acc[j]);
  block_column_sums<VEC>(dd, k, S.partial + (int64_t)blockIdx.x * k);
}

// x += alpha p, r -= alpha A p on active columns (double-float); block partials of
// <r, r>.  fp64 issues at 2 results per SM and clock, so the step sizes arrive
// as double-float pairs and the sums leave a thread by integer conversions: n = 50k, k = 12
// (one row a thread) 10.6 us, 21.2 with both in fp64.
// With S.r3 (VEC = 4), also the three bf16 parts of r = rh + rl for columns 0..15, the
// operand of the preconditioner's B^T r (as its split kernel would write them).
template <int VEC>
__global__ void k_cg_update_xr(float* __restrict__ xh, float* __restrict__ xl,
                               float* __restrict__ rh, float* __restrict__ rl,
                               const float* p, const float* Ap,
                               int64_t n, int k, CgState S) {
  pdl_enter();
  dfloat acc[VEC], a[VEC], na[VEC];
  bool on[VEC];
  {
    const int c = (int)(threadIdx.x % (k / VEC)) * VEC;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      acc[j] = {0.f, 0.f};
      on[j] = S.active[c + j] != 0;
      a[j] = S.alpha[c + j];
      na[j] = {-a[j].hi, -a[j].lo};
    }
  }
  SGP_ROWS_LOOP(row) {
    const int64_t e = row * k + c0;
    float pv[VEC], qv[VEC], xhv[VEC], xlv[VEC], rhv[VEC], rlv[VEC];
    ldf<VEC>(p + e, pv);
    ldf<VEC>(Ap + e, qv);
    ldf<VEC>(xh + e, xhv);
    ldf<VEC>(xl + e, xlv);
    ldf<VEC>(rh + e, rhv);
    ldf<VEC>(rl + e, rlv);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      if (on[j]) {
        const dfloat x = df_add({xhv[j], xlv[j]}, df_mul_f(a[j], pv[j]));
        const dfloat r = df_add({rhv[j], rlv[j]}, df_mul_f(na[j], qv[j]));
        xhv[j] = x.hi, xlv[j] = x.lo, rhv[j] = r.hi, rlv[j] = r.lo;
      }
      dfloat sq = df_two_prod(rhv[j], rhv[j]);
      sq = df_fast_two_sum(sq.hi, __fmaf_rn(2.f * rhv[j], rlv[j], sq.lo));
      acc[j] = df_add(acc[j], sq);
    }
    stf<VEC>(xh + e, xhv);
    stf<VEC>(xl + e, xlv);
    stf<VEC>(rh + e, rhv);
    stf<VEC>(rl + e, rlv);
    if constexpr (VEC == 4) {
      if (S.r3 && c0 < 16) {
        bf16 q[4][3];
#pragma unroll
        for (int j = 0; j < 4; ++j) split3(__fadd_rn(rhv[j], rlv[j]), q[j][0], q[j][1], q[j][2]);
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          uint2 w;
          w.x = (uint32_t)__bfloat16_as_ushort(q[0][part]) |
                ((uint32_t)__bfloat16_as_ushort(q[1][part]) << 16);
          w.y = (uint32_t)__bfloat16_as_ushort(q[2][part]) |
                ((uint32_t)__bfloat16_as_ushort(q[3][part]) << 16);
          *reinterpret_cast<uint2*>(S.r3 + row * 64 + part * 16 + c0) = w;
        }
      }
    }
  }
  double dd[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) dd[j] = df_to_double(acc[j]);
  block_column_sums<VEC>(dd, k, S.partial + (int64_t)blockIdx.x * k);
}

// Preconditioned CG: p = z + beta p on active columns (first == true: p = z).
template <int VEC, bool FIRST>
__global__ void k_cg_update_p_z(float* __restrict__ p, const float* z, int64_t n,
                                int k, CgState S) {
  pdl_enter();
  dfloat b[VEC];
  bool on[VEC];
  {
    const int c = (int)(threadIdx.x % (k / VEC)) * VEC;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      on[j] = S.active[c + j] != 0;
      b[j] = S.beta[c + j];
    }
  }
  SGP_ROWS_LOOP(row) {
    const int64_t e = row * k + c0;
    float pv[VEC], zv[VEC];
    ldf<VEC>(p + e, pv);
    ldf<VEC>(z + e, zv);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      if (FIRST) {
        pv[j] = zv[j];
      } else if (on[j]) {
        const dfloat t = df_add(df_mul_f(b[j], pv[j]), {zv[j], 0.f});
        pv[j] = __fadd_rn(t.hi, t.lo);
      }
    }
    stf<VEC>(p + e, pv);
  }
}

// p = r + beta p on active columns (double-float sum, rounded to fp32).
template <int VEC>
__global__ void k_cg_update_p(float* __restrict__ p, const float* rh,
                              const float* rl, int64_t n, int k, CgState S) {
  pdl_enter();
  dfloat b[VEC];
  bool on[VEC];
  {
    const int c = (int)(threadIdx.x % (k / VEC)) * VEC;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      on[j] = S.active[c + j] != 0;
      b[j] = S.beta[c + j];
    }
  }
  SGP_ROWS_LOOP(row) {
    const int64_t e = row * k + c0;
    float pv[VEC], rhv[VEC], rlv[VEC];
    ldf<VEC>(p + e, pv);
    ldf<VEC>(rh + e, rhv);
    ldf<VEC>(rl + e, rlv);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      if (on[j]) {
        const dfloat t = df_add({rhv[j], rlv[j]}, df_mul_f(b[j], pv[j]));
        pv[j] = __fadd_rn(t.hi, t.lo);
      }
    }
    stf<VEC>(p + e, pv);
  }
}

template <int VEC>
__global__ void k_cg_store_x(const float* xh, const float* xl,
                             const int32_t* __restrict__ perm, float* __restrict__ X, int kb,
                             int64_t n, int k) {
  pdl_enter();
  SGP_ROWS_LOOP(row) {
    float hv[VEC], lv[VEC];
    ldf<VEC>(xh + row * k + c0, hv);
    ldf<VEC>(xl + row * k + c0, lv);
    float* dst = X + (int64_t)perm[row] * kb + c0;
#pragma unroll
    for (int j = 0; j < VEC; ++j)
      if (c0 + j < kb) dst[j] = __fadd_rn(hv[j], lv[j]);
  }
}

}  // namespace

sgp_status run_cg(Lattice* L, const float* B, int k, int blur, float noise, float tol,
                  int max_iter, float* X, int* iters, double* rel_res, int precond_rank,
                  uint64_t seed, const LanczosRecord* rec, double* history) {
  const int64_t n = L->n;
  // The solver works on k rounded up to a multiple of 4 (zero right-hand sides in the
  // extra columns, inactive from the start), so that its vectors and the lattice values
  // are rows of float4 and the MVM takes its vectorised kernels.  One or two Lanczos probes
  // (sgp_logdet) stay as they are; their huge vertices' sums keep the caller's k's shape.
  const int kb = k;
  k = rec ? rec->cols : (k + 3) / 4 * 4;
  // CUDA graphs cannot be captured on the legacy default stream: use a private blocking
  // stream then (it is ordered with the legacy stream like any blocking stream).
  cudaStream_t st = L->stream;
  cudaStream_t own = nullptr;
  if (st == nullptr) {
    cudaError_t e = cudaStreamCreateWithFlags(&own, cudaStreamDefault);
    if (e != cudaSuccess) return cuda_status(e, "creating the CG stream");
    st = own;
  }
  struct Cleanup {
    cudaStream_t st, own;
    std::vector<void*> ptrs;
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;
    ShiftedNystrom pre;
    ~Cleanup() {
      pre.release(st);
      if (exec) (void)cudaGraphExecDestroy(exec);
      if (graph) (void)cudaGraphDestroy(graph);
      for (void* p : ptrs) (void)cudaFreeAsync(p, st);
      if (own) {
        (void)cudaStreamSynchronize(own);
        (void)cudaStreamDestroy(own);
      }
      clear_pending_error();
    }
  } cl{st, own, {}};
  auto get = [&](void** p, size_t bytes) {
    cudaError_t e = cols_malloc(L, k, p, std::max<size_t>(bytes, 16), st);
    if (e == cudaSuccess) cl.ptrs.push_back(*p);
    return e;
  };
#define CG_CHECK(expr, what)                               \
  do {                                                     \
    cudaError_t e_ = (expr);                               \
    if (e_ != cudaSuccess) return cuda_status(e_, what);   \
  } while (0)

  float *xh, *xl, *rh, *rl, *p, *Ap;
  CgState S{};
  const int vec = k % 4 == 0 ? 4 : 1;
  const int kt = rec ? kb : k;  // shapes the sums
  const int T = column_block_threads(k, vec, kt);
  const int64_t rows_per_block = T / (k / vec);
  const unsigned vblocks = (unsigned)std::min<int64_t>(kVecBlocks, std::max<int64_t>(1, ceil_div(n, rows_per_block)));
  const int64_t sblocks = slice_dot_blocks(L, k, kt);
  const bool want_pre = precond_rank > 0 && noise > 0.f && !rec;
  // bounds ShiftedNystrom::dot_blocks (its z blocks: at most one per 128-row tile)
  const int64_t pblocks = want_pre ? ceil_div(n, 128) : 0;
  CG_CHECK(get((void**)&xh, n * k * sizeof(float)), "alloc x");
  CG_CHECK(get((void**)&xl, n * k * sizeof(float)), "alloc x");
  CG_CHECK(get((void**)&rh, n * k * sizeof(float)), "alloc r");
  CG_CHECK(get((void**)&rl, n * k * sizeof(float)), "alloc r");
  CG_CHECK(get((void**)&p, n * k * sizeof(float)), "alloc p");
  CG_CHECK(get((void**)&Ap, n * k * sizeof(float)), "alloc Ap");
  CG_CHECK(get((void**)&S.partial,
               (size_t)std::max<int64_t>(std::max<int64_t>(vblocks, sblocks), pblocks) * k *
                   sizeof(double)),
           "alloc partial");
  double* scal;
  CG_CHECK(get((void**)&scal, 5 * (size_t)k * sizeof(double)), "alloc scalars");
  S.rho = scal;
  S.bnorm = scal + k;
  S.rr = scal + 2 * k;
  S.alpha = reinterpret_cast<dfloat*>(scal + 3 * k);
  S.beta = reinterpret_cast<dfloat*>(scal + 4 * k);
  int* flags;
  CG_CHECK(get((void**)&flags, 2 * (size_t)k * sizeof(int)), "alloc flags");
  S.active = flags;
  S.iters = flags + k;
  S.tol = tol;
  S.max_iter = max_iter;
  if (rec) {
    S.ha = rec->alpha;
    S.hb = rec->beta;
    S.hcap = rec->cap;
  }
  if (history && max_iter > 0) {
    CG_CHECK(get((void**)&S.hist, (size_t)max_iter * k * sizeof(double)), "alloc history");
    S.hist_cap = max_iter;
    // iterations a column does not run read back as NaN
    std::vector<double> nan((size_t)max_iter * k, std::nan(""));
    CG_CHECK(cudaMemcpyAsync(S.hist, nan.data(), nan.size() * sizeof(double),
                             cudaMemcpyHostToDevice, st),
             "clear history");
    CG_CHECK(cudaStreamSynchronize(st), "sync history");
  }
  sgp_status s = ensure_lattice_values(L, k, st);
  if (s != SGP_OK) return s;

  // the preconditioner (built before anything is captured); needs noise > 0
  bool use_pre = false;
  float* z = nullptr;
  if (want_pre) {
    s = cl.pre.build(L, precond_rank, seed, noise, blur, L->precond_power_iters, st);
    if (s != SGP_OK) return s;
    use_pre = cl.pre.ok;
    if (use_pre) CG_CHECK(get((void**)&z, n * k * sizeof(float)), "alloc z");
    // the x, r update writes the split residual the preconditioner's B^T r reads
    if (use_pre && vec == 4) S.r3 = static_cast<bf16*>(cl.pre.r3);
  }

  if (vec == 4)
    launch_pdl(k_cg_init<4>, vblocks, T, st, B, kb, L->perm, xh, xl, rh, rl, p, n, k, S);
  else
    launch_pdl(k_cg_init<1>, vblocks, T, st, B, kb, L->perm, xh, xl, rh, rl, p, n, k, S);
  auto end = [&](CgEnd what, int64_t blocks) {
    launch_pdl(k_cg_end, k, 32, st, what, (int)blocks, k, S);
    note_launches(1);
  };
  end(CG_INIT, vblocks);
  note_launches(1);
  if (use_pre) {  // z = P^-1 r, rho = <r, z>, p = z
    cl.pre.apply(rh, rl, k, z, S.partial, st);
    end(CG_RHO_INIT, cl.pre.dot_blocks());
    if (vec == 4) launch_pdl(k_cg_update_p_z<4, true>, vblocks, T, st, p, z, n, k, S);
    else launch_pdl(k_cg_update_p_z<1, true>, vblocks, T, st, p, z, n, k, S);
    note_launches(1);
  }
  CG_CHECK(cudaGetLastError(), "CG init");

  cudaEvent_t* ev = L->profile ? L->prof_ev : nullptr;
  int passes = 0;
  const CgEnd after_r = use_pre ? CG_CHECK : CG_BETA;
  auto iteration = [&]() {
    // Ap = outputscale K~ p + noise p, with the slice also summing <p, Ap>: alpha
    passes = enqueue_mvm(L, p, k, blur, L->outputscale, noise, Ap, st, ev, /*internal=*/true,
                         S.partial, kt);
    end(CG_ALPHA, sblocks);
    if (vec == 4)
      launch_pdl(k_cg_update_xr<4>, vblocks, T, st, xh, xl, rh, rl, p, Ap, n, k, S);
    else
      launch_pdl(k_cg_update_xr<1>, vblocks, T, st, xh, xl, rh, rl, p, Ap, n, k, S);
    end(after_r, vblocks);
    if (use_pre) {
      cl.pre.apply(rh, rl, k, z, S.partial, st, ev ? ev + 4 : nullptr, S.r3 != nullptr);
      end(CG_BETA_PRE, cl.pre.dot_blocks());
      if (vec == 4) launch_pdl(k_cg_update_p_z<4, false>, vblocks, T, st, p, z, n, k, S);
      else launch_pdl(k_cg_update_p_z<1, false>, vblocks, T, st, p, z, n, k, S);
    } else {
      if (vec == 4) launch_pdl(k_cg_update_p<4>, vblocks, T, st, p, rh, rl, n, k, S);
      else launch_pdl(k_cg_update_p<1>, vblocks, T, st, p, rh, rl, n, k, S);
    }
    note_launches(2);
  };

  std::vector<int> hact(k);
  const int every = std::max(1, L->check_every);
  if (max_iter > 0) {
    // the captured launches run only when the graph is replayed: count them per replay
    const int64_t before = launches_so_far();
    CG_CHECK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal), "begin capture");
    iteration();
    CG_CHECK(cudaStreamEndCapture(st, &cl.graph), "end capture");
    const int64_t per_iteration = launches_so_far() - before;
    note_launches(-per_iteration);
    CG_CHECK(cudaGraphInstantiate(&cl.exec, cl.graph, 0), "instantiate CG graph");
    CG_CHECK(cudaMemcpyAsync(hact.data(), S.active, k * sizeof(int), cudaMemcpyDeviceToHost, st),
             "read flags");
    CG_CHECK(cudaStreamSynchronize(st), "sync CG");
    int launched = 0;
    while (launched < max_iter && std::any_of(hact.begin(), hact.end(), [](int a) { return a; })) {
      const int batch = std::min(every, max_iter - launched);
      for (int b = 0; b < batch; ++b) CG_CHECK(cudaGraphLaunch(cl.exec, st), "launch CG graph");
      note_launches(per_iteration * batch);
      launched += batch;
      CG_CHECK(cudaMemcpyAsync(hact.data(), S.active, k * sizeof(int), cudaMemcpyDeviceToHost, st),
               "read flags");
      CG_CHECK(cudaStreamSynchronize(st), "sync CG");
      if (ev) {  // the events of the last replay bracket one MVM's splat, blur and slice
        float ms[kProfStages] = {};
        const int from[kProfStages] = {2, 0, 1, 4, 6}, to[kProfStages] = {0, 1, 3, 5, 7};
        for (int q = 0; q < (use_pre ? kProfStages : 3); ++q)
          CG_CHECK(cudaEventElapsedTime(&ms[q], ev[from[q]], ev[to[q]]),
                   "reading the stage timing events");
        L->prof_ms += ms[1];
        L->prof_passes += passes;
        for (int q = 0; q < kProfStages; ++q) L->prof_stage_ms[q] += ms[q];
        L->prof_mvms += 1;
      }
    }
  }
  if (vec == 4) launch_pdl(k_cg_store_x<4>, vblocks, T, st, xh, xl, L->perm, X, kb, n, k);
  else launch_pdl(k_cg_store_x<1>, vblocks, T, st, xh, xl, L->perm, X, kb, n, k);
  note_launches(1);
  CG_CHECK(cudaGetLastError(), "CG result");
  std::vector<double> hscal(2 * (size_t)k);  // ||b||, <r, r>
  std::vector<int> hit(k);
  CG_CHECK(cudaMemcpyAsync(hscal.data(), S.bnorm, hscal.size() * sizeof(double),
                           cudaMemcpyDeviceToHost, st),
           "read residuals");
  CG_CHECK(cudaMemcpyAsync(hit.data(), S.iters, k * sizeof(int), cudaMemcpyDeviceToHost, st),
           "read iterations");
  CG_CHECK(cudaStreamSynchronize(st), "sync CG");
  if (use_pre && (s = cl.pre.check(st)) != SGP_OK) return s;
  if (iters) std::copy(hit.begin(), hit.begin() + kb, iters);
  if (rel_res)
    for (int c = 0; c < kb; ++c) {  // ||r|| / ||b||; 1 before the first iteration, 0 for b = 0
      const double b = hscal[c], r = std::sqrt(hscal[k + c]);
      rel_res[c] = b == 0.0 ? 0.0 : hit[c] == 0 ? 1.0 : r / b;
    }
  if (S.hist) {  // [max_iter][k] on the device, the caller's [max_iter][kb] on the host
    std::vector<double> h((size_t)max_iter * k);
    CG_CHECK(cudaMemcpyAsync(h.data(), S.hist, h.size() * sizeof(double),
                             cudaMemcpyDeviceToHost, st),
             "read history");
    CG_CHECK(cudaStreamSynchronize(st), "sync CG");
    for (int j = 0; j < max_iter; ++j)
      std::copy(h.begin() + (size_t)j * k, h.begin() + (size_t)j * k + kb,
                history + (size_t)j * kb);
  }
  if (rec) {  // ||b_c|| and the iteration counts stay on the device for the quadrature
    CG_CHECK(cudaMemcpyAsync(rec->bnorm, S.bnorm, k * sizeof(double), cudaMemcpyDeviceToDevice,
                             st),
             "copy norms");
    CG_CHECK(cudaMemcpyAsync(rec->iters, S.iters, k * sizeof(int), cudaMemcpyDeviceToDevice, st),
             "copy iterations");
    CG_CHECK(cudaStreamSynchronize(st), "sync CG");
  }
  return SGP_OK;
#undef CG_CHECK
}

}  // namespace sgp
