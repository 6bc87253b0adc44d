// Backward of the lattice MVM  out = alpha W B W^T V  (Sec. 3.2; Sec. 4.2).
//
// For a scalar loss L with G = dL/dout:
//   dV = alpha W B^T W^T G: the transpose product on the same lattice (the sequential
//        blur's transpose runs the directions in reverse; the symmetric blur is its own).
//   dX, dl, two ways (sgp_mvm_backward's `grad`):
//   SGP_GRAD_LATTICE  the exact derivative of the product the forward computes.  It is
//        multilinear in V and in the barycentric weights w_ik, and the weights are
//        piecewise linear in the elevated point y (ranks, remainder-0 points and vertex
//        ids are piecewise constant):
//          dw_ik = alpha (<G_i, (B W^T V)[v_ik]> + <V_i, (B^T W^T G)[v_ik]>)
//          dy_ic = (dw_i[d - rank_ic] - dw_i[(D - rank_ic) mod D]) / D
//        then the transpose of the elevation y = E (x / l) (triangular basis E, scaled).
//   SGP_GRAD_FILTER   Sec. 4.2: the kernel's own input gradient
//          dL/dz_n = 2 sum_j k'_nj [(g_n . v_j) + (g_j . v_n)] (z_n - z_j),  z = x / l,
//        from one filtering of the columns [z (.) g, g, z (.) v, v] with k' = dk/d(d^2);
//        for the RBF k' = -k / 2, so the filter is the lattice operator itself.
//   Both: dX = dz / l, and dl_j = -sum_i dX_ij x_ij / l_j (fixed-order reduction).
#include <algorithm>
#include <cmath>
#include <vector>

#include "sgp_internal.cuh"
#include "values.cuh"

namespace sgp {
namespace {

constexpr int kBT = 128;
constexpr int kDlsBlocks = 2 * 152;
constexpr int kFilterChunk = 256;  // columns per filtering product
// Lattice values of two dense blurs done as one.  Symmetric gradients, apart / together (d = 9): 3.5
// MB 213 / 162 us, 7.7 MB 307 / 249, 15 MB 376 / 350, 21 MB 517 / 486, 27 MB 711 / 694, 32 MB 885 / 881.
constexpr size_t kPairBytes = 32u << 20;

template <class S, int VEC>
__device__ __forceinline__ float row_dot2(const float* g, const S* bu, const float* v,
                                          const S* bs, int k) {
  float acc = 0.f;
  if (VEC == 4) {
    for (int c = 0; c < k; c += 4) {
      const float4 gv = *reinterpret_cast<const float4*>(g + c);
      const float4 vv = *reinterpret_cast<const float4*>(v + c);
      const float4 a = Store<S>::ld4(bu + c);
      const float4 b = Store<S>::ld4(bs + c);
      acc = fmaf(gv.x, a.x, acc);
      acc = fmaf(gv.y, a.y, acc);
      acc = fmaf(gv.z, a.z, acc);
      acc = fmaf(gv.w, a.w, acc);
      acc = fmaf(vv.x, b.x, acc);
      acc = fmaf(vv.y, b.y, acc);
      acc = fmaf(vv.z, b.z, acc);
      acc = fmaf(vv.w, b.w, acc);
    }
  } else {
    for (int c = 0; c < k; ++c) {
      acc = fmaf(g[c], Store<S>::ld1(bu + c), acc);
      acc = fmaf(v[c], Store<S>::ld1(bs + c), acc);
    }
  }
  return acc;
}

// Exact derivative through the weights: one thread per point (locality order p); dX in
// the caller's order.  Rows of all four arrays are ld apart.  f[j] = scale / sqrt((j+1)(j+2)) are
// the elevation factors.
template <int MAXD, int VEC, class S>
__global__ void __launch_bounds__(kBT) k_weight_grad(int64_t n, int d, int k, int ld,
                                                     const int32_t* __restrict__ perm,
                                                     const int32_t* __restrict__ idx,
                                                     const uint8_t* __restrict__ rank,
                                                     const S* BU,
                                                     const S* BS,
                                                     const float* Vp,
                                                     const float* Gp, dfloat alpha,
                                                     const double* f,
                                                     const float* ls,
                                                     float* __restrict__ dX) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int D = d + 1;
  float dw[MAXD];
  for (int kk = 0; kk < D; ++kk) {
    const int64_t v = idx[p * D + kk];
    const float dot = row_dot2<S, VEC>(Gp + p * ld, BU + v * ld, Vp + p * ld, BS + v * ld, k);
    dw[kk] = df_times(alpha, dot);
  }
  double dy[MAXD];
  for (int c = 0; c < D; ++c) {
    const int rk = rank[p * D + c];
    dy[c] = ((double)dw[d - rk] - (double)dw[(D - rk) % D]) / (double)D;
  }
  // y_0 = sum_l a_l, y_i = sum_{l > i} a_l - i a_i, a_l = z_{l-1} f_{l-1}
  const int64_t i = perm[p];
  double below = dy[0];
  for (int l = 1; l <= d; ++l) {
    const double da = below - (double)l * dy[l];
    below += dy[l];
    dX[i * d + (l - 1)] = (float)(da * f[l - 1] / (double)ls[l - 1]);
  }
}

// Filter inputs, columns [col0, col0 + kc) of [z (.) g | g | z (.) v | v] ([n][kk],
// kk = 2 k (d + 1); column c d + t of a z-block holds g_c z_t), caller's order.
__global__ void k_filter_in(int64_t n, int d, int k, int col0, int kc,
                            const float* X, const float* ls,
                            const float* V, const float* G,
                            float* __restrict__ out) {
  pdl_enter();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * kc) return;
  const int64_t i = e / kc;
  const int q = col0 + (int)(e - i * kc);
  const int kd = k * d;
  float val;
  if (q < kd) {
    val = G[i * k + q / d] * (X[i * d + q % d] / ls[q % d]);
  } else if (q < kd + k) {
    val = G[i * k + (q - kd)];
  } else if (q < 2 * kd + k) {
    const int r = q - kd - k;
    val = V[i * k + r / d] * (X[i * d + r % d] / ls[r % d]);
  } else {
    val = V[i * k + (q - 2 * kd - k)];
  }
  out[e] = val;
}

// Accumulate the filtered columns [col0, col0 + kc) into dZ ([n][d], fp32, caller's order)
// without the factor 2 alpha k'/k: one thread per point, columns in order.
__global__ void k_filter_acc(int64_t n, int d, int k, int col0, int kc,
                             const float* X, const float* ls,
                             const float* V, const float* G,
                             const float* F, float* __restrict__ dZ) {
  pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int kd = k * d;
  float* dz = dZ + i * d;
  for (int j = 0; j < kc; ++j) {
    const int q = col0 + j;
    const float fv = F[i * kc + j];
    if (q < kd) {  // K (z (.) g): - v_c (K z_t g_c)
      dz[q % d] -= V[i * k + q / d] * fv;
    } else if (q < kd + k) {  // K g: + z_t v_c (K g_c)
      const float vc = V[i * k + (q - kd)] * fv;
      for (int t = 0; t < d; ++t) dz[t] += (X[i * d + t] / ls[t]) * vc;
    } else if (q < 2 * kd + k) {  // K (z (.) v): - g_c (K z_t v_c)
      const int r = q - kd - k;
      dz[r % d] -= G[i * k + r / d] * fv;
    } else {  // K v: + z_t g_c (K v_c)
      const float gc = G[i * k + (q - 2 * kd - k)] * fv;
      for (int t = 0; t < d; ++t) dz[t] += (X[i * d + t] / ls[t]) * gc;
    }
  }
}

__global__ void k_filter_finish(int64_t n, int d, float scale, const float* ls,
                                float* __restrict__ dX) {
  pdl_enter();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * d) return;
  dX[e] = scale * dX[e] / ls[e % d];
}

// dl_j = -sum_i dX_ij x_ij / l_j: per-block partials (thread t owns column t % d and
// rows t / d, t / d + P, ... of the block's range, P = floor(256 / d)), combined in a
// fixed order; then the blocks in a fixed order.
__global__ void __launch_bounds__(256) k_dls_partial(int64_t n, int d, const float* X,
                                                     const float* dX,
                                                     double* __restrict__ partial) {
  pdl_enter();
  __shared__ double sh[256];
  const int P = 256 / d;
  const int t = threadIdx.x;
  const int j = t % d, phase = t / d;
  const int64_t rows = ceil_div(n, (int64_t)gridDim.x);
  const int64_t r0 = (int64_t)blockIdx.x * rows;
  const int64_t r1 = std::min<int64_t>(n, r0 + rows);
  double acc = 0.0;
  if (phase < P)
    for (int64_t i = r0 + phase; i < r1; i += P) acc += (double)dX[i * d + j] * (double)X[i * d + j];
  sh[t] = acc;
  __syncthreads();
  if (t < d) {
    double s = 0.0;
    for (int ph = 0; ph < P; ++ph) s += sh[ph * d + t];
    partial[(int64_t)blockIdx.x * d + t] = s;
  }
}

__global__ void k_dls_final(int nblk, int d, const double* partial,
                            const float* ls, float* __restrict__ dls) {
  pdl_enter();
  // eight lanes a dimension, every eighth block each (304 dependent fp64 additions: 27 us)
  const int j = blockIdx.x * (blockDim.x / 8) + threadIdx.x / 8, lane = threadIdx.x % 8;
  double s = 0.0;
  if (j < d) {
#pragma unroll 8
    for (int b = lane; b < nblk; b += 8) s += partial[(int64_t)b * d + j];
  }
  for (int o = 4; o >= 1; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (j < d && lane == 0) dls[j] = (float)(-s / (double)ls[j]);
}

#define BW_CHECK(expr, what)                                  \
  do {                                                        \
    cudaError_t e_ = (expr);                                  \
    if (e_ != cudaSuccess) return cuda_status(e_, what);      \
  } while (0)

struct Work {
  cudaStream_t st;
  std::vector<void*> ptrs;
  ~Work() {
    for (void* p : ptrs) (void)cudaFreeAsync(p, st);
  }
  template <class T>
  cudaError_t get(T** p, size_t bytes, const Lattice* L = nullptr, int columns = 0) {
    bytes = std::max<size_t>(bytes, 16);
    cudaError_t e = L ? cols_malloc(L, columns, (void**)p, bytes, st) : dev_malloc((void**)p, bytes, st);
    if (e == cudaSuccess) ptrs.push_back((void*)*p);
    return e;
  }
};

template <class S, int VEC>
void launch_weight_grad(const Lattice* L, int k, int ld, const void* BU, const void* BS, const float* Vp,
                        const float* Gp, dfloat alpha, const double* f, const float* ls, float* dX,
                        cudaStream_t st) {
  const unsigned grid = (unsigned)ceil_div(L->n, kBT);
  const int D = L->D;
#define SGP_WG(MAXD)                                                                        \
  launch_pdl(k_weight_grad<MAXD, VEC, S>, grid, kBT, st, L->n, L->d, k, ld, L->perm, L->idx, L->rank, \
                                                    (const S*)BU, (const S*)BS, Vp, Gp,      \
                                                    alpha, f, ls, dX)
  if (D <= 8) SGP_WG(8);
  else if (D <= 16) SGP_WG(16);
  else if (D <= 32) SGP_WG(32);
  else if (D <= 64) SGP_WG(64);
  else SGP_WG(128);
#undef SGP_WG
  note_launches(1);
}

int transpose_blur(int blur) {
  return blur == SGP_BLUR_SEQUENTIAL ? SGP_BLUR_TRANSPOSE
         : blur == SGP_BLUR_TRANSPOSE ? SGP_BLUR_SEQUENTIAL
                                      : SGP_BLUR_SYMMETRIC;
}

// may_pair: the symmetric blur's two products may share their passes; *paired: they did.
sgp_status backward(Lattice* L, const float* X, const float* ls, const float* V, const float* G,
                    int k, int blur, float alpha, int grad, float* dV, float* dX, float* dls,
                    bool may_pair, bool* paired) {
  cudaStream_t st = L->stream;
  const int64_t n = L->n;
  const int d = L->d;
  Work w{st, {}};
  const bool want_x = dX || dls;
  float* dXw = dX;
  if (want_x && !dXw) BW_CHECK(w.get(&dXw, (size_t)n * d * sizeof(float)), "alloc dX");

  if (grad == SGP_GRAD_LATTICE) {
    sgp_status s = ensure_product(L, k, st);
    if (s != SGP_OK) return s;
    const int kp = value_cols(L, k);
    // B^T W^T G and B W^T V, each over its factor (both blurs have as many passes and the same
    // centre tap: one factor).  The symmetric blur is its own transpose, so the two can share
    // their passes as the halves of rows of 2 kp columns: half the launches, and rows of 32
    // bytes (k = 8) at random places cost DRAM 64 either way (n = 500k, d = 20, k = 8: 84 passes
    // of 22.3 us apart, 42 of 33.5 together).  Done where it takes no more memory than apart (in-place
    // blurs) or little of it.
    const int kp2 = 2 * kp;
    const size_t vb = lattice_value_bytes(L, kp), vb2 = 2 * vb;
    const bool pair = may_pair && want_x && blur == SGP_BLUR_SYMMETRIC && !L->tight_cols &&
                      kp2 <= 256 &&
                      (blur_in_place(L) || (!L->sparse && vb2 <= kPairBytes));
    *paired = pair;
    const int ld = pair ? kp2 : kp;
    const size_t one = sizeof(float);
    void *b0 = nullptr, *b1 = nullptr;
    float *Vp = nullptr, *Gp = nullptr;
    const void *BS = nullptr, *BU = nullptr;
    double scale = 1.0;
    if (pair) {
      float* part = nullptr;
      BW_CHECK(w.get(&b0, vb2, L, kp2), "alloc lattice values");
      if (!blur_in_place(L)) BW_CHECK(w.get(&b1, vb2, L, kp2), "alloc lattice values");
      BW_CHECK(w.get(&part, (size_t)L->nslots * kp2 * one, L, kp2), "alloc splat partials");
      BW_CHECK(w.get(&Gp, (size_t)n * kp2 * one, L, kp2), "alloc G, V");
      Vp = Gp + kp;
      enqueue_permute_pair(L, G, V, k, kp, Gp, st);
      BS = enqueue_splat_blur(L, Gp, kp2, k, blur, b0, b1, part, st, &scale);
      BU = static_cast<const char*>(BS) + vb / L->m;
    } else {
      BW_CHECK(w.get(&b0, vb, L, kp), "alloc lattice values");
      BW_CHECK(w.get(&b1, vb, L, kp), "alloc lattice values");
      BW_CHECK(w.get(&Vp, (size_t)n * kp * one, L, kp), "alloc V");
      BW_CHECK(w.get(&Gp, (size_t)n * kp * one, L, kp), "alloc G");
      enqueue_permute(L, G, k, kp, Gp, st);
      BS = enqueue_splat_blur(L, Gp, kp, k, transpose_blur(blur), b0, b1, L->partial, st, &scale);
    }
    const dfloat factor = split_factor(alpha * scale);
    if (dV) enqueue_slice_caller(L, BS, k, kp, ld, factor, dV, st);
    if (want_x) {
      if (!pair) {
        enqueue_permute(L, V, k, kp, Vp, st);
        BU = enqueue_splat_blur(L, Vp, kp, k, blur, L->lat[0], L->lat[1], L->partial, st, &scale);
      }
      const double scale = std::sqrt((double)(d * (d + 1))) / L->s;
      std::vector<double> hf(d);
      for (int j = 0; j < d; ++j) hf[j] = scale / std::sqrt((double)((j + 1) * (j + 2)));
      double* f = nullptr;
      BW_CHECK(w.get(&f, d * sizeof(double)), "alloc f");
      // pageable source: the call returns once hf has been staged
      BW_CHECK(cudaMemcpyAsync(f, hf.data(), d * sizeof(double), cudaMemcpyHostToDevice, st),
               "copy f");
      const bool v4 = kp % 4 == 0;
      if (L->value_dtype == SGP_VALUES_BF16) {
        if (v4) launch_weight_grad<bf16, 4>(L, kp, ld, BU, BS, Vp, Gp, factor, f, ls, dXw, st);
        else launch_weight_grad<bf16, 1>(L, kp, ld, BU, BS, Vp, Gp, factor, f, ls, dXw, st);
      } else {
        if (v4) launch_weight_grad<float, 4>(L, kp, ld, BU, BS, Vp, Gp, factor, f, ls, dXw, st);
        else launch_weight_grad<float, 1>(L, kp, ld, BU, BS, Vp, Gp, factor, f, ls, dXw, st);
      }
    }
  } else {  // SGP_GRAD_FILTER
    if (dV) {
      sgp_status s = ensure_product(L, k, st);
      if (s != SGP_OK) return s;
      enqueue_mvm(L, G, k, transpose_blur(blur), alpha, 0.f, dV, st);
    }
    if (want_x) {
      const int kk = 2 * k * (d + 1);
      const int chunk = std::min(kk, kFilterChunk);
      sgp_status s = ensure_product(L, chunk, st);
      if (s != SGP_OK) return s;
      float *in = nullptr, *F = nullptr;
      BW_CHECK(w.get(&in, (size_t)n * chunk * sizeof(float)), "alloc filter input");
      BW_CHECK(w.get(&F, (size_t)n * chunk * sizeof(float)), "alloc filter output");
      BW_CHECK(cudaMemsetAsync(dXw, 0, (size_t)n * d * sizeof(float), st), "clear dX");
      for (int col0 = 0; col0 < kk; col0 += chunk) {
        const int kc = std::min(chunk, kk - col0);
        launch_pdl(k_filter_in, (unsigned)ceil_div(n * kc, 256), 256, st, n, d, k, col0, kc, X, ls, V,
                                                                      G, in);
        enqueue_mvm(L, in, kc, blur, 1.f, 0.f, F, st);
        launch_pdl(k_filter_acc, (unsigned)ceil_div(n, kBT), kBT, st, n, d, k, col0, kc, X, ls, V, G,
                                                                 F, dXw);
        note_launches(2);
      }
      // dz = 2 alpha (k'/k) dZ with k' = -k/2 for the RBF; dX = dz / l
      launch_pdl(k_filter_finish, (unsigned)ceil_div(n * d, 256), 256, st, n, d, -alpha, ls, dXw);
      note_launches(1);
    }
  }
  if (dls) {
    double* part = nullptr;
    BW_CHECK(w.get(&part, (size_t)kDlsBlocks * d * sizeof(double)), "alloc partials");
    launch_pdl(k_dls_partial, kDlsBlocks, 256, st, n, d, X, dXw, part);
    launch_pdl(k_dls_final, (unsigned)ceil_div(d, 16), 128, st, kDlsBlocks, d, part, ls, dls);
    note_launches(2);
  }
  BW_CHECK(cudaGetLastError(), "launching the MVM backward");
  return SGP_OK;
}

}  // namespace

// Where memory is short: without pairing, then without padded rows.  (A pass that ran out of memory
// half way is done again from the start; it has written outputs only.)
sgp_status run_mvm_backward(Lattice* L, const float* X, const float* ls, const float* V,
                            const float* G, int k, int blur, float alpha, int grad, float* dV,
                            float* dX, float* dls) {
  bool paired = false;
  auto run = [&](bool may_pair) {
    return backward(L, X, ls, V, G, k, blur, alpha, grad, dV, dX, dls, may_pair, &paired);
  };
  sgp_status s = run(true);
  if (s == SGP_ERR_OOM && paired) s = run(false);
  if (s == SGP_ERR_OOM && (grad == SGP_GRAD_FILTER || padded_cols(k) != k) &&
      give_up_padding(L, L->stream))
    s = run(false);
  return s;
}

}  // namespace sgp
