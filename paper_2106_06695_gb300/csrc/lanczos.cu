// Log-determinant of A = outputscale K~ + noise I by stochastic Lanczos quadrature (the
// log-det term of Eq. gp_mll; App. A: at most 100 Lanczos iterations).
//
// For a probe z, m steps of Lanczos on (A, z / ||z||) give a symmetric tridiagonal T_m
// with z^T log(A) z ~ ||z||^2 e1^T log(T_m) e1 (Gauss quadrature of the spectral measure
// of z); averaging over probes with E[z z^T] = I estimates tr log(A) = log det A.  The
// Lanczos coefficients are read off the plain CG run on A x = z (the CG-Lanczos
// correspondence): with CG's step sizes alpha_j and ratios beta_j,
//   T[j][j]   = 1 / alpha_j + beta_{j-1} / alpha_{j-1}     (the second term absent at j = 0)
//   T[j+1][j] = sqrt(beta_j) / alpha_j.
// With q_j = 1 / alpha_j and e_j = beta_j / alpha_j, T = L U has the all-positive resolvent
// e1^T (T + t I)^-1 e1 = 1 / (t + R_0), R_j = q_j / (1 + e_j / (t + R_{j+1})), R_{m-1} =
// q_{m-1} (Stieltjes' continued fraction: no subtraction, so every value is good to a few m
// ulps), and since log x = int_0^inf (1 / (1 + t) - 1 / (x + t)) dt,
//   e1^T log(T) e1 = int_{-inf}^{inf} t (R_0 - 1) / ((1 + t) (t + R_0)) dx,  t = e^x.
// The integrand is analytic in |Im x| < pi and falls off as e^-|x|, so the trapezoidal rule
// with step h errs by e^(-2 pi^2 / h): h = 0.45 and tails cut at 1e-18 leave the rounding of
// fp64.  About 220 nodes, all independent.
#include <algorithm>
#include <cmath>
#include <vector>

#include "sgp_internal.cuh"

namespace sgp {
namespace {

constexpr int kMaxLanczos = 256;
constexpr int kSlqWarps = 8;     // node warps per probe (256 nodes: one round as a rule)
constexpr double kSlqStep = 0.45;  // trapezoid step in log t

constexpr double kQlFree = 1e-12;
constexpr int kQlSweeps = 64;  // QL iterations allowed per eigenvalue

// Whether the implicit QL iteration with Wilkinson shifts (Bowdler, Martin, Reinsch & Wilkinson
// 1968) finds all eigenvalues of the symmetric tridiagonal (diagonal d, e[i] coupling i and i + 1)
// above zero.  Overwrites d and e.
__device__ __noinline__ bool ql_positive(double* d, double* e, int m) {
  for (int l = 0; l < m; ++l) {
    for (int sweep = 0;; ++sweep) {
      int mm = l;
      for (; mm < m - 1; ++mm)
        if (fabs(e[mm]) <= 1e-15 * (fabs(d[mm]) + fabs(d[mm + 1]))) break;
      if (mm == l) break;
      if (sweep == kQlSweeps) return false;
      double g = (d[l + 1] - d[l]) / (2.0 * e[l]);  // shift from the leading 2 x 2 block
      double r = hypot(g, 1.0);
      g = d[mm] - d[l] + e[l] / (g + copysign(r, g));
      double s = 1.0, c = 1.0, p = 0.0;
      int i = mm - 1;
      for (; i >= l; --i) {
        const double f = s * e[i], b = c * e[i];
        r = hypot(f, g);
        e[i + 1] = r;
        if (r == 0.0) {  // split: deflate and restart this eigenvalue
          d[i + 1] -= p;
          e[mm] = 0.0;
          break;
        }
        s = f / r;
        c = g / r;
        g = d[i + 1] - p;
        r = (d[i] - g) * s + 2.0 * c * b;
        p = s * r;
        d[i + 1] = g + p;
        g = c * r - b;
      }
      if (r == 0.0 && i >= l) continue;
      d[l] -= p;
      e[l] = g;
      e[mm] = 0.0;
    }
    if (!(d[l] > 0.0)) return false;  // not touched again
  }
  return true;
}

// Block (w, c): warp w of probe c.  Warps 0 .. kSlqWarps - 1 sum the integrand at the nodes
// 32 w + lane (+ 256, ...), in a fixed order, into part[c][w] (scaled: the probe's value is
// the plain sum of its parts; a probe without iterations has none); warp kSlqWarps sets bad[c] when
// T is not numerically positive definite: an entry that is not finite, or an eigenvalue that the QL
// iteration rounds to zero or below.  (Every pivot of T's LDL^T is 1 / alpha_j > 0, whatever the
// operator: a singular one shows only in what rounding does to T's smallest eigenvalues.)  QL's
// eigenvalues are off by some 1e-13 ||T|| at most, so it need not run when all are above kQlFree
// ||T||, which the LDL^T of the shifted T tells: m divisions in place of some 150 m rotations.
//
// Bound by the latency of one fp64 division per step of the fraction.  The nodes are spread
// over one-warp blocks, so that a probe uses nine SMs' fp64 pipes.  It replaced an implicit
// QL iteration with one thread per probe (a serial chain of about 15,000 rotations, 21.8 ms
// for 10 probes of 100 steps); the whole log determinant at n = 46k, d = 9 went from 39.4 to
// 17.5 ms.  Against 50-digit arithmetic its values are off by 0 to 2e-16, QL's by up to 1e-12.
__global__ void __launch_bounds__(32) k_slq(const double* ha,
                                            const double* hb, int k, int cap,
                                            const int* iters,
                                            const double* bnorm,
                                            double* __restrict__ part, int* __restrict__ bad) {
  pdl_enter();
  __shared__ double al[kMaxLanczos], be[kMaxLanczos];
  const int c = blockIdx.y, w = blockIdx.x, lane = threadIdx.x;
  const int m = min(iters[c], cap);
  for (int j = lane; j < m; j += 32) {
    al[j] = ha[(int64_t)j * k + c];
    be[j] = j + 1 < m ? hb[(int64_t)j * k + c] : 0.0;
  }
  __syncwarp();
  if (w == kSlqWarps) {
    __shared__ double d[kMaxLanczos], e[kMaxLanczos];
    double norm = 0.0;
    bool ok = true;
    for (int j = lane; j < m; j += 32) {
      d[j] = 1.0 / al[j] + (j > 0 ? be[j - 1] / al[j - 1] : 0.0);
      e[j] = sqrt(be[j]) / al[j];  // 0 for the last
      norm = fmax(norm, d[j] + 2.0 * e[j]);
      ok = ok && isfinite(d[j]) && isfinite(e[j]);
    }
    // twice the largest of the rows' d + 2 e bounds what Gershgorin's circles reach
    for (int o = 16; o >= 1; o >>= 1) norm = fmax(norm, __shfl_xor_sync(0xffffffffu, norm, o));
    norm *= 2.0;
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    if (lane != 0) return;
    bool clear = true;  // T - kQlFree norm I is positive definite
    double piv = 1.0;
    for (int j = 0; j < m && ok && clear; ++j) {
      piv = d[j] - kQlFree * norm - (j > 0 ? e[j - 1] * e[j - 1] / piv : 0.0);
      clear = piv > 0.0;
    }
    bad[c] = ok && (clear || ql_positive(d, e, m)) ? 0 : 1;
    return;
  }
  double sum = 0.0;
  if (m > 0) {
    // F(0) = e1^T T^-1 e1 = alpha_0 + beta_0 (alpha_1 + beta_1 (...)) and T_00 = 1 / alpha_0
    // bound the tails (the integrand's are t (1 - F(0)) and (T_00 - 1) / t)
    double f0 = 0.0;
    for (int j = m - 1; j >= 0; --j) f0 = fma(be[j], f0, al[j]);
    const double q0 = 1.0 / al[0];
    f0 = fmin(f0, 1e300);
    const double x0 = -41.5 - log(fmax(1.0, f0)), x1 = 41.5 + log(fmax(1.0, q0));
    const double span = (x1 - x0) / kSlqStep;
    const int nodes = span >= 0.0 && span < 4096.0 ? (int)span + 2 : 0;  // NaN, Inf: see *bad
    __syncwarp();
    for (int j = lane; j < m; j += 32) {  // alpha, beta -> q, e
      const double a = al[j];
      al[j] = 1.0 / a;
      be[j] = be[j] / a;
    }
    __syncwarp();
    for (int i = 32 * w + lane; i < nodes; i += 32 * kSlqWarps) {
      const double t = exp(x0 + kSlqStep * i);
      double R = al[m - 1];
      for (int j = m - 2; j >= 0; --j) {
        const double u = t + R;
        R = al[j] * (u / (u + be[j]));
      }
      sum += (t / (1.0 + t)) * ((R - 1.0) / (t + R));
    }
  }
  for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) part[c * kSlqWarps + w] = m > 0 ? bnorm[c] * bnorm[c] * kSlqStep * sum : 0.0;
}

// sp: columns of the solver's rows (zero columns appended).
sgp_status logdet_rows(Lattice* L, const float* Z, int s, int sp, float noise, int max_lanczos,
                       float tol, double* logdet, double* quad) {
  cudaStream_t st = L->stream;
  const int cap = std::min(max_lanczos, kMaxLanczos);
  struct Bufs {
    cudaStream_t st;
    std::vector<void*> p;
    ~Bufs() {
      for (void* x : p) (void)cudaFreeAsync(x, st);
    }
  } b{st, {}};
  auto get = [&](void** x, size_t bytes) {
    cudaError_t e = dev_malloc(x, std::max<size_t>(bytes, 16), st);
    if (e == cudaSuccess) b.p.push_back(*x);
    return e;
  };
#define LZ_CHECK(expr, what)                                 \
  do {                                                       \
    cudaError_t e_ = (expr);                                 \
    if (e_ != cudaSuccess) return cuda_status(e_, what);     \
  } while (0)
  LanczosRecord rec{};
  rec.cap = cap;
  rec.cols = sp;
  float* X = nullptr;
  double* dq = nullptr;
  int* bad = nullptr;
  LZ_CHECK(get((void**)&rec.alpha, (size_t)cap * sp * sizeof(double)), "alloc Lanczos record");
  LZ_CHECK(get((void**)&rec.beta, (size_t)cap * sp * sizeof(double)), "alloc Lanczos record");
  LZ_CHECK(get((void**)&rec.bnorm, (size_t)sp * sizeof(double)), "alloc Lanczos record");
  LZ_CHECK(get((void**)&rec.iters, (size_t)sp * sizeof(int)), "alloc Lanczos record");
  LZ_CHECK(get((void**)&X, (size_t)L->n * s * sizeof(float)), "alloc CG solution");
  LZ_CHECK(get((void**)&dq, (size_t)s * kSlqWarps * sizeof(double)), "alloc quadratures");
  LZ_CHECK(get((void**)&bad, (size_t)s * sizeof(int)), "alloc flags");
  sgp_status status = run_cg(L, Z, s, SGP_BLUR_SYMMETRIC, noise, tol, cap, X, nullptr, nullptr,
                             0, 0, &rec);
  if (status != SGP_OK) return status;
  launch_pdl(k_slq, dim3(kSlqWarps + 1, (unsigned)s), 32, st, rec.alpha, rec.beta, sp, cap,
             rec.iters, rec.bnorm, dq, bad);
  note_launches(1);
  LZ_CHECK(cudaGetLastError(), "Lanczos quadrature");
  std::vector<double> hq(s, 0.0), hp((size_t)s * kSlqWarps);
  std::vector<int> hbad(s, 0);
  LZ_CHECK(cudaMemcpyAsync(hp.data(), dq, hp.size() * sizeof(double), cudaMemcpyDeviceToHost, st),
           "read quadratures");
  LZ_CHECK(cudaMemcpyAsync(hbad.data(), bad, s * sizeof(int), cudaMemcpyDeviceToHost, st),
           "read flags");
  LZ_CHECK(cudaStreamSynchronize(st), "sync Lanczos");
#undef LZ_CHECK
  for (int c = 0; c < s; ++c) {
    for (int w = 0; w < kSlqWarps; ++w) hq[c] += hp[(size_t)c * kSlqWarps + w];
    if (hbad[c]) hq[c] = std::nan("");
  }
  if (quad) std::copy(hq.begin(), hq.end(), quad);
  double sum = 0.0;
  for (double v : hq) sum += v;
  if (logdet) *logdet = sum / s;
  if (std::find(hbad.begin(), hbad.end(), 1) != hbad.end()) {
    set_error("sgp_logdet: a Lanczos tridiagonal was not numerically positive definite");
    return SGP_ERR_NONFINITE;
  }
  return SGP_OK;
}

}  // namespace

sgp_status run_logdet(Lattice* L, const float* Z, int s, float noise, int max_lanczos, float tol,
                      double* logdet, double* quad) {
  sgp_status st = logdet_rows(L, Z, s, value_cols(L, s), noise, max_lanczos, tol, logdet, quad);
  if (st == SGP_ERR_OOM && padded_cols(s) != s && give_up_padding(L, L->stream))
    st = logdet_rows(L, Z, s, s, noise, max_lanczos, tol, logdet, quad);
  return st;
}

}  // namespace sgp
