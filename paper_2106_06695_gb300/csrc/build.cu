// Lattice construction on the GPU (Sec. 3.2 "Splat"; Eq. canon_simplex).
//
//  1. k_elevate      one thread per point: z = x / l, y = E z in H_d (triangular basis),
//                    nearest remainder-0 point, rank of residuals, sum fix, barycentric
//                    weights.  Every floating-point step is a single IEEE-rounded FP64
//                    operation (explicit _rn intrinsics, file built with -fmad=false) so
//                    the integer results are identical to any other correct FP64
//                    evaluation of the same expression order.
//  2. locality order points sorted by their enclosing remainder-0 cell (lexicographic
//                    over the leading coordinates, stable), so that neighbouring work
//                    touches neighbouring vertices.
//  3. k_insert       one thread per (point, vertex): lock-free open addressing in a
//                    power-of-two table of 64-bit slots (31-bit hash tag | owner entry);
//                    the full key of a slot is recomputed from its owner entry, and
//                    atomicMin keeps the earliest entry as owner.
//  4. numbering      vertex ids = first occurrence in locality order (owner flags +
//                    exclusive scan).
//  5. k_neighbours   per vertex and direction j: ids of v +- t u_j, u_j = (d+1) e_j - 1, by
//                    looking the shifted linear hashes up in the sorted vertex hashes.
//  6. splat lists    (vertex, entry) pairs sorted stably by vertex id (radix sort) give
//                    each vertex the list of (point, weight) it gathers.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "sgp_internal.cuh"

namespace sgp {
namespace {

constexpr uint64_t kEmpty = ~0ull;

__device__ __forceinline__ uint64_t mix64(uint64_t h) {
  h ^= h >> 33;
  h *= 0xff51afd7ed558ccdull;
  h ^= h >> 33;
  h *= 0xc4ceb9fe1a85ec53ull;
  h ^= h >> 33;
  return h;
}
uint64_t host_mix64(uint64_t h) {
  h ^= h >> 33;
  h *= 0xff51afd7ed558ccdull;
  h ^= h >> 33;
  h *= 0xc4ceb9fe1a85ec53ull;
  h ^= h >> 33;
  return h;
}
uint64_t host_coord_mult(int c) { return host_mix64(0x9e3779b97f4a7c15ull * (uint64_t)(c + 1)) | 1ull; }

// Vertex hash, linear in the integer key: lin(key) = sum_c A_c key_c (mod 2^64) with odd
// per-coordinate multipliers A_c, then mixed.  A lattice step u_j = (d+1) e_j - 1 moves
// lin by (d+1) A_j - sum_c A_c, so a neighbour's hash costs O(1) from the vertex's.
// The multipliers A_c = mix64(0x9e3779b97f4a7c15 (c + 1)) | 1, one table per device
// (constant memory: the lattice kernels read them with warp-uniform c).
__constant__ uint64_t c_coord_mult[kMaxD];
__device__ __forceinline__ uint64_t coord_mult(int c) { return c_coord_mult[c]; }

__device__ __forceinline__ uint64_t lin_hash(const int* key, int D) {
  uint64_t h = 0;
  for (int c = 0; c < D; ++c) h += coord_mult(c) * (uint64_t)(int64_t)key[c];
  return h;
}

// Coordinate c of vertex k of the simplex (rem0, rank): rem0 + k, minus d+1 where the
// coordinate's rank exceeds d - k (the canonical vertex s_k, coordinates permuted).
__device__ __forceinline__ int vertex_coord(const int16_t* rem0, const uint8_t* rank, int d,
                                            int k, int c) {
  return (int)rem0[c] + k - ((int)rank[c] > d - k ? d + 1 : 0);
}

// Does the vertex of entry `e` (locality-ordered point e / D, vertex e % D) equal key?
template <int MAXD>
__device__ __forceinline__ bool entry_has_key(uint32_t e, const int* key, int d,
                                              const int32_t* perm, const int16_t* rem0,
                                              const uint8_t* rank) {
  const int D = d + 1;
  const int64_t i = perm[e / D];
  const int k = (int)(e % D);
  const int16_t* r0 = rem0 + i * D;
  const uint8_t* rk = rank + i * D;
  for (int c = 0; c < D; ++c)
    if (vertex_coord(r0, rk, d, k, c) != key[c]) return false;
  return true;
}

// ---------------------------------------------------------------------------------
// 1. Elevation, enclosing simplex, barycentric weights.
// ---------------------------------------------------------------------------------
// FP64 issues at about 2 results per SM and clock on this part, so the elevation is bound by
// its count of fp64 operations (comparisons and conversions included).  Where the result is
// the same, divisions become a multiplication with an exact correction, conversions become
// integer operations on the bits, and the rounding to a multiple of D starts from a fp32
// guess that a fp64 residual confirms: 14 fp64 operations a coordinate.

// Correctly rounded a / b from rb = RN(1 / b) (one Newton correction with an exact remainder;
// Markstein, "Computation of elementary functions on the IBM RISC System/6000", 1990).  With
// q0 = RN(a rb), |q0 - a/b| <= 2 ulp(q0).  Here b has at most 24 significant bits (a
// lengthscale, or D) and a is a float or a difference of magnitude |q0 b|, so a - q0 b is a
// multiple of ulp(q0) ulp(b) below 2^26 of them: exact in one fma.  Then q0 + r rb differs from
// a/b by at most 2^-51 ulp(q0), while a/b is at least 2^-25 ulp(q0) away from every
// rounding boundary (a - M b is a non-zero multiple of ulp(b) ulp(q0) / 2 for a 54-bit M, and
// M b = a would need more bits than a has), so the last fma rounds to RN(a/b).  a = 0 keeps
// its sign through q0.
__device__ __forceinline__ double div_rn(double a, double b, double rb) {
  const double q0 = __dmul_rn(a, rb);
  const double q = __fma_rn(__fma_rn(-q0, b, a), rb, q0);
  return (__double_as_longlong(a) << 1) == 0 ? q0 : q;
}

// x to 22 bits or more as a float (0 below 2^-126; callers bound it above).
__device__ __forceinline__ float narrow(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), m = hi & 0x7fffffffu;
  if (m < (897u << 20)) return 0.f;
  return __uint_as_float((hi & 0x80000000u) | ((m - (896u << 20)) << 3) |
                         ((uint32_t)__double2loint(x) >> 29));
}

constexpr int kElevT = 128;  // points per block

// Order-preserving integer image of a residual's fp64 bits (-0 taken as +0, no NaN here).
__device__ __forceinline__ long long rank_key(double x) {
  long long bits = __double_as_longlong(x);
  if (bits == (long long)0x8000000000000000ull) bits = 0;
  return bits ^ ((bits >> 63) & 0x7fffffffffffffffLL);
}

// (double) of an integer below 2^24 in magnitude.
__device__ __forceinline__ double exact_int(int x) {
  return widen((float)x);
}

// Nearest multiple of D to y (ties go down) as an integer, and y minus it.  False when the
// multiple lies beyond +-32000 (NaN included).
__device__ __noinline__ bool nearest_multiple_exact(double y, int D, int& r0, double& delta) {
  const double q = __ddiv_rn(y, (double)D);
  if (!(fabs(q) < 40000.0)) return false;
  const int lo = __double2int_rd(q) * D;
  const double below = __dsub_rn(y, (double)lo);            // y - down
  const double above = __dsub_rn((double)(lo + D), y);      // up - y
  const bool up = above < below;
  r0 = up ? lo + D : lo;
  delta = up ? -above : below;
  return r0 <= 32000 && r0 >= -32000;
}
// The same: a multiple whose residual is below D / 2 is the nearest one, however it was
// guessed.  The test compares the high words (2^-20 short of D / 2 at most); what it does
// not pass, ties and values beyond the range included, takes the exact path.
__device__ __forceinline__ bool nearest_multiple(double y, int D, float rD, int half_hi, int& r0,
                                                 double& delta) {
  const int y_hi = __double2hiint(y) & 0x7fffffff;
  if (y_hi < __double2hiint(32000.0)) {
    const int guess = __float2int_rn(narrow(y) * rD) * D;
    delta = __dsub_rn(y, exact_int(guess));
    if ((__double2hiint(delta) & 0x7fffffff) < half_hi && guess <= 32000 && guess >= -32000) {
      r0 = guess;
      return true;
    }
  }
  return nearest_multiple_exact(y, D, r0, delta);
}

// Range of rem0 / D per coordinate over all points, the caller's warps arriving converged;
// the plain read spares the atomic where the value would not change.
__device__ __forceinline__ void note_range(int q, int c, int* qmin, int* qmax, unsigned active,
                                           bool leader) {
  const int lo = __reduce_min_sync(active, q), hi = __reduce_max_sync(active, q);
  if (!leader) return;
  if (lo < __ldcg(qmin + c)) atomicMin(qmin + c, lo);
  if (hi > __ldcg(qmax + c)) atomicMax(qmax + c, hi);
}

// D <= MAXD <= 16: one thread per point, all per-coordinate values in registers (fully
// unrolled loops), the inputs and outputs of a block staged in shared memory so that global
// rows move coalesced, the rank-indexed weights through a conflict-free shared column.
// n = 2M, d = 11: 0.91 ms, against 2.05 ms with per-thread local arrays and fp64 divisions.
template <int MAXD>
__global__ void __launch_bounds__(kElevT) k_elevate_small(
    const float* X, const float* ls, const double* f,
    int64_t n, int d, int16_t* __restrict__ rem0_out, uint8_t* __restrict__ rank_out,
    float* __restrict__ w_out, int* __restrict__ qmin, int* __restrict__ qmax,
    unsigned* __restrict__ err, int inject_nan) {
  pdl_enter();
  __shared__ double s_l[MAXD], s_rl[MAXD], s_f[MAXD];
  __shared__ int s_bad;  // a lengthscale is not finite and positive
  __shared__ double s_v[MAXD][kElevT];  // then the block's outputs
  __shared__ float s_x[kElevT * MAXD];
  const int tid = threadIdx.x;
  const int D = d + 1;
  const double Dd = (double)D, rD = __drcp_rn(Dd);
  const float rDf = 1.f / (float)D;
  const int half_hi = __double2hiint(0.5 * Dd);
  const int64_t i0 = (int64_t)blockIdx.x * kElevT;
  const int pts = (int)min((int64_t)kElevT, n - i0);
  if (tid == 0) s_bad = 0;
  __syncthreads();
  if (tid < d) {
    const float lv = ls[tid];
    const double l = (double)lv;
    if (!isfinite(lv) || !(lv > 0.f)) s_bad = 1;
    s_l[tid] = l;
    s_rl[tid] = __drcp_rn(l);
    s_f[tid] = f[tid];
  }
  for (int q = tid; q < pts * d; q += kElevT) s_x[q] = X[i0 * d + q];
  __syncthreads();
  const bool live = tid < pts;
  bool bad = s_bad != 0;
  double y[MAXD];
  double sm = 0.0;
#pragma unroll
  for (int c = MAXD - 1; c >= 1; --c) {
    y[c] = 0.0;
    if (c > d) continue;
    const float xv = live ? s_x[tid * d + (c - 1)] : 0.f;
    if (!isfinite(xv)) bad = true;
    const double cf = __dmul_rn(div_rn(widen(xv), s_l[c - 1], s_rl[c - 1]), s_f[c - 1]);
    y[c] = __dsub_rn(sm, __dmul_rn((double)c, cf));
    sm = __dadd_rn(sm, cf);
  }
  y[0] = sm;
  if (inject_nan && i0 + tid == 0) bad = true;  // SGP_FAULT=nan_input
  if (bad) {
    if (live) atomicOr(err, ERRBIT_NONFINITE);
#pragma unroll
    for (int c = 0; c < MAXD; ++c) y[c] = 0.0;
  }
  int rem0[MAXD], rank[MAXD];
  long long key[MAXD];
  int sum = 0;
  bool range = false;
#pragma unroll
  for (int c = 0; c < MAXD; ++c) {
    rem0[c] = 0;
    key[c] = 0;
    if (c >= D) continue;
    double delta = 0.0;
    if (!nearest_multiple(y[c], D, rDf, half_hi, rem0[c], delta)) range = true;
    key[c] = rank_key(delta);
    sum += rem0[c];
  }
  if (range) {  // keep the rest of the computation in bounds; the build reports the error
    if (live) atomicOr(err, ERRBIT_RANGE);
    sum = 0;
#pragma unroll
    for (int c = 0; c < MAXD; ++c) {
      y[c] = 0.0;
      rem0[c] = 0;
      key[c] = 0;
    }
  }
  // rank: strictly larger residuals, plus equal residuals at a lower index; then move rem0
  // onto H_d (coordinate sum 0)
  const int h = sum / D;
#pragma unroll
  for (int c = 0; c < MAXD; ++c) {
    rank[c] = 0;
    if (c >= D) continue;
    int rk = h;
#pragma unroll
    for (int c2 = 0; c2 < MAXD; ++c2) {
      if (c2 == c || c2 >= D) continue;
      rk += (c2 < c ? key[c2] >= key[c] : key[c2] > key[c]) ? 1 : 0;
    }
    if (rk < 0) {
      rk += D;
      rem0[c] += D;
    } else if (rk > d) {
      rk -= D;
      rem0[c] -= D;
    }
    rank[c] = min(max(rk, 0), d);  // already true when sum(y) = 0; guards the indexing
    s_v[rank[c]][tid] = div_rn(__dsub_rn(y[c], exact_int(rem0[c])), Dd, rD);
  }
#pragma unroll
  for (int c = 0; c < MAXD; ++c) {
    if (c >= D) continue;
    // rem0 is a multiple of D: exact; idle threads repeat their warp's first point, if any
    const int first = __shfl_sync(0xffffffffu, rem0[c], 0);
    note_range((live ? rem0[c] : first) / D, c, qmin, qmax, 0xffffffffu,
               (tid & 31) == 0 && tid < pts);
  }
  // w[t] = v of rank d - t minus v of rank D - t (w[0]: plus one)
  float w[MAXD];
  {
    const double first = s_v[d][tid], last = s_v[0][tid];
    w[0] = __double2float_rn(__dadd_rn(first, __dadd_rn(1.0, -last)));
#pragma unroll
    for (int t = 1; t < MAXD; ++t)
      if (t < D) w[t] = __double2float_rn(__dsub_rn(s_v[d - t][tid], s_v[D - t][tid]));
  }
  __syncthreads();
  float* o_w = s_x;  // reuse: kElevT * D floats, then ranks and rem0 in the s_v area
  int16_t* o_r = reinterpret_cast<int16_t*>(&s_v[0][0]);
  uint8_t* o_k = reinterpret_cast<uint8_t*>(o_r + kElevT * MAXD);
  if (live) {
#pragma unroll
    for (int c = 0; c < MAXD; ++c) {
      if (c >= D) continue;
      o_w[tid * D + c] = w[c];
      o_r[tid * D + c] = (int16_t)rem0[c];
      o_k[tid * D + c] = (uint8_t)rank[c];
    }
  }
  __syncthreads();
  const int64_t e0 = i0 * D;  // a multiple of 128: 4-byte words of every output stay aligned
  const int count = pts * D;
  for (int q = tid; q < count; q += kElevT) w_out[e0 + q] = o_w[q];
  for (int q = 2 * tid; q < count; q += 2 * kElevT) {
    if (q + 1 < count) *reinterpret_cast<uint32_t*>(rem0_out + e0 + q) = *reinterpret_cast<uint32_t*>(o_r + q);
    else rem0_out[e0 + q] = o_r[q];
  }
  for (int q = 4 * tid; q < count; q += 4 * kElevT) {
    if (q + 3 < count) *reinterpret_cast<uint32_t*>(rank_out + e0 + q) = *reinterpret_cast<uint32_t*>(o_k + q);
    else
      for (int z = q; z < count; ++z) rank_out[e0 + z] = o_k[z];
  }
}

// Any D <= MAXD: one thread per point, per-coordinate values in local memory (n = 500k, d =
// 20: 0.46 ms, before 0.96; n = 60k, d = 50: 0.33 ms, before 0.48).
template <int MAXD>
__global__ void __launch_bounds__(kElevT) k_elevate(const float* X,
                                                    const float* ls,
                                                    const double* f, int64_t n,
                                                    int d, int16_t* __restrict__ rem0_out,
                                                    uint8_t* __restrict__ rank_out,
                                                    float* __restrict__ w_out,
                                                    int* __restrict__ qmin, int* __restrict__ qmax,
                                                    unsigned* __restrict__ err, int inject_nan) {
  pdl_enter();
  __shared__ double s_l[MAXD], s_rl[MAXD], s_f[MAXD];
  __shared__ int s_bad;  // a lengthscale is not finite and positive
  const int D = d + 1;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  for (int c = threadIdx.x; c < d; c += kElevT) {
    const float lv = ls[c];
    const double l = (double)lv;
    if (!isfinite(lv) || !(lv > 0.f)) s_bad = 1;
    s_l[c] = l;
    s_rl[c] = __drcp_rn(l);
    s_f[c] = f[c];
  }
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double Dd = (double)D, rD = __drcp_rn(Dd);
  const float rDf = 1.f / (float)D;
  const int half_hi = __double2hiint(0.5 * Dd);
  double y[MAXD];  // then the weights' differences by rank
  int rem0[MAXD];
  int rank[MAXD];
  bool bad = s_bad != 0;
  // y = E z, E's column j is (1, .., 1, -(j+1), 0, ..) / sqrt((j+1)(j+2)) times the scale;
  // f[j] already holds scale / sqrt((j+1)(j+2)).
  double sm = 0.0;
  for (int c = d; c >= 1; --c) {
    const float xv = X[i * d + (c - 1)];
    if (!isfinite(xv)) bad = true;
    const double cf = __dmul_rn(div_rn(widen(xv), s_l[c - 1], s_rl[c - 1]), s_f[c - 1]);
    y[c] = __dsub_rn(sm, __dmul_rn((double)c, cf));
    sm = __dadd_rn(sm, cf);
  }
  y[0] = sm;
  if (inject_nan && i == 0) bad = true;  // SGP_FAULT=nan_input
  if (bad) {
    atomicOr(err, ERRBIT_NONFINITE);
    for (int c = 0; c < D; ++c) y[c] = 0.0;
  }
  // nearest remainder-0 point coordinate by coordinate (ties go down)
  int sum = 0;
  bool range = false;
  long long key[MAXD];
  for (int c = 0; c < D; ++c) {
    double delta = 0.0;
    int r0 = 0;
    if (!nearest_multiple(y[c], D, rDf, half_hi, r0, delta)) range = true;
    rem0[c] = r0;
    key[c] = rank_key(delta);
    sum += r0;
  }
  if (range) {  // keep the rest of the computation in bounds; the build reports the error
    atomicOr(err, ERRBIT_RANGE);
    sum = 0;
    for (int c = 0; c < D; ++c) {
      y[c] = 0.0;
      rem0[c] = 0;
      key[c] = 0;
    }
  }
  // rank: strictly larger residuals, plus equal residuals at a lower index (compared through
  // their integer images, the same order at integer-compare cost)
  for (int c = 0; c < D; ++c) {
    const long long kc = key[c];
    int rk = 0;
    for (int c2 = 0; c2 < c; ++c2) rk += key[c2] >= kc ? 1 : 0;
    for (int c2 = c + 1; c2 < D; ++c2) rk += key[c2] > kc ? 1 : 0;
    rank[c] = rk;
  }
  // move rem0 onto H_d (coordinate sum 0); b holds the weights' terms by rank
  const int h = sum / D;
  double b[MAXD];
  for (int c = 0; c < D; ++c) {
    int rk = rank[c] + h;
    if (rk < 0) {
      rk += D;
      rem0[c] += D;
    } else if (rk > d) {
      rk -= D;
      rem0[c] -= D;
    }
    rk = min(max(rk, 0), d);  // already true when sum(y) = 0; guards the indexing
    rank[c] = rk;
    b[rk] = div_rn(__dsub_rn(y[c], exact_int(rem0[c])), Dd, rD);
  }
  for (int c = 0; c < D; ++c) {
    rem0_out[i * D + c] = (int16_t)rem0[c];
    rank_out[i * D + c] = (uint8_t)rank[c];
    const double w = c == 0 ? __dadd_rn(b[d], __dadd_rn(1.0, -b[0])) : __dsub_rn(b[d - c], b[D - c]);
    w_out[i * D + c] = __double2float_rn(w);
  }
  const unsigned active = __activemask();
  const bool leader = (int)(threadIdx.x & 31) == __ffs(active) - 1;
  for (int c = 0; c < D; ++c)  // rem0 is a multiple of D: exact
    note_range(rem0[c] / D, c, qmin, qmax, active, leader);
}

// ---------------------------------------------------------------------------------
// 2. Locality key: the remainder-0 cell's leading coordinates packed MSB-first.
// ---------------------------------------------------------------------------------
struct CellPack {
  int ncoord;
  int shift[kMaxD];
  int qmin[kMaxD];
};

__global__ void k_point_key(const int16_t* rem0, int64_t n, int D, CellPack pk,
                            uint32_t* __restrict__ key, uint32_t* __restrict__ val) {
  pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t k = 0;
  for (int c = 0; c < pk.ncoord; ++c)
    k |= (uint32_t)((int)rem0[i * D + c] / D - pk.qmin[c]) << pk.shift[c];
  key[i] = k;
  val[i] = (uint32_t)i;
}

// ---------------------------------------------------------------------------------
// 3. Hash insert.
// ---------------------------------------------------------------------------------
// A slot only ever goes from empty to a vertex, whose owner only decreases: it is read before an
// atomic is tried, and an entry above the owner seen there needs none (n = 628k, d = 3, where
// 2.5M entries share a few thousand vertices: 450 us with an atomic per probe).  The linear hash
// goes to hash_lo / hash_hi for the numbering.
template <int MAXD>
__global__ void __launch_bounds__(256) k_insert(const int32_t* perm,
                                                const int16_t* rem0,
                                                const uint8_t* rank, int64_t nD,
                                                int d, unsigned long long* __restrict__ table,
                                                uint64_t mask, int32_t* __restrict__ entry_slot,
                                                uint32_t* __restrict__ hash_lo,
                                                uint32_t* __restrict__ hash_hi,
                                                unsigned* __restrict__ err) {
  pdl_enter();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nD) return;
  const int D = d + 1;
  const int64_t i = perm[e / D];
  const int k = (int)(e % D);
  int key[MAXD];
  for (int c = 0; c < D; ++c) key[c] = vertex_coord(rem0 + i * D, rank + i * D, d, k, c);
  const uint64_t lin = lin_hash(key, D);
  hash_lo[e] = (uint32_t)lin;
  hash_hi[e] = (uint32_t)(lin >> 32);
  const uint64_t h = mix64(lin);
  const uint32_t tag = (uint32_t)(h >> 33);
  const unsigned long long mine = ((unsigned long long)tag << 32) | (uint32_t)e;
  uint64_t slot = h & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    unsigned long long prev = __ldcg(&table[slot]);
    if (prev == kEmpty) prev = atomicCAS(&table[slot], kEmpty, mine);
    if (prev == kEmpty) {
      entry_slot[e] = (int32_t)slot;
      return;
    }
    if ((uint32_t)(prev >> 32) == tag &&
        entry_has_key<MAXD>((uint32_t)prev, key, d, perm, rem0, rank)) {
      if (mine < prev) atomicMin(&table[slot], mine);
      entry_slot[e] = (int32_t)slot;
      return;
    }
    slot = (slot + 1) & mask;
  }
  atomicOr(err, ERRBIT_HASH_FULL);
  entry_slot[e] = -1;
}

// ---------------------------------------------------------------------------------
// 4. Numbering: owner flags, then ids by scan, then slot -> id and vertex keys.
// ---------------------------------------------------------------------------------
__global__ void k_owner_flags(const int32_t* entry_slot,
                              const unsigned long long* table, int64_t nD,
                              uint32_t* __restrict__ flags) {
  pdl_enter();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nD) return;
  const int32_t s = entry_slot[e];
  flags[e] = (s >= 0 && (uint32_t)table[s] == (uint32_t)e) ? 1u : 0u;
}

// Owners of a warp have consecutive ids, so their key rows are one piece of memory, which the
// warp writes element by element (m = 10.5M, d = 20, 441 MB: 764 us with each thread writing its
// own 42-byte row, hashing it and looking its slot up again).  An entry owns its vertex where the
// scan steps.
constexpr int kAssignThreads = 256;
__global__ void __launch_bounds__(kAssignThreads)
    k_assign_ids(const uint32_t* scanned, const uint32_t* total,
                 const int32_t* entry_slot, const int32_t* perm,
                 const int16_t* rem0, const uint8_t* rank,
                 const uint32_t* hash_lo, const uint32_t* hash_hi,
                 int64_t nD, int d, int32_t* __restrict__ slot_id, int16_t* __restrict__ keys,
                 uint64_t* __restrict__ vhash, uint32_t* __restrict__ owner) {
  pdl_enter();
  __shared__ int2 from[kAssignThreads / 32][32];  // (point, vertex) of the warp's owners in order
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int D = d + 1;
  const uint32_t id = e < nD ? scanned[e] : 0u;
  const uint32_t next = e + 1 < nD ? scanned[e + 1] : *total;
  const bool own = e < nD && next != id;
  const unsigned owners = __ballot_sync(0xffffffffu, own);
  if (owners == 0) return;
  if (own) {
    from[warp][__popc(owners & ((1u << lane) - 1u))] = make_int2(perm[e / D], (int)(e % D));
    slot_id[entry_slot[e]] = (int32_t)id;
    owner[id] = (uint32_t)e;
    vhash[id] = (uint64_t)hash_hi[e] << 32 | hash_lo[e];
  }
  __syncwarp();
  int16_t* out = keys + (int64_t)__shfl_sync(0xffffffffu, id, __ffs(owners) - 1) * D;
  const int many = __popc(owners) * D;
  int row = lane / D, c = lane - row * D;
  for (int q = lane; q < many; q += 32) {
    const int2 p = from[warp][row];
    out[q] = (int16_t)vertex_coord(rem0 + (int64_t)p.x * D, rank + (int64_t)p.x * D, d, p.y, c);
    for (c += 32; c >= D; c -= D) ++row;
  }
}

__global__ void k_entry_ids(const int32_t* entry_slot,
                            const int32_t* slot_id,
                            const int32_t* perm, const float* w_user,
                            const uint8_t* rank_user, int64_t nD, int D,
                            int32_t* __restrict__ idx, float* __restrict__ w,
                            uint8_t* __restrict__ rank) {
  pdl_enter();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nD) return;
  const int32_t s = entry_slot[e];
  const int64_t u = (int64_t)perm[e / D] * D + (e % D);
  const int32_t id = s >= 0 ? slot_id[s] : 0;  // all loads ahead of the stores
  const float wt = w_user[u];
  const uint8_t rk = rank_user[u];
  idx[e] = id;
  w[e] = wt;
  rank[e] = rk;
}

// ---------------------------------------------------------------------------------
// 5. Neighbour table.
// ---------------------------------------------------------------------------------
// A lattice step u_j moves the linear hash by a constant delta_j, so the vertices in hash
// order have their candidates v + t u_j in hash order too: a warp's 32 lookups of one
// direction fall into a few neighbouring buckets of the sorted hashes and read a few
// consecutive sectors, where probing a hash table (or a bit filter) in any other order
// touches a sector of its own for every candidate.  The index holds 32 bits of each hash
// beside its bucket, so that it stays in L2 up to some 15M vertices.  One side is looked up;
// a match is confirmed on the keys and written on both (u is v + t u_j, v is u - t u_j).
// Consecutive vertices of a simplex are one step apart (vertex k + 1 is vertex k minus u_c, c
// the coordinate of rank d - k, cyclically), so every vertex starts with the two links its
// own simplex gives it, and those need no confirmation.
// Measured, all steps of the table (the filter and table probes of every candidate that this
// replaced in brackets): n = 500k, d = 20 (m = 10.5M) 1.9 ms (5.1); n = 60k, d = 50 (m = 3.1M)
// 1.2 ms (5.0); n = 2M, d = 11 (m = 1.6M) 0.75 ms (1.4).

// Bit j % 32 of above[j / 32][v] / below[j / 32][v]: v has a neighbour v + u_j / v - u_j
// (stencil order 1).  Null: not recorded.
struct LinkBits {
  uint32_t* above;
  uint32_t* below;
};

// nbr[j][t][side][v]: the links of v's owner simplex, -1 elsewhere; up[v]: the direction along
// which v's link upwards lies.  owner[v]: its entry.
__global__ void __launch_bounds__(256) k_nbr_init(const uint32_t* owner,
                                                  const int32_t* idx,
                                                  const uint8_t* rank, int64_t m, int d,
                                                  int r, int32_t* __restrict__ nbr,
                                                  uint8_t* __restrict__ up, LinkBits lb) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= m) return;
  const int D = d + 1;
  const uint32_t e = owner[v];
  const uint32_t p = e / (uint32_t)D;
  const int k = (int)(e - p * (uint32_t)D);
  const int64_t row = (int64_t)p * D;
  // v - u_c, c of rank d - k, is vertex k + 1 (0 after d); v + u_c, c of rank d - k + 1 (0
  // for k = 0), is vertex k - 1 (d before 0)
  const int below = idx[row + (k == d ? 0 : k + 1)], above = idx[row + (k == 0 ? d : k - 1)];
  const int rk_below = d - k, rk_above = k == 0 ? 0 : d - k + 1;
  int dir = 0;
  uint32_t has_above = 0, has_below = 0;
  for (int j = 0; j < D; ++j) {
    const int rk = rank[row + j];
    if (rk == rk_above) dir = j;
    has_above |= (rk == rk_above ? 1u : 0u) << (j & 31);
    has_below |= (rk == rk_below ? 1u : 0u) << (j & 31);
    if (lb.above && ((j & 31) == 31 || j == d)) {
      lb.above[(int64_t)(j >> 5) * m + v] = has_above;
      lb.below[(int64_t)(j >> 5) * m + v] = has_below;
      has_above = has_below = 0;
    }
    int32_t* q = nbr + (int64_t)j * r * 2 * m + v;
    __stcs(q, rk == rk_below ? below : -1);
    __stcs(q + m, rk == rk_above ? above : -1);
    for (int t = 2; t <= r; ++t) {
      __stcs(q + (int64_t)(2 * t - 2) * m, -1);
      __stcs(q + (int64_t)(2 * t - 1) * m, -1);
    }
  }
  up[v] = (uint8_t)dir;
}

// The other ends of those links, where they belong to another simplex and so did not write
// theirs.  (Several simplices may write one link; they write the same id.)
__global__ void __launch_bounds__(256) k_nbr_close(const uint32_t* owner,
                                                   const int32_t* idx,
                                                   const uint8_t* rank, int64_t m,
                                                   int d, int r, int32_t* __restrict__ nbr,
                                                   LinkBits lb) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= m) return;
  const int D = d + 1;
  const uint32_t e = owner[v];
  const uint32_t p = e / (uint32_t)D;
  const int k = (int)(e - p * (uint32_t)D);
  const int64_t row = (int64_t)p * D;
#pragma unroll
  for (int side = 0; side < 2; ++side) {  // 0: the link below v, 1: the link above
    const int other = side == 0 ? (k == d ? 0 : k + 1) : (k == 0 ? d : k - 1);
    const int u = idx[row + other];
    if (owner[u] == (uint32_t)(row + other)) continue;
    const int rk = side == 0 ? d - k : (k == 0 ? 0 : d - k + 1);
    int j = 0;
    while (rank[row + j] != rk) ++j;  // ranks are a permutation of 0..d
    nbr[((int64_t)j * r * 2 + (side == 0 ? 1 : 0)) * m + u] = (int32_t)v;
    if (lb.above) atomicOr((side == 0 ? lb.above : lb.below) + (int64_t)(j >> 5) * m + u, 1u << (j & 31));
  }
}

// Sort keys: the top bits of the vertex hashes.
__global__ void k_hash_keys(const uint64_t* vhash, int64_t m, int shift,
                            uint32_t* __restrict__ key, uint32_t* __restrict__ val) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= m) return;
  key[v] = (uint32_t)(vhash[v] >> shift);
  val[v] = (uint32_t)v;
}

// Of the i-th vertex in bucket order: its hash (low and high half) and its direction up;
// start[b] = first i of bucket b (b <= buckets).
__global__ void k_hash_index(const uint32_t* key, const uint32_t* ord,
                             const uint64_t* vhash, const uint8_t* up,
                             int64_t m, int64_t buckets, uint32_t* __restrict__ low,
                             uint32_t* __restrict__ high, uint8_t* __restrict__ up_sorted,
                             uint32_t* __restrict__ start) {
  pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const uint32_t v = ord[i];
  const int64_t own = key[i], first = i == 0 ? 0 : (int64_t)key[i - 1] + 1;
  const uint64_t h = vhash[v];  // all loads ahead of the stores
  const uint8_t dir = up[v];
  low[i] = (uint32_t)h;
  high[i] = (uint32_t)(h >> 32);
  up_sorted[i] = dir;
  for (int64_t b = first; b <= own; ++b) start[b] = (uint32_t)i;
  if (i == m - 1)
    for (int64_t b = own + 1; b <= buckets; ++b) start[b] = (uint32_t)m;
}

// Does coordinate c of u equal that of v + t u_j?  Coordinates stay within +-32255 (rem0 within
// 32000, the sum fix and the vertex offset add less than 2 D), so no sum leaves int16.
__device__ __forceinline__ bool steps_to(int16_t v, int16_t u, int c, int j, int t, int D) {
  return (int)u == (int)v + t * ((c == j ? D : 0) - 1);
}

// Thread i: the i-th vertex in hash order, all directions but the one its simplex gave.  The
// bucket bounds of kNbrGroup directions are loaded together, then their first hashes, so
// that their latencies overlap; a lane walks its bucket on its own.  Matches are confirmed on
// the keys by the thread itself for D <= 16 (every row load in flight at once), by the whole
// warp, one after another, above (a lane alone would walk a row of D loads while 31 wait).
// *hits receives the number of pairs (v, v + u_j).
// Five blocks an SM (48 registers): n = 500k, d = 20 0.93 ms, 1.08 with the 54 registers it would take.
constexpr int kNbrGroup = 4;
template <bool WARP>
__global__ void __launch_bounds__(256, 5) k_neighbours(
    const int16_t* keys, const uint32_t* low,
    const uint32_t* high, const uint8_t* up,
    const uint32_t* ord, const uint32_t* start, int shift, int64_t m,
    int d, int r, uint64_t sum_A, int32_t* __restrict__ nbr, unsigned long long* __restrict__ hits,
    LinkBits lb) {
  pdl_enter();
  __shared__ uint64_t delta[kMaxD];  // hash of u_j
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int D = d + 1, lane = (int)(threadIdx.x & 31);
  for (int j = threadIdx.x; j < D; j += blockDim.x) delta[j] = (uint64_t)D * coord_mult(j) - sum_A;
  __syncthreads();
  const bool live = i < m;
  const uint64_t h = live ? (uint64_t)high[i] << 32 | low[i] : 0;
  const int given = live ? up[i] : 0;
  unsigned found = live ? 1u : 0u;  // the given pair
  for (int j0 = 0; j0 < D; j0 += kNbrGroup) {
    for (int t = 1; t <= r; ++t) {
      uint32_t want[kNbrGroup], at[kNbrGroup], p[kNbrGroup], end[kNbrGroup];
#pragma unroll
      for (int q = 0; q < kNbrGroup; ++q) {
        const uint64_t x = h + (uint64_t)t * delta[min(j0 + q, D - 1)];
        const uint32_t* s = start + (x >> shift);
        const bool on = live && j0 + q < D && (t > 1 || j0 + q != given);
        want[q] = (uint32_t)x;
        p[q] = on ? *s : 0u;
        end[q] = on ? s[1] : 0u;
      }
#pragma unroll
      for (int q = 0; q < kNbrGroup; ++q) at[q] = p[q] < end[q] ? low[p[q]] : 0u;
#pragma unroll
      for (int q = 0; q < kNbrGroup; ++q) {
        const int j = j0 + q;
        int32_t* plane = nbr + ((int64_t)j * r + (t - 1)) * 2 * m;
        bool more = true;
        while (more) {
          while (p[q] < end[q] && at[q] != want[q])
            if (++p[q] < end[q]) at[q] = low[p[q]];
          __syncwarp();
          const bool match = p[q] < end[q];
          unsigned todo = __ballot_sync(0xffffffffu, match);
          if (!todo) break;
          const uint32_t u = match ? ord[p[q]] : 0u, v = match ? ord[i] : 0u;
          bool ok = false;
          if (WARP) {
            while (todo) {
              const int src = __ffs(todo) - 1;
              todo &= todo - 1;
              const int16_t* kv = keys + (int64_t)__shfl_sync(0xffffffffu, v, src) * D;
              const int16_t* ku = keys + (int64_t)__shfl_sync(0xffffffffu, u, src) * D;
              bool same = true;
#pragma unroll
              for (int c0 = 0; c0 < kMaxD; c0 += 32)
                if (c0 < D && c0 + lane < D)
                  same = same & steps_to(kv[c0 + lane], ku[c0 + lane], c0 + lane, j, t, D);
              same = __all_sync(0xffffffffu, same);
              ok = ok || (same && lane == src);
            }
          } else if (match) {
            const int16_t *kv = keys + (int64_t)v * D, *ku = keys + (int64_t)u * D;
            ok = true;
#pragma unroll
            for (int c = 0; c < 16; ++c)
              if (c < D) ok = ok & steps_to(kv[c], ku[c], c, j, t, D);
          }
          if (ok) {
            plane[u] = (int32_t)v;
            plane[m + v] = (int32_t)u;
            if (lb.above) {
              atomicOr(lb.above + (int64_t)(j >> 5) * m + v, 1u << (j & 31));
              atomicOr(lb.below + (int64_t)(j >> 5) * m + u, 1u << (j & 31));
            }
            found += t == 1 ? 1u : 0u;
            p[q] = end[q];
          } else if (match && ++p[q] < end[q]) {  // another vertex with these hash bits
            at[q] = low[p[q]];
          }
          more = __any_sync(0xffffffffu, p[q] < end[q]);
        }
      }
    }
  }
  found = __reduce_add_sync(0xffffffffu, found);
  if (lane == 0 && found) atomicAdd(hits, (unsigned long long)found);
}

// The link bits read off the table, where they were not recorded while it was made; for r > 1,
// above = any neighbour along the direction and below = 0.
__global__ void __launch_bounds__(256) k_link_bits(const int32_t* nbr, int64_t m,
                                                   int D, int r, LinkBits lb) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= m) return;
  for (int j0 = 0; j0 < D; j0 += 32) {
    uint32_t hi = 0, lo = 0;
    for (int j = j0; j < min(j0 + 32, D); ++j) {
      const int32_t* p = nbr + (int64_t)j * 2 * r * m + v;
      if (r == 1) {
        lo |= (__ldcs(p) >= 0 ? 1u : 0u) << (j & 31);
        hi |= (__ldcs(p + m) >= 0 ? 1u : 0u) << (j & 31);
      } else {
        int any = -1;
        for (int q = 0; q < 2 * r; ++q) any = max(any, __ldcs(p + (int64_t)q * m));
        hi |= (any >= 0 ? 1u : 0u) << (j & 31);
      }
    }
    lb.above[(int64_t)(j0 >> 5) * m + v] = hi;
    lb.below[(int64_t)(j0 >> 5) * m + v] = lo;
  }
}

// counts[j]: the vertices with a neighbour along j; heads[j]: those that head a chain along j
// (one above and none below).
__global__ void __launch_bounds__(256) k_link_counts(LinkBits lb, int64_t m, int D,
                                                     unsigned long long* __restrict__ counts,
                                                     unsigned long long* __restrict__ heads) {
  pdl_enter();
  __shared__ unsigned block_count[kMaxD], block_heads[kMaxD];
  for (int j = threadIdx.x; j < D; j += blockDim.x) block_count[j] = block_heads[j] = 0;
  __syncthreads();
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < m;
       v += (int64_t)gridDim.x * blockDim.x)
    for (int w = 0; w * 32 < D; ++w) {
      const uint32_t hi = lb.above[(int64_t)w * m + v], lo = lb.below[(int64_t)w * m + v];
      for (uint32_t x = hi | lo; x; x &= x - 1) atomicAdd(&block_count[w * 32 + __ffs(x) - 1], 1u);
      for (uint32_t x = hi & ~lo; x; x &= x - 1) atomicAdd(&block_heads[w * 32 + __ffs(x) - 1], 1u);
    }
  __syncthreads();
  for (int j = threadIdx.x; j < D; j += blockDim.x) {
    if (block_count[j]) atomicAdd(&counts[j], (unsigned long long)block_count[j]);
    if (block_heads[j]) atomicAdd(&heads[j], (unsigned long long)block_heads[j]);
  }
}

// Direction lists: thread per vertex, reading its direction bits (32 directions per word).
// A block first counts, per warp and direction, its vertices with a neighbour along the
// direction, takes one slot range per direction with one atomic, then each warp writes its
// vertices at its prefix within that range.  The order of a list is immaterial to the
// blur, which updates its vertices independently.
constexpr int kFillThreads = 512;
__global__ void __launch_bounds__(kFillThreads) k_active_fill(
    LinkBits lb, int64_t m, int D, const int64_t* off,
    unsigned long long* __restrict__ fill, int32_t* __restrict__ act) {
  pdl_enter();
  constexpr int kWarps = kFillThreads / 32;
  __shared__ unsigned wpos[kWarps][kMaxD];  // counts, then each warp's offset in the list
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = v < m;
  const int lane = (int)(threadIdx.x & 31), warp = (int)(threadIdx.x >> 5);
  for (int e = threadIdx.x; e < kWarps * kMaxD; e += blockDim.x) (&wpos[0][0])[e] = 0;
  __syncthreads();
  for (int w = 0; w * 32 < D; ++w) {
    const uint32_t bits = live ? lb.above[(int64_t)w * m + v] | lb.below[(int64_t)w * m + v] : 0u;
    uint32_t seen = __reduce_or_sync(0xffffffffu, bits);
    while (seen) {
      const int b = __ffs(seen) - 1;
      seen &= seen - 1;
      const unsigned with = __ballot_sync(0xffffffffu, (bits >> b) & 1u);
      if (lane == 0) wpos[warp][w * 32 + b] = (unsigned)__popc(with);
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < D; j += blockDim.x) {
    unsigned total = 0;
    for (int q = 0; q < kWarps; ++q) total += wpos[q][j];
    if (total == 0) continue;
    unsigned run = (unsigned)atomicAdd(&fill[j], (unsigned long long)total);
    for (int q = 0; q < kWarps; ++q) {
      const unsigned c = wpos[q][j];
      wpos[q][j] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int w = 0; w * 32 < D; ++w) {
    const uint32_t bits = live ? lb.above[(int64_t)w * m + v] | lb.below[(int64_t)w * m + v] : 0u;
    uint32_t seen = __reduce_or_sync(0xffffffffu, bits);
    while (seen) {
      const int b = __ffs(seen) - 1;
      seen &= seen - 1;
      const int j = w * 32 + b;
      const bool on = (bits >> b) & 1u;
      const unsigned with = __ballot_sync(0xffffffffu, on);
      if (on) act[off[j] + wpos[warp][j] + __popc(with & ((1u << lane) - 1u))] = (int32_t)v;
    }
  }
}

// The same lists in chain order (stencil order 1): thread per vertex, for the directions in
// which it heads a chain.  Every head walks its chain for the length (all lanes at once: the
// walks are chains of dependent loads), the block takes one range of list slots and one of
// chain slots per direction, and each head walks again to write its chain.  The order of
// the chains is immaterial.  *longest: the longest chain; beyond kMaxChain the walks stop, the
// lists are incomplete and the host has k_active_fill write them.
__global__ void __launch_bounds__(kFillThreads) k_chain_fill(
    LinkBits lb, const int32_t* nbr, int64_t m, int D,
    const int64_t* off, const int64_t* chain_off,
    unsigned long long* __restrict__ fill, unsigned long long* __restrict__ chain_fill,
    int32_t* __restrict__ act, uint2* __restrict__ chain, int* __restrict__ longest) {
  pdl_enter();
  __shared__ unsigned slen[kMaxD], scnt[kMaxD];  // this block's sums, then running positions
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = v < m;
  for (int j = threadIdx.x; j < D; j += blockDim.x) slen[j] = scnt[j] = 0;
  __syncthreads();
  auto heads = [&](int w) {
    return live ? lb.above[(int64_t)w * m + v] & ~lb.below[(int64_t)w * m + v] : 0u;
  };
  // length of the chain v heads along j, as far as it matters: a chain may run over 64000 / D
  // vertices, each a dependent load (n = 3400, d = 20 with a chain of 3000: 1930 us a build,
  // 460 with the limit)
  auto length = [&](int j) {
    const int32_t* above = nbr + ((int64_t)j * 2 + 1) * m;
    unsigned len = 1;
    for (int32_t x = above[v]; x >= 0 && len <= (unsigned)kMaxChain; x = above[x]) ++len;
    return len;
  };
  int most = 0;
  for (int w = 0; w * 32 < D; ++w)
    for (uint32_t x = heads(w); x; x &= x - 1) {
      const int j = w * 32 + __ffs(x) - 1;
      const unsigned len = length(j);
      most = max(most, (int)len);
      atomicAdd(&slen[j], len);
      atomicAdd(&scnt[j], 1u);
    }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0 && most > __ldcg(longest)) atomicMax(longest, most);
  __syncthreads();
  for (int j = threadIdx.x; j < D; j += blockDim.x) {
    if (scnt[j] == 0) continue;
    slen[j] = (unsigned)atomicAdd(&fill[j], (unsigned long long)slen[j]);
    scnt[j] = (unsigned)atomicAdd(&chain_fill[j], (unsigned long long)scnt[j]);
  }
  __syncthreads();
  for (int w = 0; w * 32 < D; ++w)
    for (uint32_t x = heads(w); x; x &= x - 1) {
      const int j = w * 32 + __ffs(x) - 1;
      const unsigned len = length(j);
      const int64_t at = off[j] + atomicAdd(&slen[j], len);
      const int64_t c = chain_off[j] + atomicAdd(&scnt[j], 1u);
      const int32_t* above = nbr + ((int64_t)j * 2 + 1) * m;
      int32_t y = (int32_t)v;
      for (unsigned q = 0; q < len; ++q) {
        act[at + q] = y;
        y = above[y];
      }
      chain[c] = make_uint2((uint32_t)at, (uint32_t)(at + len));
    }
}

// ---------------------------------------------------------------------------------
// 6. Splat lists.
// ---------------------------------------------------------------------------------
__global__ void k_splat_items(const uint32_t* sorted_entries,
                              const float* w,
                              int64_t nD, int D, int2* __restrict__ items) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nD) return;
  const uint32_t e = sorted_entries[p];
  items[p] = make_int2((int)(e / D), __float_as_int(w[e]));
}

// What a vertex with the incidences [b, e) counts for: segments, partial slots, a medium and a
// huge fix-up row (SEG_KINDS running counts).
enum { SEG_ALL = 0, SEG_SLOT, SEG_MED, SEG_HUGE, SEG_KINDS };
constexpr int kSegThreads = 512;  // vertices per block
__device__ __forceinline__ void seg_counts(int b, int e, uint32_t (&c)[SEG_KINDS]) {
  const uint32_t all = (uint32_t)((e - b + kSplatSeg - 1) / kSplatSeg);
  c[SEG_ALL] = all;
  c[SEG_SLOT] = all > 1 ? all : 0u;
  c[SEG_MED] = (all > 1 && all <= (uint32_t)kSplatMedSegs) ? 1u : 0u;
  c[SEG_HUGE] = all > (uint32_t)kSplatMedSegs ? 1u : 0u;
}

// Counts of each block of vertices, sums[kind][block], with a zero behind each row (its
// exclusive scan is the row's total).  k_seg_fill counts again rather than reading offsets per
// vertex: those are 32 bytes a vertex written and read for 4 read here (m = 10.5M: 390 us for
// the counts, their scans and the fill, 90 with the block sums alone).
__global__ void __launch_bounds__(kSegThreads) k_seg_sums(const int32_t* row_ptr,
                                                          int64_t m, uint32_t* __restrict__ sums) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * kSegThreads + threadIdx.x;
  uint32_t c[SEG_KINDS] = {};
  if (v < m) seg_counts(row_ptr[v], row_ptr[v + 1], c);
  __shared__ uint32_t sum[SEG_KINDS][kSegThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < SEG_KINDS; ++q) {
    const uint32_t t = __reduce_add_sync(0xffffffffu, c[q]);
    if (lane == 0) sum[q][warp] = t;
  }
  __syncthreads();
  if (warp < SEG_KINDS) {
    const uint32_t t = __reduce_add_sync(0xffffffffu, lane < kSegThreads / 32 ? sum[warp][lane] : 0u);
    uint32_t* row = sums + (int64_t)warp * (gridDim.x + 1);
    if (lane == 0) row[blockIdx.x] = t;
    if (lane == 0 && blockIdx.x == 0) row[gridDim.x] = 0;
  }
}

// From the scanned sums: write every segment and the fix-up row lists.  A vertex of up to
// 8 segments is written by its thread, a longer one by its warp (few dense vertices may hold
// nearly all segments: n = 760k, d = 2, five vertices, 284 us with one thread each).
__global__ void __launch_bounds__(kSegThreads)
    k_seg_fill(const int32_t* row_ptr, int64_t m, const uint32_t* sums,
               int4* __restrict__ seg, int4* __restrict__ med_rows, int4* __restrict__ huge_rows) {
  pdl_enter();
  const int64_t v = (int64_t)blockIdx.x * kSegThreads + threadIdx.x;
  const bool live = v < m;
  const int b = live ? row_ptr[v] : 0, e = live ? row_ptr[v + 1] : 0;
  uint32_t count[SEG_KINDS], at[SEG_KINDS] = {};
  seg_counts(b, e, count);
  const bool several = __syncthreads_or(count[SEG_ALL] > 1);
#pragma unroll
  for (int q = 0; q < SEG_KINDS; ++q)
    if (q == SEG_ALL || several)
      at[q] = sums[(int64_t)q * (gridDim.x + 1) + blockIdx.x] + block_exclusive_scan(count[q], nullptr);
  const int c = (int)count[SEG_ALL], s0 = (int)at[SEG_ALL];
  const int slot0 = c > 1 ? (int)at[SEG_SLOT] : -1;
  auto piece = [](int vertex, int first, int end, int slot, int j) {
    const int beg = first + j * kSplatSeg;
    return make_int4(vertex, beg, min(beg + kSplatSeg, end), slot >= 0 ? slot + j : -1);
  };
  if (c <= 8)
    for (int j = 0; j < c; ++j) seg[s0 + j] = piece((int)v, b, e, slot0, j);
  for (unsigned todo = __ballot_sync(0xffffffffu, c > 8); todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1;
    const int vv = __shfl_sync(0xffffffffu, (int)v, src), bb = __shfl_sync(0xffffffffu, b, src);
    const int ee = __shfl_sync(0xffffffffu, e, src), cc = __shfl_sync(0xffffffffu, c, src);
    const int ss = __shfl_sync(0xffffffffu, s0, src), sl = __shfl_sync(0xffffffffu, slot0, src);
    for (int j = (int)(threadIdx.x & 31); j < cc; j += 32) seg[ss + j] = piece(vv, bb, ee, sl, j);
  }
  if (count[SEG_MED]) med_rows[at[SEG_MED]] = make_int4((int)v, slot0, c, 0);
  if (count[SEG_HUGE]) huge_rows[at[SEG_HUGE]] = make_int4((int)v, slot0, c, 0);
}

// Within each window of kSegWindow consecutive segments, order the segments by length,
// longest first (ties keep their order), so that the thread groups of a warp walk lists
// of similar length and finish together.  Windows keep the vertex order of the lattice
// at large, so the gathers of concurrently running warps stay local.  The splat's result
// does not depend on the order in which segments are processed.  A counting sort: ranks by
// comparison with the whole window are 128 steps a segment (10.5M segments: 238 us).
constexpr int kSegWindow = 128;
__global__ void __launch_bounds__(kSegWindow) k_seg_window_sort(const int4* in,
                                                                int64_t nseg,
                                                                int4* __restrict__ out) {
  pdl_enter();
  constexpr int kWarps = kSegWindow / 32;
  __shared__ int count[kWarps][kSplatSeg];  // [warp][kSplatSeg - length], then positions
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int b = threadIdx.x; b < kWarps * kSplatSeg; b += kSegWindow) (&count[0][0])[b] = 0;
  const int64_t s = (int64_t)blockIdx.x * kSegWindow + threadIdx.x;
  const bool live = s < nseg;
  const int4 sg = live ? in[s] : make_int4(0, 0, 0, 0);
  const int bin = live ? kSplatSeg - (sg.z - sg.y) : kSplatSeg;  // lengths are 1 .. kSplatSeg
  __syncthreads();
  const unsigned peers = __match_any_sync(0xffffffffu, bin);
  const int before = __popc(peers & ((1u << lane) - 1u));
  if (live && before == 0) count[warp][bin] = __popc(peers);
  __syncthreads();
  if (warp == 0) {
    int run = 0;
    for (int b0 = 0; b0 < kSplatSeg; b0 += 32) {
      int c[kWarps], all = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) all += c[w] = b0 + lane < kSplatSeg ? count[w][b0 + lane] : 0;
      int inc = all;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      int at = run + inc - all;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        if (b0 + lane < kSplatSeg) count[w][b0 + lane] = at;
        at += c[w];
      }
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
  }
  __syncthreads();
  if (live) out[(int64_t)blockIdx.x * kSegWindow + count[warp][bin] + before] = sg;
}

__global__ void k_iota(uint32_t* __restrict__ out, int64_t count) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < count) out[p] = (uint32_t)p;
}

__global__ void k_row_ptr(const uint32_t* sorted_ids, int64_t nD, int64_t m,
                          int32_t* __restrict__ row_ptr) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p > nD) return;
  if (p == nD) {
    row_ptr[m] = (int32_t)nD;
    return;
  }
  const uint32_t v = sorted_ids[p];
  if (p == 0 || sorted_ids[p - 1] != v) row_ptr[v] = (int32_t)p;
}

// ---------------------------------------------------------------------------------
// Host orchestration.
// ---------------------------------------------------------------------------------
template <class T>
cudaError_t dalloc(T** p, size_t count, cudaStream_t st) {
  return dev_malloc((void**)p, std::max<size_t>(count, 1) * sizeof(T), st);
}

struct Temps {
  cudaStream_t st;
  std::vector<void*> ptrs;
  ~Temps() {
    for (void* p : ptrs) (void)cudaFreeAsync(p, st);
    clear_pending_error();
  }
  template <class T>
  cudaError_t get(T** p, size_t count) {
    cudaError_t e = dalloc(p, count, st);
    if (e == cudaSuccess) ptrs.push_back((void*)*p);
    return e;
  }
};

int bits_for(uint64_t v) {  // bits needed to hold values 0..v
  int b = 0;
  while (b < 64 && (v >> b) != 0) ++b;
  return b;
}

#define SGP_DISPATCH_D(D, KERNEL, GRID, BLOCK, ST, ...)                            \
  do {                                                                              \
    if ((D) <= 8) launch_pdl(KERNEL<8>, (GRID), (BLOCK), (ST), __VA_ARGS__);             \
    else if ((D) <= 16) launch_pdl(KERNEL<16>, (GRID), (BLOCK), (ST), __VA_ARGS__);      \
    else if ((D) <= 32) launch_pdl(KERNEL<32>, (GRID), (BLOCK), (ST), __VA_ARGS__);      \
    else if ((D) <= 64) launch_pdl(KERNEL<64>, (GRID), (BLOCK), (ST), __VA_ARGS__);      \
    else launch_pdl(KERNEL<128>, (GRID), (BLOCK), (ST), __VA_ARGS__);                    \
    note_launches(1);                                                               \
  } while (0)

#define SGP_CHECK(expr, what)                                  \
  do {                                                         \
    cudaError_t e_ = (expr);                                   \
    if (e_ != cudaSuccess) return cuda_status(e_, what);       \
  } while (0)

}  // namespace

// Upload the hash multipliers to the current device once (blocking, so that every stream
// of the process sees them before its first build kernel).
static sgp_status ensure_coord_mults() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_status(e, "cudaGetDevice");
  if (dev < 0 || dev >= 64) {
    set_error("sgp_lattice_build: device ordinal out of range");
    return SGP_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return SGP_OK;
  uint64_t table[kMaxD];
  for (int c = 0; c < kMaxD; ++c) table[c] = host_coord_mult(c);
  e = cudaMemcpyToSymbol(c_coord_mult, table, sizeof(table));
  if (e != cudaSuccess) return cuda_status(e, "uploading the hash multipliers");
  done[dev] = true;
  return SGP_OK;
}

sgp_status build_lattice(Lattice* L, const float* X, const float* ls) {
  cudaStream_t st = L->stream;
  {
    const sgp_status s0 = ensure_coord_mults();
    if (s0 != SGP_OK) return s0;
  }
  const int64_t n = L->n;
  const int d = L->d, D = L->D, r = L->r;
  const int64_t nD = n * D;
  Temps tmp{st, {}};

  // per-dimension factors of the elevation: scale / sqrt((j+1)(j+2)), scale = sqrt(d(d+1))/s
  const double scale = std::sqrt((double)(d * (d + 1))) / L->s;
  std::vector<double> hf(d);
  for (int j = 0; j < d; ++j) hf[j] = scale / std::sqrt((double)((j + 1) * (j + 2)));
  double* f = nullptr;
  SGP_CHECK(tmp.get(&f, d), "alloc f");
  SGP_CHECK(cudaMemcpyAsync(f, hf.data(), d * sizeof(double), cudaMemcpyHostToDevice, st),
            "copy f");

  int16_t* rem0 = nullptr;
  uint8_t* rank = nullptr;
  float* w_user = nullptr;
  int* qmm = nullptr;  // [2][D]: min, max of rem0 / D per coordinate
  SGP_CHECK(tmp.get(&rem0, nD), "alloc rem0");
  SGP_CHECK(tmp.get(&rank, nD), "alloc rank");
  SGP_CHECK(tmp.get(&w_user, nD), "alloc w");
  SGP_CHECK(tmp.get(&qmm, 2 * D), "alloc qmm");
  {
    std::vector<int> init(2 * D);
    for (int c = 0; c < D; ++c) {
      init[c] = 1 << 30;
      init[D + c] = -(1 << 30);
    }
    SGP_CHECK(cudaMemcpyAsync(qmm, init.data(), 2 * D * sizeof(int), cudaMemcpyHostToDevice, st),
              "copy qmm");
  }
  SGP_CHECK(cudaMemsetAsync(L->err, 0, sizeof(unsigned), st), "memset err");
  {
    const unsigned grid = (unsigned)ceil_div(n, kElevT);
    const int nan = L->fault == FAULT_NAN_INPUT ? 1 : 0;
    auto go = [&](auto kernel) {
      launch_pdl(kernel, grid, kElevT, st, X, ls, f, n, d, rem0, rank, w_user, qmm, qmm + D, L->err,
                 nan);
    };
    if (D <= 4) go(k_elevate_small<4>);
    else if (D <= 8) go(k_elevate_small<8>);
    else if (D <= 12) go(k_elevate_small<12>);
    else if (D <= 16) go(k_elevate_small<16>);
    else if (D <= 32) go(k_elevate<32>);
    else if (D <= 64) go(k_elevate<64>);
    else go(k_elevate<128>);
    note_launches(1);
    SGP_CHECK(cudaGetLastError(), "k_elevate");
  }
  unsigned herr = 0;
  std::vector<int> hq(2 * D);
  SGP_CHECK(cudaMemcpyAsync(hq.data(), qmm, 2 * D * sizeof(int), cudaMemcpyDeviceToHost, st),
            "read qmm");
  SGP_CHECK(cudaMemcpyAsync(&herr, L->err, sizeof(unsigned), cudaMemcpyDeviceToHost, st),
            "read err");
  SGP_CHECK(cudaStreamSynchronize(st), "sync elevate");
  if (herr & ERRBIT_NONFINITE) {
    set_error("sgp_lattice_build: X holds NaN/Inf or a lengthscale is not a finite positive");
    return SGP_ERR_NONFINITE;
  }
  if (herr & ERRBIT_RANGE) {
    set_error("sgp_lattice_build: a lattice coordinate exceeds the int16 key range "
              "(lengthscales too small for the spread of X)");
    return SGP_ERR_RANGE;
  }

  // sort buffers, used in turn for the points, the vertex hashes and the splat lists
  uint32_t *ka, *va, *kb, *vb, *rt;
  SGP_CHECK(tmp.get(&ka, nD), "alloc sort");
  SGP_CHECK(tmp.get(&va, nD), "alloc sort");
  SGP_CHECK(tmp.get(&kb, nD), "alloc sort");
  SGP_CHECK(tmp.get(&vb, nD), "alloc sort");
  SGP_CHECK(tmp.get(&rt, radix_temp_elems(nD)), "alloc sort");

  // 2. locality order
  CellPack pk{};
  {
    int used = 0;
    for (int c = 0; c < d && c < kMaxD; ++c) {
      const int b = bits_for((uint64_t)(hq[D + c] - hq[c]));
      if (used + b > 32) break;
      pk.ncoord = c + 1;
      pk.qmin[c] = hq[c];
      used += b;
      pk.shift[c] = b > 0 ? 32 - used : 0;  // a single-valued coordinate packs to 0
    }
    launch_pdl(k_point_key, (unsigned)ceil_div(n, 256), 256, st, rem0, n, D, pk, ka, va);
    note_launches(1);
    // the packed cell occupies the top `used` bits; bits below are zero
    const bool in_alt = radix_sort_pairs(ka, va, kb, vb, n, (32 - used) & ~7, 32, rt, st);
    SGP_CHECK(dalloc(&L->perm, n, st), "alloc perm");
    SGP_CHECK(cudaMemcpyAsync(L->perm, in_alt ? vb : va, n * sizeof(int32_t),
                              cudaMemcpyDeviceToDevice, st),
              "copy perm");
    L->bytes += n * sizeof(int32_t);
  }

  // 3. hash insert
  uint64_t cap = 1024;
  if (L->fault != FAULT_HASH_FULL)  // SGP_FAULT=hash_full keeps the 1024-slot table
    while (cap < (uint64_t)(2 * nD)) cap <<= 1;
  const uint64_t mask = cap - 1;
  unsigned long long* table = nullptr;
  int32_t* entry_slot = nullptr;
  SGP_CHECK(tmp.get(&table, cap), "alloc hash table");
  SGP_CHECK(tmp.get(&entry_slot, nD), "alloc entry slots");
  SGP_CHECK(cudaMemsetAsync(table, 0xff, cap * sizeof(unsigned long long), st), "memset table");
  SGP_DISPATCH_D(D, k_insert, (unsigned)ceil_div(nD, 256), 256, st, L->perm, rem0, rank, nD, d,
                 table, mask, entry_slot, ka, va, L->err);  // ka, va: free until the sorts below
  SGP_CHECK(cudaGetLastError(), "k_insert");

  // 4. numbering
  uint32_t *flags, *scan_tmp, *total;
  SGP_CHECK(tmp.get(&flags, nD), "alloc flags");
  SGP_CHECK(tmp.get(&scan_tmp, scan_temp_elems(nD)), "alloc scan");
  SGP_CHECK(tmp.get(&total, 1), "alloc total");
  launch_pdl(k_owner_flags, (unsigned)ceil_div(nD, 256), 256, st, entry_slot, table, nD, flags);
  note_launches(1);
  exclusive_scan_u32(flags, nD, total, scan_tmp, st);
  uint32_t hm = 0;
  SGP_CHECK(cudaMemcpyAsync(&hm, total, sizeof(uint32_t), cudaMemcpyDeviceToHost, st), "read m");
  SGP_CHECK(cudaMemcpyAsync(&herr, L->err, sizeof(unsigned), cudaMemcpyDeviceToHost, st),
            "read err");
  SGP_CHECK(cudaStreamSynchronize(st), "sync insert");
  if (herr & ERRBIT_HASH_FULL) {
    set_error("sgp_lattice_build: vertex hash table full");
    return SGP_ERR_HASH_FULL;
  }
  const int64_t m = hm;
  L->m = m;
  int32_t* slot_id = nullptr;
  SGP_CHECK(tmp.get(&slot_id, cap), "alloc slot ids");
  SGP_CHECK(dalloc(&L->keys, m * D, st), "alloc keys");
  L->bytes += m * D * sizeof(int16_t);
  uint64_t* vhash = nullptr;
  SGP_CHECK(tmp.get(&vhash, m), "alloc vertex hashes");
  uint32_t* owner = nullptr;  // [m] first entry of each vertex
  SGP_CHECK(tmp.get(&owner, m), "alloc owners");
  launch_pdl(k_assign_ids, (unsigned)ceil_div(nD, kAssignThreads), kAssignThreads, st, flags, total,
             entry_slot, L->perm, rem0, rank, ka, va, nD, d, slot_id, L->keys, vhash, owner);
  note_launches(1);
  SGP_CHECK(dalloc(&L->idx, nD, st), "alloc idx");
  SGP_CHECK(dalloc(&L->w, nD, st), "alloc w");
  SGP_CHECK(dalloc(&L->rank, nD, st), "alloc rank");
  L->bytes += nD * (sizeof(int32_t) + sizeof(float) + sizeof(uint8_t));
  launch_pdl(k_entry_ids, (unsigned)ceil_div(nD, 256), 256, st, entry_slot, slot_id, L->perm, w_user,
                                                          rank, nD, D, L->idx, L->w, L->rank);
  note_launches(1);
  SGP_CHECK(cudaGetLastError(), "numbering");

  // 5. neighbour table
  const size_t nbr_count = (size_t)D * r * 2 * m;
  SGP_CHECK(dalloc(&L->nbr, nbr_count, st), "alloc nbr");
  L->bytes += nbr_count * sizeof(int32_t);
  // [D] vertices per direction, [D] list fill, pairs (v, v + u_j), [D] chains, [D] chain fill,
  // longest chain
  unsigned long long* counts = nullptr;
  SGP_CHECK(tmp.get(&counts, 4 * D + 2), "alloc counts");
  SGP_CHECK(cudaMemsetAsync(counts, 0, (4 * D + 2) * sizeof(unsigned long long), st), "clear counts");
  LinkBits lb{nullptr, nullptr};
  if (m > 0) {
    // few vertices belong to several simplices: the lattice is probably sparse, so record the
    // links while they are found (two atomics a link; sparse ones have few beyond their own
    // simplex's).  Otherwise k_link_bits reads them off the table if it turns out sparse.
    if (r == 1 && m >= nD / 4) {
      const int64_t words = (int64_t)((D + 31) / 32) * m;
      SGP_CHECK(tmp.get(&lb.above, words), "alloc link bits");
      SGP_CHECK(tmp.get(&lb.below, words), "alloc link bits");
    }
    // one to two vertices per bucket on average
    const int bits = std::min(31, std::max(1, bits_for((uint64_t)(m - 1)) - 1));
    const int64_t buckets = (int64_t)1 << bits;
    uint32_t *low = nullptr, *high = nullptr, *start = nullptr;
    uint8_t *up = nullptr, *up_sorted = nullptr;
    SGP_CHECK(tmp.get(&low, m), "alloc sorted hashes");
    SGP_CHECK(tmp.get(&high, m), "alloc sorted hashes");
    SGP_CHECK(tmp.get(&up, m), "alloc links");
    SGP_CHECK(tmp.get(&up_sorted, m), "alloc links");
    SGP_CHECK(tmp.get(&start, buckets + 1), "alloc hash buckets");
    const unsigned grid = (unsigned)ceil_div(m, 256);
    launch_pdl(k_nbr_init, grid, 256, st, owner, L->idx, L->rank, m, d, r, L->nbr, up, lb);
    launch_pdl(k_nbr_close, grid, 256, st, owner, L->idx, L->rank, m, d, r, L->nbr,
               lb);
    launch_pdl(k_hash_keys, grid, 256, st, vhash, m, 64 - bits, ka, va);
    const bool in_alt = radix_sort_pairs(ka, va, kb, vb, m, 0, bits, rt, st);
    const uint32_t* ord = in_alt ? vb : va;
    launch_pdl(k_hash_index, grid, 256, st, in_alt ? kb : ka, ord, vhash, up, m, buckets,
               low, high, up_sorted, start);
    // sum_c A_c over the D coordinates, as the kernels compute A_c
    uint64_t sum_A = 0;
    for (int c = 0; c < D; ++c) sum_A += host_coord_mult(c);
    launch_pdl(D <= 16 ? k_neighbours<false> : k_neighbours<true>, grid, 256, st, L->keys, low, high,
               up_sorted, ord, start, 64 - bits, m, d, r, sum_A, L->nbr, counts + 2 * D, lb);
    note_launches(5);
  }
  SGP_CHECK(cudaGetLastError(), "k_neighbours");

  // 6. splat lists: (vertex id, entry) sorted by id, stable in entry order
  {
    SGP_CHECK(cudaMemcpyAsync(ka, L->idx, nD * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st),
              "copy ids");
    launch_pdl(k_iota, (unsigned)ceil_div(nD, 256), 256, st, va, nD);
    note_launches(1);
    const int bits = std::max(1, bits_for((uint64_t)(m > 0 ? m - 1 : 0)));
    const bool in_alt = radix_sort_pairs(ka, va, kb, vb, nD, 0, bits, rt, st);
    const uint32_t* sorted_ids = in_alt ? kb : ka;
    const uint32_t* sorted_entries = in_alt ? vb : va;
    SGP_CHECK(dalloc(&L->items, nD, st), "alloc items");
    SGP_CHECK(dalloc(&L->row_ptr, m + 1, st), "alloc row_ptr");
    L->bytes += nD * sizeof(int2) + (m + 1) * sizeof(int32_t);
    launch_pdl(k_splat_items, (unsigned)ceil_div(nD, 256), 256, st, sorted_entries, L->w, nD, D,
                                                              L->items);
    note_launches(1);
    launch_pdl(k_row_ptr, (unsigned)ceil_div(nD + 1, 256), 256, st, sorted_ids, nD, m, L->row_ptr);
    note_launches(1);
    SGP_CHECK(cudaGetLastError(), "splat lists");
  }

  // 7. splat segments (load balance)
  unsigned long long pairs = 0;  // (v, v + u_j) pairs: at least as many active vertices
  {
    const int64_t blocks = std::max<int64_t>(1, ceil_div(m, (int64_t)kSegThreads));
    uint32_t* sums;
    SGP_CHECK(tmp.get(&sums, SEG_KINDS * (blocks + 1)), "alloc seg");
    launch_pdl(k_seg_sums, (unsigned)blocks, kSegThreads, st, L->row_ptr, m, sums);
    note_launches(1);
    exclusive_scan_rows_u32(sums, SEG_KINDS, blocks + 1, st);
    uint32_t ht[SEG_KINDS];
    SGP_CHECK(cudaMemcpy2DAsync(ht, sizeof(uint32_t), sums + blocks, (blocks + 1) * sizeof(uint32_t),
                                sizeof(uint32_t), SEG_KINDS, cudaMemcpyDeviceToHost, st),
              "read seg");
    SGP_CHECK(cudaMemcpyAsync(&pairs, counts + 2 * D, sizeof(pairs), cudaMemcpyDeviceToHost, st),
              "read pairs");
    SGP_CHECK(cudaStreamSynchronize(st), "sync seg");
    L->nseg = ht[SEG_ALL];
    L->nslots = ht[SEG_SLOT];
    L->nmed = ht[SEG_MED];
    L->nhuge = ht[SEG_HUGE];
    SGP_CHECK(dalloc(&L->seg, L->nseg, st), "alloc seg");
    SGP_CHECK(dalloc(&L->med_rows, L->nmed, st), "alloc seg");
    SGP_CHECK(dalloc(&L->huge_rows, L->nhuge, st), "alloc seg");
    L->bytes += (L->nseg + L->nmed + L->nhuge) * sizeof(int4);
    int4* seg_unsorted = nullptr;
    SGP_CHECK(tmp.get(&seg_unsorted, std::max<int64_t>(L->nseg, 1)), "alloc seg");
    launch_pdl(k_seg_fill, (unsigned)blocks, kSegThreads, st, L->row_ptr, m, sums, seg_unsorted,
               L->med_rows, L->huge_rows);
    if (L->nseg > 0)
      launch_pdl(k_seg_window_sort, (unsigned)ceil_div(L->nseg, kSegWindow), kSegWindow, st, 
          seg_unsorted, L->nseg, L->seg);
    note_launches(2);
    SGP_CHECK(cudaGetLastError(), "splat segments");
  }
  // 8. direction lists of a sparse lattice
  if ((double)pairs <= kSparseFrac * (double)D * (double)m) {
    const unsigned vgrid = (unsigned)std::max<int64_t>(1, ceil_div(m, 256));
    if (!lb.above) {
      const int64_t words = (int64_t)((D + 31) / 32) * m;
      SGP_CHECK(tmp.get(&lb.above, words), "alloc link bits");
      SGP_CHECK(tmp.get(&lb.below, words), "alloc link bits");
      launch_pdl(k_link_bits, vgrid, 256, st, L->nbr, m, D, r, lb);
      note_launches(1);
    }
    launch_pdl(k_link_counts, std::min(vgrid, 8u * 152u), 256, st, lb, m, D, counts,
               counts + 2 * D + 1);
    note_launches(1);
    std::vector<unsigned long long> hc(4 * D + 2);
    SGP_CHECK(cudaMemcpyAsync(hc.data(), counts, hc.size() * sizeof(unsigned long long),
                              cudaMemcpyDeviceToHost, st),
              "read counts");
    SGP_CHECK(cudaStreamSynchronize(st), "sync counts");
    int64_t total = 0, largest = 0;
    for (int j = 0; j < D; ++j) {
      total += (int64_t)hc[j];
      largest = std::max<int64_t>(largest, (int64_t)hc[j]);
    }
    if (m > 0 && (double)total <= kSparseFrac * (double)D * (double)m) {
      L->sparse = true;
      L->act_max = largest;
      L->act_off.assign(D + 1, 0);
      for (int j = 0; j < D; ++j) L->act_off[j + 1] = L->act_off[j] + (int64_t)hc[j];
      SGP_CHECK(dalloc(&L->act, std::max<int64_t>(total, 1), st), "alloc direction lists");
      SGP_CHECK(dalloc(&L->epoch, m, st), "alloc epochs");
      L->bytes += (size_t)total * sizeof(int32_t) + (size_t)m * sizeof(int32_t);
      SGP_CHECK(dalloc(&L->act_off_dev, 2 * (D + 1), st), "alloc list offsets");
      std::vector<int64_t> offsets(L->act_off);  // then the chains' offsets
      offsets.resize(2 * (D + 1), 0);
      for (int j = 0; j < D; ++j) offsets[D + 2 + j] = offsets[D + 1 + j] + (int64_t)hc[2 * D + 1 + j];
      SGP_CHECK(cudaMemcpyAsync(L->act_off_dev, offsets.data(), offsets.size() * sizeof(int64_t),
                                cudaMemcpyHostToDevice, st),
                "copy list offsets");
      const unsigned grid = (unsigned)ceil_div(m, kFillThreads);
      if (r == 1 && total <= (int64_t)0xffffffff) {  // chains hold 32-bit positions in the lists
        L->chain_off.assign(offsets.begin() + D + 1, offsets.end());
        const int64_t chains = L->chain_off.back();
        SGP_CHECK(dalloc(&L->chain, std::max<int64_t>(chains, 1), st), "alloc chains");
        L->bytes += (size_t)chains * sizeof(uint2);
        int* longest = reinterpret_cast<int*>(counts + 4 * D + 1);
        launch_pdl(k_chain_fill, grid, kFillThreads, st, lb, L->nbr, m, D, L->act_off_dev,
                   L->act_off_dev + D + 1, counts + D, counts + 3 * D + 1, L->act, L->chain, longest);
        SGP_CHECK(cudaMemcpyAsync(&L->chain_max, longest, sizeof(int), cudaMemcpyDeviceToHost, st),
                  "read chains");
      } else {
        launch_pdl(k_active_fill, grid, kFillThreads, st, lb, m, D, L->act_off_dev, counts + D, L->act);
      }
      note_launches(1);
      // powers of the symmetric blur's centre tap g_0 (stored rows are rescaled lazily)
      std::vector<float> pw(2 * D + 1);
      for (int q = 0; q <= 2 * D; ++q) pw[q] = (float)std::pow(L->half[0], (double)q);
      SGP_CHECK(dalloc(&L->g0pow, 2 * D + 1, st), "alloc tap powers");
      SGP_CHECK(cudaMemcpyAsync(L->g0pow, pw.data(), pw.size() * sizeof(float),
                                cudaMemcpyHostToDevice, st),
                "copy tap powers");
      SGP_CHECK(cudaGetLastError(), "direction lists");
    }
  }
  SGP_CHECK(cudaStreamSynchronize(st), "sync build");
  if (L->chain_max > kMaxChain) {  // blurred through the direction lists, without chains
    SGP_CHECK(cudaFreeAsync(L->chain, st), "free chains");
    L->chain = nullptr;
    L->bytes -= (size_t)L->chain_off.back() * sizeof(uint2);
    SGP_CHECK(cudaMemsetAsync(counts + D, 0, D * sizeof(unsigned long long), st), "clear list fill");
    launch_pdl(k_active_fill, (unsigned)ceil_div(m, kFillThreads), kFillThreads, st, lb, m, D,
               L->act_off_dev, counts + D, L->act);
    note_launches(1);
    SGP_CHECK(cudaGetLastError(), "direction lists");
    SGP_CHECK(cudaStreamSynchronize(st), "sync direction lists");
  }
  return SGP_OK;
}

}  // namespace sgp
