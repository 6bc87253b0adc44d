// The lattice MVM  out = alpha * W B W^T V + beta * V  (Sec. 3.2, Eq. ski_to_bf).
//
//   k_splat  W^T: each lattice vertex gathers w * V[point] over its list of incident
//            (point, weight) pairs, cut into segments of at most kSplatSeg items; long
//            lists are finished by an ordered fix-up.  Gathers only: deterministic.
//   k_blur   one lattice direction u_j: out[v] = c_0 in[v] + sum_t c_t (in[v - t u_j] +
//            in[v + t u_j]) with absent neighbours contributing 0 (Sec. 3.2 "Blur"); the
//            neighbour ids come from the table built with the lattice.
//   k_slice  W: each point interpolates its d+1 vertices with its barycentric weights,
//            fused with the alpha/beta epilogue.
//
// All of them are bound by memory traffic.  The caller's vectors are fp32 [rows][k]
// row-major.  Lattice values are stored as S = float or __nv_bfloat16 (SGP_VALUES_BF16:
// half the bytes of the dominant blur traffic); every sum is accumulated in fp32.
//
// Inside the operator a row has kp >= k columns (padded_cols): one or two columns as they
// are, more rounded up to a multiple of 4 with zero columns, so that every row is float4
// groups whatever k and however the caller's buffers are aligned; a thread owns 4 (2, 1)
// consecutive columns of a row, the pipelined blur 8.  At n = 50k, d = 8, k = 9 a product
// with 9 scalar columns took 100 us, with 12 padded ones 77.5 us (launches alike).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include <cuda_bf16.h>

#include "sgp_internal.cuh"
#include "values.cuh"

namespace sgp {
namespace {

constexpr int kThreads = 256;

// ---- splat ---------------------------------------------------------------------------
// Incidences and vertex rows are gathered kChunk at a time: a thread first loads the
// (point, weight) pairs or (vertex id, weight) pairs of a chunk, then issues all of the
// chunk's row loads, then accumulates in order.  The row loads of a chunk are independent,
// so kChunk of them are in flight per thread instead of one dependent pair at a time; the
// sums keep the incidence order, so results do not change with the chunking.
constexpr int kChunk = 8;

// One thread-group of G = k / VEC threads per segment of at most kSplatSeg incidences;
// blockDim.x is a multiple of G.  scale: a power of two on the vertices' values (ChainRange).
template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_splat(int64_t nseg, int G, int k,
                                                    const int4* __restrict__ seg,
                                                    const int2* __restrict__ items,
                                                    const float* V, float scale,
                                                    S* __restrict__ lat,
                                                    float* __restrict__ partial) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t s = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (s >= nseg) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  const int4 sg = __ldg(seg + s);
  typename Vt::T acc = Vt::zero();
  for (int p0 = sg.y; p0 < sg.z; p0 += kChunk) {
    int2 it[kChunk];
#pragma unroll
    for (int j = 0; j < kChunk; ++j)
      it[j] = p0 + j < sg.z ? __ldg(items + p0 + j) : make_int2(-1, 0);
    typename Vt::T row[kChunk];
#pragma unroll
    for (int j = 0; j < kChunk; ++j)
      row[j] = it[j].x >= 0 ? Vt::ld(V + (int64_t)it[j].x * k + col) : Vt::zero();
#pragma unroll
    for (int j = 0; j < kChunk; ++j)
      if (it[j].x >= 0) acc = Vt::fma(__int_as_float(it[j].y), row[j], acc);
  }
  if (sg.w < 0) Vt::sts(lat + (int64_t)sg.x * k + col, Vt::scale(scale, acc));
  else Vt::st(partial + (int64_t)sg.w * k + col, acc);
}

// Fix-up of the vertices with several segments, in one launch.  Blocks below `nhuge`: one
// vertex of more than kSplatMedSegs segments each, in `groups` (a power of two, groups G <=
// kThreads, or twice that where two products share the rows) strided partial sums and a fixed-shape shared-memory tree over them (the result
// depends on `groups` only, not on how the threads share the work).  The blocks after them:
// one thread-group per vertex of 2..kSplatMedSegs segments, summed in order.
template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_splat_fix(int nhuge, int64_t nmed, int groups, int G,
                                                        int k, const int4* __restrict__ huge_rows,
                                                        const int4* __restrict__ med_rows,
                                                        const float* partial,
                                                        float scale, S* __restrict__ lat) {
  pdl_enter();
  using Vt = Vec<VEC>;
  __shared__ typename Vt::T red[2 * kThreads];
  if ((int)blockIdx.x >= nhuge) {
    const int rows = kThreads / G;
    const int64_t q = (int64_t)((int)blockIdx.x - nhuge) * rows + threadIdx.x / G;
    if (q >= nmed || (int)threadIdx.x >= rows * G) return;
    const int col = (int)(threadIdx.x % G) * VEC;
    const int4 rw = med_rows[q];
    const float* base = partial + (int64_t)rw.y * k + col;
    typename Vt::T x[kSplatMedSegs], acc = Vt::zero();
#pragma unroll
    for (int j = 0; j < kSplatMedSegs; ++j) x[j] = j < rw.z ? Vt::ld(base + (int64_t)j * k) : Vt::zero();
#pragma unroll
    for (int j = 0; j < kSplatMedSegs; ++j)
      if (j < rw.z) acc = Vt::add(acc, x[j]);
    Vt::sts(lat + (int64_t)rw.x * k + col, Vt::scale(scale, acc));
    return;
  }
  const int4 rw = huge_rows[blockIdx.x];
  for (int q = threadIdx.x; q < groups * G; q += blockDim.x) {
    const float* base = partial + (int64_t)rw.y * k + (q % G) * VEC;
    typename Vt::T acc = Vt::zero();
    int j = q / G;
    for (; j + 15 * groups < rw.z; j += 16 * groups) {  // 16 loads in flight, summed in order
      typename Vt::T x[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) x[e] = Vt::ld(base + (int64_t)(j + e * groups) * k);
#pragma unroll
      for (int e = 0; e < 16; ++e) acc = Vt::add(acc, x[e]);
    }
    for (; j < rw.z; j += groups) acc = Vt::add(acc, Vt::ld(base + (int64_t)j * k));
    red[q] = acc;
  }
  __syncthreads();
  for (int half = groups / 2; half >= 1; half /= 2) {
    for (int q = threadIdx.x; q < half * G; q += blockDim.x)
      red[q] = Vt::add(red[q], red[q + half * G]);
    __syncthreads();
  }
  for (int q = threadIdx.x; q < G; q += blockDim.x)
    Vt::sts(lat + (int64_t)rw.x * k + q * VEC, Vt::scale(scale, red[q]));
}

// ---- blur ----------------------------------------------------------------------------
// One value per thread (any k: the fixed work area's unpadded rows).
template <class S>
__global__ void __launch_bounds__(kThreads) k_blur(int64_t m, int k, int r, Taps tp,
                                                   const int32_t* __restrict__ nbr,
                                                   const S* in, S* __restrict__ out) {
  pdl_enter();
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t v = gid / k;
  if (v >= m) return;
  const int col = (int)(gid - v * k);
  float acc = tp.t[0] * Store<S>::ld1(in + v * k + col);
  for (int t = 1; t <= r; ++t) {
    const int a = nbr[(int64_t)(2 * (t - 1)) * m + v];
    const int c = nbr[(int64_t)(2 * (t - 1) + 1) * m + v];
    float s = 0.f;
    if (a >= 0) s += Store<S>::ld1(in + (int64_t)a * k + col);
    if (c >= 0) s += Store<S>::ld1(in + (int64_t)c * k + col);
    acc = fmaf(tp.t[t], s, acc);
  }
  Store<S>::st1(out + v * k + col, acc);
}

// Rows of k = VEC CH G values.  Each thread owns VEC CH consecutive columns of U rows (R =
// stencil order): it issues all id loads, then all own and neighbour row loads, then the
// arithmetic, so 3 U row loads per order are in flight at once.  A block covers U
// consecutive runs of kThreads / G rows (coalesced per run, local per block).
template <int VEC, int CH, int U, int R, class S>
__global__ void __launch_bounds__(kThreads) k_blur_rows(int64_t m, int G, int k, Taps tp,
                                                        const int32_t* __restrict__ nbr,
                                                        const S* in,
                                                        S* __restrict__ out) {
  static_assert(CH == 1 || (CH == 2 && VEC == 4), "one group of columns per thread, or 2 x 4");
  using Vt = Vec<VEC>;
  using T = typename Vt::T;
  const int rows_per_run = blockDim.x / G;
  const int col = (int)(threadIdx.x % G) * (VEC * CH);
  int64_t v[U];
  int ia[U][R], ic[U][R];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    v[u] = ((int64_t)blockIdx.x * U + u) * rows_per_run + threadIdx.x / G;
#pragma unroll
    for (int t = 0; t < R; ++t) {
      ia[u][t] = v[u] < m ? __ldg(nbr + (int64_t)(2 * t) * m + v[u]) : -1;
      ic[u][t] = v[u] < m ? __ldg(nbr + (int64_t)(2 * t + 1) * m + v[u]) : -1;
    }
  }
  pdl_enter();  // the ids do not change: loaded before the wait
  auto load = [&](int64_t row, T* x) {
    if constexpr (CH == 2) Store<S>::ld8(in + row * k + col, x[0], x[1]);
    else x[0] = Vt::lds(in + row * k + col);
  };
  T own[U][CH], sa[U][R][CH], sc[U][R][CH];
#pragma unroll
  for (int u = 0; u < U; ++u) {
#pragma unroll
    for (int c = 0; c < CH; ++c) own[u][c] = Vt::zero();
    if (v[u] < m) load(v[u], own[u]);
#pragma unroll
    for (int t = 0; t < R; ++t) {
#pragma unroll
      for (int c = 0; c < CH; ++c) sa[u][t][c] = sc[u][t][c] = Vt::zero();
      if (ia[u][t] >= 0) load(ia[u][t], sa[u][t]);
      if (ic[u][t] >= 0) load(ic[u][t], sc[u][t]);
    }
  }
  pdl_leave();
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (v[u] >= m) continue;
    T acc[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      acc[c] = Vt::scale(tp.t[0], own[u][c]);
#pragma unroll
      for (int t = 0; t < R; ++t)
        acc[c] = Vt::fma(tp.t[t + 1], Vt::add(sa[u][t][c], sc[u][t][c]), acc[c]);
    }
    if constexpr (CH == 2) Store<S>::st8(out + v[u] * k + col, acc[0], acc[1]);
    else Vt::sts(out + v[u] * k + col, acc[0]);
  }
}

// Stencil order 1 with eight columns per thread, persistent and software-pipelined: each
// thread group walks rows v, v + stride, ...; while it combines row v, the rows of v +
// stride (own and both neighbours) and the neighbour ids of v + 2 stride are in flight, so
// the memory system sees a steady stream instead of one burst per block.  Same arithmetic
// as k_blur_rows (bitwise equal results).
//
// RO: the rows through the read-only path, not launched as a dependent (the rule at launch_pdl).
// fp32 values of kReadOnlyBytes or more blur faster so, although a launch costs 2.5 us more:
// symmetric products, read-only / ordinary loads: m = 2.24M, k = 64 (547 MiB) 6.34 / 7.14 ms, k =
// 48 (410) 5.01 / 5.11, k = 40 (342) 4.27 / 4.29, k = 32 (273) 3.25 / 3.20, k = 16 (137) 1.79 / 1.72;
// m = 440k, k = 256 (429) 5.49 / 5.93, k = 192 (322) 4.08 / 4.10.  BF16 ones do not (m = 2.24M, k =
// 192, 820 MiB: 13.12 / 13.11), nor do rows of k_blur_rows.
constexpr size_t kReadOnlyBytes = (size_t)350 << 20;
template <bool RO, class S>
__global__ void __launch_bounds__(kThreads) k_blur_pipe(int64_t m, int G, int k, Taps tp,
                                                        const int32_t* __restrict__ nbr,
                                                        const S* in,
                                                        S* __restrict__ out) {
  pdl_enter();
  const int rows_per_block = blockDim.x / G;
  const int col = (int)(threadIdx.x % G) * 8;
  const int64_t stride = (int64_t)gridDim.x * rows_per_block;
  int64_t row = (int64_t)blockIdx.x * rows_per_block + threadIdx.x / G;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto ids = [&](int64_t v, int& a, int& c) {  // neighbour ids of v - u_j, v + u_j
    if (v < m) {
      a = __ldg(nbr + v);
      c = __ldg(nbr + m + v);
    } else {
      a = c = -1;
    }
  };
  auto load = [&](int64_t v, int a, int c, float4 (&x)[3][2]) {  // own, minus, plus rows
    x[0][0] = x[0][1] = x[1][0] = x[1][1] = x[2][0] = x[2][1] = zero;
    auto row = [&](int64_t u, float4 (&y)[2]) {
      if constexpr (RO) Store<S>::ro8(in + u * k + col, y[0], y[1]);
      else Store<S>::ld8(in + u * k + col, y[0], y[1]);
    };
    if (v < m) row(v, x[0]);
    if (a >= 0) row(a, x[1]);
    if (c >= 0) row(c, x[2]);
  };
  int a0, c0, a1, c1;
  ids(row, a0, c0);
  ids(row + stride, a1, c1);
  float4 cur[3][2];
  load(row, a0, c0, cur);
  while (row < m) {
    const int64_t nrow = row + stride;
    int a2, c2;
    ids(nrow + stride, a2, c2);
    float4 nxt[3][2];
    load(nrow, a1, c1, nxt);
    float4 acc[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      acc[h] = make_float4(tp.t[0] * cur[0][h].x, tp.t[0] * cur[0][h].y, tp.t[0] * cur[0][h].z,
                           tp.t[0] * cur[0][h].w);
      acc[h].x = fmaf(tp.t[1], cur[1][h].x + cur[2][h].x, acc[h].x);
      acc[h].y = fmaf(tp.t[1], cur[1][h].y + cur[2][h].y, acc[h].y);
      acc[h].z = fmaf(tp.t[1], cur[1][h].z + cur[2][h].z, acc[h].z);
      acc[h].w = fmaf(tp.t[1], cur[1][h].w + cur[2][h].w, acc[h].w);
    }
    Store<S>::st8(out + row * k + col, acc[0], acc[1]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      cur[q][0] = nxt[q][0];
      cur[q][1] = nxt[q][1];
    }
    a1 = a2;
    c1 = c2;
    row = nrow;
  }
}

// Blocks of k_blur_pipe<RO, S> the device keeps resident (one wave), cached per device.
template <bool RO, class S>
int blur_pipe_blocks() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  int b = cache[dev].load();
  if (b > 0) return b;
  int per_sm = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_blur_pipe<RO, S>, kThreads, 0) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    clear_pending_error();
    return 152;
  }
  b = std::max(1, per_sm) * std::max(1, sms);
  cache[dev].store(b);
  return b;
}

// ---- blur of small lattices ---------------------------------------------------------------
// All passes in one launch: a cluster of thread blocks holds VEC columns of every vertex in
// its shared memory (two buffers of `rows` rows a block, vertex v in block v / rows), a
// neighbour's value is read from whichever block holds it (distributed shared memory), and a
// cluster barrier separates the passes; the column groups are independent clusters.  A pass
// of its own launch waits for a grid to drain, for the next to start, for the neighbour ids
// and then for the rows; here the ids of the next pass are loaded before the barrier and
// the rows come from shared memory.  Same arithmetic as k_blur_rows, values rounded to S after
// every pass alike (bitwise equal results).
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive;" ::: "memory");
  asm volatile("barrier.cluster.wait;" ::: "memory");
}
// VEC values of type S at shared-memory address `local` of block `rank` of the cluster.
template <int VEC, class S>
__device__ __forceinline__ typename Vec<VEC>::T ld_cluster(uint32_t local, uint32_t rank) {
  uint32_t at;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(local), "r"(rank));
  constexpr int kBytes = VEC * (int)sizeof(S);
  alignas(16) uint32_t w[4];
  if constexpr (kBytes == 16)
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(at) : "memory");
  else if constexpr (kBytes == 8)
    asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(at) : "memory");
  else if constexpr (kBytes == 4)
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(w[0]) : "r"(at) : "memory");
  else {
    uint16_t h;
    asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(h) : "r"(at) : "memory");
    w[0] = h;
  }
  return Vec<VEC>::lds(reinterpret_cast<const S*>(w));
}

struct ClusterBlur {
  int m, k, D, passes, blur, rows;  // rows: vertices per block
  Taps tp;
  const int32_t* nbr;
};

// One thread per vertex (rows <= blockDim.x).
template <int VEC, int R, class S>
__global__ void __launch_bounds__(1024) k_blur_cluster(ClusterBlur q, S* __restrict__ lat) {
  using Vt = Vec<VEC>;
  using T = typename Vt::T;
  __shared__ __align__(16) S buf[2][1024 * VEC];
  const uint32_t rank = cluster_rank();
  const int v0 = (int)rank * q.rows;
  const int l = (int)threadIdx.x, col = (int)blockIdx.y * VEC;
  const bool live = l < q.rows && v0 + l < q.m;  // the last blocks may be short or empty
  S* own = lat + (int64_t)(v0 + l) * q.k + col;
  int ids[2 * R];
  auto load_ids = [&](int t) {
    const int j = q.blur == SGP_BLUR_SEQUENTIAL ? t
                  : q.blur == SGP_BLUR_TRANSPOSE ? q.D - 1 - t
                                                 : (t < q.D ? t : 2 * q.D - 1 - t);
    const int32_t* plane = q.nbr + (int64_t)j * R * 2 * q.m + v0 + l;
#pragma unroll
    for (int e = 0; e < 2 * R; ++e) ids[e] = live ? __ldg(plane + (int64_t)e * q.m) : -1;
  };
  load_ids(0);  // the table does not change: before the wait
  pdl_enter();
  if (live) Vt::sts(buf[0] + l * VEC, Vt::lds(own));
  cluster_barrier();
  int cur = 0;
  for (int t = 0; t < q.passes; ++t) {
    if (live) {
      const uint32_t base = (uint32_t)__cvta_generic_to_shared(buf[cur]);
      T x[2 * R];
#pragma unroll
      for (int e = 0; e < 2 * R; ++e) {
        x[e] = Vt::zero();
        if (ids[e] >= 0) {
          const uint32_t b = (uint32_t)ids[e] / (uint32_t)q.rows;
          x[e] = ld_cluster<VEC, S>(
              base + ((uint32_t)ids[e] - b * (uint32_t)q.rows) * (uint32_t)(VEC * sizeof(S)), b);
        }
      }
      T acc = Vt::scale(q.tp.t[0], Vt::lds(buf[cur] + l * VEC));
#pragma unroll
      for (int e = 0; e < R; ++e) acc = Vt::fma(q.tp.t[e + 1], Vt::add(x[2 * e], x[2 * e + 1]), acc);
      Vt::sts(buf[cur ^ 1] + l * VEC, acc);
    }
    cur ^= 1;
    if (t + 1 < q.passes) load_ids(t + 1);
    cluster_barrier();
  }
  if (live) Vt::sts(own, Vt::lds(buf[cur] + l * VEC));
}

// ---- sparse blur (lattices whose direction lists are short) ------------------------------
// A vertex without a neighbour along a pass's direction is only scaled by the centre tap g0.
// With fp32 values kept as y = x / g0^t after t passes such vertices do not change, a pass is
// y[v] += (g1 / g0) (y[v - u_j] + y[v + u_j]) on the others, and the factor g0^passes is
// applied once at the end (by the caller, through its alpha).  ChainRange keeps y inside the
// range that x has.
//
// One thread-group of G threads per chain v, v + u_j, v + 2 u_j, ...: it reads every row of the
// chain once and writes it back in place, which no other group reads (chains are maximal).
// Chains have two vertices as a rule, so the first kChainRows rows are loaded together.
// Bound by memory: per active vertex one row read and written and a 4-byte id, per chain 8
// bytes.  n = 500k, d = 20, k = 8 (m = 10.5M, 1M active vertices a pass): 22 us a pass, 64.8
// with per-vertex epochs, a buffer of new rows and a store kernel (k_sparse_blur, below).
//
// LAZY: the values as k_sparse_blur keeps them, the value of x before pass t being
// pw[t - e(x)] stored[x], so that BF16 rows round exactly as there (rows kept as y round at
// other places, 1.6e-3 apart in the product).  Threads of other warps of the group may read an
// epoch after the pass has set it: the word holds the epoch and, above it, the one before.
constexpr int kChainRows = 4;
constexpr int kEpochMask = 0xffff;
template <int VEC, class S, bool LAZY>
__global__ void __launch_bounds__(kThreads) k_chain_blur(int64_t chains, int G, int k, float g0,
                                                         float tap, int t,
                                                         const uint2* __restrict__ chain,
                                                         const int32_t* __restrict__ act,
                                                         const float* __restrict__ pw,
                                                         int32_t* epoch, S* __restrict__ vals) {
  pdl_enter();
  using Vt = Vec<VEC>;
  using T = typename Vt::T;
  const int64_t q = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (q >= chains) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  const uint2 ch = __ldg(chain + q);
  T prev = Vt::zero();  // the row below the current one, before this pass
  for (int64_t p0 = ch.x; p0 < (int64_t)ch.y; p0 += kChainRows) {
    S* at[kChainRows + 1];
    T row[kChainRows + 1];  // the last one only as a neighbour
    int32_t* ep[kChainRows + 1];
    int age[kChainRows + 1];  // LAZY: the epoch before this pass
    float f[kChainRows + 1];  // and the row's factor
#pragma unroll
    for (int e = 0; e <= kChainRows; ++e) {
      const bool in = p0 + e < (int64_t)ch.y;
      const int64_t v = in ? __ldg(act + p0 + e) : 0;
      at[e] = in ? vals + v * k + col : nullptr;
      ep[e] = epoch + v;
      row[e] = Vt::zero();
    }
#pragma unroll
    for (int e = 0; e <= kChainRows; ++e)
      if (at[e]) {
        row[e] = Vt::lds(at[e]);
        if constexpr (LAZY) age[e] = *static_cast<volatile int32_t*>(ep[e]);
      }
    if constexpr (LAZY) {
#pragma unroll
      for (int e = 0; e <= kChainRows; ++e)
        if (at[e]) {
          const int now = age[e] & kEpochMask;
          age[e] = now == t + 1 ? age[e] >> 16 : now;
          f[e] = __ldg(pw + t - age[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < kChainRows; ++e) {
      if constexpr (LAZY) {
        if (at[e]) {
          const T own = Vt::scale(f[e], row[e]);
          const T sum = at[e + 1] ? Vt::fma(f[e + 1], row[e + 1], prev) : prev;
          Vt::sts(at[e], Vt::fma(tap, sum, Vt::scale(g0, own)));
          if (col == 0) *static_cast<volatile int32_t*>(ep[e]) = (t + 1) | (age[e] << 16);
          prev = own;
        }
      } else {
        if (at[e]) Vt::sts(at[e], Vt::fma(tap, Vt::add(prev, row[e + 1]), row[e]));
        prev = row[e];
      }
    }
  }
}

// df_times on VEC columns.
template <int VEC>
__device__ __forceinline__ typename Vec<VEC>::T times(dfloat a, typename Vec<VEC>::T x) {
  float* v = reinterpret_cast<float*>(&x);
#pragma unroll
  for (int j = 0; j < VEC; ++j) v[j] = df_times(a, v[j]);
  return x;
}

template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_rescale(int64_t m, int G, int k, dfloat f,
                                                      S* __restrict__ vals) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t v = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (v >= m) return;
  S* p = vals + v * k + (int)(threadIdx.x % G) * VEC;
  Vt::sts(p, times<VEC>(f, Vt::lds(p)));
}

// The general form (stencil orders above 1, chains longer than kMaxChain): stored rows carry
// a lazy factor, the value of vertex x before pass t being g0^(t - epoch[x]) stored[x].  Pass
// t (direction j) computes the new rows of the vertices on list j into tmp; a second kernel
// stores them and sets their epoch to t + 1.  After the last pass, k_sparse_finish applies
// the remaining factors.
template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_sparse_blur(int64_t count, int G, int k, int r,
                                                          Taps tp, int t,
                                                          const int32_t* __restrict__ act,
                                                          const int32_t* __restrict__ nbr_j,
                                                          int64_t m,
                                                          const int32_t* epoch,
                                                          const float* __restrict__ pw,
                                                          const S* stored,
                                                          S* __restrict__ tmp) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t a = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (a >= count) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  const int64_t v = act[a];
  auto value = [&](int64_t x) {
    const float f = pw ? pw[t - epoch[x]] : 1.f;
    return Vt::scale(f, Vt::lds(stored + x * k + col));
  };
  typename Vt::T acc = Vt::scale(tp.t[0], value(v));
  for (int q = 1; q <= r; ++q) {
    const int ua = nbr_j[(int64_t)(2 * (q - 1)) * m + v];
    const int uc = nbr_j[(int64_t)(2 * (q - 1) + 1) * m + v];
    typename Vt::T sum = Vt::zero();
    if (ua >= 0) sum = value(ua);
    if (uc >= 0) sum = Vt::add(sum, value(uc));
    acc = Vt::fma(tp.t[q], sum, acc);
  }
  Vt::sts(tmp + a * k + col, acc);
}

template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_sparse_store(int64_t count, int G, int k, int t,
                                                           const int32_t* __restrict__ act,
                                                           const S* tmp,
                                                           S* __restrict__ stored,
                                                           int32_t* __restrict__ epoch) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t a = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (a >= count) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  const int64_t v = act[a];
  Vt::sts(stored + v * k + col, Vt::lds(tmp + a * k + col));
  if (col == 0) epoch[v] = t + 1;
}

template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_sparse_finish(int64_t m, int G, int k, int P,
                                                            const int32_t* epoch,
                                                            const float* __restrict__ pw,
                                                            S* __restrict__ stored) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t v = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (v >= m) return;
  const int e = epoch[v] & kEpochMask;  // chains keep the epoch before in the upper half
  if (e == P) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  Vt::sts(stored + v * k + col, Vt::scale(pw[P - e], Vt::lds(stored + v * k + col)));
}

// ---- slice ---------------------------------------------------------------------------
// sum_c w[p][c] lat[idx[p][c]] for the VEC columns at col, in vertex order c = 0..D-1,
// loading the ids and weights of kChunk vertices before their rows.  Where a row's bytes count,
// the last D % kChunk vertices go in rounds of 4, 2 and 1 without conditions (k_slice, n = 2M, d =
// 11, k = 64: 420 us, 623 with every load under a condition); with one or two columns the
// rounds' latency counts (n = 46k, d = 9, k = 1: 33.5 us a product, 34.8 with more rounds), and
// the CG's slice of BF16 values keeps more loads in flight with conditions (n = 200k, d = 33: 62 us,
// 97 without).
template <int VEC, bool EXACT, class S>
__device__ __forceinline__ typename Vec<VEC>::T slice_row(int64_t p, int D, int k, int col,
                                                          const int32_t* __restrict__ idx,
                                                          const float* __restrict__ w,
                                                          const S* lat) {
  using Vt = Vec<VEC>;
  typename Vt::T acc = Vt::zero();
  const int64_t e0 = p * D;
  if constexpr (EXACT) {
    auto run = [&](int c0, auto count) {
      constexpr int N = decltype(count)::value;
      int id[N];
      float wt[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        id[j] = __ldg(idx + e0 + c0 + j);
        wt[j] = __ldg(w + e0 + c0 + j);
      }
      typename Vt::T row[N];
#pragma unroll
      for (int j = 0; j < N; ++j) row[j] = Vt::lds(lat + (int64_t)id[j] * k + col);
#pragma unroll
      for (int j = 0; j < N; ++j) acc = Vt::fma(wt[j], row[j], acc);
    };
    int c0 = 0;
    for (; c0 + kChunk <= D; c0 += kChunk) run(c0, std::integral_constant<int, kChunk>{});
    if (c0 + 4 <= D) {
      run(c0, std::integral_constant<int, 4>{});
      c0 += 4;
    }
    if (c0 + 2 <= D) {
      run(c0, std::integral_constant<int, 2>{});
      c0 += 2;
    }
    if (c0 < D) run(c0, std::integral_constant<int, 1>{});
  } else {
    for (int c0 = 0; c0 < D; c0 += kChunk) {
      int id[kChunk];
      float wt[kChunk];
#pragma unroll
      for (int j = 0; j < kChunk; ++j) {
        const bool in = c0 + j < D;
        id[j] = in ? __ldg(idx + e0 + c0 + j) : -1;
        wt[j] = in ? __ldg(w + e0 + c0 + j) : 0.f;
      }
      typename Vt::T row[kChunk];
#pragma unroll
      for (int j = 0; j < kChunk; ++j)
        row[j] = id[j] >= 0 ? Vt::lds(lat + (int64_t)id[j] * k + col) : Vt::zero();
#pragma unroll
      for (int j = 0; j < kChunk; ++j)
        if (id[j] >= 0) acc = Vt::fma(wt[j], row[j], acc);
    }
  }
  return acc;
}

// out = alpha W lat (+ beta Vp when beta != 0, rows of k in locality order) for the first G VEC of
// lat's k columns.  PERM: out has the caller's ko columns and row order (row perm[p]), written one
// value at a time unless WIDE (ko = G VEC, aligned rows); else out is [n][k] in locality order.
template <int VEC, bool PERM, bool WIDE, class S>
__global__ void __launch_bounds__(kThreads) k_slice(int64_t n, int G, int k, int ko, int D,
                                                    const int32_t* __restrict__ perm,
                                                    const int32_t* __restrict__ idx,
                                                    const float* __restrict__ w,
                                                    const S* lat,
                                                    const float* Vp, dfloat alpha,
                                                    float beta, float* __restrict__ out) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t p = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (p >= n) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  const typename Vt::T acc = slice_row<VEC, VEC == 4, S>(p, D, k, col, idx, w, lat);
  const int64_t i = PERM ? (int64_t)perm[p] : p;
  typename Vt::T res = times<VEC>(alpha, acc);
  if (beta != 0.f) res = Vt::fma(beta, Vt::ld(Vp + p * k + col), res);
  if constexpr (!PERM || WIDE) {
    Vt::st(out + i * (PERM ? ko : k) + col, res);
  } else {
    const float* rr = reinterpret_cast<const float*>(&res);
#pragma unroll
    for (int j = 0; j < VEC; ++j)
      if (col + j < ko) out[i * ko + col + j] = rr[j];
  }
}

// The CG's slice: V and out in locality order, out = alpha W lat + beta V, and the
// per-block column sums of V * out for <p, A p> (exact products and double-float
// accumulation per thread, fp64 across threads).  Grid-stride over points.
template <int VEC, class S>
__global__ void __launch_bounds__(kThreads) k_slice_dot(int64_t n, int G, int k, int D,
                                                        const int32_t* __restrict__ idx,
                                                        const float* __restrict__ w,
                                                        const S* lat,
                                                        const float* V, dfloat alpha,
                                                        float beta, float* __restrict__ out,
                                                        double* __restrict__ dot_partial) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int rows = blockDim.x / G;
  const int col = (int)(threadIdx.x % G) * VEC;
  dfloat d[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) d[j] = {0.f, 0.f};
  for (int64_t p = (int64_t)blockIdx.x * rows + threadIdx.x / G; p < n;
       p += (int64_t)gridDim.x * rows) {
    const typename Vt::T acc =
        slice_row<VEC, VEC == 4 && std::is_same_v<S, float>, S>(p, D, k, col, idx, w, lat);
    const typename Vt::T v = Vt::ld(V + p * k + col);
    const typename Vt::T res = Vt::fma(beta, v, times<VEC>(alpha, acc));
    Vt::st(out + p * k + col, res);
    const float* vv = reinterpret_cast<const float*>(&v);
    const float* rr = reinterpret_cast<const float*>(&res);
#pragma unroll
    for (int j = 0; j < VEC; ++j) d[j] = df_add(d[j], df_two_prod(vv[j], rr[j]));
  }
  double dd[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) dd[j] = df_to_double(d[j]);
  block_column_sums<VEC>(dd, k, dot_partial + (int64_t)blockIdx.x * k);
}

// Vp[p] = V[perm[p]]: the caller's rows (ki columns) in locality order, padded with zero
// columns to k.  WIDE: ki = k and aligned rows.
template <int VEC, bool WIDE>
__global__ void __launch_bounds__(kThreads) k_permute_rows(int64_t n, int G, int k, int ki,
                                                           const int32_t* __restrict__ perm,
                                                           const float* V,
                                                           float* __restrict__ Vp) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t p = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (p >= n) return;
  const int col = (int)(threadIdx.x % G) * VEC;
  const int64_t i = perm[p];
  typename Vt::T x = Vt::zero();
  if constexpr (WIDE) {
    x = Vt::ld(V + i * k + col);
  } else {
    float* xx = reinterpret_cast<float*>(&x);
#pragma unroll
    for (int j = 0; j < VEC; ++j)
      if (col + j < ki) xx[j] = V[i * ki + col + j];
  }
  Vt::st(Vp + p * k + col, x);
}

// Out[p] = (A[perm[p]], B[perm[p]]): the caller's rows of two arrays (ki columns each, padded with
// zero columns to kp) side by side.  VEC divides kp; WIDE: ki = kp and aligned rows.
template <int VEC, bool WIDE>
__global__ void __launch_bounds__(kThreads) k_permute_pair(int64_t n, int G, int kp, int ki,
                                                           const int32_t* __restrict__ perm,
                                                           const float* A,
                                                           const float* B,
                                                           float* __restrict__ out) {
  pdl_enter();
  using Vt = Vec<VEC>;
  const int64_t p = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G;
  if (p >= n) return;
  const int at = (int)(threadIdx.x % G) * VEC;
  const float* src = at < kp ? A : B;
  const int col = at < kp ? at : at - kp;
  const int64_t i = perm[p];
  typename Vt::T x = Vt::zero();
  if constexpr (WIDE) {
    x = Vt::ld(src + i * ki + col);
  } else {
    float* xx = reinterpret_cast<float*>(&x);
#pragma unroll
    for (int j = 0; j < VEC; ++j)
      if (col + j < ki) xx[j] = src[i * ki + col + j];
  }
  Vt::st(out + p * 2 * kp + at, x);
}

// Columns per thread and launch shape for rows of kp columns in library buffers (16-byte
// aligned): a whole number of G-thread rows per block.
struct RowShape {
  int vec, G, threads;
  unsigned blocks;  // for `rows` rows
};
RowShape row_shape(int64_t rows, int kp) {
  RowShape q;
  q.vec = kp % 4 == 0 ? 4 : kp == 2 ? 2 : 1;
  q.G = kp / q.vec;
  q.threads = q.G * (kThreads / q.G);
  q.blocks = (unsigned)ceil_div(rows, q.threads / q.G);
  return q;
}
// The direction lists' kernels read 2 r + 1 rows a vertex one after another, so rows of one thread
// leave a short list with too few warps: rows of two columns, and short lists of four, go a
// column a thread.  Log determinants of 15 steps (d = 33, order 3, 10,000 vertices a list):
// two probes 3.39 ms, 4.06 with two columns a thread; three (rows of four) 3.29, 3.54 with
// four.  Lists of 54,000 (d = 20, order 2): 2.95 and 3.08 ms, of 80,000 (d = 33, order 3): 7.79 and
// 6.53.
RowShape list_shape(int64_t rows, int kp) {
  RowShape q = row_shape(rows, kp);
  if (kp == 2 || (kp == 4 && rows <= 1 << 16)) {
    q.vec = 1;
    q.G = kp;
    q.threads = kThreads;
    q.blocks = (unsigned)ceil_div(rows, kThreads / kp);
  }
  return q;
}
bool wide_ok(int k, int kp, const void* user) {
  return k == kp && (uintptr_t)user % (kp % 4 == 0 ? 16 : kp == 2 ? 8 : 4) == 0;
}
// Calls f(std::integral_constant<int, vec>).
template <class F>
void by_vec(int vec, F f) {
  if (vec == 4) f(std::integral_constant<int, 4>{});
  else if (vec == 2) f(std::integral_constant<int, 2>{});
  else f(std::integral_constant<int, 1>{});
}

// ---- launchers -----------------------------------------------------------------------
// scale: a power of two on the splatted values (1 but for fp32 chains).
// kt: the column count that fixes the shape of the huge vertices' summation tree (the
// caller's k, so that neither padding nor a second product beside it changes a result); kp is
// at most twice kt rounded up.
template <class S>
void launch_splat_t(const Lattice* L, const float* V, int kp, int kt, float scale, S* lat,
                    float* partial, cudaStream_t st) {
  by_vec(row_shape(1, kp).vec, [&](auto vec) {
    constexpr int VEC = decltype(vec)::value;
    const RowShape q = row_shape(L->nseg, kp);
    launch_pdl(k_splat<VEC, S>, q.blocks, q.threads, st, L->nseg, q.G, kp, L->seg, L->items, V,
               scale, lat, partial);
    note_launches(1);
    if (L->nmed > 0 || L->nhuge > 0) {
      const int gt = kt % 4 == 0 ? kt / 4 : kt;
      int groups = 1;
      while (groups * 2 * gt <= kThreads) groups *= 2;
      const int64_t med_blocks = ceil_div(L->nmed, kThreads / q.G);
      launch_pdl(k_splat_fix<VEC, S>, (unsigned)(L->nhuge + med_blocks), kThreads, st, (int)L->nhuge,
                 L->nmed, groups, q.G, kp, L->huge_rows, L->med_rows, partial, scale, lat);
      note_launches(1);
    }
  });
}

template <int VEC, int CH, int U, class S>
void launch_blur_rows(const Lattice* L, const int32_t* nbr, const Taps& taps, const S* in,
                      S* out, int k, cudaStream_t st) {
  const int G = k / (VEC * CH);
  const int threads = G * (kThreads / G);  // a whole number of rows per run
  const int64_t runs = ceil_div(L->m, threads / G);
  const unsigned grid = (unsigned)ceil_div(runs, U);
  switch (L->r) {
    case 1: launch_pdl(k_blur_rows<VEC, CH, U, 1, S>, grid, threads, st, L->m, G, k, taps, nbr, in, out); break;
    case 2: launch_pdl(k_blur_rows<VEC, CH, U, 2, S>, grid, threads, st, L->m, G, k, taps, nbr, in, out); break;
    case 3: launch_pdl(k_blur_rows<VEC, CH, U, 3, S>, grid, threads, st, L->m, G, k, taps, nbr, in, out); break;
    default: launch_pdl(k_blur_rows<VEC, CH, U, 4, S>, grid, threads, st, L->m, G, k, taps, nbr, in, out); break;
  }
}

template <class S>
void launch_blur_t(const Lattice* L, int j, const Taps& taps, const S* in, S* out, int k,
                   cudaStream_t st) {
  const int32_t* nbr = L->nbr + (size_t)j * L->r * 2 * L->m;
  if (k % 8 == 0 && k / 8 <= kThreads && L->r == 1) {  // eight columns, pipelined rows
    const int G = k / 8, threads = G * (kThreads / G);
    const int64_t most = ceil_div(L->m, threads / G);
    bool done = false;
    if constexpr (std::is_same_v<S, float>) {
      if ((size_t)L->m * k * sizeof(float) >= kReadOnlyBytes) {  // not as a dependent
        const unsigned blocks = (unsigned)std::min<int64_t>(blur_pipe_blocks<true, S>(), most);
        k_blur_pipe<true, S><<<blocks, threads, 0, st>>>(L->m, G, k, taps, nbr, in, out);
        done = true;
      }
    }
    if (!done) {
      const unsigned blocks = (unsigned)std::min<int64_t>(blur_pipe_blocks<false, S>(), most);
      launch_pdl(k_blur_pipe<false, S>, blocks, threads, st, L->m, G, k, taps, nbr, in, out);
    }
  } else if (k % 8 == 0 && k / 8 <= kThreads) {  // eight columns of two rows per thread
    launch_blur_rows<4, 2, 2, S>(L, nbr, taps, in, out, k, st);
  } else if (k % 4 == 0 && k / 4 <= kThreads) {
    launch_blur_rows<4, 1, 2, S>(L, nbr, taps, in, out, k, st);
  } else if (k == 2) {
    launch_blur_rows<2, 1, 2, S>(L, nbr, taps, in, out, k, st);
  } else if (k == 1) {
    launch_blur_rows<1, 1, 2, S>(L, nbr, taps, in, out, k, st);
  } else {
    launch_pdl(k_blur<S>, (unsigned)ceil_div(L->m * k, kThreads), kThreads, st, L->m, k, L->r, taps, nbr,
                                                                          in, out);
  }
  note_launches(1);
}

// out = alpha W lat + beta Vp (Vp in locality order, rows of kp).  PERM: out is the caller's
// [n][k]; else [n][kp] in locality order.  lat_cols: columns of a row of lat (0: kp).
template <bool PERM, class S>
void launch_slice_t(const Lattice* L, const S* lat, const float* Vp, int k, int kp, dfloat alpha,
                    float beta, float* out, cudaStream_t st, int lat_cols = 0) {
  if (lat_cols == 0) lat_cols = kp;
  const RowShape q = row_shape(L->n, kp);
  if (!Vp) beta = 0.f;
  by_vec(q.vec, [&](auto vec) {
    constexpr int VEC = decltype(vec)::value;
    if (!PERM || wide_ok(k, kp, out))
      launch_pdl(k_slice<VEC, PERM, true, S>, q.blocks, q.threads, st, L->n, q.G, lat_cols, k, L->D,
                 L->perm, L->idx, L->w, lat, Vp, alpha, beta, out);
    else
      launch_pdl(k_slice<VEC, PERM, false, S>, q.blocks, q.threads, st, L->n, q.G, lat_cols, k, L->D,
                 L->perm, L->idx, L->w, lat, Vp, alpha, beta, out);
  });
  note_launches(1);
}

template <class S>
void launch_slice_dot(const Lattice* L, const S* lat, const float* V, int k, int kt, dfloat alpha,
                      float beta, float* out, double* dot_partial, cudaStream_t st) {
  const int vec = k % 4 == 0 ? 4 : 1;
  const int T = column_block_threads(k, vec, kt);
  const unsigned grid = (unsigned)slice_dot_blocks(L, k, kt);
  if (vec == 4)
    launch_pdl(k_slice_dot<4, S>, grid, T, st, L->n, k / 4, k, L->D, L->idx, L->w, lat, V, alpha, beta,
                                          out, dot_partial);
  else
    launch_pdl(k_slice_dot<1, S>, grid, T, st, L->n, k, k, L->D, L->idx, L->w, lat, V, alpha, beta, out,
                                          dot_partial);
  note_launches(1);
}

void launch_permute(const Lattice* L, const float* V, int k, int kp, float* Vp, cudaStream_t st) {
  const RowShape q = row_shape(L->n, kp);
  by_vec(q.vec, [&](auto vec) {
    constexpr int VEC = decltype(vec)::value;
    if (wide_ok(k, kp, V))
      launch_pdl(k_permute_rows<VEC, true>, q.blocks, q.threads, st, L->n, q.G, kp, k, L->perm, V, Vp);
    else
      launch_pdl(k_permute_rows<VEC, false>, q.blocks, q.threads, st, L->n, q.G, kp, k, L->perm, V, Vp);
  });
  note_launches(1);
}

// The cluster blur takes lattices of up to 16 blocks of 1024 vertices and up to 8 column
// groups (as many clusters are resident at once).  Measured, symmetric product with d = 8, k =
// 16, clusters of 16 / a launch a pass: m = 5.9k 34 / 55 us, 10.8k (k = 12) 41 / 61 us, 17k (d = 9,
// k = 2) 52 / 62 us; beyond, remote shared-memory reads cost more than a launch (m = 51k: 107 /
// 62 us with several vertices a thread).  Blocks of 64 vertices or more: smaller clusters
// were never faster (m = 1k, d = 4: 38 us with one block, 31 with 16).
constexpr int kClusterBlocks = 16, kClusterRows = 1024, kClusterGroups = 8;

// Launch configuration of one cluster per column group; at: room for its two attributes.
cudaLaunchConfig_t cluster_config(int blocks, int groups, int rows, cudaStream_t st,
                                  cudaLaunchAttribute (&at)[2]) {
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)blocks;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks, (unsigned)groups);
  cfg.blockDim = (unsigned)(ceil_div(rows, 32) * 32);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

// Whether the current device can hold the largest cluster (on a partitioned one it may have
// too few SMs together): asked before the first launch, because inside a stream capture a
// launch is only recorded and would fail when the graph runs.
template <int VEC, int R, class S>
bool cluster_fits() {
  static std::atomic<int> cache[64];  // 0: not asked yet, 1: fits, 2: does not
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  if (const int c = cache[dev].load()) return c == 1;
  if (cudaPeekAtLastError() != cudaSuccess) return false;  // left for the caller's check
  auto kernel = k_blur_cluster<VEC, R, S>;
  cudaLaunchAttribute at[2]{};
  const cudaLaunchConfig_t cfg = cluster_config(kClusterBlocks, 1, kClusterRows, nullptr, at);
  int clusters = 0;
  const bool fits =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
          cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0;
  if (!fits) clear_pending_error();  // of these two calls
  cache[dev].store(fits ? 1 : 2);
  return fits;
}

// All passes on lat0 by k_blur_cluster; false when the lattice is not of its size, or the device
// has no room for its clusters.
template <class S>
bool blur_cluster_t(const Lattice* L, int blur, int passes, const Taps& tp, S* lat0, int k,
                    cudaStream_t st) {
  const RowShape shape = row_shape(L->m, k);
  if (L->m > kClusterBlocks * kClusterRows || shape.G > kClusterGroups || L->r > 2 ||
      L->fault == FAULT_NO_CLUSTER)
    return false;
  int blocks = 1;
  while (blocks < kClusterBlocks && L->m > 64 * blocks) blocks *= 2;
  const ClusterBlur q{(int)L->m, k, L->D, passes, blur, (int)ceil_div(L->m, blocks), tp, L->nbr};
  bool done = false;
  by_vec(shape.vec, [&](auto vec) {
    constexpr int VEC = decltype(vec)::value;
    auto go = [&](auto order) {
      constexpr int R = decltype(order)::value;
      if (!cluster_fits<VEC, R, S>()) return;
      cudaLaunchAttribute at[2]{};
      const cudaLaunchConfig_t cfg = cluster_config(blocks, shape.G, q.rows, st, at);
      (void)cudaLaunchKernelEx(&cfg, k_blur_cluster<VEC, R, S>, q, lat0);  // as launch_pdl
      done = true;
    };
    if (L->r == 1) go(std::integral_constant<int, 1>{});
    else go(std::integral_constant<int, 2>{});
  });
  if (done) note_launches(1);
  return done;
}

// Sparse blurs run on chains (else on the direction lists).
bool chains_ok(const Lattice* L) { return L->chain_max > 0 && L->chain_max <= kMaxChain; }

// Centre and side tap of one pass.
double tap0(const Lattice* L, int blur) { return (blur == SGP_BLUR_SYMMETRIC ? L->half : L->coef)[0]; }
double tap1(const Lattice* L, int blur) { return (blur == SGP_BLUR_SYMMETRIC ? L->half : L->coef)[1]; }
int pass_count(const Lattice* L, int blur) { return blur == SGP_BLUR_SYMMETRIC ? 2 * L->D : L->D; }

// The values y = x / g0^t of fp32 chains grow past x by g0^-t (400 at d = 50 and the default
// spacing, 3e22 at a spacing of 0.25): a product whose x has room in fp32 must not overflow in
// y, nor its alpha g0^t underflow.  So the splat takes 2^-exponent off (exact, and no bit of a
// product differs for it), with 2^exponent >= g0^-t, and the values are multiplied by g0^run
// every `run` passes so that exponent <= 12 (never below 142 passes at the default spacing):
// |y| <= |x|, and x down to 2^-114 keeps its 24 bits.
struct ChainRange {
  int run = 0;       // passes between rescalings (0: the values are x itself)
  int exponent = 0;
};
template <class S>
ChainRange chain_range(const Lattice* L, int blur, bool dense) {
  const double g0 = tap0(L, blur);
  if (!L->sparse || dense || !chains_ok(L) || std::is_same_v<S, bf16> || g0 >= 1.0) return {};
  constexpr double kMaxExponent = 12.0;
  const double bits = -std::log2(g0);  // growth of a pass
  const int P = pass_count(L, blur);
  const int most = std::max(1, (int)std::min<double>(P, kMaxExponent / bits));
  const int runs = (P + most - 1) / most;
  ChainRange c;
  c.run = (P + runs - 1) / runs;
  c.exponent = (int)std::ceil(c.run * bits);
  return c;
}

// The blur passes of `blur` on the splatted values in lat0 (lat1: ping-pong buffer);
// returns the buffer that holds the result divided by *scale.  Sparse lattices use their
// chains or direction lists (lat1 unused) unless `dense` is set.
template <class S>
S* blur_passes_t(const Lattice* L, int blur, S* lat0, S* lat1, int k, cudaStream_t st,
                 int* passes_out, bool dense, double* scale) {
  *scale = 1.0;
  Taps c{}, g{};
  for (int t = 0; t <= L->r; ++t) {
    c.t[t] = (float)L->coef[t];
    g.t[t] = (float)L->half[t];
  }
  const int D = L->D;
  const int P = blur == SGP_BLUR_SYMMETRIC ? 2 * D : D;
  auto dir = [&](int t) {
    if (blur == SGP_BLUR_SEQUENTIAL) return t;
    if (blur == SGP_BLUR_TRANSPOSE) return D - 1 - t;
    return t < D ? t : 2 * D - 1 - t;
  };
  const Taps& tp = blur == SGP_BLUR_SYMMETRIC ? g : c;
  if (passes_out) *passes_out = P;
  if (!L->sparse || dense) {
    if (blur_cluster_t<S>(L, blur, P, tp, lat0, k, st)) return lat0;
    S* a = lat0;
    S* b = lat1;
    for (int t = 0; t < P; ++t) {
      launch_blur_t<S>(L, dir(t), tp, a, b, k, st);
      S* x = a;
      a = b;
      b = x;
    }
    return a;
  }
  const float* pw = tp.t[0] == 1.f ? nullptr : L->g0pow;
  // BF16 chains keep the lazy factors of the direction lists (none when the centre tap is 1)
  const bool lazy = pw && (!chains_ok(L) || std::is_same_v<S, bf16>);
  if (lazy) cudaMemsetAsync(L->epoch, 0, (size_t)L->m * sizeof(int32_t), st);
  auto finish = [&] {
    const RowShape q = row_shape(L->m, k);
    by_vec(q.vec, [&](auto vec) {
      launch_pdl(k_sparse_finish<decltype(vec)::value, S>, q.blocks, q.threads, st, L->m, q.G, k, P,
                 L->epoch, pw, lat0);
    });
    note_launches(1);
  };
  if (chains_ok(L)) {
    const double g0 = tap0(L, blur), g1 = tap1(L, blur);
    const ChainRange range = chain_range<S>(L, blur, dense);
    int owed = 0;  // passes whose factor has not been applied
    by_vec(row_shape(1, k).vec, [&](auto vec) {
      constexpr int VEC = decltype(vec)::value;
      for (int t = 0; t < P; ++t) {
        const int j = dir(t);
        const int64_t count = L->chain_off[j + 1] - L->chain_off[j];
        if (range.run > 0 && owed == range.run) {
          const RowShape q = row_shape(L->m, k);
          launch_pdl(k_rescale<VEC, S>, q.blocks, q.threads, st, L->m, q.G, k,
                     split_factor(std::pow(g0, owed)), lat0);
          note_launches(1);
          owed = 0;
        }
        ++owed;
        if (count == 0) continue;
        const RowShape q = row_shape(count, k);
        const uint2* chain = L->chain + L->chain_off[j];
        auto pass = [&](auto keep, float own, float tap) {
          launch_pdl(k_chain_blur<VEC, S, decltype(keep)::value>, q.blocks, q.threads, st, count,
                     q.G, k, own, tap, t, chain, L->act, pw, L->epoch, lat0);
        };
        if (lazy) pass(std::is_same<S, bf16>{}, tp.t[0], tp.t[1]);
        else pass(std::false_type{}, 1.f, (float)(g1 / g0));
        note_launches(1);
      }
    });
    if (lazy) finish();
    else *scale = std::ldexp(std::pow(g0, owed), range.exponent);
    return lat0;
  }
  S* tmp = static_cast<S*>(L->act_tmp);
  for (int t = 0; t < P; ++t) {
    const int j = dir(t);
    const int64_t count = L->act_off[j + 1] - L->act_off[j];
    if (count == 0) continue;
    const int32_t* act = L->act + L->act_off[j];
    const int32_t* nbr_j = L->nbr + (size_t)j * L->r * 2 * L->m;
    const RowShape q = list_shape(count, k);
    by_vec(q.vec, [&](auto vec) {
      constexpr int VEC = decltype(vec)::value;
      launch_pdl(k_sparse_blur<VEC, S>, q.blocks, q.threads, st, count, q.G, k, L->r, tp, t, act,
                 nbr_j, L->m, L->epoch, pw, lat0, tmp);
      launch_pdl(k_sparse_store<VEC, S>, q.blocks, q.threads, st, count, q.G, k, t, act, tmp, lat0,
                 L->epoch);
      note_launches(2);
    });
  }
  if (pw) finish();
  return lat0;
}

// The whole operator with explicit buffers, whose rows have kp columns.  internal: V and out
// are [n][kp] in locality order; else V and out are the caller's [n][k] and V is first
// gathered into `vperm`.  kt: see launch_splat_t.
template <class S>
int enqueue_t(const Lattice* L, const float* V, int k, int kp, int kt, int blur, float alpha,
              float beta, float* out, S* lat0, S* lat1, float* partial, float* vperm,
              cudaStream_t st, cudaEvent_t* ev, bool internal, double* dot_partial = nullptr,
              bool dense = false) {
  const float* src = V;
  if (!internal) {
    launch_permute(L, V, k, kp, vperm, st);
    src = vperm;
  }
  if (ev) cudaEventRecordWithFlags(ev[2], st, cudaEventRecordExternal);
  const float take = std::ldexp(1.f, -chain_range<S>(L, blur, dense).exponent);
  launch_splat_t<S>(L, src, kp, kt, take, lat0, partial, st);
  // External: inside a stream capture this becomes an event-record node of the graph
  if (ev) cudaEventRecordWithFlags(ev[0], st, cudaEventRecordExternal);
  int passes = 0;
  double scale = 1.0;
  S* a = blur_passes_t<S>(L, blur, lat0, lat1, kp, st, &passes, dense, &scale);
  const dfloat factor = split_factor(alpha * scale);
  if (ev) cudaEventRecordWithFlags(ev[1], st, cudaEventRecordExternal);
  if (internal && dot_partial) launch_slice_dot<S>(L, a, V, kp, kt, factor, beta, out, dot_partial, st);
  else if (internal) launch_slice_t<false, S>(L, a, V, kp, kp, factor, beta, out, st);
  else launch_slice_t<true, S>(L, a, src, k, kp, factor, beta, out, st);
  if (ev) cudaEventRecordWithFlags(ev[3], st, cudaEventRecordExternal);
  return passes;
}

// Splat (locality-ordered input, rows of kp) and blur only; returns the buffer holding the
// result.
template <class S>
S* splat_blur_t(const Lattice* L, const float* Vp, int kp, int kt, int blur, S* lat0, S* lat1,
                float* partial, cudaStream_t st, double* scale) {
  const float take = std::ldexp(1.f, -chain_range<S>(L, blur, false).exponent);
  launch_splat_t<S>(L, Vp, kp, kt, take, lat0, partial, st);
  return blur_passes_t<S>(L, blur, lat0, lat1, kp, st, nullptr, false, scale);
}

size_t value_size(const Lattice* L) {
  return L->value_dtype == SGP_VALUES_BF16 ? sizeof(bf16) : sizeof(float);
}

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

size_t mvm_work_bytes(const Lattice* L, int k) {
  return 2 * round256((size_t)L->m * k * value_size(L)) +
         round256((size_t)L->nslots * k * sizeof(float)) + round256((size_t)L->n * k * sizeof(float));
}

void release_lattice_values(Lattice* L, cudaStream_t st) {
  void** bufs[4] = {(void**)&L->lat[0], (void**)&L->lat[1], (void**)&L->partial,
                    (void**)&L->vperm};
  for (void** b : bufs) {
    if (*b) cudaFreeAsync(*b, st);
    *b = nullptr;
  }
  L->bytes -= L->lat_bytes;
  L->lat_bytes = 0;
  L->lat_elems = 0;
  L->vperm_elems = 0;
}

sgp_status ensure_lattice_values(Lattice* L, int k, cudaStream_t st) {
  if (L->sparse && (!chains_ok(L) || L->table_blur) &&
      L->act_tmp_elems < (size_t)L->act_max * k) {
    if (L->act_tmp) cudaFreeAsync(L->act_tmp, st);
    L->act_tmp = nullptr;
    L->act_tmp_elems = 0;  // if there is no room now, a narrower product asks again
    const size_t bytes = std::max<size_t>((size_t)L->act_max * k * value_size(L), 16);
    cudaError_t e = cols_malloc(L, k, &L->act_tmp, bytes, st);
    if (e != cudaSuccess) return cuda_status(e, "allocating the sparse blur buffer");
    L->act_tmp_elems = (size_t)L->act_max * k;
  }
  if (L->lat_elems >= (size_t)L->m * k && L->lat[0] && L->vperm_elems >= (size_t)L->n * k)
    return SGP_OK;
  release_lattice_values(L, st);
  void** bufs[4] = {(void**)&L->lat[0], (void**)&L->lat[1], (void**)&L->partial,
                    (void**)&L->vperm};
  const size_t vbytes = (size_t)L->m * k * value_size(L);
  const size_t sizes[4] = {vbytes, vbytes, (size_t)L->nslots * k * sizeof(float),
                           (size_t)L->n * k * sizeof(float)};
  for (int b = 0; b < 4; ++b) {
    cudaError_t e = cols_malloc(L, k, bufs[b], std::max<size_t>(sizes[b], 16), st);
    if (e != cudaSuccess) return cuda_status(e, "allocating lattice values");
  }
  L->lat_elems = (size_t)L->m * k;
  L->vperm_elems = (size_t)L->n * k;
  L->lat_bytes = sizes[0] + sizes[1] + sizes[2] + sizes[3];
  L->bytes += L->lat_bytes;
  return SGP_OK;
}

int enqueue_mvm(const Lattice* L, const float* V, int k, int blur, float alpha, float beta,
                float* out, cudaStream_t st, cudaEvent_t* ev, bool internal, double* dot_partial,
                int tree_k) {
  const int kp = internal ? k : value_cols(L, k);
  const int kt = tree_k > 0 ? tree_k : k;
  if (L->value_dtype == SGP_VALUES_BF16)
    return enqueue_t<bf16>(L, V, k, kp, kt, blur, alpha, beta, out, (bf16*)L->lat[0],
                           (bf16*)L->lat[1], L->partial, L->vperm, st, ev, internal, dot_partial);
  return enqueue_t<float>(L, V, k, kp, kt, blur, alpha, beta, out, (float*)L->lat[0],
                          (float*)L->lat[1], L->partial, L->vperm, st, ev, internal, dot_partial);
}

void enqueue_mvm_bf16_values(const Lattice* L, const float* V, int k, int blur, float alpha,
                             float* out, cudaStream_t st) {
  enqueue_t<bf16>(L, V, k, k, k, blur, alpha, 0.f, out, (bf16*)L->lat[0], (bf16*)L->lat[1],
                  L->partial, L->vperm, st, nullptr, /*internal=*/true);
}

int64_t slice_dot_blocks(const Lattice* L, int k, int tree_k) {
  const int vec = k % 4 == 0 ? 4 : 1;
  const int G = k / vec;
  const int T = column_block_threads(k, vec, tree_k);
  // one wave: as many blocks as the device keeps resident (a grid-stride kernel whose
  // grid exceeds that runs a second, mostly idle wave)
  int per_sm = 0, sms = 0, dev = 0;
  const void* fn = vec == 4 ? (L->value_dtype == SGP_VALUES_BF16
                                   ? (const void*)k_slice_dot<4, bf16>
                                   : (const void*)k_slice_dot<4, float>)
                            : (L->value_dtype == SGP_VALUES_BF16
                                   ? (const void*)k_slice_dot<1, bf16>
                                   : (const void*)k_slice_dot<1, float>);
  int64_t resident = kVecBlocks;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, T, 0) == cudaSuccess &&
      per_sm > 0)
    resident = (int64_t)per_sm * sms;
  else
    (void)cudaGetLastError();
  return std::min<int64_t>(resident, std::max<int64_t>(1, ceil_div(L->n, T / G)));
}

void enqueue_mvm_into(const Lattice* L, const float* V_user, int k, int blur, float alpha,
                      float beta, float* out, void* work, cudaStream_t st) {
  char* w = static_cast<char*>(work);
  const size_t vb = round256((size_t)L->m * k * value_size(L));
  void* lat0 = w;
  void* lat1 = w + vb;
  float* partial = reinterpret_cast<float*>(w + 2 * vb);
  float* vperm = reinterpret_cast<float*>(w + 2 * vb + round256((size_t)L->nslots * k * sizeof(float)));
  // the fixed work area holds no direction-list buffers: dense passes
  if (L->value_dtype == SGP_VALUES_BF16)
    enqueue_t<bf16>(L, V_user, k, k, k, blur, alpha, beta, out, (bf16*)lat0, (bf16*)lat1, partial, vperm,
                    st, nullptr, false, nullptr, /*dense=*/true);
  else
    enqueue_t<float>(L, V_user, k, k, k, blur, alpha, beta, out, (float*)lat0, (float*)lat1, partial,
                     vperm, st, nullptr, false, nullptr, /*dense=*/true);
}

void* enqueue_splat_blur(const Lattice* L, const float* Vp, int kp, int kt, int blur, void* lat0,
                         void* lat1, float* partial, cudaStream_t st, double* scale) {
  if (L->value_dtype == SGP_VALUES_BF16)
    return splat_blur_t<bf16>(L, Vp, kp, kt, blur, (bf16*)lat0, (bf16*)lat1, partial, st, scale);
  return splat_blur_t<float>(L, Vp, kp, kt, blur, (float*)lat0, (float*)lat1, partial, st, scale);
}

void enqueue_permute(const Lattice* L, const float* V, int k, int kp, float* Vp, cudaStream_t st) {
  launch_permute(L, V, k, kp, Vp, st);
}

void enqueue_permute_pair(const Lattice* L, const float* A, const float* B, int k, int kp,
                          float* out, cudaStream_t st) {
  const int vec = kp % 4 == 0 ? 4 : 1;
  const int G = 2 * kp / vec, rows = kThreads / G;
  const unsigned blocks = (unsigned)ceil_div(L->n, rows);
  auto go = [&](auto kernel) {
    launch_pdl(kernel, blocks, rows * G, st, L->n, G, kp, k, L->perm, A, B, out);
  };
  if (vec == 4 && wide_ok(k, kp, A) && wide_ok(k, kp, B)) go(k_permute_pair<4, true>);
  else if (vec == 4) go(k_permute_pair<4, false>);
  else go(k_permute_pair<1, false>);
  note_launches(1);
}

bool blur_in_place(const Lattice* L) { return L->sparse && chains_ok(L); }

void enqueue_slice_caller(const Lattice* L, const void* lat, int k, int kp, int lat_cols,
                          dfloat alpha, float* out, cudaStream_t st) {
  if (L->value_dtype == SGP_VALUES_BF16)
    launch_slice_t<true, bf16>(L, (const bf16*)lat, nullptr, k, kp, alpha, 0.f, out, st, lat_cols);
  else
    launch_slice_t<true, float>(L, (const float*)lat, nullptr, k, kp, alpha, 0.f, out, st, lat_cols);
}

size_t lattice_value_bytes(const Lattice* L, int k) { return (size_t)L->m * k * value_size(L); }

int padded_cols(int k) { return k <= 2 ? k : (k + 3) / 4 * 4; }

int value_cols(const Lattice* L, int k) { return L->tight_cols ? k : padded_cols(k); }

bool give_up_padding(Lattice* L, cudaStream_t st) {
  if (L->tight_cols) return false;
  L->tight_cols = true;
  release_lattice_values(L, st);
  return true;
}

sgp_status ensure_product(Lattice* L, int k, cudaStream_t st) {
  sgp_status s = ensure_lattice_values(L, value_cols(L, k), st);
  if (s == SGP_ERR_OOM && padded_cols(k) != k && give_up_padding(L, st))
    s = ensure_lattice_values(L, k, st);
  return s;
}

sgp_status run_mvm(Lattice* L, const float* V, int k, int blur, float alpha, float beta,
                   float* out) {
  sgp_status s = ensure_product(L, k, L->stream);
  if (s != SGP_OK) return s;
  enqueue_mvm(L, V, k, blur, alpha, beta, out, L->stream);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "launching the lattice MVM");
  return SGP_OK;
}

}  // namespace sgp
