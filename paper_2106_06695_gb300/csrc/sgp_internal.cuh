// Internal declarations of the sm_103a Simplex-GP library (not part of the C-ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <string>
#include <utility>
#include <vector>

#include "../../include/sgp.h"

namespace sgp {

// Device error word bits, OR-ed by kernels and read back by the host.
enum : unsigned {
  ERRBIT_NONFINITE = 1u,
  ERRBIT_RANGE = 2u,
  ERRBIT_HASH_FULL = 4u,
};

// Faults injected on the host through SGP_FAULT (tests of the error paths).
enum { FAULT_NONE = 0, FAULT_OOM, FAULT_CUDA, FAULT_HASH_FULL, FAULT_NAN_INPUT, FAULT_NO_CLUSTER };
int injected_fault(int* columns);  // *columns: sgp_lattice::fault_cols

// NVTX range for the lifetime of a scope (timeline profilers; no-op without one).
struct NvtxRange {
  explicit NvtxRange(const char* name);
  ~NvtxRange();
};

constexpr int kMaxOrder = 4;  // stencil order r
constexpr int kMaxD = 128;    // d + 1
constexpr int kMaxK = 256;    // right-hand sides per call
constexpr int kProfStages = 5;     // splat, blur, slice, B^T r, z (sgp_profile_read_stages)
constexpr int kSplatSeg = 32;      // splat items per segment
constexpr int kSplatMedSegs = 16;  // segments a single thread-group sums in the fix-up
// A lattice blurs in sparse mode when the direction lists hold at most this fraction of
// the D m (vertex, direction) pairs.
constexpr double kSparseFrac = 0.3;
// Chains longer than this are not walked by one thread group: the lattice is blurred through
// the direction lists then.
constexpr int kMaxChain = 64;

// Stencil taps passed by value to the blur kernels.
struct Taps {
  float t[kMaxOrder + 1];
};

}  // namespace sgp

// The lattice handle: every array below is device memory owned by the handle.
struct sgp_lattice {
  int64_t n = 0;
  int d = 0, D = 0, r = 1;
  int kernel = 0;
  int64_t m = 0;
  double s = 0.0;
  double coef[sgp::kMaxOrder + 1] = {};
  double half[sgp::kMaxOrder + 1] = {};
  float outputscale = 1.f;
  int value_dtype = 0;
  int check_every = 8;
  int precond_rank = 0;
  int precond_power_iters = 1;
  uint64_t precond_seed = 0;
  int fault = 0;  // sgp::FAULT_* injected by SGP_FAULT into this lattice's construction
  int fault_cols = 0;  // > 0: buffers of more columns than this fail to allocate (SGP_FAULT)
  int device = -1;  // CUDA device current at build time (the arrays live there)
  cudaStream_t stream = nullptr;

  // Points are processed in a locality order p = 0..n-1; perm[p] is the caller's index.
  int32_t* perm = nullptr;   // [n]
  int32_t* idx = nullptr;    // [n][D] vertex id of vertex k of point perm[p]
  float* w = nullptr;        // [n][D] barycentric weight, same order
  int32_t* row_ptr = nullptr;  // [m+1] splat lists: vertex v gathers items[row_ptr[v]..]
  int2* items = nullptr;       // [n*D] (locality-ordered point index p, weight bits)
  // Splat work split into segments of at most kSplatSeg items (load balance: a dense
  // cluster gives a vertex thousands of points).  seg[s] = (vertex, begin, end, slot):
  // slot < 0 writes the vertex directly, else the partial goes to partial[slot] and a
  // fix-up sums a vertex's partials in order.  med_rows / huge_rows: (vertex, first slot,
  // number of slots) of vertices with 2..kSplatMedSegs / more segments.
  int4* seg = nullptr;
  int64_t nseg = 0;
  int4* med_rows = nullptr;
  int64_t nmed = 0;
  int4* huge_rows = nullptr;
  int64_t nhuge = 0;
  int64_t nslots = 0;
  float* partial = nullptr;  // [nslots][k], sized with the lattice values
  float* vperm = nullptr;    // [n][k] the caller's V in locality order (public MVMs)
  int32_t* nbr = nullptr;      // [D][r][2][m] neighbour id of v - t u_j (0) / v + t u_j (1)
  int16_t* keys = nullptr;     // [m][D] vertex coordinates
  // Sparse lattices (few vertices with a neighbour along each direction, e.g. isolated
  // simplices at high d): act[act_off[j] .. act_off[j+1]) lists the vertices with at least
  // one neighbour along direction j, and the blur updates only those (sgp::kSparseFrac).
  bool sparse = false;
  int32_t* act = nullptr;
  std::vector<int64_t> act_off;  // [D + 1], host
  int64_t* act_off_dev = nullptr;  // [D + 1], device copy
  int64_t act_max = 0;           // largest list
  // Stencil order 1: each list is ordered by chains (maximal runs v, v + u_j, v + 2 u_j, ...);
  // chain[chain_off[j] .. chain_off[j+1]) holds (begin, end) of direction j's chains in act.
  uint2* chain = nullptr;
  std::vector<int64_t> chain_off;  // [D + 1], host
  int chain_max = 0;  // longest chain, kMaxChain + 1 for any longer one; 0: no chains (order > 1)
  bool table_blur = false;       // blurred by the server's table kernels too (needs act_tmp)
  int32_t* epoch = nullptr;      // [m] pass after which a vertex's stored row was written
  void* act_tmp = nullptr;       // [act_max][k] new values of one pass
  size_t act_tmp_elems = 0;
  float* g0pow = nullptr;        // [2D + 1] powers of the symmetric blur's centre tap
  uint8_t* rank = nullptr;     // [n][D] rank of each elevated coordinate, locality order
  unsigned* err = nullptr;     // device error word

  // Lattice values (fp32 or bf16 per value_dtype), allocated on first use, grown on demand.
  void* lat[2] = {nullptr, nullptr};
  size_t lat_elems = 0;
  size_t lat_bytes = 0;  // value buffers + splat partials + permuted input
  size_t vperm_elems = 0;
  bool tight_cols = false;  // products use unpadded rows (value_cols): memory was short

  // Optional blur timing: events bracket the blur passes of one MVM inside the CG graph
  // and are read at every flag check (sgp_profile_blur / sgp_profile_read).
  // prof_ev: [0] after the splat, [1] after the blur, [2] before the splat, [3] after the
  // slice of the MVM inside the CG graph; [4] .. [7] around the preconditioner's B^T r
  // kernel ([4], [5]) and its z kernel ([6], [7]).
  int profile = 0;
  cudaEvent_t prof_ev[8] = {};
  double prof_ms = 0.0;
  int64_t prof_passes = 0;
  double prof_stage_ms[sgp::kProfStages] = {};  // SGP_STAGE_* order
  int64_t prof_mvms = 0;

  size_t bytes = 0;
};

namespace sgp {

using Lattice = ::sgp_lattice;

// An unevaluated sum of two fp32 numbers (the arithmetic stands below).
struct dfloat {
  float hi, lo;
};
// A factor to 48 bits; lo = 0 for an fp32 number.
inline dfloat split_factor(double x) {
  const float hi = (float)x;
  const float lo = (float)(x - (double)hi);
  return {hi, std::isfinite(lo) ? lo : 0.f};
}

// ---- error reporting and launch accounting (api.cu) ----
void set_error(const std::string& msg);
sgp_status cuda_status(cudaError_t e, const char* what);
// Clear a pending non-sticky runtime error left by earlier calls of this thread (ours or
// the caller's), so that the launch checks of the current call report only its own
// launches.  A sticky error (a failed context) is returned again by the next call anyway.
void clear_pending_error();
// Count kernels enqueued by this library (graph replays count every kernel node).
void note_launches(int64_t count);
int64_t launches_so_far();
// Stream-ordered device allocation from the library's pool on the current device (freed
// with cudaFreeAsync; freed blocks stay mapped for reuse until sgp_trim_memory).
cudaError_t dev_malloc(void** p, size_t bytes, cudaStream_t st);
// The same for a buffer of `columns` columns that a call on L may fail to get.
cudaError_t cols_malloc(const sgp_lattice* L, int columns, void** p, size_t bytes, cudaStream_t st);

// ---- programmatic dependent launch ----
// Back-to-back dependent kernels on one stream start about 4.1 us apart on GB300 when each
// launch waits for the previous grid to drain, and 1.4-1.6 us apart when it is set up
// beforehand and only waits for the data (measured: 200 dependent kernels of 152 blocks,
// legacy and created streams; inside a graph 1.15 and 0.94 us).  launch_pdl marks a launch as
// such a dependent; every block of a kernel launched with it calls pdl_enter(), which waits until
// all work before this grid has completed and is visible.  What keeps the order that ordinary
// launches have:
//  - Nothing is written before the wait.
//  - Read before it are only arrays that do not change after the build (neighbour ids), and data
//    whose last writer is a grid that the grid right before this one has itself waited for, so
//    at least two launches back (the server's table kernels: the list stands at SLOT_AHEAD).
//  - What grids of the same stream write is read by ordinary loads: neither __ldg nor pointers
//    that are const and __restrict__.  Those stand for data that do not change while the kernel
//    runs, and a dependent runs already while the writer does; the compiler might also move
//    such a load ahead of the wait.  Only the arrays that are fixed after the build (and the
//    server's table) are declared so, and only a kernel that is launched the ordinary way may
//    load others so (k_blur_pipe<RO = true>).
// Dependents are not let in early (griddepcontrol.launch_dependents
// at the top of each kernel): their waiting blocks take slots from the running grid (a
// product at n = 50k, d = 8, k = 9: 63 us without, 78 us with it; eight CG iterations at n =
// 86k, d = 8: 998 and 1154 us).  After the last loads are issued it does no harm (pdl_leave).
template <class... P, class... A>
inline void launch_pdl_smem(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                            cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);  // read by cudaGetLastError
}
template <class... P, class... A>
inline void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A&&... args) {
  launch_pdl_smem(kernel, grid, block, 0, st, std::forward<A>(args)...);
}
// Lets the next grid in: only where this grid has nothing left to load.
__device__ __forceinline__ void pdl_leave() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- stencils (stencil.cpp) ----
// Spacing s and taps c[0..r] (kernel values k(t s)) and g[0..r] (half-kernel taps).
// Returns false when the kernel id or order is invalid.
bool make_stencil(int kernel, int r, double spacing_override, double* s, double* coef,
                  double* half);

// ---- primitives (scan_sort.cu) ----
// Exclusive scan of n uint32 values in place; *total (device, may be null) receives the
// sum.  `tmp` must hold scan_temp_elems(n) uint32.
size_t scan_temp_elems(int64_t n);
void exclusive_scan_u32(uint32_t* data, int64_t n, uint32_t* total, uint32_t* tmp,
                        cudaStream_t st);
// Exclusive scans in place of `rows` rows of n values, one block each (block sums).
void exclusive_scan_rows_u32(uint32_t* data, int rows, int64_t n, cudaStream_t st);
// Stable LSD radix sort of (key, value) pairs by bits begin .. end - 1 of the key (8 at a
// time, so up to 7 more).  Uses the *_alt buffers as ping-pong storage; returns true when the
// result ended in *_alt.
size_t radix_temp_elems(int64_t n);
bool radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt,
                      int64_t n, int begin, int end, uint32_t* tmp, cudaStream_t st);

// ---- lattice construction (build.cu) ----
sgp_status build_lattice(Lattice* L, const float* X, const float* ls);

// ---- MVM (mvm.cu) ----
// Make sure the lattice value buffers, splat partials and permuted-input buffer hold
// what a k-column product needs (allocated on `st`).
sgp_status ensure_lattice_values(Lattice* L, int k, cudaStream_t st);
// Columns of a row inside the operator for a caller's k (zero columns appended), and what
// this lattice uses (k itself once the padded buffers did not fit).
int padded_cols(int k);
int value_cols(const Lattice* L, int k);
// No room for zero columns: from now on this lattice's products go without, and the value
// buffers are given back.  False when it was so before.
bool give_up_padding(Lattice* L, cudaStream_t st);
// ensure_lattice_values for a public k-column product (value_cols columns).
sgp_status ensure_product(Lattice* L, int k, cudaStream_t st);
// Enqueue out = alpha * W B W^T V + beta * V on `st` (buffers must be ready: ensure_product,
// or ensure_lattice_values when internal).  With internal = false, V and out are the
// caller's [n][k] in the caller's point order (V is first permuted into locality order);
// with internal = true both are [n][k] in locality order (CG; 16-byte aligned rows or k <=
// 2).  When `ev` is given, ev[0] / ev[1] are recorded around the blur passes.  tree_k > 0:
// the column count that shapes the huge vertices' sums (k otherwise).  Returns the number of
// blur passes.
int enqueue_mvm(const Lattice* L, const float* V, int k, int blur, float alpha, float beta,
                float* out, cudaStream_t st, cudaEvent_t* ev = nullptr, bool internal = false,
                double* dot_partial = nullptr, int tree_k = 0);
// out = alpha K V (V and out in locality order) with the lattice values held in bf16 whatever
// the lattice's value type, in the lattice's own value buffers, which
// ensure_lattice_values(L, k) must have sized (a bf16 value takes half the room of an fp32
// one); every sum stays fp32.
void enqueue_mvm_bf16_values(const Lattice* L, const float* V, int k, int blur, float alpha,
                             float* out, cudaStream_t st);
// With internal = true and dot_partial set, the slice also writes per-block column sums of
// V * out (the CG's <p, A p>) to dot_partial[block][k]; this many blocks (grid-stride).
// tree_k as enqueue_mvm's.
int64_t slice_dot_blocks(const Lattice* L, int k, int tree_k);
constexpr int kVecBlocks = 8 * 152;  // blocks of the grid-stride column-owning kernels
// Bytes of work space one k-column product needs (value buffers, partials, permuted
// input, each rounded up to 256 bytes).
size_t mvm_work_bytes(const Lattice* L, int k);
// As enqueue_mvm (caller's point order) with all work space carved out of `work`
// (mvm_work_bytes(L, k) bytes, 256-byte aligned); allocates nothing.
void enqueue_mvm_into(const Lattice* L, const float* V, int k, int blur, float alpha,
                      float beta, float* out, void* work, cudaStream_t st);
// Pieces of the operator for the backward: splat a locality-ordered Vp (rows of kp) and blur
// it (the result ends in the returned buffer, lat0 or lat1, of the handle's value type; kt
// as enqueue_mvm's tree_k; the blurred values are *scale times what the buffer holds); gather
// the caller's rows of k into locality-ordered rows of kp (two arrays: side by side, 2 kp
// columns); out (caller's order, rows of k) = alpha W lat, the first kp of lat's lat_cols columns.
void* enqueue_splat_blur(const Lattice* L, const float* Vp, int kp, int kt, int blur, void* lat0,
                         void* lat1, float* partial, cudaStream_t st, double* scale);
void enqueue_permute(const Lattice* L, const float* V, int k, int kp, float* Vp, cudaStream_t st);
void enqueue_permute_pair(const Lattice* L, const float* A, const float* B, int k, int kp,
                          float* out, cudaStream_t st);
bool blur_in_place(const Lattice* L);  // enqueue_splat_blur needs no second buffer (lat1)
void enqueue_slice_caller(const Lattice* L, const void* lat, int k, int kp, int lat_cols,
                          dfloat alpha, float* out, cudaStream_t st);
size_t lattice_value_bytes(const Lattice* L, int k);
// Full operator on the handle's stream, allocating value buffers when needed.
sgp_status run_mvm(Lattice* L, const float* V, int k, int blur, float alpha, float beta,
                   float* out);

// ---- Nystrom preconditioners of the CG (server: nystrom.cu + serve.cu; library: precond.cu) ----
constexpr int kMaxRank = 128;       // server requests (kb_* ring kernels)
constexpr int kMaxLibRank = 4096;   // library CG (ShiftedNystrom)

// Large-rank shifted Nystrom preconditioner of the library CG (precond.cu):
// P = B B^T + tau I with B B^T a rank-l Nystrom approximation of outputscale K~ (q power
// iterations) and tau = lambda_min(B^T B) + noise.
struct ShiftedNystrom {
  int l = 0, ld = 0;
  int64_t n = 0;
  float tau = 0.f;
  bool ok = false;
  // [n][ld] bf16 (the factor rounded to bf16; P is defined by these values), locality
  // order, padding columns zero
  void* B = nullptr;
  float* Minv = nullptr;   // [ld][ld] fp32 (tau I + B^T B)^-1 of the stored B, zero padded
  float* tpart = nullptr;  // [bt_splits][ld][16] B^T r partials
  float* tvec = nullptr;   // [ld][16]
  void* u = nullptr;       // [3][16][ld] bf16: Minv B^T r split in three bf16 parts
  void* r3 = nullptr;      // [ldr][64] bf16: r split in three bf16 parts (columns 16 p + c
                           // hold part p of column c; 48..63 zero)
  int* err = nullptr;      // set when a per-iteration kernel's bounded wait gave up
  int64_t ldr = 0;         // n rounded up to 64
  int bt_splits = 0;
  int64_t bt_rows = 0;
  int z_blocks = 0;
  // TMA maps: B as [n][ld] in 128 x 64 boxes (A of B u) and 64 x 64 boxes (A of B^T r),
  // u as [48][ld] in 48 x 64 boxes and r3 as [n][64] in 64 x 64 boxes
  CUtensorMap map_b_k, map_b_mn, map_u, map_r;
  std::vector<void*> ptrs;
  sgp_status build(Lattice* L, int rank, uint64_t seed, float noise, int blur, int power_iters,
                   cudaStream_t st);
  // partial rows apply() writes per column: one per block of the z kernel
  int64_t dot_blocks() const;
  // z = P^-1 r (r = rh + rl, locality order [n][k]) and per-block column sums of r z into
  // dot[block][c] (fp64).  split_ready: r3 already holds the split of columns 0..15 of r
  // (written by the CG's x, r update).
  void apply(const float* rh, const float* rl, int k, float* z, double* dot, cudaStream_t st,
             cudaEvent_t* ev = nullptr, bool split_ready = false) const;
  // SGP_ERR_CUDA when a per-iteration kernel gave up waiting (synchronizes st)
  sgp_status check(cudaStream_t st) const;
  void release(cudaStream_t st);
};

// Nystrom factor of the training block of a joint lattice's operator, for the GP
// posterior server: A = outputscale K~ restricted to the rows p with perm[p] < n_train
// (the other rows are masked: zero sketch rows, zero rows of Y and B).  The l sketch
// columns go through the lattice kp at a time (V, KV: [n][kp] device scratch, lattice
// values already sized for kp columns), so that no l-column value buffer is needed.
// Writes B (fp32 [n][ld], locality order, columns l..ld-1 zero) into Bh and
// (noise I + B^T B)^-1 (fp64 [l][l]) into Minv; scratch: nystrom_masked_scratch_bytes(l, n)
// device bytes.  Enqueued on st; *status_dev (device int) is set to 1 when a Cholesky
// pivot fails (the factor must then not be used); the caller reads it.
size_t nystrom_masked_scratch_bytes(int l, int64_t n);
sgp_status nystrom_build_masked(Lattice* L, int64_t n_train, int l, int ld, uint64_t seed,
                                float noise, int kp, float* V, float* KV, float* Bh,
                                double* Minv, void* scratch, int* status_dev, cudaStream_t st);

// ---- backward (backward.cu) ----
sgp_status run_mvm_backward(Lattice* L, const float* X, const float* ls, const float* V,
                            const float* G, int k, int blur, float alpha, int grad, float* dV,
                            float* dX, float* dls);

// ---- CG (cg.cu) ----
// Device buffers that receive the CG coefficients of every column for the Lanczos
// quadrature: alpha_j / beta_j of column c at [j][cols] for j < cap, ||b_c|| and the
// iteration count per column.  cols: what the solver rounds k up to (padded_cols(k), or k
// itself where memory is short).
struct LanczosRecord {
  int cols;
  double* alpha;
  double* beta;
  int cap;
  double* bnorm;
  int* iters;
};
// precond_rank > 0: preconditioned CG with a rank-precond_rank Nystrom preconditioner
// (not with a Lanczos record, which needs the plain CG's coefficients).
sgp_status run_cg(Lattice* L, const float* B, int k, int blur, float noise, float tol,
                  int max_iter, float* X, int* iters, double* rel_res, int precond_rank = 0,
                  uint64_t seed = 0, const LanczosRecord* rec = nullptr,
                  double* history = nullptr);
// log det(outputscale K~ + noise I) by stochastic Lanczos quadrature over the probe
// columns Z (device [n][s], caller's order); quad (host [s], may be null) receives each
// probe's ||z||^2 e1^T log(T) e1 (lanczos.cu).
sgp_status run_logdet(Lattice* L, const float* Z, int s, float noise, int max_lanczos,
                      float tol, double* logdet, double* quad);

__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Exclusive block scan of one value per thread; returns the block total in *total.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_sums[32];
  __shared__ uint32_t block_total;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  const int nwarps = blockDim.x >> 5;
  if (warp == 0) {
    uint32_t s = lane < nwarps ? warp_sums[lane] : 0u;
    uint32_t si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, si, o);
      if (lane >= o) si += t;
    }
    if (lane < nwarps) warp_sums[lane] = si - s;
    if (lane == 31) block_total = si;  // nwarps <= 32
  }
  __syncthreads();
  const uint32_t res = warp_sums[warp] + inc - v;
  if (total) *total = block_total;
  __syncthreads();
  return res;
}

// Per-column sums of per-thread fp64 partials inside one block, for kernels whose threads
// own VEC consecutive columns of one row: thread t owns columns (t % G) VEC .. + VEC - 1
// of block row t / G, with G = k / VEC threads per row and blockDim.x a multiple of G.
// The block's column sums go to out[0..k), rows in order (the order is part of the CG's
// results).  Every thread of the block must call it; k <= blockDim.x.
template <int VEC>
__device__ __forceinline__ void block_column_sums(const double (&acc)[VEC], int k, double* out) {
  __shared__ double s[256 * VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) s[threadIdx.x * VEC + j] = acc[j];
  __syncthreads();
  const int rows = (int)blockDim.x / (k / VEC);
  if ((int)threadIdx.x < k) {
    double t = 0.0;
    int r = 0;
    for (; r + 8 <= rows; r += 8) {  // loads ahead of the additions
      double x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = s[(r + q) * k + threadIdx.x];
#pragma unroll
      for (int q = 0; q < 8; ++q) t += x[q];
    }
    for (; r < rows; ++r) t += s[r * k + threadIdx.x];
    out[threadIdx.x] = t;
  }
}

// Whether ||r|| / ||b|| = sqrt(rr) / bnorm (fp64) is at most tol or not finite.  Decided in
// fp32 unless the two are within 1e-4 of each other (or out of fp32's range): a square root
// and a division in fp64 are some 60 dependent operations of a narrow pipe, 2 us.
__device__ __forceinline__ bool cg_stops(double rr, double bnorm, float tol) {
  const float r = (float)rr, b = (float)bnorm;
  const float lim = tol * b * (tol * b);
  if (r > 1e-30f && r < 1e30f && lim < 1e30f && lim > 1e-30f) {
    if (r > lim * 1.0002f) return false;
    if (r < lim * 0.9998f) return true;
  }
  const double rel = sqrt(rr) / bnorm;
  return rel <= (double)tol || !isfinite(rel);
}

// ---- double-float arithmetic -------------------------------------------------------
// FP64 throughput on this part is a small fraction of FP32, so quantities that need more
// than fp32 precision per element (CG iterate and residual, dot-product accumulation) are
// kept as unevaluated sums hi + lo of two fp32 numbers and updated with error-free
// transformations: TwoSum (Knuth), FastTwoSum (Dekker, |a| >= |b|) and TwoProd through a
// fused multiply-add.  The _rn intrinsics keep the compiler from contracting or
// reordering the steps.  About 48 significant bits.

__device__ __forceinline__ dfloat df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ dfloat df_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ dfloat df_two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
// (a.hi + a.lo) + (b.hi + b.lo)
__device__ __forceinline__ dfloat df_add(dfloat a, dfloat b) {
  const dfloat s = df_two_sum(a.hi, b.hi);
  const float e = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return df_fast_two_sum(s.hi, e);
}
// (a.hi + a.lo) * b
__device__ __forceinline__ dfloat df_mul_f(dfloat a, float b) {
  const dfloat p = df_two_prod(a.hi, b);
  return df_fast_two_sum(p.hi, __fmaf_rn(a.lo, b, p.lo));
}
// (a.hi + a.lo) x with one rounding of the result, for factors: an fp32 factor alone would put its
// own rounding error, up to 6e-8, on every value alike.  a.lo = 0 but where the blur leaves a
// power of the centre tap to the factor; infinities stay what a.hi x makes them.
__device__ __forceinline__ float df_times(dfloat a, float x) {
  const float low = a.lo * x, high = a.hi * x;
  return a.lo != 0.f && !isinf(low) ? __fmaf_rn(a.hi, x, low) : high;
}
__device__ __forceinline__ dfloat df_from_double(double x) {
  const float hi = (float)x;
  return {hi, (float)(x - (double)hi)};
}
// (double)x by integer operations (conversions share the narrow fp64 pipe).
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), e = (u >> 23) & 255u;
  if (e - 1u >= 254u) return (u << 1) == 0 ? __hiloint2double((int)u, 0) : (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))),
                          (int)(u << 29));
}
__device__ __forceinline__ double df_to_double(dfloat a) { return widen(a.hi) + widen(a.lo); }

// Threads per block for the column-owning kernels: a whole number of rows of G threads (k <=
// 256, so at least k of them).  caller_k < k: what k was rounded up from, where the sums may
// follow it.  One thread a row means 256 additions in order a block (13 us), so three
// columns rounded up to four keep the 85 rows they would have apart (log determinant of one
// point, 3 probes: 544 us with 256 rows, 422 with 85).
inline int column_block_threads(int k, int vec, int caller_k) {
  const int G = k / vec;
  return G * (G == 1 && caller_k < k ? 256 / caller_k : 256 / G);
}

}  // namespace sgp
