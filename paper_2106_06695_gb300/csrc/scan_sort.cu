// Device-wide exclusive scan and stable LSD radix sort, used while numbering lattice
// vertices and grouping point/vertex incidences by vertex during the build.
#include "sgp_internal.cuh"

namespace sgp {
namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortBatches = 8;                       // 32-item batches per warp
constexpr int kSortTile = kSortThreads * kSortBatches;  // 4096 items per block
constexpr int kSortSelf = 128;  // up to this many blocks the scatter sums the histograms itself

__global__ void k_scan_reduce(const uint32_t* data, int64_t n,
                              uint32_t* __restrict__ block_sums) {
  pdl_enter();
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i)
    if (base + i < n) s += data[base + i];
  uint32_t total;
  block_exclusive_scan(s, &total);
  if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

// Exclusive scan in place of the rows of n sums, a block each.
__global__ void k_scan_top(uint32_t* __restrict__ block_sums, int64_t nb) {
  pdl_enter();
  block_sums += blockIdx.y * nb;
  uint32_t carry = 0;
  for (int64_t base = 0; base < nb; base += kScanTile) {
    const int64_t my = base + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      v[i] = (my + i < nb) ? block_sums[my + i] : 0u;
      s += v[i];
    }
    uint32_t tile_total;
    uint32_t run = carry + block_exclusive_scan(s, &tile_total);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
      if (my + i < nb) block_sums[my + i] = run;
      run += v[i];
    }
    carry += tile_total;
  }
}

// SELF: the block adds up the sums of the blocks before it, one a thread (up to kScanThreads
// blocks; a launch less than with k_scan_top, 2.5 us).
template <bool SELF>
__global__ void k_scan_down(uint32_t* __restrict__ data, int64_t n,
                            const uint32_t* block_sums,
                            uint32_t* __restrict__ total) {
  pdl_enter();
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = (base + i < n) ? data[base + i] : 0u;
    s += v[i];
  }
  uint32_t before;
  if (SELF) block_exclusive_scan(threadIdx.x < blockIdx.x ? block_sums[threadIdx.x] : 0u, &before);
  else before = block_sums[blockIdx.x];
  uint32_t mine;
  uint32_t run = before + block_exclusive_scan(s, &mine);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < n) data[base + i] = run;
    run += v[i];
  }
  if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1 && total) *total = before + mine;
}

// Digit counts of each block's items: [digit][block] for the scan, [block][digit] with SELF.
template <bool SELF>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t* keys,
                                                             int64_t n, int shift,
                                                             uint32_t* __restrict__ hist,
                                                             int64_t nblk) {
  pdl_enter();
  __shared__ uint32_t h[256];
  if (threadIdx.x < 256) h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kSortTile;
  uint32_t key[kSortBatches];
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b) {
    const int64_t e = base + b * kSortThreads + threadIdx.x;
    key[b] = e < n ? keys[e] : 0u;
  }
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b)
    if (base + b * kSortThreads + threadIdx.x < n) atomicAdd(&h[(key[b] >> shift) & 255u], 1u);
  __syncthreads();
  if (threadIdx.x < 256)
    hist[SELF ? (int64_t)blockIdx.x * 256 + threadIdx.x : (int64_t)threadIdx.x * nblk + blockIdx.x] =
        h[threadIdx.x];
}

// Stable scatter.  Each warp owns a contiguous run of kSortBatches * 32 items and ranks it in
// order, lanes with the same digit by lane within a batch; the items then go through shared
// memory in digit order, so that a block writes runs of 16 items of a digit instead of single
// ones.  Bound by the ranking (a match over the warp and a shared-memory update per 32 items).
// 460k items (113 blocks): 30 us a pass of 5 kernels before, 15 now; 10.5M: 128 and 134.
//
// offs: start of each digit's items of this block ([digit][block], scanned).  SELF: offs holds
// the counts ([block][digit], at most kSortSelf blocks) and the block adds up what it needs of
// them, 1.5 us in place of the three launches of a scan.
template <bool SELF>
__global__ void __launch_bounds__(kSortThreads)
    k_radix_scatter(const uint32_t* kin, const uint32_t* vin,
                    uint32_t* __restrict__ kout, uint32_t* __restrict__ vout, int64_t n, int shift,
                    const uint32_t* offs, int64_t nblk) {
  pdl_enter();
  __shared__ uint32_t cnt[kSortWarps][256];
  __shared__ uint32_t item[kSortTile];
  __shared__ uint32_t goff[256];  // global position of a digit's items minus the one in `item`
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tile = (int64_t)blockIdx.x * kSortTile;
  const int many = (int)(n - tile < kSortTile ? n - tile : kSortTile);
  const int own = warp * (kSortBatches * 32) + lane;  // of the warp's first batch, in the tile
  uint32_t key[kSortBatches], val[kSortBatches], rank[kSortBatches];
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b) {
    const bool in = own + b * 32 < many;
    key[b] = in ? kin[tile + own + b * 32] : 0u;
    val[b] = in ? vin[tile + own + b * 32] : 0u;
  }
  // digit q = threadIdx.x % 256: items of all blocks, and of the blocks before this one, in
  // half of the blocks (threadIdx.x / 256)
  uint32_t all = 0, before = 0;
  if (SELF) {
    const int q = threadIdx.x & 255;
#pragma unroll 16
    for (int b = threadIdx.x >> 8; b < (int)nblk; b += 2) {
      const uint32_t c = offs[b * 256 + q];
      all += c;
      if (b < (int)blockIdx.x) before += c;
    }
  }
  for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortThreads) (&cnt[0][0])[i] = 0u;
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b) {
    const bool in = own + b * 32 < many;
    const uint32_t dig = in ? (key[b] >> shift) & 255u : 256u;
    const unsigned peers = __match_any_sync(0xffffffffu, dig);
    const int first = __ffs(peers) - 1;
    uint32_t start = 0;
    if (in && lane == first) {
      start = cnt[warp][dig];
      cnt[warp][dig] = start + __popc(peers);
    }
    rank[b] = __shfl_sync(0xffffffffu, start, first) + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
  }
  __syncthreads();
  // counts before each warp, then positions in the tile and in the output
  uint32_t run = 0;
  if (threadIdx.x < 256) {
    for (int w = 0; w < kSortWarps; ++w) {
      const uint32_t c = cnt[w][threadIdx.x];
      cnt[w][threadIdx.x] = run;
      run += c;
    }
  }
  const uint32_t local = block_exclusive_scan(threadIdx.x < 256 ? run : 0u, nullptr);
  if (threadIdx.x < 256)
    for (int w = 0; w < kSortWarps; ++w) cnt[w][threadIdx.x] += local;
  if (SELF) {
    if (threadIdx.x >= 256) {  // halves together
      item[threadIdx.x & 255] = all;
      item[256 + (threadIdx.x & 255)] = before;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
      all += item[threadIdx.x];
      before += item[256 + threadIdx.x];
    }
    const uint32_t base = block_exclusive_scan(threadIdx.x < 256 ? all : 0u, nullptr);
    if (threadIdx.x < 256) goff[threadIdx.x] = base + before - local;
  } else if (threadIdx.x < 256) {
    goff[threadIdx.x] = offs[(int64_t)threadIdx.x * nblk + blockIdx.x] - local;
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b) {
    if (own + b * 32 >= many) continue;
    rank[b] += cnt[warp][(key[b] >> shift) & 255u];  // position in the tile, by digit
    item[rank[b]] = key[b];
  }
  __syncthreads();
  uint32_t to[kSortBatches];
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b) {
    const int i = b * kSortThreads + threadIdx.x;
    if (i >= many) continue;
    const uint32_t k = item[i];
    to[b] = goff[(k >> shift) & 255u] + (uint32_t)i;
    kout[to[b]] = k;
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b)
    if (own + b * 32 < many) item[rank[b]] = val[b];
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kSortBatches; ++b) {
    const int i = b * kSortThreads + threadIdx.x;
    if (i < many) vout[to[b]] = item[i];
  }
}

}  // namespace

size_t scan_temp_elems(int64_t n) { return (size_t)ceil_div(n > 0 ? n : 1, kScanTile); }

void exclusive_scan_u32(uint32_t* data, int64_t n, uint32_t* total, uint32_t* tmp,
                        cudaStream_t st) {
  if (n <= 0) {
    if (total) cudaMemsetAsync(total, 0, sizeof(uint32_t), st);
    return;
  }
  const int64_t nb = ceil_div(n, kScanTile);
  launch_pdl(k_scan_reduce, (unsigned)nb, kScanThreads, st, data, n, tmp);
  if (nb <= kScanThreads) {
    launch_pdl(k_scan_down<true>, (unsigned)nb, kScanThreads, st, data, n, tmp, total);
    note_launches(2);
    return;
  }
  launch_pdl(k_scan_top, 1, kScanThreads, st, tmp, nb);
  launch_pdl(k_scan_down<false>, (unsigned)nb, kScanThreads, st, data, n, tmp, total);
  note_launches(3);
}

void exclusive_scan_rows_u32(uint32_t* data, int rows, int64_t n, cudaStream_t st) {
  launch_pdl(k_scan_top, dim3(1, (unsigned)rows), kScanThreads, st, data, n);
  note_launches(1);
}

size_t radix_temp_elems(int64_t n) {
  const int64_t nblk = ceil_div(n > 0 ? n : 1, 2048);  // at least as many as the sort's blocks
  return (size_t)(256 * nblk) + scan_temp_elems(256 * nblk);
}

bool radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt,
                      int64_t n, int begin, int end, uint32_t* tmp, cudaStream_t st) {
  if (n <= 1 || begin >= end) return false;
  const int64_t nblk = ceil_div(n, kSortTile);
  const bool self = nblk <= kSortSelf;
  uint32_t* hist = tmp;
  uint32_t* scan_tmp = tmp + 256 * nblk;
  bool alt = false;
  for (int shift = begin; shift < end; shift += 8) {
    const uint32_t* kin = alt ? keys_alt : keys;
    const uint32_t* vin = alt ? vals_alt : vals;
    uint32_t* kout = alt ? keys : keys_alt;
    uint32_t* vout = alt ? vals : vals_alt;
    launch_pdl(self ? k_radix_hist<true> : k_radix_hist<false>, (unsigned)nblk, kSortThreads, st,
               kin, n, shift, hist, nblk);
    if (!self) exclusive_scan_u32(hist, 256 * nblk, nullptr, scan_tmp, st);
    launch_pdl(self ? k_radix_scatter<true> : k_radix_scatter<false>, (unsigned)nblk, kSortThreads,
               st, kin, vin, kout, vout, n, shift, hist, nblk);
    note_launches(2);
    alt = !alt;
  }
  return alt;
}

}  // namespace sgp
