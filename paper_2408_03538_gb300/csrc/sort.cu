// Prefix sums and a stable LSD radix sort of (uint32 or uint64 key, int32 value) pairs.
//
// Used by the BVH build (Morton keys, Sec. 4.4) and by the splat rasteriser: depth order of the splats,
// then the (splat, tile) pairs by tile (front-to-back order of Eq. 4).
#include "common.cuh"
#include "internal.h"

namespace prtgs {

// ------------------------------------------------------------------------------------------
// Three-phase prefix sum over uint32: per-block totals, a scan of the block totals in one
// block, then per-block scans with their offsets.
// ------------------------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* smem_warp, uint32_t& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) smem_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < (int)(blockDim.x >> 5) ? smem_warp[lane] : 0u;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += y;
    }
    smem_warp[lane] = w;  // inclusive warp totals
  }
  __syncthreads();
  total = smem_warp[(blockDim.x >> 5) - 1];
  uint32_t before = warp > 0 ? smem_warp[warp - 1] : 0u;
  __syncthreads();
  return before + x - v;
}

// in[i], or in[idx[i]] with an index
__device__ __forceinline__ uint32_t scan_in(const uint32_t* in, const int32_t* idx, int64_t i) {
  return in[idx ? (int64_t)idx[i] : i];
}

// Up to kScanSmall elements in one block (one launch; three launches of the general form take longer than
// the sums themselves there: a frame of 4,000 splats, with two scans, 64 us and 70; of 8,000 103 and 101; one block for
// 16,000 150 and 127).
constexpr int kScanSmall = 8192;
__global__ void __launch_bounds__(1024) k_scan_small(const uint32_t* in, const int32_t* __restrict__ idx, uint32_t* out,
                                                     int n, int exclusive, uint32_t* __restrict__ total, uint32_t cap) {
  __shared__ uint32_t sw[32];
  constexpr int kItems = kScanSmall / 1024;
  const int base = threadIdx.x * kItems;
  uint32_t v[kItems];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    v[k] = base + k < n ? scan_in(in, idx, base + k) : 0u;
    s += v[k];
  }
  uint32_t sum;
  uint32_t run = block_exclusive_scan(s, sw, sum);
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    if (base + k < n) out[base + k] = exclusive ? run : run + v[k];
    run += v[k];
  }
  if (threadIdx.x == 0 && total) *total = min(sum, cap);
}

__global__ void k_scan_reduce(const uint32_t* __restrict__ in, const int32_t* __restrict__ idx, int64_t n,
                              uint32_t* __restrict__ block_sums) {
  __shared__ uint32_t sw[32];
  int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k)
    if (base + k < n) s += scan_in(in, idx, base + k);
  uint32_t total;
  block_exclusive_scan(s, sw, total);
  if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

__global__ void k_scan_block_sums(uint32_t* __restrict__ sums, int64_t nb, uint32_t* __restrict__ grand_total,
                                  uint32_t cap) {
  __shared__ uint32_t sw[32];
  uint32_t carry = 0;
  for (int64_t base = 0; base < nb; base += blockDim.x) {
    int64_t i = base + threadIdx.x;
    uint32_t v = i < nb ? sums[i] : 0u;
    uint32_t total;
    uint32_t ex = block_exclusive_scan(v, sw, total);
    if (i < nb) sums[i] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0 && grand_total) *grand_total = min(carry, cap);
}

__global__ void k_scan_apply(const uint32_t* in, const int32_t* __restrict__ idx, uint32_t* out, int64_t n,
                             const uint32_t* __restrict__ block_offsets, int exclusive) {
  __shared__ uint32_t sw[32];
  int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = (base + k < n) ? scan_in(in, idx, base + k) : 0u;
    s += v[k];
  }
  uint32_t total;
  uint32_t run = block_exclusive_scan(s, sw, total) + block_offsets[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    if (base + k < n) out[base + k] = exclusive ? run : run + v[k];
    run += v[k];
  }
}

size_t scan_workspace(int64_t n) {
  int64_t nb = (n + kScanTile - 1) / kScanTile;
  return align_up(sizeof(uint32_t) * (size_t)(nb > 0 ? nb : 1));
}

// idx (nullable): sums of in[idx[i]] (out must then not be in); total (nullable): the grand total, at most cap.
int scan_u32(const uint32_t* in, uint32_t* out, int64_t n, bool exclusive, uint32_t* total, void* ws,
             cudaStream_t stream, const int32_t* idx, uint32_t cap) {
  if (n <= 0) {
    if (total) cudaMemsetAsync(total, 0, sizeof(uint32_t), stream);
    return PRTGS_OK;
  }
  int64_t nb = (n + kScanTile - 1) / kScanTile;
  uint32_t* sums = static_cast<uint32_t*>(ws);
  if (n <= kScanSmall) {
    k_scan_small<<<1, 1024, 0, counted(stream)>>>(in, idx, out, (int)n, exclusive ? 1 : 0, total, cap);
    PRTGS_CHECK_LAUNCH();
    return PRTGS_OK;
  }
  k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, counted(stream)>>>(in, idx, n, sums);
  k_scan_block_sums<<<1, 1024, 0, counted(stream)>>>(sums, nb, total, cap);
  k_scan_apply<<<(unsigned)nb, kScanThreads, 0, counted(stream)>>>(in, idx, out, n, sums, exclusive ? 1 : 0);
  PRTGS_CHECK_LAUNCH();
  return PRTGS_OK;
}

// ------------------------------------------------------------------------------------------
// Stable LSD radix sort, digits of at most 8 bits. One pass = digit histograms per tile of 4,096 (or
// 2,048 64-bit) keys, their prefix sums, and a stable scatter: a warp ranks its own contiguous part of the tile
// (eight ballots, one per bit, counters in shared memory, no block barrier), the tile is put in digit order in
// shared memory, and runs of one digit leave it as coalesced writes. 25 M pairs in two passes, the second writing
// 12 bytes a pair: 383 us at three blocks an SM; 515 with __match_any_sync, whose time grows with the distinct
// digits of a round; 483 with the values loaded after the ranks; 659 at two blocks, 447 at four (which spill).
// Up to kSelfTiles tiles a scatter block sums the histograms itself, which saves three launches a pass (a BVH build of
// 262k keys, 128 tiles, 171 us and 179 with the scan; of 524k, 256 tiles, 255 and 251; a frame of 300k splats and 964k
// pairs, 236 tiles, 203 and 219). Up to kSmallSort keys are sorted over all digits in one launch (4,096 keys of a BVH
// 72 us and 80; 8,192 in one block 97 and 84).
// The element count may live on the device (d_count), so the whole sort can be enqueued
// without a host round trip; tiles past the count do no work.
// ------------------------------------------------------------------------------------------
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSelfTiles = 256;
constexpr int kSmallSort = 4096;
template <class K>
struct SortShape {
  static constexpr int kItems = sizeof(K) == 8 ? 8 : 16;
  static constexpr int kTile = kSortThreads * kItems;
};

__device__ __forceinline__ int64_t sort_count(const uint32_t* d_count, int64_t capacity) {
  if (!d_count) return capacity;
  int64_t c = (int64_t)*d_count;
  return c < capacity ? c : capacity;
}

// A sorted key with its value's 32 low bits behind it.
template <class K>
__device__ __forceinline__ uint64_t wide_key(K k, float low) {
  return ((uint64_t)k << 32) | __float_as_uint(low);
}

// Digit counts of a tile. Its keys are all loaded before the first count: loads between the shared-memory atomics wait
// for them (25 M keys in two passes 140 us, 61 like this; four private histograms per block change nothing).
// hist: [tile][256] when self (the scatter blocks sum it), else [256][tile] for one exclusive scan.
template <class K>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const K* __restrict__ keys, int64_t capacity,
                                                             const uint32_t* d_count, int shift, unsigned mask, int n_tiles,
                                                             int self, uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t n = sort_count(d_count, capacity);
  const int64_t base = (int64_t)blockIdx.x * SortShape<K>::kTile;
  K key[SortShape<K>::kItems];
#pragma unroll
  for (int r = 0; r < SortShape<K>::kItems; ++r) {
    const int64_t i = base + r * kSortThreads + threadIdx.x;
    key[r] = i < n ? keys[i] : (K)0;
  }
#pragma unroll
  for (int r = 0; r < SortShape<K>::kItems; ++r)
    if (base + r * kSortThreads + threadIdx.x < n) atomicAdd(&h[(unsigned)(key[r] >> shift) & mask], 1u);
  __syncthreads();
  if (self) hist[(int64_t)blockIdx.x * 256 + threadIdx.x] = h[threadIdx.x];
  else if (threadIdx.x <= mask) hist[(int64_t)threadIdx.x * n_tiles + blockIdx.x] = h[threadIdx.x];
}

// Ranks of a warp's keys (round by round, in order) among the warp's keys of the same digit; cnt: the warp's
// 256 counters, zero before, the digit counts after.
template <class K, int ITEMS>
__device__ __forceinline__ void warp_ranks(const K (&key)[ITEMS], int rounds, int64_t first, int64_t n, int shift,
                                           unsigned mask, uint32_t* cnt, unsigned (&rank)[ITEMS]) {
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (r >= rounds) break;  // uniform
    const bool valid = first + r * 32 + lane < n;
    const unsigned digit = (unsigned)(key[r] >> shift) & mask;
    unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int bit = 0; bit < 8; ++bit) {
      const unsigned ones = __ballot_sync(0xffffffffu, (digit >> bit) & 1u);
      peers &= (digit >> bit) & 1u ? ones : ~ones;
    }
    const int leader = __ffs(peers) - 1;  // (an invalid lane's peers are the valid lanes of its digit, or none)
    unsigned old = 0;
    if (valid && lane == leader) {
      old = cnt[digit];
      cnt[digit] = old + __popc(peers);
    }
    rank[r] = __shfl_sync(0xffffffffu, old, leader & 31) + __popc(peers & lt_mask);
    __syncwarp();
  }
}

template <class K>
__global__ void __launch_bounds__(kSortThreads, 3) k_radix_scatter(const K* __restrict__ keys_in,
                                                                const int32_t* __restrict__ vals_in,
                                                                K* __restrict__ keys_out, int32_t* __restrict__ vals_out,
                                                                int64_t capacity, const uint32_t* d_count, int shift,
                                                                unsigned mask, int n_tiles, int self,
                                                                const uint32_t* __restrict__ hist,
                                                                const float* __restrict__ low,
                                                                uint64_t* __restrict__ wide_out) {
  constexpr int ITEMS = SortShape<K>::kItems, TILE = SortShape<K>::kTile;
  __shared__ K skey[TILE];
  __shared__ int32_t sval[TILE];
  __shared__ uint32_t cnt[kSortWarps][256];
  __shared__ uint32_t dstart[256];
  __shared__ int64_t gofs[256];
  __shared__ uint32_t sw[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t n = sort_count(d_count, capacity);
  const int64_t base = (int64_t)blockIdx.x * TILE;
  if (base >= n) return;  // uniform over the block
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) cnt[w][tid] = 0;
  const int64_t first = base + warp * 32 * ITEMS;
  K key[ITEMS];
  unsigned rank[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int64_t i = first + r * 32 + lane;
    key[r] = i < n ? keys_in[i] : (K)0;
  }
  int32_t val[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int64_t i = first + r * 32 + lane;
    val[r] = i < n ? (vals_in ? vals_in[i] : (int32_t)i) : 0;
  }
  __syncthreads();
  warp_ranks<K, ITEMS>(key, ITEMS, first, n, shift, mask, cnt[warp], rank);
  __syncthreads();
  uint32_t run = 0;  // this thread's digit: counts in front of each warp, and in all
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    const uint32_t c = cnt[w][tid];
    cnt[w][tid] = run;
    run += c;
  }
  uint32_t all;
  const uint32_t ds = block_exclusive_scan(run, sw, all);
  int64_t gbase;
  if (self) {
    uint32_t total = 0, before = 0;
#pragma unroll 8
    for (int t = 0; t < n_tiles; ++t) {
      const uint32_t c = hist[(int64_t)t * 256 + tid];
      total += c;
      before += t < (int)blockIdx.x ? c : 0u;
    }
    gbase = (int64_t)block_exclusive_scan(total, sw, all) + before;
  } else {
    gbase = tid <= mask ? hist[(int64_t)tid * n_tiles + blockIdx.x] : 0;
  }
  dstart[tid] = ds;
  gofs[tid] = gbase - ds;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (first + r * 32 + lane < n) {
      const unsigned d = (unsigned)(key[r] >> shift) & mask;
      const uint32_t lp = dstart[d] + cnt[warp][d] + rank[r];
      skey[lp] = key[r];
      sval[lp] = val[r];
    }
  }
  __syncthreads();
  const int m = (int)(n - base < TILE ? n - base : TILE);
  for (int i = tid; i < m; i += kSortThreads) {
    const K k = skey[i];
    const int64_t dst = gofs[(unsigned)(k >> shift) & mask] + i;
    if (dst < n) {  // always true when the histograms are consistent
      const int32_t v = sval[i];
      if (wide_out) wide_out[dst] = wide_key(k, low[v]);
      else keys_out[dst] = k;
      vals_out[dst] = v;
    }
  }
}

// Every digit of up to kSmallSort pairs in one block.
template <class K>
__global__ void __launch_bounds__(kSortThreads) k_radix_small(const K* __restrict__ keys_in,
                                                              const int32_t* __restrict__ vals_in,
                                                              K* __restrict__ keys_out, int32_t* __restrict__ vals_out,
                                                              int64_t capacity, const uint32_t* d_count, int begin_bit,
                                                              int end_bit, int width, const float* __restrict__ low,
                                                              uint64_t* __restrict__ wide_out) {
  constexpr int ITEMS = kSmallSort / kSortThreads;
  extern __shared__ unsigned char sort_smem[];
  K* skey = reinterpret_cast<K*>(sort_smem);
  int32_t* sval = reinterpret_cast<int32_t*>(skey + kSmallSort);
  __shared__ uint32_t cnt[kSortWarps][256];
  __shared__ uint32_t dstart[256];
  __shared__ uint32_t sw[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = (int)sort_count(d_count, capacity);
  const int rounds = (n + kSortThreads - 1) / kSortThreads;  // per warp: a contiguous part of the pairs
  const int first = warp * 32 * rounds;
  K key[ITEMS];
  int32_t val[ITEMS];
  unsigned rank[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int i = first + r * 32 + lane;
    const bool on = r < rounds && i < n;
    key[r] = on ? keys_in[i] : (K)0;
    val[r] = on ? (vals_in ? vals_in[i] : i) : 0;
  }
  for (int bit = begin_bit; bit < end_bit; bit += width) {
    const unsigned mask = (1u << min(width, end_bit - bit)) - 1u;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) cnt[w][tid] = 0;
    __syncthreads();
    warp_ranks<K, ITEMS>(key, rounds, first, n, bit, mask, cnt[warp], rank);
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
      const uint32_t c = cnt[w][tid];
      cnt[w][tid] = run;
      run += c;
    }
    uint32_t all;
    dstart[tid] = block_exclusive_scan(run, sw, all);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (r < rounds && first + r * 32 + lane < n) {
        const unsigned d = (unsigned)(key[r] >> bit) & mask;
        const uint32_t lp = dstart[d] + cnt[warp][d] + rank[r];
        skey[lp] = key[r];
        sval[lp] = val[r];
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const int i = first + r * 32 + lane;
      if (r < rounds && i < n) {
        key[r] = skey[i];
        val[r] = sval[i];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int i = first + r * 32 + lane;
    if (r < rounds && i < n) {
      if (wide_out) wide_out[i] = wide_key(key[r], low[val[r]]);
      else keys_out[i] = key[r];
      vals_out[i] = val[r];
    }
  }
}

template <class K>
static int64_t sort_tiles(int64_t capacity) {
  const int64_t t = (capacity + SortShape<K>::kTile - 1) / SortShape<K>::kTile;
  return t > 1 ? t : 1;
}

size_t radix_sort_workspace(int64_t capacity) {
  const int64_t tiles = sort_tiles<uint64_t>(capacity);  // the smaller tiles: enough for either key
  return align_up(sizeof(uint32_t) * 256 * (size_t)tiles) + scan_workspace(256 * tiles);
}

template <class K>
static int radix_sort_t(const K* keys_x, const int32_t* vals_x, K* keys_f, int32_t* vals_f, K* keys_y, int32_t* vals_y,
                        int64_t capacity, const uint32_t* d_count, int begin_bit, int end_bit, void* ws,
                        cudaStream_t stream, const float* low = nullptr, uint64_t* wide = nullptr) {
  if (capacity <= 0) return PRTGS_OK;
  const int bits = end_bit > begin_bit ? end_bit - begin_bit : 1;
  const int passes = (bits + 7) / 8;
  const int width = (bits + passes - 1) / passes;
  if (capacity <= kSmallSort) {
    const int smem = kSmallSort * (int)(sizeof(K) + sizeof(int32_t));
    cudaFuncSetAttribute(k_radix_small<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    k_radix_small<K><<<1, kSortThreads, smem, counted(stream)>>>(keys_x, vals_x, keys_f, vals_f, capacity, d_count,
                                                                 begin_bit, begin_bit + bits, width, low, wide);
    PRTGS_CHECK_LAUNCH();
    return PRTGS_OK;
  }
  const int tiles = (int)sort_tiles<K>(capacity);
  const int self = tiles <= kSelfTiles;
  Carver c(ws);
  uint32_t* hist = c.take<uint32_t>(256 * (size_t)tiles);
  void* scan_ws = c.take<char>(scan_workspace(256 * (int64_t)tiles));
  const K* ksrc = keys_x;
  const int32_t* vsrc = vals_x;
  for (int p = 0; p < passes; ++p) {
    // the last pass must land in the final buffers
    const bool to_f = ((passes - 1 - p) % 2) == 0;
    K* kdst = to_f ? keys_f : keys_y;
    int32_t* vdst = to_f ? vals_f : vals_y;
    const int shift = begin_bit + width * p;
    const int w = begin_bit + bits - shift < width ? begin_bit + bits - shift : width;
    const unsigned mask = (1u << w) - 1u;
    k_radix_hist<K><<<tiles, kSortThreads, 0, counted(stream)>>>(ksrc, capacity, d_count, shift, mask, tiles, self, hist);
    if (!self) {
      const int rc = scan_u32(hist, hist, ((int64_t)mask + 1) * tiles, true, nullptr, scan_ws, stream);
      if (rc != PRTGS_OK) return rc;
    }
    k_radix_scatter<K><<<tiles, kSortThreads, 0, counted(stream)>>>(ksrc, vsrc, kdst, vdst, capacity, d_count, shift, mask,
                                                                    tiles, self, hist, low, p == passes - 1 ? wide : nullptr);
    PRTGS_CHECK_LAUNCH();
    ksrc = kdst;
    vsrc = vdst;
  }
  return PRTGS_OK;
}

int radix_sort_pairs(const uint64_t* keys_x, const int32_t* vals_x, uint64_t* keys_f, int32_t* vals_f,
                     uint64_t* keys_y, int32_t* vals_y, int64_t capacity, const uint32_t* d_count, int begin_bit,
                     int end_bit, void* ws, cudaStream_t stream) {
  return radix_sort_t<uint64_t>(keys_x, vals_x, keys_f, vals_f, keys_y, vals_y, capacity, d_count, begin_bit, end_bit, ws,
                                stream);
}

int radix_sort_pairs(const uint32_t* keys_x, const int32_t* vals_x, uint32_t* keys_f, int32_t* vals_f,
                     uint32_t* keys_y, int32_t* vals_y, int64_t capacity, const uint32_t* d_count, int begin_bit,
                     int end_bit, void* ws, cudaStream_t stream, const float* low, uint64_t* wide) {
  return radix_sort_t<uint32_t>(keys_x, vals_x, keys_f, vals_f, keys_y, vals_y, capacity, d_count, begin_bit, end_bit, ws,
                                stream, low, wide);
}

}  // namespace prtgs
