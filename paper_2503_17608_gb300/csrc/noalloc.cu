// Stable partition of slot indices by key without any device allocation.
//
// The step loop partitions track slots by next action with per-tile key
// counts kept in memory the context allocates. This file offers the same
// partition as a stand-alone call whose only working memory is a fixed
// file-scope device array, for callers that must not allocate device memory
// themselves: code that runs while another framework's caching allocator
// owns the device memory, or latency-critical host loops that cannot afford
// cudaMalloc/cudaFree (cudaFree synchronises the whole device).
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "celer_gb.h"

namespace {

constexpr int kNaThreads = 256;
constexpr int kNaPer = 16;                          // consecutive slots per thread: one 16-byte load of keys
constexpr int kNaTile = kNaThreads * kNaPer;        // slots per tile
constexpr uint32_t kNaMaxSlots = 1u << 20;          // largest n accepted
constexpr int kNaMaxKeys = 16;                      // largest n_keys accepted
constexpr uint32_t kNaMaxTiles = kNaMaxSlots / kNaTile;
constexpr int kNaMaxDevices = 64;

// Keys per tile, tile major: 256 x 16 x 4 bytes = 16 KiB, held by every
// device that loads the library.
__device__ __align__(256) uint32_t g_partition_scratch[kNaMaxKeys * kNaMaxTiles];

// Device address of g_partition_scratch per device ordinal, looked up once
// per process. cudaDeviceReset destroys the context this address belongs to,
// so the entry point must not be called on a device after it was reset.
uint32_t* g_scratch_ptr[kNaMaxDevices] = {};
std::mutex g_scratch_mutex;

cudaError_t scratch_for_current_device(uint32_t** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kNaMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_ptr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_partition_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = static_cast<uint32_t*>(ptr);
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

// The partition is bound by launches and latencies (5 MB at the largest n, 0.7
// us at the copy rate): two launches, or one when a single tile holds every
// slot, and no pass over the counts on its own. Tiles of 4,096 slots make at
// most 256 x 16 counts, few enough for every block of the second launch to sum
// those of the tiles before it. 2^20 slots and 9 keys: 12.3 us a call; with
// tiles of 256 slots and a scan by one block in between 44.8 us.

// A thread's 16 consecutive keys, 0xFF past the end and for keys out of range.
__device__ __forceinline__ void load_keys(const uint8_t* keys, uint32_t n, int n_keys, uint32_t first, uint8_t (&k)[kNaPer]) {
  uint32_t w[4];
  if (first + kNaPer <= n && (reinterpret_cast<uintptr_t>(keys) & 15u) == 0u) {
    const uint4 v = *reinterpret_cast<const uint4*>(keys + first);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
#pragma unroll
    for (int i = 0; i < kNaPer; ++i) k[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
  } else {
#pragma unroll
    for (int i = 0; i < kNaPer; ++i) k[i] = first + i < n ? keys[first + i] : (uint8_t)0xFF;
  }
#pragma unroll
  for (int i = 0; i < kNaPer; ++i)
    if ((int)k[i] >= n_keys) k[i] = 0xFF;
}

// Key counts of 16 keys in eight words of two 16-bit fields: word j holds keys
// 2j and 2j + 1 (a block's counts, at most 4,096, fit).
__device__ __forceinline__ void count_keys(const uint8_t (&k)[kNaPer], uint32_t (&h)[8]) {
  unsigned long long lo = 0, hi = 0;  // keys 0-7 and 8-15, 8 bits each (at most 16 per thread)
#pragma unroll
  for (int i = 0; i < kNaPer; ++i) {
    const unsigned long long one = 1ull << (8 * (k[i] & 7));
    lo += k[i] < 8 ? one : 0ull;
    hi += (k[i] & 0xF8) == 8 ? one : 0ull;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t a = (uint32_t)(lo >> (16 * j)) & 0xFFFFu, b = (uint32_t)(hi >> (16 * j)) & 0xFFFFu;
    h[j] = (a & 0xFFu) | (a >> 8 << 16);
    h[4 + j] = (b & 0xFFu) | (b >> 8 << 16);
  }
}

// First launch: keys per tile (every (tile, key) entry is written, so the
// scratch needs no clearing between calls).
__global__ void __launch_bounds__(kNaThreads) k_na_count(const uint8_t* keys, uint32_t n, int n_keys, uint32_t* counts) {
  __shared__ uint32_t s_cnt[kNaThreads / 32][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint8_t k[kNaPer];
  load_keys(keys, n, n_keys, blockIdx.x * kNaTile + threadIdx.x * kNaPer, k);
  uint32_t h[8];
  count_keys(k, h);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t sum = __reduce_add_sync(0xffffffffu, h[j]);  // both fields at once: no carry, at most 512 each
    if (lane == j) s_cnt[warp][j] = sum;
  }
  __syncthreads();
  if (threadIdx.x < kNaMaxKeys) {
    const int j = threadIdx.x >> 1, sh = (threadIdx.x & 1) * 16;
    uint32_t sum = 0;
#pragma unroll
    for (int w = 0; w < kNaThreads / 32; ++w) sum += (s_cnt[w][j] >> sh) & 0xFFFFu;
    counts[blockIdx.x * kNaMaxKeys + threadIdx.x] = sum;
  }
}

// Second launch: every block sums the counts of the tiles before its own (and
// of all tiles, for the keys' offsets), sorts its tile by key in shared
// memory and writes each key's run to its place. Slots whose key is skip_key
// (or not below n_keys) are left out of perm; offsets[k] = first position of
// key k, offsets[n_keys] = the number of slots whose key is below n_keys.
__global__ void __launch_bounds__(kNaThreads) k_na_scatter(const uint8_t* keys, uint32_t n, int n_keys, uint32_t n_tiles,
                                                           const uint32_t* counts, int skip_key, uint32_t* perm,
                                                           uint32_t* offsets) {
  constexpr int kWarps = kNaThreads / 32, kRows = kNaThreads / kNaMaxKeys;
  __shared__ uint32_t s_row[2][kRows][kNaMaxKeys];
  __shared__ uint32_t s_warp[kWarps][8];
  __shared__ uint16_t s_pos[kNaMaxKeys][kNaThreads];
  __shared__ uint32_t s_sorted[kNaTile];
  __shared__ uint32_t s_global[kNaMaxKeys], s_local[kNaMaxKeys + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tile = blockIdx.x, first = tile * kNaTile + threadIdx.x * kNaPer;
  uint8_t k[kNaPer];
  load_keys(keys, n, n_keys, first, k);
  {  // counts of the tiles before this one, and of all tiles
    const uint32_t key = threadIdx.x % kNaMaxKeys, row = threadIdx.x / kNaMaxKeys;
    uint32_t before = 0, all = 0;
    if (n_tiles > 1) {
#pragma unroll 8
      for (uint32_t t = row; t < n_tiles; t += kRows) {
        const uint32_t v = counts[t * kNaMaxKeys + key];
        all += v;
        before += t < tile ? v : 0u;
      }
    }
    s_row[0][row][key] = before;
    s_row[1][row][key] = all;
  }
  uint32_t h[8], incl[8];
  count_keys(k, h);
#pragma unroll
  for (int j = 0; j < 8; ++j) incl[j] = h[j];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl[j], o);
      if (lane >= o) incl[j] += v;
    }
  if (lane == 31)
#pragma unroll
    for (int j = 0; j < 8; ++j) s_warp[warp][j] = incl[j];
  __syncthreads();
  if (warp == 0) {
    // one lane per key: the tile's runs, and their places
    const int key = lane & (kNaMaxKeys - 1);
    uint32_t mine = 0, before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) mine += (s_warp[w][key >> 1] >> (16 * (key & 1))) & 0xFFFFu;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      before += s_row[0][r][key];
      all += s_row[1][r][key];
    }
    if (n_tiles == 1) all = mine;
    uint32_t li = mine, gi = all;
#pragma unroll
    for (int o = 1; o < kNaMaxKeys; o <<= 1) {
      const uint32_t a = __shfl_up_sync(0xffffffffu, li, o, kNaMaxKeys), b = __shfl_up_sync(0xffffffffu, gi, o, kNaMaxKeys);
      if (key >= o) {
        li += a;
        gi += b;
      }
    }
    if (lane < kNaMaxKeys) {
      s_local[key] = li - mine;
      s_global[key] = gi - all + before;
      if (key == kNaMaxKeys - 1) s_local[kNaMaxKeys] = li;
      if (tile == 0) {
        if (key < n_keys) offsets[key] = gi - all;
        if (key == n_keys - 1) offsets[n_keys] = gi;
      }
    }
  }
  __syncthreads();
  // this thread's first place per key within the tile's sorted order
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint32_t p = incl[j] - h[j];
    for (int w = 0; w < warp; ++w) p += s_warp[w][j];
    s_pos[2 * j][threadIdx.x] = (uint16_t)(s_local[2 * j] + (p & 0xFFFFu));
    s_pos[2 * j + 1][threadIdx.x] = (uint16_t)(s_local[2 * j + 1] + (p >> 16));
  }
#pragma unroll
  for (int i = 0; i < kNaPer; ++i) {
    if (k[i] != 0xFF) {
      const uint16_t p = s_pos[k[i]][threadIdx.x]++;
      s_sorted[p] = ((uint32_t)k[i] << 16) | (threadIdx.x * kNaPer + i);
    }
  }
  __syncthreads();
  const uint32_t in_range = s_local[kNaMaxKeys];
  for (uint32_t i = threadIdx.x; i < in_range; i += kNaThreads) {
    const uint32_t v = s_sorted[i], key = v >> 16;
    if ((int)key != skip_key) perm[s_global[key] + (i - s_local[key])] = tile * kNaTile + (v & 0xFFFFu);
  }
}

}  // namespace

extern "C" celer_status celer_partition_keys_noalloc(const uint8_t* d_keys, uint64_t n, int n_keys, int skip_key,
                                                     uint32_t* d_perm, uint32_t* d_offsets, void* cuda_stream) {
  if (!d_offsets || (n > 0 && (!d_keys || !d_perm))) return CELER_ERR_INVALID;
  if (n > kNaMaxSlots || n_keys < 1 || n_keys > kNaMaxKeys || skip_key >= n_keys) return CELER_ERR_INVALID;
  // An error left pending by earlier work on this thread is not ours to
  // report or clear: launch nothing and leave it in place.
  if (cudaPeekAtLastError() != cudaSuccess) return CELER_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (n == 0) {  // every offset is 0; d_perm is not touched
    return cudaMemsetAsync(d_offsets, 0, sizeof(uint32_t) * (size_t)(n_keys + 1), s) == cudaSuccess ? CELER_OK
                                                                                              : CELER_ERR_CUDA;
  }
  uint32_t* scratch = nullptr;
  if (scratch_for_current_device(&scratch) != cudaSuccess) return CELER_ERR_CUDA;
  const uint32_t n_tiles = (uint32_t)((n + kNaTile - 1) / kNaTile);
  if (n_tiles > 1) k_na_count<<<n_tiles, kNaThreads, 0, s>>>(d_keys, (uint32_t)n, n_keys, scratch);
  k_na_scatter<<<n_tiles, kNaThreads, 0, s>>>(d_keys, (uint32_t)n, n_keys, n_tiles, scratch, skip_key, d_perm, d_offsets);
  // nothing was pending before the launches, so an error now is theirs
  return cudaGetLastError() == cudaSuccess ? CELER_OK : CELER_ERR_CUDA;
}
