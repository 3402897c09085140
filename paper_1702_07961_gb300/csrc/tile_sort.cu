// tile_sort.cu -- the whole-array base case: one CTA per tile, running the
// CTA body of tile_sort.cuh.
#include "tile_sort.cuh"

namespace mms {

// The sort's first kernel clears the workspace's status word (errors are recorded
// by later kernels only): a memset of its own cost a launch of 2 us and more.
__device__ __forceinline__ void clear_status_word(int* status) {
  if (status != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *status = kDevOk;
}

template <typename KeyT, int WARPS, bool XIN, bool XOUT>
__global__ void __launch_bounds__(WARPS * 32, (TileMinBlocks<KeyT, WARPS>::value))
    tile_sort_kernel(const KeyT* in, KeyT* out, long long n, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  constexpr int T = WARPS * kBlockItems;
  griddep_wait();                                 // the keys: whatever ran before on the stream
  griddep_launch_dependents();                    // the first splitter may get resident early
  clear_status_word(status);
  tile_sort_tile<KeyT, WARPS, XIN, sizeof(KeyT) == 4>(in, out, n, (long long)blockIdx.x * T, XOUT, smem_raw);
}

// Base case of the key-value sort: 32-bit keys -> sorted tiles of unique
// 64-bit composites (ordered key << 32 | position in the array).
template <int WARPS, bool XIN>
__global__ void __launch_bounds__(WARPS * 32, (TileMinBlocks<uint64_t, WARPS>::value))
    tile_sort_composite_kernel(const uint32_t* in, uint64_t* out, long long n,
                               int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  constexpr int T = WARPS * kBlockItems;
  griddep_wait();
  griddep_launch_dependents();
  clear_status_word(status);
  tile_sort_composite_tile<WARPS, XIN, false>(in, out, n, (long long)blockIdx.x * T, 0, smem_raw);
}

size_t tile_sort_smem_bytes(int key_bytes, int warps) {
  return (size_t)key_bytes * warps * kBlockItems;
}

template <typename KeyT, int WARPS, bool XIN, bool XOUT>
static cudaError_t launch_tile_sort_t(const void* in, void* out, long long n, int* status,
                                      cudaStream_t s) {
  constexpr size_t smem = sizeof(KeyT) * WARPS * kBlockItems;   // no attribute: at most 48 KB
  static_assert(smem <= 48 * 1024, "a larger tile needs the shared-memory attribute");
  const long long T = (long long)WARPS * kBlockItems;
  const unsigned grid = (unsigned)((n + T - 1) / T);
  return launch_k(tile_sort_kernel<KeyT, WARPS, XIN, XOUT>, dim3(grid), dim3(WARPS * 32), smem, s,
                  true, static_cast<const KeyT*>(in), static_cast<KeyT*>(out), n, status);
}

template <int WARPS>
static cudaError_t launch_tile_sort_w(int key_bytes, bool xin, bool xout, const void* in, void* out,
                                      long long n, int* status, cudaStream_t s) {
  if (!valid_tile_warps(key_bytes, WARPS)) return cudaErrorInvalidValue;
  if constexpr (WARPS != 2) {
    if (key_bytes == 4) {
      if (xin && xout) return launch_tile_sort_t<uint32_t, WARPS, true, true>(in, out, n, status, s);
      if (xin) return launch_tile_sort_t<uint32_t, WARPS, true, false>(in, out, n, status, s);
      return launch_tile_sort_t<uint32_t, WARPS, false, false>(in, out, n, status, s);
    }
  }
  if constexpr (WARPS != 8) return launch_tile_sort_t<uint64_t, WARPS, false, false>(in, out, n, status, s);
  return cudaErrorInvalidValue;
}

template <int WARPS, bool XIN>
static cudaError_t launch_composite_t(const void* in, void* out, long long n, int* status,
                                      cudaStream_t s) {
  constexpr size_t smem = sizeof(uint64_t) * WARPS * kBlockItems;
  static_assert(smem <= 48 * 1024, "a larger tile needs the shared-memory attribute");
  const long long T = (long long)WARPS * kBlockItems;
  const unsigned grid = (unsigned)((n + T - 1) / T);
  return launch_k(tile_sort_composite_kernel<WARPS, XIN>, dim3(grid), dim3(WARPS * 32), smem, s,
                  true, static_cast<const uint32_t*>(in), static_cast<uint64_t*>(out), n, status);
}

cudaError_t launch_tile_sort_composite(int tile_warps, bool xin, const void* keys32, void* out64,
                                       long long n, int* status, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (tile_warps == 4)
    return xin ? launch_composite_t<4, true>(keys32, out64, n, status, s) : launch_composite_t<4, false>(keys32, out64, n, status, s);
  if (tile_warps == 2)
    return xin ? launch_composite_t<2, true>(keys32, out64, n, status, s) : launch_composite_t<2, false>(keys32, out64, n, status, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_tile_sort(int key_bytes, int tile_warps, bool xin, bool xout, const void* in,
                             void* out, long long n, int* status, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  switch (tile_warps) {
    case 2: return launch_tile_sort_w<2>(key_bytes, xin, xout, in, out, n, status, s);
    case 4: return launch_tile_sort_w<4>(key_bytes, xin, xout, in, out, n, status, s);
    case 8: return launch_tile_sort_w<8>(key_bytes, xin, xout, in, out, n, status, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mms
