// splitter.cu -- the whole-array splitter: one warp per output tile of a
// merge round, running splitter_row of splitter.cuh.
#include "splitter.cuh"

namespace mms {

// Warps per splitter CTA: on GB300 2 and 4 measure the same, 8 is 1 to 3%
// slower (10^8 u32 keys, and 2 * 10^7 u64).
constexpr int kSplitterWarps = 4;

// Rows up to which the splitter is launched with programmatic stream serialization.
// Behind a merge pass it then starts on SMs whose memory is set up as shared
// memory, and a row's samples of a step do not fit the L1 that is left: from
// 2^23 keys on the gap saved costs more than it gives (10^8 u32 keys 2669 -> 2539
// us without it, 16.8 * 10^6 451 -> 404, 2^23 256 -> 215; 2^21 93 either way; 2^20 78
// without, 66 with).
constexpr long long kSplitterPdlTiles = 192;

// Rows from which 8-byte keys with more than 4 runs take stride halving (K2 = 0).  Up to
// about one wave of warps a row's chain of steps counts, and windows take a third of the steps;
// beyond it the sectors, and 32 M samples of 8 bytes a step are twice a halving level's
// share.  Sorts of u64 keys, us, windows / halving, random and 1% swapped keys: 6 * 10^6 (1465 rows) 355 / 379, 357 / 365;
// 1.2 * 10^7 (2930) 709 / 721, 664 / 643; 1.6 * 10^7 (3907) 910 / 909, 863 / 807; 10^8 6338 / 6309, 5431 / 4967.
// 4-byte keys stay with windows: 10^8 random u32 keys' splitters 264 / 307.
constexpr unsigned kHalvingRows = 3584;

// CTAs per SM the splitter is compiled for: 40 warps (48 registers), 32 with more than 16
// runs, whose window is twice as large.  The search waits for loads, so warps count: left
// to itself the compiler takes 40 to 64 and spills some (6 * 10^6 pairs of 4-byte keys 411 -> 414
// us, 10^8 u32 keys' splitters 262 -> 266); for 48 warps it spills more (268).
constexpr int splitter_ctas(int k2) { return k2 == 32 ? 8 : 10; }   // 48 registers halving, too

template <typename KeyT, int K2, typename Idx>
__global__ void __launch_bounds__(32 * kSplitterWarps, splitter_ctas(K2))
    splitter_kernel(const KeyT* in, long long n, long long run_len, int K,
                    long long S, unsigned tpg, unsigned ntiles, long long* table) {
  griddep_wait();                                 // the runs are the previous kernel's output
  griddep_launch_dependents();
  const unsigned t = blockIdx.x * kSplitterWarps + (threadIdx.x >> 5);
  if (t >= ntiles) return;                        // uniform over the warp
  splitter_row<KeyT, K2, Idx>(in, n, run_len, K, S, t / tpg, t % tpg, table + (long long)t * K);
}

template <typename KeyT, int K2>
static cudaError_t launch_k2(const void* in, long long n, long long run_len, int K, long long S,
                             unsigned tpg, unsigned ntiles, long long* table, cudaStream_t s,
                             bool pdl) {
  const unsigned grid = (ntiles + kSplitterWarps - 1) / kSplitterWarps;
  const KeyT* kin = static_cast<const KeyT*>(in);
  if (n < (K2 == 0 ? 1ll << 30 : 1ll << 31))      // counts and positions fit 32 bits
    return launch_k(splitter_kernel<KeyT, K2, int>, dim3(grid), dim3(32 * kSplitterWarps), 0, s, pdl, kin, n, run_len,
                    K, S, tpg, ntiles, table);
  if constexpr (sizeof(KeyT) == 8 && K2 > 4)
    return cudaErrorInvalidValue;                 // so many rows have taken K2 = 0
  else
    return launch_k(splitter_kernel<KeyT, K2, long long>, dim3(grid), dim3(32 * kSplitterWarps), 0, s, pdl, kin, n,
                    run_len, K, S, tpg, ntiles, table);
}

template <typename KeyT>
static cudaError_t launch_key(const void* in, long long n, long long run_len, int K, long long S,
                              unsigned tpg, unsigned ntiles, long long* table, cudaStream_t s, bool pdl) {
  if constexpr (sizeof(KeyT) == 8)
    if (K > 4 && ntiles >= kHalvingRows)
      return launch_k2<KeyT, 0>(in, n, run_len, K, S, tpg, ntiles, table, s, pdl);
  switch (pow2_ceil(K)) {
    case 2: return launch_k2<KeyT, 2>(in, n, run_len, K, S, tpg, ntiles, table, s, pdl);
    case 4: return launch_k2<KeyT, 4>(in, n, run_len, K, S, tpg, ntiles, table, s, pdl);
    case 8: return launch_k2<KeyT, 8>(in, n, run_len, K, S, tpg, ntiles, table, s, pdl);
    case 16: return launch_k2<KeyT, 16>(in, n, run_len, K, S, tpg, ntiles, table, s, pdl);
    default: return launch_k2<KeyT, 32>(in, n, run_len, K, S, tpg, ntiles, table, s, pdl);
  }
}

// One output tile per warp.
cudaError_t launch_splitter(int key_bytes, long long S, const void* in, long long n,
                            long long run_len, int K, long long* table, cudaStream_t s, bool pdl) {
  const long long ntiles = num_tiles(S, n, run_len, K);
  if (ntiles <= 0) return cudaSuccess;
  if (K < 2 || K > kMaxFanout || ntiles > 0x7FFFFFFFll) return cudaErrorInvalidValue;
  if (ntiles > kSplitterPdlTiles) pdl = false;
  long long tpg = tiles_per_group(S, run_len, K);
  if (tpg > 0xFFFFFFFFll) tpg = 0xFFFFFFFFll;     // more than the grid: every tile is in group 0
  if (key_bytes == 4) return launch_key<uint32_t>(in, n, run_len, K, S, (unsigned)tpg, (unsigned)ntiles, table, s, pdl);
  return launch_key<uint64_t>(in, n, run_len, K, S, (unsigned)tpg, (unsigned)ntiles, table, s, pdl);
}

}  // namespace mms
