// tile_sort.cuh -- the CTA body of the base case of GPU Multiway Mergesort
// (Sec. 4.3 "Internal Memory Sort"), shared by the whole-array base case and
// the segmented (batched) one: a tile of T = 1024 * WARPS consecutive keys is
// sorted on its own, producing a sorted run the K-way merge rounds start from.
//
// The paper's base case is a per-warp shearsort of a 32 x 32 grid, extended
// by bitonic merges between warps.  Here each lane sorts the 32 keys it loaded
// with an in-register sorting network, the warp finishes its 1024 keys with
// bitonic merges through conflict-free transposes in its share of the tile
// buffer (the row/column transposes of shearsort, swizzled), and the CTA
// merges the warps' blocks with the same conflict-free networks, in place.  HBM traffic: one coalesced 128-bit read and one coalesced
// 128-bit write of every key.
#pragma once

#include <type_traits>

#include "mms_common.cuh"
#include "mms_kernels.cuh"

namespace mms {

// Sorting network over a lane's 32 registers (ascending): Batcher's odd-even
// merge sort (K. E. Batcher, "Sorting networks and their applications",
// AFIPS 1968), 191 compare-exchanges in 15 stages against the bitonic
// sorter's 240.  Stage (p, k) of the network compares items x and x + k for
// x = j + i with j running from k mod p in steps of 2k and i from 0 to k - 1,
// whenever both lie in the same block of 2p items.  Every index is a
// compile-time constant once the loops are unrolled, so each compare-exchange
// is register to register; within a stage the mix's share of the pairs takes the
// multiply-add form (by their ordinal in the stage), as in the other networks.
template <typename KeyT, typename M>
__device__ __forceinline__ void lane_sort32(KeyT (&v)[32], const M& c) {
#pragma unroll
  for (int lp = 0; lp < 5; ++lp) {
#pragma unroll
    for (int lk = lp; lk >= 0; --lk) {
      const int p = 1 << lp, k = 1 << lk;
      const int j0 = k & (p - 1);                      // first j of the stage: k mod p
      int ord = 0;                                     // ordinal of the pair in its stage
#pragma unroll
      for (int x = 0; x < 31; ++x) {                   // x = j + i, j = j0 + 2kt, i < k
        if (x + k < 32 && x >= j0 && ((x - j0) & (2 * k - 1)) < k &&
            (x >> (lp + 1)) == ((x + k) >> (lp + 1))) {
          cas_mix(v[x], v[x + k], ord, c);
          ++ord;
        }
      }
    }
  }
}

// Blocked -> striped through `scratch` (aligned to a row, 1024 items), with the
// second half of every block of 2h rows read backwards (h a power of two, 1 ..
// 16).  On return register k of lane l holds item 32k + l of the sequence in
// which every block is its first h rows in order followed by its last h rows in
// reverse, each from column 31 down: a bitonic sequence when both halves are
// ascending, so an ascending half-cleaner cascade sorts it, with no per-lane
// directions.  A lane of a second half writes its row to the mirrored place
// (row l ^ (h - 1)), as 16-byte chunks XOR-swizzled by that place & 7; register k
// is then column l, or 31 - l, of row k.  The writes and the reads (32 distinct words of one row) have no
// bank conflicts.
template <typename KeyT>
__device__ __forceinline__ void blocked_to_striped_rev(KeyT (&v)[32], KeyT* scratch, int h,
                                                       int lane) {
  constexpr int E = Vec16<KeyT>::E;
  constexpr uint32_t SZ = sizeof(KeyT), RB = 32 * SZ;
  const uint32_t sb = smem_u32addr(scratch);
  const uint32_t place = (lane & h) ? lane ^ (h - 1) : lane;
  const uint32_t row = (sb + place * RB) ^ ((place & 7) << 4);
#pragma unroll
  for (int ch = 0; ch < 32 / E; ++ch) sts128(row ^ (ch << 4), &v[ch * E]);
  __syncwarp();
  // Column offsets: c[k] = lane, mirrored when k has bit h, swizzled by k & 7;
  // c[k] follows from c[k without its lowest bit] by one XOR.
  uint32_t mir[5];
#pragma unroll
  for (int b = 0; b < 5; ++b) mir[b] = (h >> b) & 1 ? 31 * SZ : 0u;
  uint32_t c[32];
  c[0] = sb ^ (lane * SZ);
#pragma unroll
  for (int k = 1; k < 32; ++k) {
    const int p = k & (k - 1);                                 // k without its lowest bit
    const int b = (k & -k) == 1 ? 0 : (k & -k) == 2 ? 1 : (k & -k) == 4 ? 2 : (k & -k) == 8 ? 3 : 4;
    c[k] = c[p] ^ mir[b] ^ (uint32_t)(E * ((k & 7) ^ (p & 7)) * SZ);
  }
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = lds_at<KeyT>(c[k] + k * RB);
  __syncwarp();
}

// Blocked layout -> `out` (aligned to a row, 1024 items) in order: the rows
// go out swizzled, come back as consecutive 16-byte chunks (chunk 32q + lane in
// registers), and those are stored in their places; all conflict-free.
template <typename KeyT>
__device__ __forceinline__ void blocked_to_linear(KeyT (&v)[32], KeyT* out, int lane) {
  constexpr int E = Vec16<KeyT>::E;
  constexpr int CPR = 32 / E;                                  // chunks of a row: 8 or 16
  constexpr uint32_t RB = 32 * sizeof(KeyT);
  const uint32_t sb = smem_u32addr(out);
  const uint32_t row = (sb + lane * RB) ^ ((lane & 7) << 4);
#pragma unroll
  for (int ch = 0; ch < CPR; ++ch) sts128(row ^ (ch << 4), &v[ch * E]);
  __syncwarp();
#pragma unroll
  for (int q = 0; q < CPR; ++q) {
    const uint32_t r = (uint32_t)(q * (32 / CPR)) + (uint32_t)lane / CPR;   // row of chunk 32q + lane
    lds_chunk(sb + r * RB + ((((uint32_t)lane % CPR) ^ (r & 7)) << 4), &v[q * E]);
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < CPR; ++q) sts128(sb + ((32 * q + lane) << 4), &v[q * E]);
}

template <typename KeyT, bool XIN>
__device__ __forceinline__ KeyT xform_in(KeyT k) {
  if constexpr (XIN) return (KeyT)f32_to_ordered((uint32_t)k);
  return k;
}
// Writes the sorted tile src[0, m) to global memory: one TMA bulk store of the
// 16-byte-aligned body, plain stores for the < 16-byte tail.  Every thread
// must call it (it contains a barrier).
template <typename KeyT>
__device__ __forceinline__ void cta_store_tile(const KeyT* src, KeyT* dst, int m) {
  constexpr int E = 16 / sizeof(KeyT);
  // A destination off the 16-byte grid (a segment of a batch may start
  // anywhere) is written with plain coalesced stores.
  const int body = (((uintptr_t)dst & 15u) == 0) ? m / E * E : 0;
  fence_proxy_async_smem();
  __syncthreads();
  if (threadIdx.x == 0 && body > 0) bulk_s2g_and_wait(dst, src, (unsigned)(body * sizeof(KeyT)));
  for (int i = body + (int)threadIdx.x; i < m; i += blockDim.x) dst[i] = src[i];
}

// Everything after the load: v (32 keys per lane, any assignment) to the sorted
// tile in shared memory, first min(T, n - base) entries of the returned buffer.
// Each lane sorts its 32 keys (a row).  Then a level merges pairs of sorted
// blocks of 32h keys by one bitonic cascade -- strides of 32 and more between
// registers in the striped layout, the rest inside the lane -- with h = 1 .. 16
// inside each warp's 1024 keys and h = 32, 64, .. across the CTA:
//   - warp levels come to the striped layout by a transpose in the warp's own
//     part of the buffer that reads every second half backwards;
//   - CTA levels by writing the blocks out in order and reading the window of
//     the warp's output block (its co-ranks found by the merge-path search).
// The tile is sorted in place in one buffer of 1024 * WARPS keys (aligned to
// 1024 bytes): a barrier separates a CTA level's reads from its writes, and
// half the shared memory lets four CTAs of 8-byte keys on an SM.  A short tile
// is padded with the all-ones key (pads sort last, and one that ties with a
// real key is bit-identical to it) and takes only the CTA levels its keys need.
//
// The levels are loops, not unrolled.  With 8-byte keys all of them share one
// body: unrolled they were 161 KB of code, and a warp waited for its next
// instruction longer than for anything else (2.05 of 6.5 warps per issue;
// with four warps to a CTA no two warps of a scheduler run the same code at the
// same time).  2 * 10^7 8-byte keys: 396 us unrolled, 279 us as one 49 KB body,
// 262 us with every pair's second key taken from the sums (kTileMad64Pairs).
// With 4-byte keys the warp levels and the CTA levels are a body each, and the
// CTA levels use the directed last stages, which store in order at once:
// 16.8 * 10^6 keys 117 us unrolled, 104 us as one body, 101 us as two, 98.5 us so.
// Bound at that size: issue 69%, ALU 72%, shared-memory wavefronts 75% (4-byte), ALU 86%
// before the sums (8-byte).
// xout: write the last level's output as floats.
template <typename KeyT, int WARPS>
__device__ __forceinline__ KeyT* tile_sort_smem(KeyT (&v)[32], long long n, long long base,
                                                bool xout, unsigned char* smem_raw) {
  constexpr int T = WARPS * kBlockItems;
  KeyT* buf = reinterpret_cast<KeyT*>(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  KeyT* own = buf + warp * kBlockItems;
  const long long rem = n - base;
  const int m = rem >= T ? T : (int)rem;
  const TileMix c = mad_ones<TileMix>();

  // From the striped layout, bitonic blocks of 2h rows, to sorted rows of the blocked layout.
  auto network = [&](int h, auto flip) {
    if (h >= 16) striped_stage<16>(v, c);            // strides 32h .. 32, at most 512
    if (h >= 8) striped_stage<8>(v, c);
    if (h >= 4) striped_stage<4>(v, c);
    if (h >= 2) striped_stage<2>(v, c);
    striped_stage<1>(v, c);
    striped_to_blocked(v, own, 32, lane);
    blocked_stages<decltype(flip)::value>(v, lane, c);   // strides 16 .. 1
  };
  auto to_floats = [&]() {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = (KeyT)ordered_to_f32((uint32_t)v[j]);
  };
  // Loads the window of the warp's block of the merge of sequences of len keys.
  auto load_window = [&](int len) {
    const int first = warp * kBlockItems & ~(2 * len - 1);   // the pair the block lies in
    const int d0 = warp * kBlockItems - first;
    const KeyT* A = buf + first;
    const KeyT* B = A + len;
    int a0, a1;
    warp_corank_pair(A, len, B, len, d0, kBlockItems, lane, a0, a1);
    warp_load_bitonic_full(A + a0, a1 - a0, B + (d0 - a0), v, lane);
  };

  lane_sort32(v, c);
  // The previous tile of a persistent CTA has been read out of shared memory
  // before the warps use it as transpose scratch.
  __syncthreads();
  if constexpr (sizeof(KeyT) == 8) {
#pragma unroll 1
    for (int h = 1;; h *= 2) {
      if (h <= 16) {
        blocked_to_striped_rev(v, own, h, lane);
      } else {
        const bool last = 32 * h >= m;               // uniform over the CTA
        blocked_to_linear(v, own, lane);
        __syncthreads();
        if (last) return buf;
        load_window(32 * h);
        __syncthreads();
      }
      network(h, std::false_type{});
    }
  } else {
#pragma unroll 1
    for (int h = 1; h <= 16; h *= 2) {
      blocked_to_striped_rev(v, own, h, lane);
      network(h, std::false_type{});
    }
    if (kBlockItems >= m && xout) to_floats();
    blocked_to_linear(v, own, lane);
#pragma unroll 1
    for (int len = kBlockItems; len < m; len *= 2) {
      __syncthreads();
      load_window(len);
      __syncthreads();
      network(16, std::true_type{});
      warp_store_block<KeyT>(own, kBlockItems, v, lane, xout && 2 * len >= m);
    }
    __syncthreads();
    return buf;
  }
}

// Whether this warp lies past the last sequence that a short tile of m keys
// comes to in its levels; it then has kept all of tile_sort_smem's barriers.  300
// keys in a tile of 8192: 7.3 -> 6.4 us, and more with other tiles on the SM (a batch of
// 700 arrays of 2^8 to 2^14 keys: 47.8 -> 41.2 us).  4-byte tiles pay nothing for the
// question, 8-byte tiles 2%: whole arrays of those (SHORT false), whose last tile alone is
// short, do not ask it.
__device__ __forceinline__ bool tile_idle_warp(int m) {
  int region = kBlockItems;
  while (region < m) region *= 2;
  if (warp_index() * kBlockItems < region) return false;
  __syncthreads();
  for (int len = kBlockItems; len < m; len *= 2) {
    __syncthreads();
    __syncthreads();
  }
  __syncthreads();
  return true;
}

// Loads this warp's 1024 keys of the tile of 1024 * WARPS keys that starts at
// `base` (32 per lane, any assignment; pads past n), through the float order
// transform when XIN.
template <typename KeyT, int WARPS, bool XIN>
__device__ __forceinline__ void tile_load(const KeyT* in, long long n, long long base,
                                          KeyT (&v)[32]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wbase = base + (long long)warp * kBlockItems;
  const long long rem = n - wbase;
  const int cnt = rem <= 0 ? 0 : (rem >= kBlockItems ? kBlockItems : (int)rem);

  using V = Vec16<KeyT>;
  constexpr int NV = 32 / V::E;          // 16-byte vectors per lane
  if (cnt == kBlockItems && ((uintptr_t)(in + wbase) & 15u) == 0) {
    const typename V::T* src = reinterpret_cast<const typename V::T*>(in + wbase);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const typename V::T x = src[q * 32 + lane];
      KeyT t[V::E];
      V::unpack(x, t);
#pragma unroll
      for (int c = 0; c < V::E; ++c) v[q * V::E + c] = xform_in<KeyT, XIN>(t[c]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
#pragma unroll
      for (int c = 0; c < V::E; ++c) {
        const int e = q * 32 * V::E + lane * V::E + c;
        v[q * V::E + c] = e < cnt ? xform_in<KeyT, XIN>(in[wbase + e]) : key_pad<KeyT>();
      }
    }
  }
}

// Sorts the tile of 1024 * WARPS keys of in[0, n) that starts at `base` into
// the same positions of out (in == out allowed): the CTA body of the base case.
template <typename KeyT, int WARPS, bool XIN, bool SHORT>
__device__ __forceinline__ void tile_sort_tile(const KeyT* in, KeyT* out, long long n,
                                               long long base, bool xout,
                                               unsigned char* smem_raw) {
  constexpr int T = WARPS * kBlockItems;
  const long long rem = n - base;
  const int m = rem >= T ? T : (int)rem;
  if (!SHORT || !tile_idle_warp(m)) {
    KeyT v[32];
    tile_load<KeyT, WARPS, XIN>(in, n, base, v);
    tile_sort_smem<KeyT, WARPS>(v, n, base, xout, smem_raw);
  }
  cta_store_tile(reinterpret_cast<KeyT*>(smem_raw), out + base, m);
}

// Base case of the key-value sort: 32-bit keys (floats through the order
// transform when XIN) are read and turned into unique 64-bit composites
// (ordered key << 32 | pos0 + position in the array), whose ascending order is the
// stable key order; tiles of composites are then sorted like 64-bit keys.
template <int WARPS, bool XIN, bool SHORT>
__device__ __forceinline__ void tile_sort_composite_tile(const uint32_t* in,
                                                         uint64_t* out, long long n,
                                                         long long base, long long pos0,
                                                         unsigned char* smem_raw) {
  constexpr int T = WARPS * kBlockItems;
  const long long trem = n - base;
  const int m = trem >= T ? T : (int)trem;
  if (!SHORT || !tile_idle_warp(m)) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long wbase = base + (long long)warp * kBlockItems;
    const long long rem = n - wbase;
    const int cnt = rem <= 0 ? 0 : (rem >= kBlockItems ? kBlockItems : (int)rem);
    uint64_t v[32];
    if (cnt == kBlockItems && ((uintptr_t)(in + wbase) & 15u) == 0) {
      const uint4* src = reinterpret_cast<const uint4*>(in + wbase);
  #pragma unroll
      for (int q = 0; q < 8; ++q) {
        const uint4 x = src[q * 32 + lane];
        const uint32_t k[4] = {x.x, x.y, x.z, x.w};
  #pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t key = XIN ? f32_to_ordered(k[c]) : k[c];
          const uint64_t pos = (uint64_t)(pos0 + wbase + q * 128 + lane * 4 + c);
          v[q * 4 + c] = ((uint64_t)key << 32) | pos;
        }
      }
    } else {
  #pragma unroll
      for (int q = 0; q < 8; ++q) {
  #pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int e = q * 128 + lane * 4 + c;
          uint64_t x = key_pad<uint64_t>();
          if (e < cnt) {
            const uint32_t key = XIN ? f32_to_ordered(in[wbase + e]) : in[wbase + e];
            x = ((uint64_t)key << 32) | (uint64_t)(pos0 + wbase + e);
          }
          v[q * 4 + c] = x;
        }
      }
    }
    tile_sort_smem<uint64_t, WARPS>(v, n, base, false, smem_raw);
  }
  cta_store_tile(reinterpret_cast<uint64_t*>(smem_raw), out + base, m);
}

}  // namespace mms
