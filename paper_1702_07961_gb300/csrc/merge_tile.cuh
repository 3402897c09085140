// merge_tile.cuh -- the CTA body of one K-way merge round (Sec. 4.2 "I/O
// Efficient Merging", Sec. 5.1 I/O analysis), shared by the whole-array merge
// pass and the segmented (batched) merge pass.
//
// One CTA produces one output tile of S = 1024 * WARPS items of its group of K
// runs.  The splitter table gives, for the tile's start and end, the pivot in
// every run (Sec. 4.1), so the tile's inputs are K contiguous segments whose
// lengths sum to S.  The CTA:
//   1. stages the K segments into shared memory with 1-D TMA bulk copies
//      (cp.async.bulk between 16-byte boundaries, one mbarrier; plain loads
//      only where a boundary would lie past the end of the array), so every
//      input byte is read from HBM once;
//   2. merges them along a binary merge tree of ceil(log2 K') levels, K' <= K
//      the runs the group holds (the paper's minBlockHeap has the same
//      levels), one level at a time: every
//      tree node of the level (a pair of sequences) is cut into 1024-item
//      output blocks, the blocks of the level are dealt to the warps (its
//      full-size blocks first, then the small last blocks of its nodes,
//      which a smaller network merges), and a CTA barrier separates the
//      levels.  A node's output is written into the
//      span its segments were staged in, alternating between two buffers by
//      level; every segment span carries 16 items of slack (a node that merges has
//      two segments at least) so that a node's last, partial block can use its
//      output region as transpose space.
//      Each block is merged by the conflict-free warp bitonic block merge;
//   3. writes the tile, from registers (4-byte keys) or with one TMA bulk
//      store, so every output byte is written once: 2 * S * sizeof(key) bytes
//      of HBM traffic per tile.
//
// What bounds it (16.8 * 10^6 f32 keys, K = 16, 97.6 -> 94.6 us): issue 60%,
// ALU 57%, shared-memory wavefronts 55% of peak; the largest stall is the level
// barriers (2.5 of about 9.4 warp cycles per instruction issued), and shared
// memory holds three CTAs an SM.  2 * 10^7 u64 keys, K = 8, 182 -> 172 us:
// issue 47%, ALU 68%.
#pragma once

#include "mms_common.cuh"
#include "mms_kernels.cuh"
#include "splitter.cuh"

namespace mms {

// Control area after a merge CTA's mbarrier, written by the planning warps for
// the whole CTA (ints): four scalars, four per tree level (its first item, the
// end of its network items, the end of its items, unused), and the items, 16
// bytes each.  An item is one output block of a node:
//   x: offset of the node's sequence A | its length << 16,   y: the same of B,
//   z: offset of the node's output | the block's start in it << 16,   w: the block's size.
constexpr int kCtlLevels = 0, kCtlWant = 2, kCtlErr = 3;
constexpr int kCtlLevel0 = 4;                        // level lv at kCtlLevel0 + 4 * lv
constexpr int kCtlItems = 32;
constexpr int kMaxItems = 72;                        // 71 at most: 8 per level, and one per node, with K = 32
constexpr int kCtlInts = kCtlItems + 4 * kMaxItems;
constexpr size_t kMergeCtlBytes = sizeof(int) * kCtlInts;

// Shared-memory geometry of a merge CTA for fanout K.  X: the staged
// segments, each at a 16-byte aligned span start R_r (up to 2E-2 items of
// alignment slack and 16 items of transpose slack per segment: a node that runs a
// network has two segments at least, and its last block may use 31 items past
// its end), and the odd tree levels' inputs; Y: the same spans, one buffer per
// level parity.  Three CTAs fit an SM up to K = 32.
template <typename KeyT, int WARPS>
struct MergeGeom {
  static constexpr int E = Vec16<KeyT>::E;
  static constexpr int S = WARPS * kBlockItems;
  static constexpr int kSlack = 16;
  __host__ __device__ static constexpr int cap(int K) {
    return S + (K * (2 * E - 2 + kSlack) + E - 1) / E * E + E;
  }
  // control block: mbarrier (16 bytes with padding), then the control area
  __host__ __device__ static constexpr size_t bytes(int K) {
    return sizeof(KeyT) * 2 * (size_t)cap(K) + 16 + kMergeCtlBytes;
  }
  // The partition variant adds, after the control area, the offset and the length of every
  // staged segment and its pivot rows: row b (b <= WARPS) holds, per segment,
  // the items of the tile's first 1024 b outputs.
  static constexpr size_t kRowBytes = sizeof(int) * 32 * (WARPS + 3);
  __host__ __device__ static constexpr size_t bytes_partition(int K) { return bytes(K) + kRowBytes; }
};
// An SM's 228 KB, of which every CTA takes 1 KB beside its own.
static_assert(3 * (MergeGeom<uint32_t, 8>::bytes(kMaxFanout) + 1024) <= 228 * 1024, "three CTAs an SM");
static_assert(3 * (MergeGeom<uint64_t, 4>::bytes(kMaxFanout) + 1024) <= 228 * 1024, "three CTAs an SM");

// Segment bounds of the tile in run `lane` (lanes < K): from the pivot rows,
// or the run's ends for a group's first / last tile.  Warp 0 issues these
// loads first thing, so they are in flight across the CTA's setup.
__device__ __forceinline__ void merge_tile_pivots(long long n, long long run_len, int K,
                                                  long long g, long long j,
                                                  const long long* lo_row,
                                                  const long long* hi_row, int S,
                                                  int lane, long long& lo, long long& hi) {
  const long long gstart = g * run_len * K;
  const long long grest = n - gstart;
  const long long gsize = grest < run_len * K ? grest : run_len * K;
  long long rlen = n - (gstart + (long long)lane * run_len);
  rlen = rlen < 0 ? 0 : (rlen > run_len ? run_len : rlen);
  lo = 0;
  hi = 0;
  if (lane < K) {
    lo = (j == 0) ? 0 : lo_row[lane];
    hi = ((j + 1) * S < gsize) ? hi_row[lane] : rlen;   // not the group's last tile
  }
}

// Plans output tile j of group g, whose segment bounds in run `lane` are lo
// and hi (from merge_tile_pivots), and stages its segments into `stage`: one
// warp, one lane per run and one per merge-tree node.  Starts the bulk copies
// on `bar`, loads the items no bulk copy covers, and writes the items and
// the scalars (levels, tile size, error) into `ctl`; the caller's CTA
// barrier publishes the plain loads and the table, the barrier's phase the
// copies.  On segment bounds that fail their check, ctl's error scalar is set
// and nothing is staged.
// `part` splits the work between two warps that both call this with the same
// bounds: bit 0 stages the segments (and writes the tile size and error
// scalars), bit 1 writes the items (and the levels' bounds).  The
// two halves need only the segment lengths and spans, which both compute, so a
// CTA can start the copies and build the table at the same time.
template <typename KeyT, int WARPS>
__device__ __forceinline__ void merge_plan_warp(const KeyT* in, long long n,
                                                long long run_len, int K, long long g,
                                                long long j, long long lo, long long hi, int S,
                                                KeyT* stage, int* ctl, uint64_t* bar, int lane,
                                                int part = 3, int* segs = nullptr) {
  using G = MergeGeom<KeyT, WARPS>;
  constexpr int E = G::E;
  const long long gstart = g * run_len * K;
  const long long grest = n - gstart;
  const long long gsize = grest < run_len * K ? grest : run_len * K;
  const bool act = lane < K;
  const long long rstart = gstart + (long long)lane * run_len;
  long long rlen = n - rstart;
  rlen = rlen < 0 ? 0 : (rlen > run_len ? run_len : rlen);
  // The pivot rows must describe segments inside their runs whose lengths
  // sum to this tile's size; anything else would overrun the staging buffer.
  // Each segment is checked against S first, so the sum fits 32 bits.
  const long long want = (gsize - j * S) < S ? (gsize - j * S) : S;
  const bool bad_seg = act && (lo < 0 || hi < lo || hi > rlen || hi - lo > S);
  const int len32 = (act && !bad_seg) ? (int)(hi - lo) : 0;
  const int sum = (int)__reduce_add_sync(0xffffffffu, (unsigned)len32);
  const bool bad = __any_sync(0xffffffffu, bad_seg) || sum != want || K > kMaxFanout || K < 2 ||
                   S > G::S || S < kBlockItems || (smem_u32addr(stage) & 15u) != 0;
  if (lane == 0 && (part & 1)) {
    ctl[kCtlWant] = (int)want;
    ctl[kCtlErr] = bad ? 1 : 0;
  }
  if (!bad) {
    const long long gsrc = rstart + lo;              // first item, index into `in`
    const int len = act ? (int)(hi - lo) : 0;
    // `in` itself may sit off the 16-byte grid (a segment of a batch): the
    // bulk copies align on absolute addresses.
    const int in_mis = (int)(((uintptr_t)in / sizeof(KeyT)) & (E - 1));
    const int head = act ? (int)((in_mis + gsrc) % E) : 0;   // items copied before the segment
    const int span = (head + len + E - 1) / E * E + G::kSlack;   // staged span + transpose slack
    // One scan over (span, len) packed into 16-bit halves: both totals stay
    // below 2^16 (the spans sum to at most the buffer capacity).
    static_assert(G::cap(kMaxFanout) < (1 << 16), "packed span scan needs cap < 2^16");
    int incl = span | (len << 16);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    const int R = (incl & 0xFFFF) - span;            // span start of segment `lane`
    const int lpre = (incl >> 16) - len;             // items in segments before `lane`
    // Bulk part: from gsrc - head to the first 16-byte boundary (of absolute
    // addresses) at or past the segment's end.  The span rounds up to that
    // boundary, so the few items past the segment land in its own span and
    // are never read.  Where that boundary lies past the end of `in`, the
    // copy stops at the last boundary inside the segment and plain loads
    // fetch the rest (at most one tile per pass).
    const long long bulk_lo = gsrc - head;
    const long long bulk_up = (in_mis + gsrc + len + E - 1) / E * E - in_mis;
    const long long bulk_hi = bulk_up <= n ? bulk_up : (in_mis + gsrc + len) / E * E - in_mis;
    const unsigned bulk_bytes = (act && len > 0 && bulk_hi > bulk_lo)
                                    ? (unsigned)((bulk_hi - bulk_lo) * sizeof(KeyT))
                                    : 0u;
    // Items no bulk copy covers, one segment at a time, consecutive lanes ->
    // consecutive words.
    auto plain_tail = [&]() {
      for (int r = 0; r < K; ++r) {
        const long long s_src = __shfl_sync(0xffffffffu, gsrc, r);
        const int s_len = __shfl_sync(0xffffffffu, len, r);
        const int s_off = __shfl_sync(0xffffffffu, R + head, r);
        const long long s_bhi = __shfl_sync(0xffffffffu, bulk_hi, r);
        const long long s_blo = __shfl_sync(0xffffffffu, bulk_lo, r);
        const long long from = (s_bhi > s_blo) ? s_bhi : s_src;   // first item not bulk-copied
        const long long e = from + lane;
        if (e < s_src + s_len) stage[s_off + (int)(e - s_src)] = in[e];
      }
    };
    if (part & 1) {
      const unsigned total = __reduce_add_sync(0xffffffffu, bulk_bytes);
      if (lane == 0) mbar_arrive_expect_tx(bar, total);
      __syncwarp();
      if (bulk_bytes) bulk_g2s(stage + R, in + bulk_lo, bulk_bytes, bar);
      if (__any_sync(0xffffffffu, act && len > 0 && bulk_hi < gsrc + len)) plain_tail();
    }
    if (!(part & 2)) return;
    if (segs != nullptr) {                           // for the partition variant
      segs[lane] = R + head;
      segs[32 + lane] = len;
    }
    // Merge-tree nodes, one per lane, in level order: node (level l >= 1,
    // pair q) merges child A = segments [q*2^l, q*2^l + 2^(l-1)) and child
    // B = the rest of [q*2^l, (q+1)*2^l) (segments past the group's runs are
    // empty).
    // The tree spans the group's runs that exist: the last group of a round
    // (or a round's only group) may hold fewer than K, and empty leaves would
    // add levels that only copy.  At least two leaves, so that the tile is
    // always merged into span start 0.
    const int kruns = __popc(__ballot_sync(0xffffffffu, act && rlen > 0));
    int nl = 0, nnodes = 0, c_level = 0, c_pair = 0;
    {
      int cnt = kruns > 2 ? kruns : 2, idx = 0;
      for (int l = 1; cnt > 1; ++l) {
        const int pairs = (cnt + 1) >> 1;
        if (lane >= idx && lane < idx + pairs) {
          c_level = l;
          c_pair = lane - idx;
        }
        idx += pairs;
        cnt = pairs;
        nl = l;
      }
      nnodes = idx;
    }
    const bool is_node = lane < nnodes;
    const int first = c_pair << c_level;             // first segment of the node
    const int mid = first + (1 << (c_level > 0 ? c_level - 1 : 0));
    const int last = first + (1 << c_level);
    auto seg_pre = [&](int sg) {                     // items in segments [0, sg)
      const int ss = sg < K ? sg : K;
      const int v = __shfl_sync(0xffffffffu, lpre, ss & 31);
      return ss >= K ? (int)want : v;
    };
    const int pf = seg_pre(first), pm = seg_pre(mid), pl = seg_pre(last);
    const int rf = __shfl_sync(0xffffffffu, R, first & 31);
    const int hf = __shfl_sync(0xffffffffu, head, first & 31);
    const int rm = __shfl_sync(0xffffffffu, R, mid & 31);
    const int hm = __shfl_sync(0xffffffffu, head, mid & 31);
    const int lenA = is_node ? pm - pf : 0;
    const int lenB = is_node ? pl - pm : 0;
    const int nb = (lenA + lenB + kBlockItems - 1) / kBlockItems;
    // A node's last block is "small" when it holds at most kSmallBlockMax
    // items; it is merged by the small network, after every full-size block
    // of its level, so that the level's big blocks are dealt first and the
    // cheap ones fill in.  So are the blocks of a node with an empty child, which
    // are copies.  Items of a level: its nodes' big blocks in node order,
    // then the others in node order; levels follow each other.
    // Inclusive scans over the nodes (lanes, in level order) of both counts
    // give every node its first item of each kind: with n0 / n1 the first /
    // last node of the node's level,
    //   first big item = big blocks before the node + others before n0,
    //   first other    = big blocks up to n1 + others before the node.
    const int tail = lenA + lenB - (nb - 1) * kBlockItems;
    const int small = (lenA == 0 || lenB == 0) ? nb : (nb > 0 && tail <= kSmallBlockMax) ? 1 : 0;
    const int nbig = nb - small;
    int sbig = nbig, ssm = small;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, sbig, o);
      const int y = __shfl_up_sync(0xffffffffu, ssm, o);
      if (lane >= o) {
        sbig += x;
        ssm += y;
      }
    }
    const unsigned same_level = __match_any_sync(0xffffffffu, is_node ? c_level : -1);
    const int n0 = __ffs(same_level) - 1, n1 = 31 - __clz(same_level);
    const int small_before_n0 = __shfl_sync(0xffffffffu, ssm - small, n0);
    const int big_upto_n1 = __shfl_sync(0xffffffffu, sbig, n1);
    const int small_upto_n1 = __shfl_sync(0xffffffffu, ssm, n1);
    const int offA = (c_level == 1) ? rf + hf : rf;                      // staged segment
    const int offB = (mid < K) ? ((c_level == 1) ? rm + hm : rm) : 0;    // vs. child output
    const int first_big = (sbig - nbig) + small_before_n0;
    const int first_other = big_upto_n1 + (ssm - small);
    if (is_node) {
      int4* items = reinterpret_cast<int4*>(ctl + kCtlItems);
      for (int blk = 0; blk < nb; ++blk) {
        const int at = blk < nbig ? first_big + blk : first_other + (blk - nbig);
        const int left = lenA + lenB - blk * kBlockItems;
        if (at < kMaxItems)
          items[at] = make_int4(offA | (lenA << 16), offB | (lenB << 16), rf | ((blk * kBlockItems) << 16),
                                left < kBlockItems ? left : kBlockItems);
      }
      if (lane == n0) {
        int* lv = ctl + kCtlLevel0 + 4 * c_level;
        lv[0] = first_big;
        lv[2] = big_upto_n1 + small_upto_n1;
      }
      if (lane == n1) ctl[kCtlLevel0 + 4 * c_level + 1] = first_big + nbig;
    }
    if (lane == 0) ctl[kCtlLevels] = nl;
  }
}

// Merges a staged tile level by level and writes it to dstg: run by the
// WARPS merging warps (threads 0 .. 32 * WARPS - 1).  bufX holds the staged
// segments, bufY is the other level buffer; `ctl` is the tile's control area.
// sync() is a barrier over exactly the merging warps; the caller has made the
// staged data and the control area visible to them.
//
// A level's items are dealt to the warps round-robin: first the network
// items, then the small and the copied blocks; a barrier ends the level.  Each
// lane reads the item's 16 bytes (in place of the ballots and shuffles that looked a
// node up: 350 cycles of an item's 3500 with one CTA on the SM).
//
// The last stages of a block run in the blocked layout.  It leaves it in order:
// the rows go to their place swizzled, come back as consecutive 16-byte chunks, and
// are stored once more -- or, where the root's blocks are all network items and the
// tile lies on the 16-byte grid, straight to global memory, with no barrier,
// bulk store and wait after them: passes of 16.8 * 10^6 u32 keys 37.1 / 54.3 / 73.4 /
// 92.3 us to 35.0 / 52.3 / 71.0 / 89.9 (K = 2, 4, 8, 16; K = 32, now three CTAs to an SM,
// 149.9 to 122.3).  With 8-byte keys the last stages are directed
// instead (a compare's predicate takes a direction for nothing), which stores in
// place at once; their tile goes out by the bulk store.
template <typename KeyT, int WARPS, typename Sync>
__device__ __forceinline__ void merge_levels(KeyT* bufX, KeyT* bufY, const int* ctl,
                                             KeyT* dstg, bool xout, Sync sync) {
  constexpr int E = Vec16<KeyT>::E;
  constexpr uint32_t RB = 32 * sizeof(KeyT);
  constexpr bool LINEAR = sizeof(KeyT) == 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nl = ctl[kCtlLevels];
  const long long want = ctl[kCtlWant];
  const int4* items = reinterpret_cast<const int4*>(ctl + kCtlItems);
  bool direct = false;                                  // the root's blocks go straight out
  if constexpr (LINEAR) {
    const int4 root = *reinterpret_cast<const int4*>(ctl + kCtlLevel0 + 4 * nl);
    direct = root.y == root.z && ((uintptr_t)dstg & 15u) == 0;
  }
  for (int lv = 1; lv <= nl; ++lv) {
    const int4 info = *reinterpret_cast<const int4*>(ctl + kCtlLevel0 + 4 * lv);
    const KeyT* src = (lv & 1) ? bufX : bufY;           // level lv reads level lv-1's buffer
    KeyT* dst = (lv & 1) ? bufY : bufX;
    const bool xo = xout && lv == nl;
    for (int at = info.x + warp; at < info.z; at += WARPS) {
      const bool big = at < info.y;
      const int4 it = items[at];
      const int lenA = it.x >> 16, lenB = it.y >> 16, d0 = it.z >> 16, m = it.w;
      const KeyT* A = src + (it.x & 0xFFFF);
      const KeyT* B = src + (it.y & 0xFFFF);
      KeyT* o = dst + (it.z & 0xFFFF) + d0;
      if (!big && (lenA == 0 || lenB == 0)) {
        // One child is empty (a node over runs past the group's last, or a
        // tile that takes nothing from one side): the block is a copy, made
        // with 32 consecutive keys per access instead of a merge network.
        const KeyT* from = (lenB == 0 ? A : B) + d0;
        for (int i = lane; i < m; i += 32) {
          const KeyT v = from[i];
          o[i] = xo ? (KeyT)ordered_to_f32((uint32_t)v) : v;
        }
        __syncwarp();
        continue;
      }
      int a0, a1;
      block_coranks(A, lenA, B, lenB, d0, m, lane, a0, a1);
      const int X = a1 - a0;
      if (!big) {
        warp_merge_small<KeyT>(A + a0, X, B + (d0 - a0), m - X, o, lane, xo);
        __syncwarp();
        continue;
      }
      if constexpr (!LINEAR) {
        warp_merge_block<KeyT, MergeMix>(A + a0, X, B + (d0 - a0), m - X, o, lane, xo);
        __syncwarp();
        continue;
      }
      KeyT v[32];
      warp_load_bitonic(A + a0, X, B + (d0 - a0), m - X, v, lane);
      warp_bitonic_1024<MergeMix, false>(v, o, (m + 31) >> 5, lane);
      const uint32_t ob = smem_u32addr(o), r = (uint32_t)lane & 7, g = (uint32_t)lane >> 3;
      if (32 * lane < m) {
#pragma unroll
        for (int ch = 0; ch < 32 / E; ++ch) sts128(ob + lane * RB + ((ch ^ r) << 4), &v[ch * E]);
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 32 / E; ++q)                  // chunk 32q + lane: row 4q + g, place r
        if (32 * E * q + E * lane < m)
          lds_chunk(ob + (4 * q + g) * RB + ((r ^ g ^ (4 * (q & 1))) << 4), &v[q * E]);
      if (xo) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = (KeyT)ordered_to_f32((uint32_t)v[j]);
      }
      if (direct && lv == nl) {
        KeyT* og = dstg + d0;
#pragma unroll
        for (int q = 0; q < 32 / E; ++q) {
          const int pos = 32 * E * q + E * lane;
          if (pos + E <= m)
            *reinterpret_cast<typename Vec16<KeyT>::T*>(og + pos) = Vec16<KeyT>::pack(&v[q * E]);
        }
        if (m % E != 0) {                               // the chunk that straddles the end
#pragma unroll
          for (int q = 0; q < 32 / E; ++q) {
            const int pos = 32 * E * q + E * lane;
#pragma unroll
            for (int w = 0; w < E - 1; ++w)
              if (pos + w < m && pos + E > m) og[pos + w] = v[q * E + w];
          }
        }
        continue;                                       // its item is the warp's last of the tile
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 32 / E; ++q)
        sts128_if_le(ob + ((32 * q + lane) << 4), &v[q * E], 32 * E * q + E * lane + E, m);
      if (m % E != 0) {
#pragma unroll
        for (int q = 0; q < 32 / E; ++q) {
          const int pos = 32 * E * q + E * lane;
#pragma unroll
          for (int w = 0; w < E - 1; ++w)
            if (pos + w < m && pos + E > m) sts_addr(ob + (uint32_t)((pos + w) * sizeof(KeyT)), v[q * E + w]);
        }
      }
      __syncwarp();
    }
    if (direct && lv == nl) {
      fence_proxy_async_smem();                         // before a next tile's bulk copies
      return;
    }
    sync();
  }
  // The root node's output is the tile, at span start 0 of the last level's buffer.
  const KeyT* res = (nl & 1) ? bufY : bufX;
  const int m = (int)want;
  const int body = (((uintptr_t)dstg & 15u) == 0) ? m / E * E : 0;   // off-grid: plain stores
  fence_proxy_async_smem();
  sync();
  if (threadIdx.x == 0 && body > 0) bulk_s2g_and_wait(dstg, res, (unsigned)(body * sizeof(KeyT)));
  for (int i = body + (int)threadIdx.x; i < m; i += WARPS * 32) dstg[i] = res[i];
}

// The heap-free variant of the merge (Sec. 7, future work: multiway merging
// driven by the parallel partitioning alone, with no merge tree shared by the
// CTA).  The tile's output is cut into 1024-item blocks, one per warp.
//   1. Warp b finds the pivots of block start 1024 b in every staged segment
//      with the splitter's own search (the multi-sequence selection of
//      Sec. 4.1, multiseq_pivot, here over shared memory), and writes them as
//      row b of `rows`; one CTA barrier publishes the rows.
//   2. The warp's block is then the merge of its K pieces (segment r from
//      row b to row b + 1), which the warp merges alone: pairs of pieces, then
//      pairs of their outputs, along the same binary tree over the runs as the
//      CTA tree, with no barrier between its levels.  The first level reads the
//      staged pieces and writes its outputs packed into the warp's own
//      1024-item region of bufY; later levels merge adjacent outputs back into
//      their own span.  Merges of at most 1024 items at any offset take the
//      register-and-shuffle network of the smallest power of two that holds
//      them (warp_merge_any); the last level, whose output is the whole block
//      at its 16-byte aligned start, takes the transposed 1024-item network.
// bufX holds the staged segments (their offsets and lengths stand before the
// pivot rows), bufY receives the tile; the final store is the same as the
// tree's.
// A warp whose pivot rows do not describe pieces inside their segments that
// add up to its block records kDevErrInternal in dev_err and merges nothing,
// so every shared-memory access stays inside the warp's spans.
template <typename KeyT, int WARPS, typename Sync>
__device__ __forceinline__ void merge_partition_blocks(const KeyT* bufX, KeyT* bufY, const int* ctl,
                                                       int* rows, KeyT* dstg, bool xout,
                                                       int* dev_err, Sync sync) {
  constexpr int E = Vec16<KeyT>::E;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nl = ctl[kCtlLevels];                    // levels of the tree over the runs (>= 1)
  const int want = ctl[kCtlWant];                    // items of the tile
  const int nleaf = 1 << nl;                         // segments, empty past the group's runs
  const int seg_off = lane < nleaf ? rows[lane] : 0;
  const int seg_len = lane < nleaf ? rows[32 + lane] : 0;
  rows += 64;
  const int nblk = (want + kBlockItems - 1) / kBlockItems;
  if (warp == 0) {
    rows[lane] = 0;
    rows[nblk * 32 + lane] = seg_len;
  } else if (warp < nblk) {
    const int k = warp * kBlockItems;
    int d;
    if (nleaf == 2) {
      // Two segments: the search is the merge-path co-rank (ties from the
      // lower run, as in the order of Sec. 4.1).
      const int o0 = __shfl_sync(0xffffffffu, seg_off, 0), l0 = __shfl_sync(0xffffffffu, seg_len, 0);
      const int o1 = __shfl_sync(0xffffffffu, seg_off, 1), l1 = __shfl_sync(0xffffffffu, seg_len, 1);
      const int a = warp_corank(bufX + o0, l0, bufX + o1, l1, k, lane);
      d = lane == 0 ? a : (lane == 1 ? k - a : 0);
    } else {
      d = multiseq_pivot<KeyT, int>(bufX + seg_off, seg_len, lane < nleaf, nleaf, k, 0xffffffffu);
    }
    rows[warp * 32 + lane] = d;
  }
  sync();
  bool rows_ok = true;
  if (warp < nblk) {
    const int r0 = rows[warp * 32 + lane], r1 = rows[(warp + 1) * 32 + lane];
    const int bm = (want - warp * kBlockItems) < kBlockItems ? (want - warp * kBlockItems) : kBlockItems;
    const bool bad = lane < nleaf && (r0 < 0 || r1 < r0 || r1 > seg_len);
    const int sum = (int)__reduce_add_sync(0xffffffffu, (lane < nleaf && !bad) ? (unsigned)(r1 - r0) : 0u);
    rows_ok = !__any_sync(0xffffffffu, bad) && sum == bm;
    if (!rows_ok && lane == 0) set_device_error(dev_err, kDevErrInternal);
  }
  if (warp < nblk && rows_ok) {
    KeyT* blk = bufY + warp * kBlockItems;
    const int r0 = rows[warp * 32 + lane];
    int off = seg_off + r0;                          // lane q: sequence q of the level (bufX
    int len = rows[(warp + 1) * 32 + lane] - r0;     // offsets at level 1, then blk offsets)
    if (lane >= nleaf) len = 0;
    for (int l = 1; l <= nl; ++l) {
      const int npairs = nleaf >> l;
      const int la = __shfl_sync(0xffffffffu, len, (2 * lane) & 31);
      const int lb = __shfl_sync(0xffffffffu, len, (2 * lane + 1) & 31);
      const int oa = __shfl_sync(0xffffffffu, off, (2 * lane) & 31);
      const int ob = __shfl_sync(0xffffffffu, off, (2 * lane + 1) & 31);
      const int olen = lane < npairs ? la + lb : 0;
      int incl = olen;                               // outputs packed in pair order
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      const int ooff = incl - olen;
      const KeyT* src = (l == 1) ? bufX : blk;
      const bool root = l == nl;
      const bool xo = xout && root;
      for (int p = 0; p < npairs; ++p) {
        const int a = __shfl_sync(0xffffffffu, la, p);
        const int b = __shfl_sync(0xffffffffu, lb, p);
        const int m = a + b;
        if (m == 0) continue;                        // uniform over the warp
        const KeyT* A = src + __shfl_sync(0xffffffffu, oa, p);
        const KeyT* B = src + __shfl_sync(0xffffffffu, ob, p);
        KeyT* out = blk + __shfl_sync(0xffffffffu, ooff, p);
        if (a == 0 || b == 0) {
          // One side empty: a copy at the first level; later levels hold
          // the items in place already (only the float transform remains).
          if (l == 1 || xo) {
            const KeyT* from = a ? A : B;
            for (int i = lane; i < m; i += 32) {
              const KeyT v = from[i];
              out[i] = xo ? (KeyT)ordered_to_f32((uint32_t)v) : v;
            }
          }
        } else if (root && m > kSmallBlockMax) {
          if (l == 1)
            warp_merge_block<KeyT, MergeMix, false>(A, a, B, b, out, lane, xo);
          else
            warp_merge_block<KeyT, MergeMix, true>(A, a, B, b, out, lane, xo);
        } else {
          warp_merge_any<KeyT>(A, a, B, b, out, lane, xo);
        }
        __syncwarp();
      }
      off = ooff;
      len = olen;
    }
  }
  const int body = (((uintptr_t)dstg & 15u) == 0) ? want / E * E : 0;   // off-grid: plain stores
  fence_proxy_async_smem();
  sync();
  if (threadIdx.x == 0 && body > 0) bulk_s2g_and_wait(dstg, bufY, (unsigned)(body * sizeof(KeyT)));
  for (int i = body + (int)threadIdx.x; i < want; i += WARPS * 32) dstg[i] = bufY[i];
}

// Merges output tile j (of S items, a multiple of 1024 and at most
// 1024 * WARPS) of group g of `in` (n items in sorted runs of run_len, K runs
// per group) into `out`: the CTA body of a merge round, one tile at a time.
// lo_row and hi_row are the pivot rows of the tile's start and end (read only
// when the tile is not its group's first / last).  `bar` is an initialised
// mbarrier of this CTA whose next phase completes with parity `phase`.
// `xout` undoes the float transform on the tile's last level.  Returns false,
// with the error recorded, when the CTA must stop (a pivot row fails its
// check or the staging wait ran out); the decision is uniform over the CTA.
// test_timeout (a test hook; bar[1] then holds an initialised mbarrier): once
// the staged data has arrived, thread 0 also waits on bar[1] for 16 bytes no
// copy delivers, with a limit of about a millisecond, so the CTA takes the
// time-out path with no copy in flight.
// PARTITION: merge with the heap-free variant above instead of the CTA tree
// (shared memory of MergeGeom::bytes_partition).
template <typename KeyT, int WARPS, bool PARTITION = false>
__device__ __forceinline__ bool merge_tile(const KeyT* in, KeyT* out,
                                           long long n, long long run_len, int K, long long g,
                                           long long j, const long long* lo_row,
                                           const long long* hi_row, bool xout,
                                           int* dev_err, unsigned char* smem_raw, uint64_t* bar,
                                           unsigned phase, int S, bool test_timeout = false) {
  using G = MergeGeom<KeyT, WARPS>;
  const int cap = G::cap(K);
  KeyT* bufX = reinterpret_cast<KeyT*>(smem_raw);
  KeyT* bufY = bufX + cap;
  int* ctl = reinterpret_cast<int*>(bar + 2);          // the control area (see above)
  // Every thread is past the previous tile (whose store has read its shared
  // memory) before the staging copies overwrite the buffer.
  // Warp 0 stages the segments while warp 1 lists the tree's blocks.
  long long lo = 0, hi = 0;
  if ((threadIdx.x >> 5) < 2)
    merge_tile_pivots(n, run_len, K, g, j, lo_row, hi_row, S, threadIdx.x & 31, lo, hi);
  __syncthreads();
  // One thread polls the staging barrier; the others wait at the CTA barrier
  // (no issue slots spent polling), which also orders the staged data, the
  // plainly loaded items and the control area before every warp's reads.  The list is
  // ready before the data is, so it costs the tile nothing.
  bool ok = true;
  if ((threadIdx.x >> 5) < 2)
    merge_plan_warp<KeyT, WARPS>(in, n, run_len, K, g, j, lo, hi, S, bufX, ctl, bar,
                                 threadIdx.x & 31, (threadIdx.x >> 5) == 0 ? 1 : 2,
                                 PARTITION ? ctl + kCtlInts : nullptr);
  if (threadIdx.x == 0 && !ctl[kCtlErr]) {             // written by this thread
    ok = mbar_wait_bounded(bar, phase);
    if (test_timeout && ok) {
      mbar_arrive_expect_tx(bar + 1, 16u);
      ok = mbar_wait_bounded(bar + 1, 0u, 2000000ll);
    }
  }
  const bool late = __syncthreads_or(!ok);
  if (ctl[kCtlErr] || (smem_u32addr(smem_raw) & 1023u) != 0) {
    if (threadIdx.x == 0) set_device_error(dev_err, kDevErrInternal);
    return false;                                      // uniform over the CTA
  }
  if (late) {
    if (threadIdx.x == 0) set_device_error(dev_err, kDevErrTimeout);
    return false;
  }
  if constexpr (PARTITION)
    merge_partition_blocks<KeyT, WARPS>(bufX, bufY, ctl, ctl + kCtlInts,
                                        out + g * run_len * K + j * S, xout, dev_err,
                                        []() { __syncthreads(); });
  else
    merge_levels<KeyT, WARPS>(bufX, bufY, ctl, out + g * run_len * K + j * S, xout,
                              []() { __syncthreads(); });
  return true;
}

}  // namespace mms
