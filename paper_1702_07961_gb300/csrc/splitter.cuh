// splitter.cuh -- parallel partitioning of a K-way merge round (Sec. 4.1),
// shared by the whole-array splitter and the segmented (batched) one.
//
// For every output tile j of every group of K sorted runs, one warp finds the pivot indices
// c[r] (r < K): the number of items run r contributes to the group's first j*S
// outputs under the strict order (key, run, position).  That
// order makes the pivots unique even with repeated keys (the paper's
// non-overlap condition, read on the composite key) and equals a stable merge.
//
// Two searches.  window_pivot: windows of samples, sorted across the warp (described there).
// multiseq_pivot, one lane per run (K <= 32), for large sorts of 8-byte keys and, on
// segments in shared memory, for the partition variant: stride halving on regular samples.  At
// stride s the lane group holds the exact pivots d of the s-sample problem -- the
// items at positions s-1, 2s-1, ... of every run -- for rank floor(k/s).
// Halving s adds one candidate per run just above its pivot; the pivots of the
// s/2-sample problem for rank floor(2k/s) are then the floor(2k/s) smallest of
// (old selection expanded) + (candidates), found by dropping the largest items
// from the top with arg-max reductions over the lane group.  At s = 1 the sample problem is
// the whole problem.  About log2(k) rounds of two independent loads per lane.
// Positions past a run's end are padding items ordered after every real item
// (by run, then position).
#pragma once

#include "mms_common.cuh"
#include "mms_kernels.cuh"

namespace mms {

template <typename KeyT>
struct Item {
  KeyT key;
  bool pad;
};

template <typename KeyT, typename Idx>
__device__ __forceinline__ Item<KeyT> load_item(const KeyT* run, Idx len, Idx pos) {
  Item<KeyT> it;
  it.pad = pos >= len;
  it.key = it.pad ? KeyT(0) : run[pos];
  return it;
}

// a (run ra) strictly before b (run rb), ra != rb.
template <typename KeyT>
__device__ __forceinline__ bool before_cross(const Item<KeyT>& a, int ra, const Item<KeyT>& b,
                                             int rb) {
  if (a.pad != b.pad) return b.pad;
  if (!a.pad && a.key != b.key) return a.key < b.key;
  return ra < rb;
}

// Every reduction below runs over one lane group: the lanes of the mask gm
// (W consecutive lanes aligned to W; all of them execute the call).  A warp
// holds 32 / W groups, each working on its own output tile.
__device__ __forceinline__ uint32_t grp_max_u32(unsigned gm, uint32_t v) {
  return __reduce_max_sync(gm, v);
}
__device__ __forceinline__ uint32_t grp_min_u32(unsigned gm, uint32_t v) {
  return __reduce_min_sync(gm, v);
}

// Lanes with `cond` whose key equals the maximum key among them.
__device__ __forceinline__ unsigned lanes_with_max(unsigned gm, bool cond, uint32_t key) {
  const uint32_t mx = grp_max_u32(gm, cond ? key : 0u);
  return __ballot_sync(gm, cond && key == mx);
}
__device__ __forceinline__ unsigned lanes_with_max(unsigned gm, bool cond, uint64_t key) {
  const uint32_t hi = (uint32_t)(key >> 32), lo = (uint32_t)key;
  const uint32_t mh = grp_max_u32(gm, cond ? hi : 0u);
  const bool c2 = cond && hi == mh;
  const uint32_t ml = grp_max_u32(gm, c2 ? lo : 0u);
  return __ballot_sync(gm, c2 && lo == ml);
}
__device__ __forceinline__ unsigned lanes_with_min(unsigned gm, bool cond, uint32_t key) {
  const uint32_t mn = grp_min_u32(gm, cond ? key : 0xffffffffu);
  return __ballot_sync(gm, cond && key == mn);
}
__device__ __forceinline__ unsigned lanes_with_min(unsigned gm, bool cond, uint64_t key) {
  const uint32_t hi = (uint32_t)(key >> 32), lo = (uint32_t)key;
  const uint32_t mh = grp_min_u32(gm, cond ? hi : 0xffffffffu);
  const bool c2 = cond && hi == mh;
  const uint32_t ml = grp_min_u32(gm, c2 ? lo : 0xffffffffu);
  return __ballot_sync(gm, c2 && lo == ml);
}

// Lane holding the largest item among lanes with `cond` (runs compare by
// (pad, key, run)); -1 if none.  Lane numbers are the warp's.
template <typename KeyT>
__device__ __forceinline__ int grp_argmax(unsigned gm, bool cond, const Item<KeyT>& it) {
  if constexpr (sizeof(KeyT) == 4) {
    // One max over the keys with pads raised to the all-ones key, then the
    // lanes holding that maximum: a pad among them wins (pads come after
    // every real key, an all-ones real key included), else the highest lane
    // (the largest run index).  The pad ballot does not wait for the max.
    const uint32_t kk = cond ? (it.pad ? 0xffffffffu : (uint32_t)it.key) : 0u;
    const uint32_t mx = grp_max_u32(gm, kk);
    const unsigned padm = __ballot_sync(gm, cond && it.pad);
    const unsigned m = __ballot_sync(gm, cond && kk == mx);
    const unsigned mp = m & padm;
    return m ? 31 - __clz(mp ? mp : m) : -1;
  } else {
    const unsigned any = __ballot_sync(gm, cond);
    if (!any) return -1;
    const unsigned pads = __ballot_sync(gm, cond && it.pad);
    if (pads) return 31 - __clz(pads);
    return 31 - __clz(lanes_with_max(gm, cond, it.key));
  }
}

// grp_argmax when no lane of the group holds a pad: one max and one ballot
// (4-byte keys), or the two-word maximum (8-byte keys).
template <typename KeyT>
__device__ __forceinline__ int grp_argmax_real(unsigned gm, bool cond, KeyT key) {
  if constexpr (sizeof(KeyT) == 4) {
    const uint32_t mx = grp_max_u32(gm, cond ? (uint32_t)key : 0u);
    const unsigned m = __ballot_sync(gm, cond && (uint32_t)key == mx);
    return m ? 31 - __clz(m) : -1;
  } else {
    if (!__ballot_sync(gm, cond)) return -1;
    return 31 - __clz(lanes_with_max(gm, cond, key));
  }
}

template <typename KeyT>
__device__ __forceinline__ int grp_argmin(unsigned gm, bool cond, const Item<KeyT>& it) {
  const unsigned any = __ballot_sync(gm, cond);
  if (!any) return -1;
  const unsigned reals = __ballot_sync(gm, cond && !it.pad);
  if (!reals) return __ffs(any) - 1;
  return __ffs(lanes_with_min(gm, cond && !it.pad, it.key)) - 1;
}

template <typename KeyT>
__device__ __forceinline__ Item<KeyT> shfl_item(unsigned gm, const Item<KeyT>& it, int src) {
  Item<KeyT> o;
  o.key = __shfl_sync(gm, it.key, src);
  o.pad = __shfl_sync(gm, (int)it.pad, src) != 0;
  return o;
}

// Stride halving: the lanes of the group (lane gb + r on run r, act for
// r < K) return the number of items each run contributes to the first k of
// the K runs' merge under the order (key, run, position).  `run` and `rlen`
// are the lane's run and its length (rlen = 0 when !act); the runs may lie in
// global or in shared memory.  Arguments other than run / rlen / act are
// uniform over the lane group; every lane of it must call.
// UNSWITCH: one drop loop per arg-max form (no pad test inside the loop): in the splitter
// kernel 10^8 u64 keys sort in 6309 us with it, 6321 without; in the much larger partition
// merge kernel it is slower.
template <typename KeyT, typename Idx, bool UNSWITCH = false>
__device__ __forceinline__ Idx multiseq_pivot(const KeyT* run, Idx rlen, bool act, int K, Idx k,
                                              unsigned gm) {
  const int lane = threadIdx.x & 31;
  Idx d = 0;                  // selected samples of this run at the current stride
  Item<KeyT> e{KeyT(0), false};  // the d-th sample (position d*s-1) when d >= 1
  const int T = 64 - __clzll((long long)k);
  bool pad_prev = true;       // the previous level had a pad candidate (so e may be a pad)
  for (int lev = T; lev >= 1; --lev) {
    const int sh = lev - 1;                     // s2 = 2^sh
    const Idx kp = k >> sh;
    const Idx dd = 2 * d;
    Item<KeyT> o = load_item(run, rlen, ((dd + 1) << sh) - 1);
    Item<KeyT> z{KeyT(0), false};
    if (d >= 1) z = load_item(run, rlen, ((dd - 1) << sh) - 1);
    // The largest selected item (lane mz's e) needs none of the new loads:
    // its reduction overlaps them.  e is a pad only if the previous level had
    // a pad candidate.
    const bool hasZ = act && d >= 1;
    const int mz = pad_prev ? grp_argmax(gm, hasZ, e) : grp_argmax_real(gm, hasZ, e.key);
    Item<KeyT> zmax{KeyT(0), false};
    if (mz >= 0) zmax = pad_prev ? shfl_item(gm, e, mz) : Item<KeyT>{__shfl_sync(gm, e.key, mz), false};
    // Pads at this level: o is a lane's highest position, so when no o is a
    // pad, no item of the level is (e, z and any deeper item lie below o).
    const bool any_pad = __any_sync(gm, act && o.pad);
    // Items to drop: (sum of the lanes' 2d + 1) - kp.  The lanes hold the
    // pivots of rank k >> lev, so the d sum to k >> (sh + 1) and the count is
    // K minus the low bit of kp: K - 1 or K, with no reduction.
    const Idx jrem = (Idx)K - (kp & 1);
    Idx cnt = dd + 1;

    // Candidates above every selected item are dropped first, in one step.
    bool above = act;
    if (mz >= 0) {
      if (any_pad) {
        above = act && (lane == mz || before_cross(zmax, mz, o, lane));
      } else {                                  // no pads: keys, then runs
        above = act && (lane == mz || zmax.key < o.key || (zmax.key == o.key && mz < lane));
      }
    }
    const unsigned abovem = __ballot_sync(gm, above);
    const Idx u = __popc(abovem);
    Idx pops;
    if (u <= jrem) {
      if (above) cnt = dd;
      pops = jrem - u;
    } else {                                    // keep only the smallest candidate
      const int mn = grp_argmin(gm, above, o);
      if (above && lane != mn) cnt = dd;
      pops = 0;
    }
    // Remaining drops one at a time from the largest current top.  The first
    // needs no reduction: the largest top is lane mz's e (every candidate
    // above it was dropped, mz's own included), and mz then falls back to z.
    Item<KeyT> top = (cnt == dd + 1) ? o : e;
    if (mz >= 0 && pops > 0) {                  // uniform over the group
      if (lane == mz) {
        cnt = dd - 1;                           // d >= 1 on lane mz, so cnt >= 1
        top = z;
      }
      pops -= 1;
    }
    auto drop = [&](int w) {
      if (lane == w) {
        cnt -= 1;
        if (cnt >= 1) {
          if (cnt == dd)
            top = e;
          else if (cnt == dd - 1)
            top = z;
          else
            top = load_item(run, rlen, (cnt << sh) - 1);
        }
      }
    };
    if constexpr (UNSWITCH) {
      if (any_pad) {
        for (Idx p = 0; p < pops; ++p) drop(grp_argmax(gm, act && cnt >= 1, top));
      } else {
        for (Idx p = 0; p < pops; ++p) drop(grp_argmax_real(gm, act && cnt >= 1, top.key));
      }
    } else {
      for (Idx p = 0; p < pops; ++p)
        drop(any_pad ? grp_argmax(gm, act && cnt >= 1, top)
                     : grp_argmax_real(gm, act && cnt >= 1, top.key));
    }
    d = cnt;
    e = top;
    pad_prev = any_pad;
  }
  return d;
}

// The splitter kernels' search by windows: the same pivots by the same idea --
// exact pivots of the s-sample problem, s shrinking to 1 -- but with a window
// of W samples of every run held across the warp, so that a step divides s by
// W / 2 instead of 2 and its drops are found together, not one arg-max at a
// time.  One warp per row.  SUB = 32 / K2 lanes share a run (K2: K rounded up
// to a power of two); register m of sub-lane b holds the sample
// f = top - W + 1 + b * M + m of the run, counted from 1, which is the item at
// position f * s - 1.
//
//   - Let c be the run's pivot at stride s' = s * W / 2, exact for the rank
//     floor(k / s').  Sample c + 1 of stride s' was left out there, so at least
//     floor(k / s') + 1 samples of stride s' come no later, each with W / 2 samples
//     of stride s at or below it: more than floor(k / s).  So the pivot at
//     stride s is at most top = min(c * W / 2 + W / 2 - 1, len / s).
//   - D = max(0, sum of the tops - floor(k / s)) samples must go, the largest
//     ones.  The 32 M windowed samples are sorted across the warp (bitonic
//     merges of the windows, which are sorted already); the D-th largest is the
//     threshold, and every lane compares its own samples with it.
//   - A run whose whole window goes may have to give up more: it is deep.  Every run's
//     coarser pivot left part of a sample behind, and where the runs overlap little (nearly
//     sorted keys, few distinct ones) the one run that holds the boundary gives all of
//     that back, up to D of its samples (D < 16 M).  Of the deep runs, that whose lowest windowed
//     sample is the largest, r, loses its window for certain (samples not yet seen are all
//     smaller).  Either it moves on by that window and the selection is repeated, or
//     (kLongWindow) its next 16 M samples, more than it can lose, take the place of the
//     lower half of the sorted order, which cannot reach the D largest, and one bitonic
//     merge gives the threshold again; if another run is still deep then, all that lies above the
//     largest of their lowest samples has been seen and goes for certain, and the step takes
//     another turn.  About 1% of the steps of 16 random runs come here, 0.1% with 8, and most of
//     those of nearly sorted ones, which took 3.2 loads a step with 16 runs moved a window a
//     turn: 10^8 u32 keys with 1% of them swapped, splitters 631 -> 330 us.
//   - The first stride is the least power of W / 2 at which every run has at most W
//     samples; there top = len / s and the windows are all there is.
//
// Ties are broken by (run, position), so the pivots are those of multiseq_pivot.
//
// What bounds it: up to about 3000 rows (one wave of warps) a chain of
// log(run_len) / log(W / 2) steps, each a load (700 cycles and more) and a sort of
// about as long; above that the 32 M sectors a step reads.  Against stride halving (log2(K *
// run_len) levels, each a load and about K / 2 arg-maxes of 250 cycles) on random keys: both
// splitters of 2^20 u32 keys 41 -> 25 us, the three of 16.8 * 10^6 85 -> 59 us, the four of
// 3 * 10^8 926 -> 811 us; with 8-byte keys large sorts keep stride halving (splitter.cu).  Finding the threshold by
// quickselect instead of sorting took 500 cycles a round of 5 to 7 rounds and was no faster
// than stride halving.

// Samples per lane.  More samples take fewer, longer steps and read more
// sectors: with K = 8, 4 against 2 measured 12.3 against 18.4 us at 2^20 u32 keys and
// 62 against 70 us at 10^8; with K = 4, 1 against 4 18.5 against 28.5 us at 2 * 10^7 u64.
__host__ __device__ constexpr int pivot_regs(int k2) {
  return k2 == 32 ? 8 : k2 >= 8 ? 4 : 1;
}

// One bitonic merge level: sorted sequences of N / 2 elements become sorted ones of
// N, element e of the warp in register e % M of lane e / M, all ascending.  The
// first stage compares e with its mirror image in the block of N.
template <int N, int M, typename KeyT>
__device__ __forceinline__ void window_merge(KeyT (&v)[M], int lane) {
  KeyT y[M];
#pragma unroll
  for (int s = N / 2; s >= 1; s >>= 1) {
    if (s >= M) {                                  // between lanes
      const bool upper = (lane & (s / M)) != 0;
#pragma unroll
      for (int m = 0; m < M; ++m)
        y[m] = s == N / 2 ? __shfl_xor_sync(0xffffffffu, v[M - 1 - m], N / M - 1)
                          : __shfl_xor_sync(0xffffffffu, v[m], s / M);
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = (y[m] < v[m]) != upper ? y[m] : v[m];
    } else {
#pragma unroll
      for (int m = 0; m < M; ++m)
        if ((m & s) == 0) cas(v[m], v[m + s]);
    }
  }
}

// Sorted sequences of N elements to one of 32 M.
template <int N, int M, typename KeyT>
__device__ __forceinline__ void window_sort(KeyT (&v)[M], int lane) {
  if constexpr (N < 32 * M) {
    window_merge<2 * N, M>(v, lane);
    window_sort<2 * N, M>(v, lane);
  }
}

// Element `at` of the sorted windows.  In PTX, because a choice by a run-time index is
// compiled as an array in local memory.
template <int M>
__device__ __forceinline__ uint32_t window_at(const uint32_t (&v)[M], int at) {
  uint32_t t = v[0];
#pragma unroll
  for (int m = 1; m < M; ++m)
    asm("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %2, %3;\n\tselp.b32 %0, %1, %0, p;\n\t}\n"
        : "+r"(t)
        : "r"(v[m]), "r"(at & (M - 1)), "r"(m));
  return __shfl_sync(0xffffffffu, t, at / M);
}
template <int M>
__device__ __forceinline__ uint64_t window_at(const uint64_t (&v)[M], int at) {
  uint64_t t = v[0];
#pragma unroll
  for (int m = 1; m < M; ++m)
    asm("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %2, %3;\n\tselp.b64 %0, %1, %0, p;\n\t}\n"
        : "+l"(t)
        : "l"(v[m]), "r"(at & (M - 1)), "r"(m));
  return __shfl_sync(0xffffffffu, t, at / M);
}

// `run` and `rlen`: the run of this lane (lane / SUB) and its length, 0 past
// the K runs; maxlen: an upper bound of the lengths; k <= their sum.  All 32
// lanes call, k and maxlen uniform.  Returns the run's pivot on each of its
// lanes.  Idx as for multiseq_pivot (positions never pass the run's end).
template <typename KeyT, int K2, typename Idx>
__device__ __forceinline__ Idx window_pivot(const KeyT* run, Idx rlen, Idx maxlen, Idx k) {
  constexpr int SUB = 32 / K2;
  constexpr int M = pivot_regs(K2);
  constexpr int W = SUB * M;
  constexpr int B = W == 4 ? 1 : W == 8 ? 2 : W == 16 ? 3 : W == 32 ? 4 : 5;   // log2(W / 2)
  static_assert(W == (2 << B), "windows of 4 to 64 samples");
  // Whether a deep run goes on by 16 M samples at once or by a window a turn.  With 8 runs it
  // rarely moves twice; with 8-byte keys the code alone made small sorts slower (3 * 10^6 pairs
  // of 8-byte keys 473 -> 491 us with K = 16, 6 * 10^6 900 -> 917 with K = 8).
  constexpr bool kLongWindow = K2 >= 16 && sizeof(KeyT) == 4;
  const int lane = threadIdx.x & 31, sub = lane % SUB;
  if (k == 0) return 0;
  int sh = 0;
  while ((maxlen >> sh) > W) sh += B;
  Idx top = rlen >> sh;
  for (;;) {
    int D = (int)(__reduce_add_sync(0xffffffffu, sub == 0 ? (unsigned)top : 0u) - (unsigned)(k >> sh));
    int gone = 0;
    // Sorted runs need K2 / 2 turns at most (D < K2 * W / 2, and another turn comes after W
    // drops or more); after K2 the search gives up on runs that are not sorted.
    for (int turn = 0; D > 0 && turn < K2; ++turn) {
      KeyT w[M], v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const Idx f = top - (Idx)(W - 1 - m - sub * M);
        w[m] = f >= 1 ? run[(f << sh) - 1] : KeyT(0);
        v[m] = w[m];
      }
      window_sort<W, M>(v, lane);

      // Drops the `need` largest of the windows and of `extra` equal samples of run r
      // that lie below its window: sets gone, returns how many of the extra ones go.
      auto drop = [&](KeyT t, int need, int extra, int r) {
        unsigned X[M], E[M];
        int eq = extra;
#pragma unroll
        for (int m = 0; m < M; ++m) {
          X[m] = __ballot_sync(0xffffffffu, w[m] > t);
          E[m] = __ballot_sync(0xffffffffu, w[m] == t && top >= (Idx)(W - m - sub * M));
          need -= __popc(X[m]);
          eq += __popc(E[m]);
        }
        int left = extra;
        if (need >= eq) {
#pragma unroll
          for (int m = 0; m < M; ++m) X[m] |= E[m];
        } else {                                   // of equal keys, those of the later runs and places
          int above = lane / SUB < r ? extra : 0;
          left = need;
#pragma unroll
          for (int m = 0; m < M; ++m) {
            above += __popc(E[m] & ~(0xffffffffu >> (31 - lane)));
            if (extra > 0) left -= __popc(E[m] >> (r * SUB));
          }
          left = left < 0 ? 0 : left < extra ? left : extra;
#pragma unroll
          for (int m = M - 1; m >= 0; --m) {
            const bool mine = (E[m] >> lane) & 1u;
            X[m] |= __ballot_sync(0xffffffffu, mine && above < need);
            above += mine;
          }
        }
        gone = 0;
#pragma unroll
        for (int m = 0; m < M; ++m) gone += __popc((X[m] >> (lane - sub)) & (unsigned)((1ull << SUB) - 1));
        return left;
      };

      drop(window_at<M>(v, 32 * M - D), D, 0, -1);   // the D largest start there
      bool deep = sub == 0 && gone == W && top > W;  // its lane holds the run's lowest sample
      if (!__any_sync(0xffffffffu, deep)) break;

      const int at = 31 - __clz(lanes_with_max(0xffffffffu, deep, w[0]));
      if constexpr (!kLongWindow) {
        if (lane / SUB == at / SUB) top -= W;
        D -= W;
        gone = 0;
        continue;
      }
      // Run r, that of the largest such sample, goes on below its window: the next 16 M
      // samples (more than it can lose) take the place of the lower half.
      const KeyT* rrun = reinterpret_cast<const KeyT*>(__shfl_sync(0xffffffffu, (unsigned long long)run, at));
      const Idx below = __shfl_sync(0xffffffffu, top, at) - W;
      KeyT x[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const Idx f = below - (Idx)(16 * M - 1 - m - lane * M);
        x[m] = lane < 16 && f >= 1 ? rrun[(f << sh) - 1] : KeyT(0);
        v[m] = lane < 16 ? x[m] : v[m];
      }
      window_merge<32 * M, M>(v, lane);
      const KeyT t = window_at<M>(v, 32 * M - D);
      int more = 0, extra = 0;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        more += __popc(__ballot_sync(0xffffffffu, x[m] > t));
        extra += __popc(__ballot_sync(0xffffffffu, x[m] == t && lane < 16 && below >= (Idx)(16 * M - m - lane * M)));
      }
      more += drop(t, D - more, extra, at / SUB);
      deep = deep && gone == W && lane != at;
      if (!__any_sync(0xffffffffu, deep)) {
        if (lane / SUB == at / SUB) gone += more;
        break;
      }
      // Another run may have to go on too.  All that lies above the largest of their
      // lowest samples has been seen and goes for certain.
      const int at2 = 31 - __clz(lanes_with_max(0xffffffffu, deep, w[0]));
      const KeyT low = __shfl_sync(0xffffffffu, w[0], at2);
      more = W;
#pragma unroll
      for (int m = 0; m < M; ++m) more += __popc(__ballot_sync(0xffffffffu, x[m] > low));
      if (lane / SUB == at / SUB) top -= more;
      if (lane / SUB == at2 / SUB) top -= W;
      D -= more + W;
      gone = 0;
    }
    top -= gone;
    if (sh == 0) return top;
    sh -= B;
    const Idx cap = rlen >> sh;
    top = (top << B) + ((1 << B) - 1);
    top = top < cap ? top : cap;
  }
}

// Pivots of output tile j of group g, found by one warp: row[r] receives the
// number of items of run r among the group's first j * S outputs.  Arguments
// are uniform over the warp.  Idx is the type of the counts and positions of
// the search: int when n < 2^31, long long otherwise.  K2: K rounded up to a power of two;
// 0: the search by stride halving, with any K <= 32, whose positions take int when n < 2^30
// only (every position probed stays below 2n).
template <typename KeyT, int K2, typename Idx = long long>
__device__ __forceinline__ void splitter_row(const KeyT* in, long long n,
                                             long long run_len, int K, long long S, long long g,
                                             long long j, long long* row) {
  constexpr int SUB = K2 == 0 ? 1 : 32 / (K2 == 0 ? 1 : K2);
  const int lane = threadIdx.x & 31;
  const int rr = lane / SUB;                    // run of this lane
  const bool act = rr < K;
  const long long rstart = g * run_len * K + (long long)rr * run_len;
  long long rlen64 = n - rstart;
  rlen64 = rlen64 < 0 ? 0 : (rlen64 > run_len ? run_len : rlen64);
  const Idx rlen = act ? (Idx)rlen64 : Idx(0);
  const KeyT* run = in + (act ? rstart : 0);
  Idx d;
  if constexpr (K2 == 0)
    d = multiseq_pivot<KeyT, Idx, true>(run, rlen, act, K, (Idx)(j * S), 0xffffffffu);
  else
    d = window_pivot<KeyT, K2, Idx>(run, rlen, (Idx)(run_len < n ? run_len : n), (Idx)(j * S));
  if (act && lane % SUB == 0) row[rr] = d;
}

// K rounded up to a power of two (K in 2..32), for the dispatch on K2.
__host__ __device__ inline int pow2_ceil(int K) {
  int k2 = 2;
  while (k2 < K) k2 *= 2;
  return k2;
}

}  // namespace mms
