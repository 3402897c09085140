"""Host model of a merge CTA's plan as it is (merge_tile.cuh: merge_plan_warp
and MergeGeom; mms_common.cuh: warp_corank_pair).

A segment's span carries 16 items of slack.  That suffices because only a node
that merges uses space past its output (the rows of its last block, up to 31
items), and such a node has two segments at least; a node with an empty child is
copied, item for item.  The model lays out random tiles and checks, for every
fanout and number of runs the group holds:
  * the spans fit the capacity, and three CTAs fit an SM with any fanout;
  * every node writes inside its own segments' spans;
  * the block list is complete, without gaps, at most 71 long, network blocks
    before small and copied ones in every level.
The two-sided co-rank search is replayed for its result and its rounds.
"""
import numpy as np
import pytest

BLOCK, SMALL, SLACK, MAX_ITEMS = 1024, 256, 16, 72


def cap(S, K, E):
    return S + (K * (2 * E - 2 + SLACK) + E - 1) // E * E + E


def nodes_of(kruns):
    out, cnt, level = [], max(kruns, 2), 1
    while cnt > 1:
        cnt = (cnt + 1) // 2
        out += [(level, q) for q in range(cnt)]
        level += 1
    return out


def random_lengths(g, kruns, S):
    want = int(g.integers(1, S + 1)) if g.random() < 0.5 else S
    kind = g.integers(0, 3)
    if kind == 0:                                          # anywhere, many empty
        cuts = np.sort(g.integers(0, want + 1, kruns - 1))
    elif kind == 1:                                        # all from one or two runs
        cuts = np.sort(g.choice([0, want // 3, want], kruns - 1))
    else:
        cuts = np.arange(1, kruns) * want // kruns
    return np.diff(np.concatenate([[0], cuts, [want]])).astype(int)


@pytest.mark.parametrize("size", [4, 8])
@pytest.mark.parametrize("K", [2, 3, 5, 8, 11, 16, 27, 32])
def test_layout_and_block_list(size, K):
    g = np.random.default_rng(100 * size + K)
    E, S = 16 // size, 8192 if size == 4 else 4096
    for trial in range(150):
        kruns = int(g.integers(1, K + 1))
        lens = np.zeros(K, dtype=int)
        lens[:kruns] = random_lengths(g, kruns, S)
        heads = g.integers(0, E, K)
        spans = (heads + lens + E - 1) // E * E + SLACK
        R = np.concatenate([[0], np.cumsum(spans)])
        assert R[-1] <= cap(S, K, E) and np.all(R % E == 0)
        pre = np.concatenate([[0], np.cumsum(lens)])
        first_of = 0
        for lv in range(1, 1 + max(level for level, _ in nodes_of(kruns))):
            network, others, outs = [], [], []
            for level, q in nodes_of(kruns):
                if level != lv:
                    continue
                a, m, b = (min(x, K) for x in (q << lv, (q << lv) + (1 << (lv - 1)), (q + 1) << lv))
                lenA, lenB = pre[m] - pre[a], pre[b] - pre[m]
                L = int(lenA + lenB)
                blocks = [(int(R[a]), d, min(BLOCK, L - d)) for d in range(0, L, BLOCK)]
                copied = lenA == 0 or lenB == 0
                small = blocks if copied else blocks[-1:] if blocks and blocks[-1][2] <= SMALL else []
                network += blocks[:len(blocks) - len(small)]
                others += small
                used = L if copied else max(-(-L // 32) * 32, L)
                assert R[a] + used <= R[b], "past its own segments' spans"
                outs.append((int(R[a]), int(R[a]) + used))
            assert all(x[1] <= y[0] for x, y in zip(outs, outs[1:]))
            assert sum(m for _, _, m in network + others) == pre[-1]
            first_of += len(network) + len(others)
        assert first_of <= MAX_ITEMS - 1


def test_three_ctas_fit_an_sm():
    ctl = 4 * (32 + 4 * MAX_ITEMS)
    for size, S in ((4, 8192), (8, 4096)):
        for K in range(2, 33):
            assert 3 * (size * 2 * cap(S, K, 16 // size) + 16 + ctl + 1024) <= 228 * 1024


def corank_pair(A, B, d, m):
    """Both searches of warp_corank_pair, and the rounds they take together."""
    state = []
    for dd in (d, d + m):
        state.append([max(0, dd - len(B)), min(dd, len(A)), dd])
    rounds = 0
    while any(hi > lo for lo, hi, _ in state):
        rounds += 1
        for s in state:
            lo, hi, dd = s
            step = ((hi - lo + 15) >> 4) | 1
            hit = -1
            for lane in range(16):
                i = lo + lane * step
                if i >= hi or A[i] > B[dd - 1 - i]:
                    hit = lane
                    break
            top = lo + hit * step
            s[0] = lo + 15 * step + 1 if hit < 0 else lo if hit == 0 else top - step + 1
            s[1] = hi if hit < 0 else min(top, hi)
    return state[0][0], state[1][0], rounds


def rounds_for(r):
    """Rounds that a range of r positions takes at worst: a round leaves at most its step less one,
    or what lies past the last probe."""
    n = 0
    while r > 0:
        step = ((r + 15) >> 4) | 1
        r = max(step - 1, r - 15 * step - 1)
        n += 1
    return n


def test_corank_pair():
    g = np.random.default_rng(1)
    for trial in range(300):
        a, b = int(g.integers(0, 4097)), int(g.integers(0, 4097))
        A, B = np.sort(g.integers(0, 200, a)), np.sort(g.integers(0, 200, b))
        m = int(g.integers(0, min(1024, a + b) + 1))
        d = int(g.integers(0, a + b - m + 1))
        want = [int(np.sum(np.argsort(np.concatenate([A, B]), kind="stable")[:k] < a)) for k in (d, d + m)]
        c0, c1, rounds = corank_pair(A, B, d, m)
        assert [c0, c1] == want and rounds <= rounds_for(max(a, b))
    assert rounds_for(4368) == 3 and rounds_for(4369) == 4
