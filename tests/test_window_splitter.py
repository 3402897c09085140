"""The splitter's window search on runs that drive it off its usual path: one
run holding most of a level's largest samples (the window moves down), runs
that do not overlap, ties everywhere, short and empty last runs.  Whole
numbers against the oracle's brute-force table: equal, no tolerance."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def runs_of(kind, K, run_len, last, dtype, seed):
    g = np.random.default_rng(seed)
    top = np.iinfo(dtype).max
    out = []
    for r in range(K):
        n = run_len if r < K - 1 else last
        if kind == "scales":          # every run over a range of its own size
            x = g.integers(0, 1 << (4 + 3 * (r % 8)), n)
        elif kind == "one dense":     # run K // 2 crowds the upper values of the others
            x = g.integers(900, 1000, n) if r == K // 2 else g.integers(0, 1000, n)
        elif kind == "disjoint up":
            x = r * run_len + np.arange(n)
        elif kind == "nearly sorted":  # disjoint runs but for one sample in ten, which lies anywhere
            x = np.where(g.random(n) < 0.1, g.integers(0, K * run_len, n), r * run_len + np.arange(n))
        elif kind == "two dense":      # two runs hold the upper values, with ties
            x = g.integers(990, 1000, n) if r in (1, K // 2 + 1) else g.integers(0, 1000, n)
        elif kind == "disjoint down":
            x = (K - r) * run_len + np.arange(n)
        else:                         # "ties": two values, the largest key among them
            x = np.where(g.random(n) < 0.5, dtype(7), dtype(top))
        out.append(np.sort(x.astype(dtype)))
    return np.concatenate(out)


@pytest.mark.parametrize("dtype", [np.uint32, np.uint64])
@pytest.mark.parametrize("kind", ["scales", "one dense", "two dense", "disjoint up", "disjoint down", "nearly sorted", "ties"])
@pytest.mark.parametrize("K,mult", [(2, 1), (5, 3), (8, 1), (11, 2), (16, 1), (27, 1), (32, 2)])
def test_tables(gpu, dtype, kind, K, mult):
    import torch
    kt = gpu.KEY_U32 if dtype == np.uint32 else gpu.KEY_U64
    S = gpu.tile_items(kt)
    run_len = S * mult
    pre = np.concatenate([runs_of(kind, K, run_len, run_len, dtype, K),      # a full group, then a ragged one
                          runs_of(kind, (K + 1) // 2, run_len, run_len // 2 + 3, dtype, K + 1)])
    view = {np.uint32: np.int32, np.uint64: np.int64}[dtype]
    got = gpu.splitter(torch.from_numpy(pre.view(view)).cuda(), run_len, K, kt=kt).cpu().numpy()
    want = oracle.splitter_table(pre, run_len, K, S)
    assert np.array_equal(got, want)
