"""8-byte keys of many rows take the splitter's stride halving, of few its window
search: one table over many groups of runs equals the tables of its groups, on
either side of the line, and where the halving table is small enough to ask,
the oracle's.  Runs that drive the searches off their usual path, groups that
are ragged, ties.  Whole numbers: equal, no tolerance."""
import numpy as np
import pytest

import oracle
from test_window_splitter import runs_of

pytestmark = pytest.mark.gpu

LINE = 3584                                      # rows from which stride halving runs (splitter.cu)


def table(gpu, keys, run_len, K):
    import torch
    return gpu.splitter(torch.from_numpy(keys.view(np.int64)).cuda(), run_len, K, kt=gpu.KEY_U64).cpu().numpy()


@pytest.mark.parametrize("K,mult", [(5, 3), (8, 1), (11, 2), (16, 4), (27, 5), (32, 1)])
@pytest.mark.parametrize("kind", ["scales", "two dense", "disjoint down", "nearly sorted", "ties"])
def test_one_table_equals_its_groups(gpu, kind, K, mult):
    S = gpu.tile_items(gpu.KEY_U64)
    run_len = S * mult
    per_group = K * mult                         # rows of a full group
    groups = [runs_of(kind, K, run_len, run_len, np.uint64, g) for g in range(3)]
    tail = runs_of(kind, max(1, K // 2), run_len, run_len // 2 + 3, np.uint64, 9)
    count = LINE // per_group + 1
    big = np.concatenate([groups[i % 3] for i in range(count)] + [tail])
    rows = [table(gpu, g, run_len, K) for g in groups]
    assert all(len(r) == per_group < LINE for r in rows)
    want = np.concatenate([rows[i % 3] for i in range(count)] + [table(gpu, tail, run_len, K)])
    got = table(gpu, big, run_len, K)
    assert len(got) >= LINE and np.array_equal(got, want)
    few = np.concatenate([groups[i % 3] for i in range((LINE - 1) // per_group)])      # just below the line
    assert np.array_equal(table(gpu, few, run_len, K), np.concatenate([rows[i % 3] for i in range((LINE - 1) // per_group)]))


def test_against_the_oracle(gpu):
    S = gpu.tile_items(gpu.KEY_U64)
    keys = np.concatenate([runs_of("two dense", 8, S, S, np.uint64, g) for g in range(LINE // 8 + 1)])
    assert np.array_equal(table(gpu, keys, S, 8), oracle.splitter_table(keys, S, 8, S))
