"""Sorts captured where their first kernel, which is launched to start early,
has more than one thing before it, or one of this library's kernels: behind
the join of two streams, and behind another sort.  Each replay runs on new
keys and equals the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

N = 8192 * 3 + 5


def dev(a):
    import torch
    return torch.from_numpy(a.view(np.int32)).cuda()


def host(t):
    return t.cpu().numpy().view(np.uint32)


def batch_parts(gpu, n):
    import torch
    off = np.array([0, 100, 100, n], dtype=np.int64)
    ws = torch.full((gpu.segmented_workspace_bytes(gpu.KEY_U32, n, 3),), 1, dtype=torch.uint8, device="cuda")
    return off, torch.from_numpy(off).cuda(), ws


@pytest.mark.parametrize("kind", ["one array", "batch"])
@pytest.mark.parametrize("last", ["copy", "sort"])
def test_behind_a_join(gpu, kind, last):
    """Two streams each fill a half of the keys; `last` is what each ends with
    (a copy, or a sort of its half, whose last kernel is one of the library's)."""
    import torch
    src, k = dev(synth.uniform(N, 1)), dev(synth.uniform(N, 2))
    h = 8192 * 2
    halves = [(0, h), (h, N)]
    ws = torch.full((gpu.workspace_bytes(gpu.KEY_U32, N),), 1, dtype=torch.uint8, device="cuda")
    wh = [torch.full((gpu.workspace_bytes(gpu.KEY_U32, N),), 1, dtype=torch.uint8, device="cuda") for _ in halves]
    off, o, wb = batch_parts(gpu, N)
    side = torch.cuda.Stream()

    def fill(i):
        a, b = halves[i]
        k[a:b].copy_(src[a:b])
        if last == "sort":
            gpu.sort_keys(k[a:b], workspace=wh[i], kt=gpu.KEY_U32)

    def work():
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            fill(1)
        fill(0)
        main.wait_stream(side)
        if kind == "batch":
            gpu.segmented_sort(k, o, workspace=wb, kt=gpu.KEY_U32)
        else:
            gpu.sort_keys(k, workspace=ws, kt=gpu.KEY_U32)

    work()                                          # loads the kernels, and the same uncaptured
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        work()
    for seed in (3, 4):
        keys = synth.uniform(N, seed)
        src.copy_(dev(keys))
        g.replay()
        torch.cuda.synchronize()
        if kind == "batch":
            gpu.workspace_status(wb)
            halved = keys if last == "copy" else np.concatenate([oracle.sort(keys[a:b].copy())[0] for a, b in halves])
            want, _ = oracle.segmented_sort(halved, off)
        else:
            gpu.workspace_status(ws)
            want, _ = oracle.sort(keys)
        assert np.array_equal(host(k), want)


@pytest.mark.parametrize("first", [1500, 8192 * 2 + 1])
def test_sort_behind_a_sort(gpu, first):
    """A sort whose input another sort's kernels have just written."""
    import torch
    src, k = dev(synth.uniform(N, 5)), dev(synth.uniform(N, 6))
    ws = torch.full((gpu.workspace_bytes(gpu.KEY_U32, N),), 1, dtype=torch.uint8, device="cuda")

    def work():
        k.copy_(src)
        gpu.sort_keys(k[:first], workspace=ws, kt=gpu.KEY_U32)
        gpu.sort_keys(k, workspace=ws, kt=gpu.KEY_U32)

    work()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        work()
    for seed in (7, 8):
        keys = synth.uniform(N, seed)
        src.copy_(dev(keys))
        g.replay()
        gpu.workspace_status(ws)
        assert np.array_equal(host(k), oracle.sort(keys)[0])
