"""Sorts captured into a CUDA graph by the caller, behind a copy node and first
in the graph: a replay on new keys equals the oracle, and the workspace's
status word, which starts as garbage, reads clean (the first kernel clears it)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("behind_copy", [True, False])
@pytest.mark.parametrize("n", [2, 1500, 8192, 8193, 100003])
def test_sort_keys(gpu, n, behind_copy):
    import torch
    a, b = (synth.uniform(n, s, np.uint32) for s in (n, n + 1))
    src = torch.from_numpy(a.view(np.int32)).cuda()
    k = src.clone()
    ws = torch.full((gpu.workspace_bytes(gpu.KEY_U32, n),), 1, dtype=torch.uint8, device="cuda")
    gpu.sort_keys(k, workspace=ws, kt=gpu.KEY_U32)            # loads the kernels before the capture
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        if behind_copy:
            k.copy_(src)
        gpu.sort_keys(k, workspace=ws, kt=gpu.KEY_U32)
    for keys in (b, a):
        new = torch.from_numpy(keys.view(np.int32)).cuda()
        (src if behind_copy else k).copy_(new)
        ws.fill_(1)
        g.replay()
        gpu.workspace_status(ws)
        want, _ = oracle.sort(keys)
        assert np.array_equal(k.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("n", [2, 4097, 20011])
def test_sort_pairs(gpu, n):
    import torch
    keys = synth.uniform(n, n, np.uint32) % np.uint32(1000)
    src = torch.from_numpy(keys.view(np.int32)).cuda()
    k, v = src.clone(), torch.arange(n, dtype=torch.int32, device="cuda")
    vs = v.clone()
    ws = torch.full((gpu.workspace_bytes(gpu.KEY_U32, n, True),), 1, dtype=torch.uint8, device="cuda")
    gpu.sort_pairs(k, v, workspace=ws, kt=gpu.KEY_U32)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        k.copy_(src)
        v.copy_(vs)
        gpu.sort_pairs(k, v, workspace=ws, kt=gpu.KEY_U32)
    for _ in range(2):
        ws.fill_(1)
        g.replay()
        gpu.workspace_status(ws)
        want, idx = oracle.sort(keys, synth.index_payload(n))
        assert np.array_equal(k.cpu().numpy().view(np.uint32), want)
        assert np.array_equal(v.cpu().numpy().view(np.uint32), idx)
