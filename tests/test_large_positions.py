"""Sorts whose positions need more than 31 bits: from 2^31 keys on the splitter
counts in 64 bits, whole arrays and batches alike.  The keys are i -> i * m mod
n over an array of n (m prime to n), so that each array must sort to iota."""
import math

import numpy as np
import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

STEP = 1 << 27
N = (1 << 31) + 12345


def fill(t, n):
    """t[i] = i * m mod n, in chunks."""
    import torch
    m = 2654435761
    while n and math.gcd(m, n) != 1:
        m += 2
    for a in range(0, n, STEP):
        i = torch.arange(a, min(n, a + STEP), dtype=torch.int64, device=t.device)
        t[a:a + i.numel()] = (i * (m % n) % n).to(t.dtype)      # both factors below n: no overflow


def is_iota(t):
    import torch
    for a in range(0, t.numel(), STEP):
        b = min(t.numel(), a + STEP)
        want = torch.arange(a, b, dtype=torch.int64, device=t.device)
        if not torch.equal(t[a:b].to(torch.int64) & 0xFFFFFFFF, want):
            return False
    return True


@pytest.mark.parametrize("dtype", ["u32", "u64"])
def test_one_array(gpu, dtype):
    import torch
    kt, td = (gpu.KEY_U32, torch.int32) if dtype == "u32" else (gpu.KEY_U64, torch.int64)
    t = torch.empty(N, dtype=td, device="cuda")
    fill(t, N)
    ws = torch.empty(gpu.workspace_bytes(kt, N), dtype=torch.uint8, device="cuda")
    gpu.sort_keys(t, workspace=ws, kt=kt)
    gpu.workspace_status(ws)
    assert is_iota(t)


def test_batch(gpu):
    import torch
    sizes = [5, (1 << 31) - 70000, 0, 90001]                    # 2^31 + 20006 in all
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    t = torch.empty(int(off[-1]), dtype=torch.int32, device="cuda")
    for a, n in zip(off, sizes):
        fill(t[a:a + n], n)
    o = torch.from_numpy(off).cuda()
    ws = torch.empty(gpu.segmented_workspace_bytes(gpu.KEY_U32, t.numel(), len(sizes)), dtype=torch.uint8, device="cuda")
    gpu.segmented_sort(t, o, workspace=ws, kt=gpu.KEY_U32)
    gpu.workspace_status(ws)
    for a, n in zip(off, sizes):
        assert is_iota(t[a:a + n])
