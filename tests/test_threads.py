"""Sorts from two host threads at once, each with its own stream, buffers and
workspace, whose plans launch the same kernels with different fanouts: every
call succeeds and every result equals the oracle's (mms.h: calls on distinct
streams with distinct buffers and workspaces may run concurrently)."""
import threading

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

ROUNDS = 300


def both(jobs):
    """Runs the jobs' bodies at once, ROUNDS times each; the errors they raised."""
    errors = []
    gate = threading.Barrier(len(jobs))

    def body(job):
        try:
            gate.wait()
            for _ in range(ROUNDS):
                job()
        except Exception as e:  # noqa: BLE001 - reported by the caller's assert
            errors.append(repr(e))

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


@pytest.mark.parametrize("variant", ["tree", "partition", "pipelined"])
@pytest.mark.parametrize("dtype", [np.uint32, np.uint64])
def test_whole_arrays(gpu, dtype, variant):
    import torch
    kt = gpu.KEY_U32 if dtype == np.uint32 else gpu.KEY_U64
    view = np.int32 if dtype == np.uint32 else np.int64
    mv = {"tree": gpu.MERGE_TREE, "partition": gpu.MERGE_PARTITION, "pipelined": gpu.MERGE_PIPELINED}[variant]
    n = 20 * gpu.tile_items(kt) + 77
    keys = synth.uniform(n, 5, dtype)
    want, _ = oracle.sort(keys)
    src = torch.from_numpy(keys.view(view)).cuda()
    bufs, jobs = [], []
    for fanout in (2, 32):
        s, k = torch.cuda.Stream(), src.clone()
        ws = torch.zeros(gpu.workspace_bytes(kt, n), dtype=torch.uint8, device="cuda")

        def job(s=s, k=k, ws=ws, fanout=fanout):
            gpu.sort_keys(k, fanout=fanout, workspace=ws, stream=s, kt=kt, merge_variant=mv)

        bufs.append(k)
        jobs.append(job)
    torch.cuda.synchronize()
    errors = both(jobs)
    torch.cuda.synchronize()
    assert not errors, errors
    for k in bufs:
        assert np.array_equal(k.cpu().numpy().view(dtype), want)


def test_batches(gpu):
    import torch
    sizes = np.array([100000, 3, 70001, 9000], dtype=np.int64)
    off = synth.offsets_of(sizes)
    keys = synth.uniform(int(off[-1]), 6, np.uint32)
    want, _ = oracle.segmented_sort(keys, off)
    src = torch.from_numpy(keys.view(np.int32)).cuda()
    o = torch.from_numpy(off).cuda()
    bufs, jobs = [], []
    for fanout in (2, 32):
        s, k = torch.cuda.Stream(), src.clone()
        table = {c: fanout for c in range(33)}
        ws = torch.zeros(gpu.segmented_workspace_bytes(gpu.KEY_U32, keys.size, sizes.size, False, table),
                         dtype=torch.uint8, device="cuda")

        def job(s=s, k=k, ws=ws, table=table):
            gpu.segmented_sort(k, o, workspace=ws, stream=s, kt=gpu.KEY_U32, class_fanout=table)

        bufs.append(k)
        jobs.append(job)
    torch.cuda.synchronize()
    errors = both(jobs)
    torch.cuda.synchronize()
    assert not errors, errors
    for k in bufs:
        assert np.array_equal(k.cpu().numpy().view(np.uint32), want)
