"""A batch with a segment above the declared maximum, of a size class whose
fanout is larger than any that the merge rounds were launched for: it is merged
with the largest of those, within their shared memory.  With rounds to spare it
comes out sorted; where they do not suffice the status word says so, and the
other segments are sorted all the same."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu



@pytest.mark.parametrize("tiles,fits", [(13, True), (16, True), (17, False), (40, False)])
@pytest.mark.parametrize("values", [False, True])
def test_batch(gpu, tiles, fits, values):
    import torch
    tile = 4096 if values else 8192
    big = tiles * tile - 77
    sizes = np.array([700, 5 * tile, big, 3, 2 * tile + 1], dtype=np.int64)
    table = {c: (4 if (1 << c) <= 8 * tile else 32) for c in range(33)}          # 8 tiles: two rounds of 4
    off = synth.offsets_of(sizes)
    keys = synth.uniform(int(off[-1]), tiles, np.uint32) % np.uint32(5000)
    vals = synth.index_payload(keys.size)
    k = torch.from_numpy(keys.view(np.int32)).cuda()
    v = torch.from_numpy(vals.view(np.int32)).cuda() if values else None
    o = torch.from_numpy(off).cuda()
    ws = torch.zeros(gpu.segmented_workspace_bytes(gpu.KEY_U32, keys.size, sizes.size, values, table, 8 * tile),
                     dtype=torch.uint8, device="cuda")
    gpu.segmented_sort(k, o, v, workspace=ws, kt=gpu.KEY_U32, class_fanout=table, max_segment_items=8 * tile)
    if fits:
        gpu.workspace_status(ws)
    else:
        with pytest.raises(gpu.MMSError):
            gpu.workspace_status(ws)
    got_k = k.cpu().numpy().view(np.uint32)
    want_k, want_v = oracle.segmented_sort(keys, off, vals)
    for a, b in zip(off[:-1], off[1:]):
        if fits or b - a != big:
            assert np.array_equal(got_k[a:b], want_k[a:b])
            if values:
                assert np.array_equal(v.cpu().numpy().view(np.uint32)[a:b], want_v[a:b])
