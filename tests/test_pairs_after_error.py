"""A key-value batch whose offsets leave items out: the status word reports it,
the well-formed segments are sorted as ever, and the value gathers stay inside
the batch although the left-out items' workspace was never written (here all
bits set, which as a position lies far outside every array)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.uint32, np.float32, np.uint64])
def test_offsets_that_end_early(gpu, dtype):
    import ctypes

    import torch
    n, off = 20011, np.array([0, 4000, 9000, 15000], dtype=np.int64)      # 9000 .. n belongs to no good segment
    keys = synth.normal_f32(n, 1) if dtype == np.float32 else synth.uniform(n, 1, dtype) % dtype(1000)
    kt = {np.uint32: gpu.KEY_U32, np.float32: gpu.KEY_F32, np.uint64: gpu.KEY_U64}[dtype]
    view = {np.uint32: np.int32, np.float32: np.float32, np.uint64: np.int64}[dtype]
    o = torch.from_numpy(off).cuda()
    k = torch.from_numpy(keys.view(view)).cuda()
    v = torch.from_numpy(synth.index_payload(n).view(np.int32)).cuda()
    ws = torch.full((gpu.segmented_workspace_bytes(kt, n, 3, True),), 0xFF, dtype=torch.uint8, device="cuda")
    opts = gpu._seg_opts()
    st = gpu.load().mms_segmented_sort(kt, gpu._ptr(k), gpu._ptr(v), gpu._ptr(o), 3, n, gpu._ptr(ws), ws.numel(),
                                       gpu._stream_handle(None), ctypes.byref(opts))
    assert st == 0
    with pytest.raises(gpu.MMSError):
        gpu.workspace_status(ws)
    bits = np.uint64 if dtype == np.uint64 else np.uint32
    got_k, got_v = k.cpu().numpy().view(bits), v.cpu().numpy().view(np.uint32)
    for a, b in ((0, 4000), (4000, 9000)):
        want_k, want_v = oracle.sort(keys[a:b].copy(), synth.index_payload(n)[a:b].copy())
        assert np.array_equal(got_k[a:b], want_k.view(bits))
        assert np.array_equal(got_v[a:b], want_v)
    assert np.all(got_v < n)                       # gathered from inside the batch
