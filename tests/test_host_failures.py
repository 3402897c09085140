"""What a sort queues after one of its CUDA calls has failed, with a runtime
that runs nothing in the real one's place (fake_cudart.cc).  A workspace that
the library allocated is always given back, and its status word is forwarded
to the per-device word only once what clears that word has been queued."""
import ctypes
import glob
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1702_07961_gb300 import _build_lib as b
    objs = lambda: sorted(glob.glob(os.path.join(b.BUILD, "*.o")))           # noqa: E731
    b.build(force=len(objs()) < len(glob.glob(os.path.join(b.CSRC, "*.cu"))))
    so = str(tmp_path_factory.mktemp("fake") / "libmms_fake.so")
    cuda = os.path.dirname(os.path.dirname(b._nvcc())) or "/usr/local/cuda"
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                           "-o", so, os.path.join(HERE, "fake_cudart.cc"), *objs()])
    L = ctypes.CDLL(so)
    L.fake_log.restype = ctypes.c_char_p
    return L


def sort(fake, kind, kt, n, fail, base_items=0):
    """Status and log of one sort without a workspace whose calls matching `fail` fail."""
    import paper_1702_07961_gb300 as mms
    fake.fake_reset(fail.encode())
    o = mms._opts(0, base_items=base_items)
    at, zero = ctypes.c_void_p(1 << 20), ctypes.c_size_t(0)
    if kind == "keys":
        st = fake.mms_sort_keys_ex(kt, at, ctypes.c_size_t(n), None, zero, None, ctypes.byref(o))
    else:
        st = fake.mms_sort_pairs_ex(kt, at, at, ctypes.c_size_t(n), None, zero, None, ctypes.byref(o))
    return st, fake.fake_log().decode().split()


# kind, key type, keys, what fails, base_items; whether the word has been cleared by then
BEFORE = [("keys", 0, 100000, "tile_sort", 0), ("keys", 1, 100000, "tile_sort", 0), ("keys", 0, 100000, "memset", 16384),
          ("pairs", 0, 100000, "copy", 0), ("pairs", 2, 100, "tile_sort", 0), ("pairs", 1, 100000, "u64_split", 0),
          ("pairs", 1, 100000, "tile_sort", 0)]
AFTER = [("keys", 0, 100000, "splitter", 0), ("keys", 1, 100000, "merge_pass", 0), ("keys", 0, 100000, "tile_sort", 16384),
         ("pairs", 0, 100000, "pairs_finalize", 0), ("pairs", 1, 100000, "u64_mid", 0), ("pairs", 1, 100000, "u64_out", 0),
         ("keys", 0, 100000, "nothing", 0), ("pairs", 1, 100000, "nothing", 0)]


@pytest.mark.parametrize("case", BEFORE + AFTER, ids=lambda c: f"{c[0]}-{c[1]}-{c[3]}-{c[4]}")
def test_status_word(fake, case):
    st, log = sort(fake, *case[:3], case[3], case[4])
    assert (st == 0) == (case[3] == "nothing")
    assert log.count("malloc") == 1 and log.count("free") == 1 and log[-1] == "free"
    assert any("forward_status" in x for x in log) == (case in AFTER)
