"""Performance cases: the sorts a user of this library asks for, through the package's public calls.

Four kinds of call:

* ``keys``: ``sort_keys`` on one array of u32, u64 or f32 keys;
* ``noalloc``: ``sort_keys_noalloc``, for callers that may not allocate;
* ``pairs``: ``sort_pairs``, keys with a 32-bit payload, stable;
* ``batch``: many arrays of uneven size back to back, by one direct
  ``segmented_sort`` call or by replaying a ``SegmentedGraph``.

The calls sort in place, so every pass first copies the unsorted input over the
buffer it sorts, which stands for the new keys that a program has each time.
A case's fields say everything but the values, which come from the seed.  Keys
are held as int32 / int64 (unsigned keys' bits) or float32 tensors; float
results are returned as their bits, because totalOrder tells NaN payloads and
the two zeros apart.
"""
import math
import os

import numpy as np
import torch

import paper_1702_07961_gb300 as mms
from paper_1702_07961_gb300 import autotune

KT = {"u32": mms.KEY_U32, "u64": mms.KEY_U64, "f32": mms.KEY_F32}
DTYPE = {"u32": torch.int32, "u64": torch.int64, "f32": torch.float32}
KEY_BYTES = {"u32": 4, "u64": 8, "f32": 4}


def listed():
    return [
        # The smallest request of the serving mix (2^10 keys and up): one tile, latency only.
        {"name": "keys u32 1500", "kind": "keys", "key": "u32", "n": 1500, "input": "uniform",
         "workspace": True, "offset": 0},
        # A caller that may not allocate (fixed library scratch), mid-size float keys with -0.0 and NaNs.
        {"name": "noalloc f32 100003", "kind": "noalloc", "key": "f32", "n": 100003, "input": "normal", "offset": 0},
        # The plain single-array configuration: 2^20 uniform keys, the library allocating its workspace.
        {"name": "keys u32 2^20", "kind": "keys", "key": "u32", "n": 1 << 20, "input": "uniform",
         "workspace": False, "offset": 0},
        # Float keys of an odd length, from a tensor slice that starts off the 16-byte grid.
        {"name": "keys f32 16777259", "kind": "keys", "key": "f32", "n": 16777259, "input": "normal",
         "workspace": True, "offset": 3},
        # 8-byte keys, uniform over the whole range.
        {"name": "keys u64 20000003", "kind": "keys", "key": "u64", "n": 20000003, "input": "uniform",
         "workspace": True, "offset": 0},
        # The paper's workload and the benchmark's: a random permutation of 10^8 4-byte integers.
        {"name": "keys u32 10^8", "kind": "keys", "key": "u32", "n": 10**8, "input": "permutation",
         "workspace": True, "offset": 0},
        # Nearly sorted data: a sorted list with 10^5 random pairs swapped.
        {"name": "keys u32 nearly sorted", "kind": "keys", "key": "u32", "n": 30000000, "input": "swaps",
         "swaps": 100000, "workspace": True, "offset": 0},
        # A small request with a payload (the serving mix: half of its requests carry values).
        {"name": "pairs f32 20011", "kind": "pairs", "key": "f32", "n": 20011, "input": "normal",
         "workspace": True, "offset": 0},
        # Sorting rows by a 4-byte key: the payload is the row's index; keys repeat.
        {"name": "pairs u32 30000000", "kind": "pairs", "key": "u32", "n": 30000000, "input": "uniform",
         "workspace": True, "offset": 0},
        # The same with 8-byte keys.
        {"name": "pairs u64 6000001", "kind": "pairs", "key": "u64", "n": 6000001, "input": "uniform",
         "workspace": True, "offset": 0},
        # The batched configuration: arrays of 2^8 to 2^20 keys with payloads, one graph launch, tuned fanouts.
        {"name": "batch pairs u32 2000", "kind": "batch", "key": "u32", "arrays": 2000, "lo": 256, "hi": 1 << 20,
         "sizes": 3, "values": True, "graph": True},
        # Coalesced small requests as the server forms them: one direct call, key-only, the default fanouts.
        {"name": "batch keys f32 700", "kind": "batch", "key": "f32", "arrays": 700, "lo": 256, "hi": 1 << 14,
         "sizes": 5, "values": False, "graph": False},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["keys", "keys", "keys", "noalloc", "pairs", "pairs", "batch", "batch"])
    key = rng.choice(["u32", "u64", "f32"])
    if kind == "batch":
        lo = _log_uniform(rng, 1, 2000)
        hi = _log_uniform(rng, 4 * lo, 1 << 20)
        values = rng.random() < 0.5
        # as many arrays as keep the batch within the largest listed one
        mean = (hi - lo) / math.log(hi / lo)
        most = 1.2e8 if not values else 8e7 if key != "u64" else 2e7
        return {"kind": "batch", "key": key, "arrays": _log_uniform(rng, 20, max(40, min(20000, int(most / mean)))),
                "lo": lo, "hi": hi, "sizes": rng.randrange(1, 10**6), "values": values, "graph": rng.random() < 0.5}
    if kind == "noalloc":
        n = _log_uniform(rng, 1000, (1 << 19) if key == "u64" else (1 << 20))
        return {"kind": kind, "key": key, "n": n, "input": "normal" if key == "f32" else "uniform",
                "offset": rng.randrange(4)}
    top = {"keys": {"u32": 10**8, "f32": 10**8, "u64": 4 * 10**7}, "pairs": {"u32": 3 * 10**7, "f32": 3 * 10**7, "u64": 8 * 10**6}}
    c = {"kind": kind, "key": key, "n": _log_uniform(rng, 1000, top[kind][key]),
         "input": "normal" if key == "f32" else rng.choice(["uniform", "permutation", "swaps", "interleaved"]),
         "workspace": rng.random() < 0.7, "offset": rng.choice([0, 0, 0, 1, 2, 3])}
    if c["input"] == "swaps":
        c["swaps"] = min(c["n"] // 2, _log_uniform(rng, 1, 10**7))
    elif c["input"] == "interleaved":
        c["runs"] = rng.choice([2, 4, 8, 16, 32])
        c["stride"] = rng.choice([1, 32, 33])
    return c


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _wide(v, key):
    """Small whole numbers as keys of the type (8-byte keys carry them in both halves)."""
    return (v << 32) | v if key == "u64" else v.to(torch.int32)


def _normal(n, g):
    """N(0,1) with about 1% duplicates, 0.1% -0.0 and 0.01% NaNs (of both signs, some with payloads)."""
    x = torch.randn(n, generator=g, device="cuda")
    b = x.view(torch.int32)

    def some(k):
        return torch.randint(0, n, (k,), generator=g, device="cuda")

    m = n // 100                                      # every 100th key repeats some other key
    if m:
        first = int(torch.randint(0, 100, (1,), generator=g, device="cuda"))
        b[first:first + 100 * (m - 1) + 1:100] = b[some(m)]
    b[some(max(1, n // 1000))] = -(1 << 31)
    nan = some(max(4, n // 10000))
    b[nan] = 0x7FC00000
    b[nan[: nan.numel() // 4]] = -(1 << 31) | 0x7FC00000
    b[nan[-1]] = 0x7F800001 + 12345
    return x


def _values(case, n, g):
    key, kind = case["key"], case.get("input", "uniform" if case["key"] != "f32" else "normal")
    if kind == "normal":
        return _normal(n, g)
    if kind == "uniform":
        if key == "u64":
            return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), generator=g, device="cuda")
        return torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda", dtype=torch.int32)
    # the others hold distinct whole numbers that follow each other from a start that the seed picks
    start = int(torch.randint(0, 1 << 20, (1,), generator=g, device="cuda"))
    if kind == "permutation":
        return _wide(start + torch.randperm(n, generator=g, device="cuda"), key)
    if kind == "swaps":
        a = torch.arange(n, device="cuda")
        r = case["swaps"]
        p = torch.randperm(n, generator=g, device="cuda")[: 2 * r]
        a[p[:r]], a[p[r:]] = p[r:].clone(), p[:r].clone()
        return _wide(start + a, key)
    # K ascending runs dealt out in chunks of `stride`
    p = torch.arange(n, device="cuda")
    K, s = case["runs"], case["stride"]
    c = p // s
    return _wide(start + ((c // K) * s + p % s) * K + c % K, key)


def _sizes(case):
    g = np.random.default_rng(case["sizes"])
    x = np.exp(g.uniform(math.log(case["lo"]), math.log(case["hi"] + 1), size=case["arrays"]))
    return np.clip(np.floor(x).astype(np.int64), case["lo"], case["hi"])


def _tuned():
    """The committed fanout table and tile width of the batched key-value configuration, as its users load them."""
    return autotune.load_table(os.path.join(os.path.dirname(mms.__file__), "tuned", "batched_u32_pairs.json"))


def _keys_and_payload(case, seed):
    """(keys, payload or None, sizes or None) of a case."""
    g = _gen(seed)
    sizes = _sizes(case) if case["kind"] == "batch" else None
    n = int(sizes.sum()) if sizes is not None else case["n"]
    keys = _values(case, n, g)
    has = case["kind"] == "pairs" or case.get("values", False)
    vals = torch.arange(n, device="cuda", dtype=torch.int32) if has else None
    return keys, vals, sizes


def _slice(src, offset):
    """A buffer for src's values that starts `offset` elements into its allocation."""
    return torch.empty(src.numel() + offset, dtype=src.dtype, device=src.device)[offset:]


def prepare(case, seed):
    keys, vals, sizes = _keys_and_payload(case, seed)
    kt = KT[case["key"]]
    off = case.get("offset", 0)
    st = {"case": case, "kt": kt, "src": keys, "vsrc": vals, "keys": _slice(keys, off),
          "vals": None if vals is None else _slice(vals, off), "ws": None}
    n = keys.numel()
    if case["kind"] in ("keys", "pairs"):
        if case["workspace"]:
            st["ws"] = torch.empty(mms.workspace_bytes(kt, n, vals is not None), dtype=torch.uint8, device="cuda")
    elif case["kind"] == "batch":
        o = np.zeros(sizes.size + 1, dtype=np.int64)
        np.cumsum(sizes, out=o[1:])
        st["offsets"] = torch.from_numpy(o).cuda()
        st["mx"] = int(sizes.max())
        tile, st["fanout"] = 0, None
        if case["values"] and case["key"] != "u64":
            st["fanout"], tile = _tuned()
        st["tile"] = tile
        st["ws"] = torch.empty(mms.segmented_workspace_bytes(kt, n, sizes.size, vals is not None, st["fanout"], st["mx"], tile),
                               dtype=torch.uint8, device="cuda")
        if case["graph"]:
            st["graph"] = mms.SegmentedGraph(st["keys"], st["offsets"], st["vals"], workspace=st["ws"], kt=kt,
                                             class_fanout=st["fanout"], max_segment_items=st["mx"], tile_items=tile)
    return st


def run(st):
    case, keys, vals = st["case"], st["keys"], st["vals"]
    keys.copy_(st["src"])
    if vals is not None:
        vals.copy_(st["vsrc"])
    kind = case["kind"]
    if kind == "keys":
        mms.sort_keys(keys, workspace=st["ws"], kt=st["kt"])
    elif kind == "noalloc":
        mms.sort_keys_noalloc(keys, kt=st["kt"])
    elif kind == "pairs":
        mms.sort_pairs(keys, vals, workspace=st["ws"], kt=st["kt"])
    elif case["graph"]:
        st["graph"].launch()
    else:
        mms.segmented_sort(keys, st["offsets"], vals, workspace=st["ws"], kt=st["kt"], class_fanout=st["fanout"],
                           max_segment_items=st["mx"], tile_items=st["tile"])
    return _out(keys, vals)


def _out(keys, vals):
    keys = keys.view(torch.int32) if keys.dtype == torch.float32 else keys
    return [keys] if vals is None else [keys, vals]


def work(case):
    """Every key (and payload) read once and written once; sorting does no floating-point work."""
    n = int(_sizes(case).sum()) if case["kind"] == "batch" else case["n"]
    item = KEY_BYTES[case["key"]] + (4 if case["kind"] == "pairs" or case.get("values") else 0)
    return {"bytes": 2.0 * n * item, "flops": 0.0}


def exact(case, seed):
    """A stable sort by plain torch: of the keys mapped to signed 64-bit integers in their order."""
    keys, vals, sizes = _keys_and_payload(case, seed)
    if case["key"] == "u64":
        order = keys ^ (-(1 << 63))
    else:
        b = keys.view(torch.int32).to(torch.int64)
        order = torch.where(b < 0, ~b, b + (1 << 31)) & 0xFFFFFFFF if case["key"] == "f32" else b & 0xFFFFFFFF
    at = torch.sort(order, stable=True).indices
    del order
    if sizes is not None:                                   # then stably by array
        seg = torch.repeat_interleave(torch.arange(sizes.size, device="cuda", dtype=torch.int32), torch.from_numpy(sizes).cuda())
        at = at[torch.sort(seg[at], stable=True).indices]
    return _out(keys[at], None if vals is None else vals[at])
