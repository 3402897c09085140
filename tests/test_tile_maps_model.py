"""Host model of the tile sort's warp levels as they are (tile_sort.cuh:
blocked_to_striped_rev, blocked_to_linear; mms_common.cuh: store_striped4,
load_row), on a byte-addressed buffer, for 4- and 8-byte keys.

It replays the address arithmetic -- rows of a second half stored at their
mirrored place, column offsets built up one XOR a row, the stmatrix addresses
(8-byte keys: low halves, then high halves, 128 bytes on), the word-by-word
stores of a short block, the way out in order -- and checks that each map is
the transpose it is meant to be, that the levels sort 1024 keys, and that every
access is free of bank conflicts: 16-byte accesses by quarters of a warp, 8-byte
ones by halves, 4-byte ones by warps.
"""
import numpy as np
import pytest

LANES = range(32)
DTYPE = {4: np.uint32, 8: np.uint64}


class Shared:
    def __init__(self, size):
        self.size, self.RB, self.E = size, 32 * size, 16 // size
        self.buf = np.zeros(32 * self.RB, dtype=np.uint8)

    def access(self, addr, width):
        """One instruction: the lanes' addresses, `width` bytes each."""
        addr = np.asarray(addr)
        assert np.all(addr % width == 0) and addr.min() >= 0 and addr.max() + width <= self.buf.size
        for a in addr.reshape(-1, 32 if width == 4 else 128 // width):
            assert len(set(a % 128 // width)) == a.size, "bank conflict"

    def store(self, addr, keys):
        """keys[lane]: the item or items of the lane."""
        keys = np.ascontiguousarray(keys)
        rows = keys.reshape(len(addr), -1).view(np.uint8)
        self.access(addr, rows.shape[1])
        for a, r in zip(addr, rows):
            self.buf[a:a + r.size] = r

    def load(self, addr, dtype, count=1):
        width = np.dtype(dtype).itemsize * count
        self.access(addr, width)
        return np.array([self.buf[a:a + width].view(dtype) for a in addr])


def striped_rev(blocked, h, size):
    """Registers k of lane l after blocked_to_striped_rev."""
    m = Shared(size)
    place = [(l ^ (h - 1)) if l & h else l for l in LANES]
    row = [(p * m.RB) ^ ((p & 7) << 4) for p in place]
    for ch in range(32 // m.E):
        m.store([r ^ (ch << 4) for r in row], blocked[:, ch * m.E:(ch + 1) * m.E])
    mir = [31 * size if (h >> b) & 1 else 0 for b in range(5)]
    c = [np.arange(32) * size]
    out = np.empty((32, 32), dtype=DTYPE[size])
    for k in range(32):
        if k:
            p = k & (k - 1)
            b = (k & -k).bit_length() - 1
            c.append(c[p] ^ mir[b] ^ (m.E * ((k & 7) ^ (p & 7)) * size))
        out[k] = m.load(c[k] + k * m.RB, DTYPE[size])[:, 0]
    return out


def to_blocked(striped, size, rows=32):
    """Lane l's row l after striped_to_blocked with `rows` rows wanted."""
    m = Shared(size)
    halves = striped.view(np.uint32).reshape(32, 32, size // 4)                  # row, lane, half
    for q in range(8):
        nr = rows - 4 * q
        for half in range(size // 4):
            if nr >= 4:                                                          # stmatrix: lane T holds an address
                addr = [(4 * q + (t >> 3)) * m.RB + (((t & 7) ^ (t >> 3) ^ 4 * (q & 1)) << 4) + 128 * half for t in LANES]
                m.store(addr, np.stack([halves[4 * q + (t >> 3), 4 * (t & 7):4 * (t & 7) + 4, half] for t in LANES]))
            else:
                for k in range(max(0, nr)):
                    addr = [(4 * q + k) * m.RB + ((l ^ (4 * (k + 4 * (q & 1)))) << 2) + 128 * half for l in LANES]
                    m.store(addr, halves[4 * q + k, :, half])
    out = np.empty((32, 32, size // 4), dtype=np.uint32)
    for ch in range(8):
        for half in range(size // 4):
            addr = [l * m.RB + ((ch ^ (l & 7)) << 4) + 128 * half for l in LANES]
            out[:, 4 * ch:4 * ch + 4, half] = m.load(addr, np.uint32, 4)
    return out.reshape(32, -1).view(DTYPE[size])


def to_linear(blocked, size):
    m = Shared(size)
    cpr = 32 // m.E
    for ch in range(cpr):
        m.store([((l * m.RB) ^ ((l & 7) << 4)) ^ (ch << 4) for l in LANES], blocked[:, ch * m.E:(ch + 1) * m.E])
    regs = []
    for q in range(cpr):
        r = [q * (32 // cpr) + l // cpr for l in LANES]
        regs.append(m.load([r[l] * m.RB + (((l % cpr) ^ (r[l] & 7)) << 4) for l in LANES], DTYPE[size], m.E))
    for q in range(cpr):
        m.store([(32 * q + l) << 4 for l in LANES], regs[q])
    return m.buf.view(DTYPE[size])


def keys_of(size, seed, distinct=True):
    g = np.random.default_rng(seed)
    top = 1 << (8 * size - 1)
    return (g.integers(0, top, 1024) if distinct else g.integers(0, 7, 1024) * (top // 7)).astype(DTYPE[size])


@pytest.mark.parametrize("size", [4, 8])
@pytest.mark.parametrize("h", [1, 2, 4, 8, 16])
def test_second_halves_come_reversed(size, h):
    rows = keys_of(size, h).reshape(32, 32)
    got = striped_rev(rows, h, size)
    for b in range(0, 32, 2 * h):
        want = np.concatenate([rows[b:b + h].reshape(-1), rows[b + h:b + 2 * h].reshape(-1)[::-1]])
        assert np.array_equal(got[b:b + 2 * h].reshape(-1), want)


@pytest.mark.parametrize("size", [4, 8])
@pytest.mark.parametrize("rows", [1, 2, 3, 4, 5, 7, 8, 22, 31, 32])
def test_striped_to_blocked(size, rows):
    x = keys_of(size, 3).reshape(32, 32)
    assert np.array_equal(to_blocked(x, size, rows)[:rows], x[:rows])


@pytest.mark.parametrize("size", [4, 8])
def test_blocked_to_linear(size):
    x = keys_of(size, 4)
    assert np.array_equal(to_linear(x.reshape(32, 32), size), x)


@pytest.mark.parametrize("size", [4, 8])
@pytest.mark.parametrize("distinct", [True, False])
def test_the_levels_sort(size, distinct):
    keys = keys_of(size, 5, distinct)
    v = np.sort(keys.reshape(32, 32), axis=1)

    def half_cleaners(x, s):
        while s >= 1:
            for k in range(32):
                if not k & s:
                    x[k], x[k + s] = np.minimum(x[k], x[k + s]), np.maximum(x[k], x[k + s])
            s //= 2

    for h in (1, 2, 4, 8, 16):
        v = striped_rev(v, h, size)
        half_cleaners(v, h)                                                      # strides 32 h .. 32
        v = to_blocked(v, size)
        half_cleaners(v.T, 16)                                                   # strides 16 .. 1, inside the lane
    assert np.array_equal(to_linear(v, size), np.sort(keys))
