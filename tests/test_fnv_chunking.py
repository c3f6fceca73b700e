"""The arithmetic the parallel second level of the tree digest rests on, restated on the
host and checked against the oracle's literal FNV-1a-64 (no GPU): a chain over a byte
stream cut into chunks, combined from per-chunk low-byte tables, a low-word run from each
chunk's starting low byte, a scan of the low word and a fold of the high word, equals the
serial chain.  A wrong derivation (a dropped d term, the high word's carry, the wrong power
of p, the packed 16-bit lanes) fails here before any kernel runs."""
import struct

import numpy as np
import pytest

import oracle

M32 = 0xFFFFFFFF
P = 0x1B3  # FNV-1a-64's prime is 2^40 + 0x1b3


def step(lo, hi, b):
    """One byte on the split state: x = lo ^ b; x p = low32(x 0x1b3) + (hi 0x1b3 + (x << 8) +
    high32(x 0x1b3)) 2^32 mod 2^64."""
    x = lo ^ b
    w = x * P
    return w & M32, (hi * P + (w >> 32) + (x << 8)) & M32


def run(lo, hi, data):
    for b in data:
        lo, hi = step(lo, hi, b)
    return lo, hi


def low_byte_table(chunk):
    """l_end for all 256 starting low bytes, four starts per 'thread' in two registers of two
    16-bit lanes, multiplier 0xb3 (= p mod 256); the mask of one step merged into the next."""
    mask = 0x00FF00FF
    out = [0] * 256
    for tid in range(64):
        r0 = tid | (tid + 64) << 16
        r1 = (tid + 128) | (tid + 192) << 16
        for b in chunk:
            bb = b | b << 16
            r0 = (((r0 & mask) ^ bb) * 0xB3) & M32
            r1 = (((r1 & mask) ^ bb) * 0xB3) & M32
        out[tid], out[tid + 64] = r0 & 0xFF, (r0 >> 16) & 0xFF
        out[tid + 128], out[tid + 192] = r1 & 0xFF, (r1 >> 16) & 0xFF
    return out


def chunked(head, stream, m):
    """FNV-1a-64 of head + stream with the stream cut into chunks of m bytes."""
    lo, hi = run(0x84222325, 0xCBF29CE4, head)
    chunks = [stream[i:i + m] for i in range(0, len(stream), m)]
    tabs = [low_byte_table(c) for c in chunks]
    ls, l = [], lo & 0xFF                       # walk the low byte through the tables
    for t in tabs:
        ls.append(l)
        l = t[l]
    bparts = []                                 # B from the starting low byte alone
    for c, l0 in zip(chunks, ls):
        lo_end = l0
        for b in c:
            lo_end = ((lo_end ^ b) * P) & M32
        bparts.append((lo_end - pow(P, len(c), 1 << 32) * l0) & M32)
    starts = []                                 # lo at every chunk start
    for c, bp in zip(chunks, bparts):
        starts.append(lo)
        lo = (pow(P, len(c), 1 << 32) * lo + bp) & M32
    for c, s, l0 in zip(chunks, starts, ls):    # the walk saw the true low bytes
        assert s & 0xFF == l0
    for c, s in zip(chunks, starts):            # hi folded over H from each true start
        _, h = run(s, 0, c)
        hi = (pow(P, len(c), 1 << 32) * hi + h) & M32
    return hi << 32 | lo


@pytest.mark.parametrize("nwords,m", [(1, 8), (2, 8), (5, 16), (9, 24), (40, 64), (64, 512)])
def test_chunked_chain_equals_the_serial_digest(nwords, m):
    rng = np.random.default_rng(nwords * 1000 + m)
    for trial in range(4):
        words = rng.integers(0, 2 ** 63, nwords, dtype=np.uint64) * (1 + trial % 2)
        if trial == 2:
            words[:] = 0
        if trial == 3:
            words[:] = np.uint64(2 ** 64 - 1)
        n = int(rng.integers(0, 2 ** 40))
        head = struct.pack("<Q", n)
        stream = words.astype("<u8").tobytes()
        assert chunked(head, stream, m) == oracle.fnv1a64(head + stream)


def test_chunked_chain_over_real_leaf_digests():
    """The second level proper: the stream is LE64 of the 4096-byte leaf digests."""
    rng = np.random.default_rng(3)
    data = rng.integers(0, 256, 4096 * 37 + 11, dtype=np.uint8)
    leaves = [oracle.fnv1a64(data[i:i + 4096]) for i in range(0, data.size, 4096)]
    stream = struct.pack("<%dQ" % len(leaves), *leaves)
    assert chunked(struct.pack("<Q", data.size), stream, 8 * 5) == oracle.fnv_tree(data)


# ----------------------------------------------------------------------------- nibble by nibble

M64 = (1 << 64) - 1
PRIME = 0x100000001B3


def chain(h, data):
    for b in data:
        h = ((h ^ b) * PRIME) & M64
    return h


def nibble_tables(chunk, nib=None):
    """The packed lanes of the chunk passes: the low nibble from starts 0..7 (eight-bit lanes,
    multiplier 3), or with `nib` the high nibble from starts nib + 16 j (sixteen-bit lanes)."""
    if nib is None:
        regs, mask, mul, rep, width = [0x03020100, 0x07060504], 0x0F0F0F0F, 3, 0x01010101, 8
    else:
        regs = [(nib + 32 * i) | (nib + 32 * i + 16) << 16 for i in range(4)]
        mask, mul, rep, width = 0x00FF00FF, 0xB3, 0x00010001, 16
    for b in chunk:
        for i, r in enumerate(regs):
            u = (r ^ (b * rep)) & mask
            assert all((u >> s & ((1 << width) - 1)) * mul < 1 << width for s in range(0, 32, width))
            regs[i] = (u * mul) & 0xFFFFFFFF
    lanes = [r >> s for r in regs for s in range(0, 32, width)]
    return [v & 15 if nib is None else v >> 4 & 15 for v in lanes]


def through(table, s):
    return table[s & 7] ^ (s & 8)


def chained(head, stream, m):
    """h after `stream` from state `head`, in chunks of m bytes: low nibbles, high nibbles, the
    64-bit sums D, the fold."""
    chunks = [stream[i:i + m] for i in range(0, len(stream), m)]
    low, s = [], head & 15
    for c in chunks:
        low.append(s)
        s = through(nibble_tables(c), s)
    start, s = [], head >> 4 & 15
    for c, nib in zip(chunks, low):
        start.append(nib | s << 4)
        s = through(nibble_tables(c, nib), s)
    h = head
    for c, l in zip(chunks, start):
        assert h & 0xFF == l
        pm = pow(PRIME, len(c), 1 << 64)
        h = (pm * h + chain(l, c) - pm * l) & M64
    return h


@pytest.mark.parametrize("n,m", [(1, 8), (7, 8), (8, 8), (1000, 24), (700, 256)])
def test_nibble_chunks_equal_the_serial_chain(n, m):
    rng = np.random.default_rng(n + m)
    for fill in (None, 0, 255):
        data = rng.integers(0, 256, n, dtype=np.uint8) if fill is None else np.full(n, fill, np.uint8)
        assert chained(0xCBF29CE484222325, data.tobytes(), m) == oracle.fnv1a64(data)
    tables = [nibble_tables(data.tobytes())] + [nibble_tables(data.tobytes(), k) for k in range(16)]
    for t, table in enumerate(tables):  # the 8 starts that are not run follow from the 8 that are
        for s in range(16):
            l = s if t == 0 else (t - 1) | s << 4
            end = chain(l, data.tobytes())
            assert through(table, s) == (end & 15 if t == 0 else end >> 4 & 15)
