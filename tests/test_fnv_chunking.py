"""The arithmetic of the parallel FNV-1a-64 chains (the literal digest, and the second level of
the tree digest), restated on the host and checked against the oracle's literal FNV-1a-64 (no GPU):
a byte stream cut into chunks; per chunk a table of the low nibble from 8 starts and one of the
high nibble from 8 more; the tables composed in runs and walked; a 64-bit run per chunk from its
starting low byte; and the runs' sums, each by Horner's rule, moved to the end by powers of p^m.
A wrong derivation (a dropped d term, a lane that carries into the next, the wrong power of p, a
composition in the wrong order) fails here before any kernel runs."""
import struct

import numpy as np
import pytest

import oracle

M64 = (1 << 64) - 1
PRIME = 0x100000001B3
OFFSET = 0xCBF29CE484222325
IDENTITY = 0x76543210


def chain(h, data):
    for b in data:
        h = ((h ^ b) * PRIME) & M64
    return h


def table_of(chunk, nib=None):
    """The packed lanes of the chunk passes: the low nibble from starts 0..7 (eight-bit lanes,
    multiplier 3), or with `nib` the high nibble from starts nib + 16 j (sixteen-bit lanes); the
    nibble at the end for start j in bits 4j..4j+3."""
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
    return sum((v & 15 if nib is None else v >> 4 & 15) << (4 * j) for j, v in enumerate(lanes))


def through(table, s):
    return (table >> ((s & 7) << 2) & 15) ^ (s & 8)


def then(a, b):
    """The table of `a` followed by `b`."""
    t = a & 0x88888888
    for j in range(8):
        t ^= (b >> ((a >> (4 * j) & 7) << 2) & 15) << (4 * j)
    return t


def runs(n, walkers):
    """The contiguous shares of n items that `walkers` threads take."""
    per = -(-n // walkers)
    return [(min(n, w * per), min(n, (w + 1) * per)) for w in range(walkers)]


def walk(tables, s, walkers):
    """The state before every table from s: each walker composes its run, the composed tables are
    walked, and each walker walks its run from there."""
    starts = []
    for a, e in runs(len(tables), walkers):
        g, mine = IDENTITY, s
        for t in tables[a:e]:
            g = then(g, t)
            starts.append(mine)
            mine = through(t, mine)
        s = through(g, s)
    return starts


def fold(head, sums, lengths, m, walkers):
    """h = p^m h + D over the chunks: runs of whole chunks, their sum, then the last chunk."""
    pm, whole, h = pow(PRIME, m, 1 << 64), len(sums) - 1, 0
    for a, e in runs(whole, walkers):
        part = 0
        for d in sums[a:e]:
            part = (part * pm + d) & M64
        h += part * pow(pm, whole - e, 1 << 64)
    h = (h + head * pow(pm, whole, 1 << 64)) & M64
    return (h * pow(PRIME, lengths[-1], 1 << 64) + sums[-1]) & M64


def chained(head, stream, m, walkers):
    """h after `stream` from state `head`, in chunks of m bytes."""
    chunks = [stream[i:i + m] for i in range(0, len(stream), m)]
    low = walk([table_of(c) for c in chunks], head & 15, walkers)
    high = walk([table_of(c, nib) for c, nib in zip(chunks, low)], head >> 4 & 15, walkers)
    sums, true = [], head
    for c, lo, hi in zip(chunks, low, high):
        start = lo | hi << 4
        assert true & 0xFF == start  # the walks saw the true low bytes
        true = chain(true, c)
        sums.append((chain(start, c) - pow(PRIME, len(c), 1 << 64) * start) & M64)
    return fold(head, sums, [len(c) for c in chunks], m, walkers)


@pytest.mark.parametrize("n,m", [(1, 8), (7, 8), (8, 8), (1000, 24), (700, 256)])
def test_chunks_equal_the_serial_chain(n, m):
    rng = np.random.default_rng(n + m)
    for fill in (None, 0, 255):
        data = rng.integers(0, 256, n, dtype=np.uint8) if fill is None else np.full(n, fill, np.uint8)
        for walkers in (1, 4, 32):
            assert chained(OFFSET, data.tobytes(), m, walkers) == oracle.fnv1a64(data)
    tables = [table_of(data.tobytes())] + [table_of(data.tobytes(), k) for k in range(16)]
    for t, table in enumerate(tables):  # the 8 starts that are not run follow from the 8 that are
        for s in range(16):
            start = s if t == 0 else (t - 1) | s << 4
            end = chain(start, data.tobytes())
            assert through(table, s) == (end & 15 if t == 0 else end >> 4 & 15)


def test_tables_compose():
    rng = np.random.default_rng(5)
    for _ in range(20):
        a, b = rng.integers(0, 256, 9, dtype=np.uint8).tobytes(), rng.integers(0, 256, 5, dtype=np.uint8).tobytes()
        assert then(table_of(a), table_of(b)) == table_of(a + b)
        assert then(IDENTITY, table_of(a)) == table_of(a) == then(table_of(a), IDENTITY)


def test_chunked_chain_over_real_leaf_digests():
    """The second level proper: LE64 of the length, then the 4096-byte leaf digests; and a leaf in
    the 128-byte shares of a warp's lanes, the last one short and lanes behind it empty."""
    rng = np.random.default_rng(3)
    data = rng.integers(0, 256, 4096 * 37 + 11, dtype=np.uint8)
    leaves = [oracle.fnv1a64(data[i:i + 4096]) for i in range(0, data.size, 4096)]
    stream = struct.pack("<%dQ" % len(leaves), *leaves)
    assert chained(chain(OFFSET, struct.pack("<Q", data.size)), stream, 8 * 5, 3) == oracle.fnv_tree(data)
    for n in (1, 128, 129, 4000, 4096):
        assert chained(OFFSET, data[:n].tobytes(), 128, 32) == oracle.fnv1a64(data[:n])
