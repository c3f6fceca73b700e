"""The work that users of this framework have it do, as cases for timing it.

A case is a dict of plain values.  Its `op` names the path, and its `shapes` the tensors:

  op "pass"       Handle.pass_: one GEMV per matrix over weights that are resident in HBM.
                  `dtype` is the weights' type; `cols` is 0 for one token, or the T of a batch
                  of T activation columns.  Output: every y.
  op "digest"     Handle.checksum / wt.checksum_noalloc: the FNV-1a-64 digest of every tensor.
                  `kind` is "tree", "noalloc" or "plain".  Output: every digest.
  op "first_use"  checkpoint files in the page cache -> first use: open, allocation and ingest,
                  the event-gated pass, every y back on the host, close.  Outputs: every y and
                  the ingested tensors.

  shapes "uniform"  `n` matrices of `M` x `K`
  shapes "decoder"  `layers` decoder layers (q, k, v, o, gate, up, down; [out, in]) of width
                    `d`, `kv` key/value rows and `ffn` rows; embed and head if `vocab` > 0
  shapes "many"     the first `n` matrices of the many-small checkpoint
  shapes "spread"   `n` buffers of `lo` to `hi` bytes, log-uniform from the seed `pick`
"""
import math
import os
import random
import shutil
import tempfile

import numpy as np
import torch

from paper_2608_12114_gb300 import pipeline, synth, wt

DTYPES = {"f32": (wt.WT_F32, torch.float32, 4), "bf16": (wt.WT_BF16, torch.bfloat16, 2),
          "f16": (wt.WT_F16, torch.float16, 2), "i8": (wt.WT_I8, torch.int8, 1)}
LARGE = dict(shapes="decoder", d=4096, kv=1024, ffn=14336)
MID = dict(shapes="decoder", d=2560, kv=2560, ffn=6912)


def listed():
    return [
        # the smallest pass: eight fp32 256 x 256 matrices; a call's fixed cost
        dict(name="pass_tiny_f32", op="pass", shapes="uniform", n=8, M=256, K=256, dtype="f32", cols=0),
        # one 16 MiB matrix, the middle of the size sweep
        dict(name="pass_16mib_bf16", op="pass", shapes="uniform", n=1, M=4096, K=2048, dtype="bf16", cols=0),
        # one token through every matrix of the large decoder, 16 GB: the headline pass
        dict(name="pass_decoder_bf16", op="pass", dtype="bf16", cols=0, layers=32, vocab=128256, **LARGE),
        # the same through 1253 small matrices of 32 to 2048 columns
        dict(name="pass_many_bf16", op="pass", shapes="many", n=1253, dtype="bf16", cols=0),
        # a small decoder whose gated FFN has the unrounded width 8/3 d: rows of 2731 elements
        # (no multiple of 16 bytes) in its down projections
        dict(name="pass_ragged_f16", op="pass", shapes="decoder", layers=8, d=1024, kv=256, ffn=2731, vocab=0,
             dtype="f16", cols=0),
        # one token through int8 layers with fp16 row scales; down rows have 14336 weights
        dict(name="pass_layers_i8", op="pass", dtype="i8", cols=0, layers=4, vocab=0, **LARGE),
        # a batch of 16 tokens through bf16 layers
        dict(name="batch16_layers_bf16", op="pass", dtype="bf16", cols=16, layers=2, vocab=0, **LARGE),
        # a batch of 8 tokens through one int8 layer of the mid decoder
        dict(name="batch8_layer_i8", op="pass", dtype="i8", cols=8, layers=1, vocab=0, **MID),
        # digests that confirm an ingest: two layers, embed and head of the large decoder
        dict(name="digest_decoder", op="digest", kind="tree", dtype="bf16", layers=2, vocab=128256, **LARGE),
        # ... and the 1253 matrices of the many-small checkpoint
        dict(name="digest_many", op="digest", kind="tree", shapes="many", n=1253, dtype="bf16"),
        # the literal digest, as other tools compute it over a tensor's bytes: eight of 16 MiB
        dict(name="digest_plain", op="digest", kind="plain", shapes="uniform", n=8, M=4096, K=2048, dtype="bf16"),
        # checkpoint files -> first use: two layers, embed and head of a mid decoder
        dict(name="first_use_mid", op="first_use", dtype="bf16", layers=2, vocab=8000, **MID),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A row length: a multiple of 64 mostly, of 16, or any."""
    k = _log(rng, lo, hi)
    step = rng.choice((64, 64, 16, 1))
    return max(step, k // step * step)


def _decoder(rng, most):
    d = max(256, _log(rng, 256, 5120) // 64 * 64)
    ffn = rng.choice((3 * d, 7 * d // 2, 8 * d // 3, 27 * d // 10))
    c = dict(shapes="decoder", d=d, kv=max(64, d // rng.choice((1, 4, 8))), ffn=ffn, vocab=0, layers=1)
    layer = 2 * (2 * d * d + 2 * c["kv"] * d + 3 * d * ffn)
    c["layers"] = max(1, min(32, _log(rng, 1, 32), most // layer))
    return c


def draw(rng):
    op = rng.choice(("pass",) * 7 + ("batch",) * 4 + ("digest",) * 4 + ("first_use",))
    if op in ("pass", "batch"):
        c = dict(op="pass", dtype=rng.choice(("f32", "bf16", "bf16", "f16", "i8") if op == "pass" else ("bf16", "f16", "i8")),
                 cols=0 if op == "pass" else rng.randint(1, 16))
        s = rng.choice(("uniform", "uniform", "decoder", "many"))
        if s == "uniform":
            c.update(shapes=s, n=_log(rng, 1, 64), M=_log(rng, 64, 32768), K=_width(rng, 32, 32768))
            c["M"] = max(16, min(c["M"], (2 << 30) // (4 * c["n"] * c["K"])))
        elif s == "decoder":
            c.update(_decoder(rng, 2 << 30))
        else:
            c.update(shapes=s, n=_log(rng, 40, 1253))
        return c
    if op == "digest":
        c = dict(op="digest", kind=rng.choice(("tree", "tree", "noalloc", "plain")), dtype="bf16")
        if c["kind"] == "plain":
            c.update(shapes="spread", n=_log(rng, 1, 48), lo=64, hi=_log(rng, 1 << 12, 1 << 23), pick=rng.randint(0, 999))
        elif rng.random() < 0.5:
            c.update(shapes="spread", n=_log(rng, 1, 600), lo=1, hi=_log(rng, 1 << 12, 1 << 24), pick=rng.randint(0, 999))
        else:
            c.update(_decoder(rng, 2 << 30))
        return c
    c = dict(op="first_use", dtype="bf16", **_decoder(rng, 256 << 20))
    c["vocab"] = _log(rng, 256, 8000)
    return c


# ------------------------------------------------------------------------------ inputs

def _matrices(case):
    s = case["shapes"]
    if s == "uniform":
        return [(case["M"], case["K"])] * case["n"]
    if s == "many":
        return synth.many_shapes(1253)[:case["n"]]
    d, kv, ffn, V = case["d"], case["kv"], case["ffn"], case["vocab"]
    layer = [(d, d), (kv, d), (kv, d), (d, d), (ffn, d), (ffn, d), (d, ffn)]
    return [(V, d)] * (V > 0) + layer * case["layers"] + [(V, d)] * (V > 0)


def _buffers(case):
    """The sizes of a digest case's buffers, in bytes."""
    if case["shapes"] != "spread":
        return [2 * M * K for M, K in _matrices(case)]
    rng = random.Random(case["pick"])
    return [_log(rng, case["lo"], case["hi"]) for _ in range(case["n"])]


def _offsets(sizes, align=256):
    """Offsets of buffers of these sizes in one slab, each 256-byte aligned, and its size."""
    offs, pos = [], 0
    for n in sizes:
        offs.append(pos)
        pos += -(-n // align) * align
    return offs, max(pos, align)


def _normal(n, dtype, std, g):
    t = torch.empty(n, dtype=dtype, device="cuda")
    step = 1 << 28
    for i in range(0, n, step):
        t[i:i + step].normal_(0.0, std, generator=g)
    return t


class _Pass:
    """Weights, activations and outputs of a pass, in device memory."""

    def __init__(self, case, seed):
        g = torch.Generator("cuda").manual_seed(int(seed))
        self.dt, tdt, es = DTYPES[case["dtype"]]
        self.T = max(1, case["cols"])
        self.mats = _matrices(case)
        self.offs, total = _offsets([M * K * es for M, K in self.mats])
        if case["dtype"] == "i8":
            self.w = torch.randint(-127, 128, (total,), dtype=torch.int8, device="cuda", generator=g)
            so, st = _offsets([2 * M for M, _ in self.mats])
            self.s = (torch.rand(st // 2, device="cuda", generator=g) * 0.0018 + 0.0002).to(torch.float16)
            self.soffs = [o // 2 for o in so]
        else:
            self.w = _normal(total // es, tdt, 0.02, g)
            self.s, self.soffs = None, None
        self.x = {K: _normal(self.T * K, torch.float16 if case["dtype"] == "i8" else tdt, 1.0, g)
                  for K in dict.fromkeys(K for _, K in self.mats)}
        self.es = es
        self.rows = [M * self.T for M, _ in self.mats]
        self.y = torch.empty(sum(self.rows), dtype=torch.float32, device="cuda")

    def weight(self, i):
        M, K = self.mats[i]
        o = self.offs[i] // self.es
        return self.w[o:o + M * K].view(M, K)


class _Digest:
    """Buffers to digest, in one device slab."""

    def __init__(self, case, seed):
        g = torch.Generator("cuda").manual_seed(int(seed))
        self.sizes = _buffers(case)
        self.offs, total = _offsets(self.sizes)
        self.slab = _normal(total // 2, torch.bfloat16, 0.02, g).view(torch.uint8)
        self.out = torch.zeros(len(self.sizes), dtype=torch.int64, device="cuda")


class _Files:
    """A checkpoint's files (in the page cache after they are written) and the host side of a step."""

    def __init__(self, case, seed):
        g = torch.Generator("cuda").manual_seed(int(seed))
        self.dir = tempfile.mkdtemp(prefix="wt_cases_")
        mats, tensors = _matrices(case), []
        for i, (M, K) in enumerate(mats):
            v = _normal(M * K, torch.bfloat16, 0.02, g).view(torch.int16).cpu().numpy().view(np.uint16)
            tensors.append(synth.TensorSpec("w%d" % i, synth.DT_BF16, (M, K), 2 * i // len(mats), fill="array", array=v))
        self.paths = [os.path.join(self.dir, "part%d.wt" % f) for f in range(tensors[-1].file + 1)]
        synth.write_files(synth.Checkpoint("cases", self.paths, tensors, []))
        self.w = [(t.array, t.shape) for t in tensors]
        self.x = {K: _normal(K, torch.bfloat16, 1.0, g) for K in dict.fromkeys(K for _, K in mats)}

    def __del__(self):
        shutil.rmtree(self.dir, ignore_errors=True)


def prepare(case, seed):
    if case["op"] == "pass":
        s = _Pass(case, seed)
        s.h = wt.Handle([])
        yo = np.cumsum([0] + s.rows)
        s.descs = np.zeros(len(s.mats), wt.DESC_DTYPE)
        for i, (M, K) in enumerate(s.mats):
            s.descs[i] = (s.w.data_ptr() + s.offs[i], s.dt, case["cols"], M, K, s.x[K].data_ptr(),
                          s.y.data_ptr() + 4 * int(yo[i]), 0, 0 if s.s is None else s.s.data_ptr() + 2 * s.soffs[i])
        return s
    if case["op"] == "digest":
        s = _Digest(case, seed)
        s.kind = case["kind"]
        s.h = wt.Handle([])
        s.ptrs = [s.slab.data_ptr() + o for o in s.offs]
        return s
    s = _Files(case, seed)
    s.w = None
    with wt.Handle(s.paths, wt.WT_OPEN_HOST_ONLY) as h:
        mats = pipeline.matrices(h)
        s.x_host = pipeline.host_inputs(mats)
        for (K, _), (o, n) in pipeline.io_layout(mats)[0].items():
            s.x_host[o:o + n] = s.x[K].view(torch.uint8).cpu()
        s.y_host = torch.empty(int(mats.M.sum()), dtype=torch.float32, pin_memory=True)
    s.ingest, s.consume = torch.cuda.Stream(), torch.cuda.Stream(priority=-1)
    return s


def run(s):
    if isinstance(s, _Pass):
        s.h.pass_(s.descs, torch.cuda.current_stream().cuda_stream)
        return s.y
    if isinstance(s, _Digest):
        st = torch.cuda.current_stream().cuda_stream
        if s.kind == "noalloc":
            wt.checksum_noalloc(s.ptrs, s.sizes, s.out.data_ptr(), st)
        else:
            s.h.checksum(s.ptrs, s.sizes, s.out.data_ptr(), st, plain=s.kind == "plain")
        return s.out
    h = wt.Handle(s.paths)
    mats = pipeline.matrices(h)
    dev, events, _ = pipeline.DeviceCheckpoint.stream_in(h, mats, wt.WT_ADOPT_GATHER, s.ingest.cuda_stream, io=True)
    with torch.cuda.stream(s.consume):
        dev.io_x().copy_(s.x_host, non_blocking=True)
        ys = dev.io_outputs()
        h.pass_(dev.descs(dev.io_inputs(), ys, events), s.consume.cuda_stream)
        s.y_host.copy_(ys.buf, non_blocking=True)
    s.consume.synchronize()
    h.close()
    n = len(mats)
    some = range(n) if n <= 60 else sorted({i * (n - 1) // 59 for i in range(60)})
    return {"y": s.y_host, "weights": [dev.bufs[k] for k in some]}


# ------------------------------------------------------------------------------ what is asked of it

def work(case):
    if case["op"] == "digest":
        return {"bytes": sum(_buffers(case)) + 8 * len(_buffers(case)), "flops": 0}
    mats = _matrices(case)
    es = DTYPES[case["dtype"]][2]
    T = max(1, case.get("cols", 0))
    xes = 2 if case["dtype"] == "i8" else es
    w = sum(M * K for M, K in mats)
    rows = sum(M for M, _ in mats)
    xs = sum(set(K for _, K in mats))
    b = w * es + T * xs * xes + 4 * T * rows + (2 * rows if case["dtype"] == "i8" else 0)
    if case["op"] == "first_use":
        b += w * es  # read from the page cache, written to HBM
    return {"bytes": b, "flops": 2 * w * T}


def tolerance(case):
    """Digests and ingested bytes are exact.  The y are fp32 sums of exact products: against
    64-bit sums they are off by 5e-8 to 1.5e-7 (2-norm) where CUDA cores sum them, and by up
    to 9.2e-6 (bf16, 16 columns, rows of 14336) where tensor cores do."""
    if case["op"] == "digest":
        return "exact"
    tensor_cores = case.get("cols", 0) > 0 or case["dtype"] == "i8"
    return {"rel": 4e-5 if tensor_cores else 1e-6, "differ": 0.0}


def _fnv_bytes(data, h=0xcbf29ce484222325):
    for b in data:
        h = ((h ^ b) * 0x100000001b3) & 0xffffffffffffffff
    return h


def _leaf_digests(buf):
    """FNV-1a-64 of each 4096-byte leaf of a uint8 device tensor, as Python integers."""
    n = buf.numel()
    full = n // 4096
    out = []
    if full:
        rows = buf[:full * 4096].view(full, 4096).t().contiguous()
        h = torch.full((full,), 0xcbf29ce484222325 - (1 << 64), dtype=torch.int64, device=buf.device)
        for i in range(4096):
            h.bitwise_xor_(rows[i].to(torch.int64)).mul_(0x100000001b3)
        out = [v & 0xffffffffffffffff for v in h.tolist()]
    if n % 4096:
        out.append(_fnv_bytes(buf[full * 4096:].cpu().numpy().tobytes()))
    return out


def exact(case, seed):
    if case["op"] == "digest":
        s = _Digest(case, seed)
        if case["kind"] == "plain" and sum(s.sizes) > 1 << 25:
            return None
        if len(s.sizes) > 64 and case["kind"] != "plain":
            return None  # thousands of leaf launches for each buffer
        got = []
        for o, n in zip(s.offs, s.sizes):
            buf = s.slab[o:o + n]
            if case["kind"] == "plain":
                got.append(_fnv_bytes(buf.cpu().numpy().tobytes()))
            else:
                words = np.array([n] + _leaf_digests(buf), dtype="<u8")
                got.append(_fnv_bytes(words.tobytes()))
        return torch.from_numpy(np.array(got, np.uint64).view(np.int64))
    if case["op"] == "first_use":
        f = _Files(case, seed)
        y = []
        for w, (M, K) in f.w:
            W = torch.from_numpy(w.view(np.int16)).cuda().view(torch.bfloat16).view(M, K)
            y.append(torch.mv(W.double(), f.x[K].double()))
        some = len(f.w) if len(f.w) <= 60 else len({i * (len(f.w) - 1) // 59 for i in range(60)})
        return {"y": torch.cat(y).cpu(), "weights": [None] * some}
    s = _Pass(case, seed)
    y = []
    for i, (M, K) in enumerate(s.mats):
        W, X = s.weight(i), s.x[K].view(s.T, K).double()
        step = max(1, (1 << 28) // K)
        Y = torch.cat([X @ W[r:r + step].double().t() for r in range(0, M, step)], dim=1)
        if s.s is not None:
            Y *= s.s[s.soffs[i]:s.soffs[i] + M].double()
        y.append(Y.reshape(-1))
    return torch.cat(y)
