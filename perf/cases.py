"""Measured cases of the decompression library, through its public entry points.

Inputs are the seeded synthetic FASTQ and order-2 Markov texts of the tests and the benchmark
(paper_1905_07224_gb300.synth), compressed by the host zlib.  Sizes follow the repository's own
configurations: the 1 MiB FASTQ file at level 6, the 256 MiB FASTQ files, the batch of members of
log-uniform size at levels 1/6/9, the served pool with whole members and byte ranges, the streamed
member -- scaled so that the inputs can be made in seconds.
"""
from __future__ import annotations

import math
import os
import random
import zlib
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1905_07224_gb300 import pgz, synth

KIB, MIB = 1 << 10, 1 << 20
# compressed / decompressed bytes of the synthetic texts, for work()
_RATIO = {("fastq", 1): 0.52, ("fastq", 6): 0.49, ("fastq", 9): 0.48, ("markov", 1): 0.78, ("markov", 6): 0.81,
          ("markov", 9): 0.81}


def listed():
    return [
        # a small record block decoded inside another program's loop, with no allocation allowed
        {"name": "noalloc_64k", "kind": "noalloc", "text": "fastq", "bytes": 65521, "read": 100, "level": 6},
        # one small FASTQ file, default settings: a single latency-bound call
        {"name": "file_1m", "kind": "file", "text": "fastq", "bytes": 1048576, "read": 100, "level": 6, "tail": 0,
         "parts": 0},
        # one ordinary text file at the strongest level, ragged size, with the determined-tail option
        {"name": "file_12m_markov", "kind": "file", "text": "markov", "bytes": 12 * MIB + 12345, "read": 0, "level": 9,
         "tail": 1, "parts": 0},
        # one large sequencing file at the fast level, cut into 1024 parts
        {"name": "file_256m", "kind": "file", "text": "fastq", "bytes": 256 * MIB, "read": 150, "level": 1, "tail": 0,
         "parts": 1024},
        # blocked gzip (BGZF): the usual container of sequencing tools, hundreds of small members
        {"name": "bgzf_40m", "kind": "bgzf", "text": "fastq", "bytes": 40 * MIB + 777, "read": 150, "level": 6},
        # two large files at levels 1 and 9, planned once and replayed as a graph, parts in one wave
        {"name": "graph_2x96m", "kind": "graph", "bytes": 96 * MIB, "read": 150},
        # many members of very different sizes, levels 1/6/9, FASTQ and Markov text, in one batch
        {"name": "batch_96", "kind": "batch", "members": 96, "lo": 64 * KIB, "hi": 8 * MIB, "chunk": 65536, "wpb": 4,
         "pipe": 0},
        # the same from pinned host memory, large enough for overlapped groups
        {"name": "host_batch_24", "kind": "host", "members": 24, "lo": 8 * MIB, "hi": 32 * MIB},
        # a host-resident member decoded in segments with bounded device memory
        {"name": "stream_64m", "kind": "stream", "bytes": 64 * MIB + 4321, "read": 150, "level": 6, "segment": 8 * MIB},
        # byte ranges of one indexed resident member
        {"name": "ranges_64m", "kind": "ranges", "bytes": 64 * MIB, "read": 150, "level": 6, "count": 8,
         "lo": 4 * KIB, "hi": MIB},
        # random access: from a bit offset to the member's end, and the DNA reads in the symbols
        {"name": "at_12m", "kind": "at", "bytes": 12 * MIB, "read": 150, "level": 6, "from": 0.6},
        # a served mix of whole members and byte ranges over resident files
        {"name": "served_40", "kind": "served", "files": 20, "lo": 64 * KIB, "hi": 12 * MIB, "requests": 40, "slots": 4},
    ]


def _logint(rng: random.Random, lo: int, hi: int) -> int:
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng: random.Random):
    kind = rng.choice(["noalloc", "file", "file", "bgzf", "graph", "batch", "batch", "host", "stream", "ranges", "at",
                       "served"])
    level = rng.choice([1, 6, 9])
    read = rng.choice([75, 100, 150, 250])
    if kind == "noalloc":
        return {"kind": kind, "text": rng.choice(["fastq", "markov"]), "bytes": _logint(rng, 8 * KIB, 3 * MIB),
                "read": read, "level": level}
    if kind == "file":
        text = rng.choice(["fastq", "fastq", "markov"])
        n = _logint(rng, 64 * KIB, (128 if text == "fastq" else 12) * MIB)
        return {"kind": kind, "text": text, "bytes": n, "read": read, "level": level, "tail": rng.choice([0, 0, 1]),
                "parts": rng.choice([0, 0, 0, max(1, n // 262144)])}
    if kind == "bgzf":
        return {"kind": kind, "text": "fastq", "bytes": _logint(rng, 256 * KIB, 64 * MIB), "read": read, "level": level}
    if kind == "graph":
        return {"kind": kind, "bytes": _logint(rng, 4 * MIB, 96 * MIB), "read": read}
    if kind == "batch":
        return {"kind": kind, "members": rng.randint(5, 128), "lo": _logint(rng, 16 * KIB, 256 * KIB),
                "hi": _logint(rng, MIB, 8 * MIB), "chunk": rng.choice([32768, 65536, 100000, 131072]),
                "wpb": rng.choice([2, 4, 8]), "pipe": rng.choice([0, 1])}
    if kind == "host":
        return {"kind": kind, "members": rng.randint(2, 24), "lo": _logint(rng, 64 * KIB, 4 * MIB),
                "hi": _logint(rng, 6 * MIB, 24 * MIB)}
    if kind == "stream":
        return {"kind": kind, "bytes": _logint(rng, 8 * MIB, 96 * MIB), "read": read, "level": level,
                "segment": _logint(rng, 2 * MIB, 32 * MIB)}
    if kind == "ranges":
        return {"kind": kind, "bytes": _logint(rng, 4 * MIB, 96 * MIB), "read": read, "level": level,
                "count": rng.randint(1, 12), "lo": _logint(rng, KIB, 16 * KIB), "hi": _logint(rng, 64 * KIB, 2 * MIB)}
    if kind == "at":
        return {"kind": kind, "bytes": _logint(rng, MIB, 16 * MIB), "read": read, "level": level,
                "from": rng.uniform(0.5, 0.95)}
    return {"kind": kind, "files": rng.randint(4, 24), "lo": 64 * KIB, "hi": _logint(rng, MIB, 12 * MIB),
            "requests": rng.randint(8, 48), "slots": rng.choice([2, 4])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_PIECE = 4 * MIB


def _pool():
    return ThreadPoolExecutor(max(1, len(os.sched_getaffinity(0))))


def _texts(specs):
    """One text per (kind, bytes, read length, seed); drawn in pieces over threads."""
    with _pool() as pool:
        fut = []
        for kind, n, read, seed in specs:
            if kind == "markov":
                fut.append([pool.submit(synth.markov, n, seed)])
            else:
                fut.append([pool.submit(synth.fastq, min(_PIECE, n - a), read, 0.001, seed * 1009 + a // _PIECE)
                            for a in range(0, n, _PIECE)])
        return [b"".join(f.result() for f in fs) for fs in fut]


def _deflate(job):
    data, dic, level, last = job
    c = zlib.compressobj(level, zlib.DEFLATED, -15, 8, zlib.Z_DEFAULT_STRATEGY, *([dic] if dic else []))
    return c.compress(data) + c.flush(zlib.Z_FINISH if last else zlib.Z_SYNC_FLUSH)


def _gzips(texts, levels):
    """One gzip member per text; a text above one piece is deflated in pieces over threads, as pigz does."""
    with _pool() as pool:
        fut = []
        for data, level in zip(texts, levels):
            n = len(data)
            fut.append((data, [pool.submit(_deflate, (data[a:a + _PIECE], data[max(0, a - 32768):a] if a else b"",
                                                      level, a + _PIECE >= n)) for a in range(0, max(n, 1), _PIECE)]))
        out = []
        for data, fs in fut:
            out.append(bytes([0x1F, 0x8B, 8, 0, 0, 0, 0, 0, 0, 255]) + b"".join(f.result() for f in fs) +
                       (zlib.crc32(data) & 0xFFFFFFFF).to_bytes(4, "little") +
                       (len(data) & 0xFFFFFFFF).to_bytes(4, "little"))
        return out


def _bgzf(data, level):
    with _pool() as pool:
        step = 64 * 65280
        fs = [pool.submit(synth.bgzf_compress, data[a:a + step], level, 65280, a + step >= len(data))
              for a in range(0, len(data), step)]
        return b"".join(f.result() for f in fs)


def _member_specs(case, seed):
    """(kind, bytes, read length, seed) and level of the members of a batch, log-uniform sizes."""
    r = random.Random(case["members"] * 7919 + case["lo"] + case["hi"])
    specs, levels = [], []
    for k in range(case["members"]):
        kind = "markov" if case["kind"] == "batch" and k % 4 == 3 else "fastq"
        specs.append((kind, _logint(r, case["lo"], case["hi"]), 150, seed * 131 + k))
        levels.append(r.choice([1, 6, 9]) if case["kind"] == "batch" else 1)
    return specs, levels


def _dev(data: bytes):
    return torch.from_numpy(np.frombuffer(data, dtype=np.uint8).copy()).cuda()


def _arena(sizes, host):
    """One zeroed output buffer and its slices, each starting on a 256-byte boundary."""
    offs = [0]
    for n in sizes:
        offs.append(offs[-1] + (n + 255) // 256 * 256)
    kw = {"pin_memory": True} if host else {"device": "cuda"}
    whole = torch.zeros(offs[-1], dtype=torch.uint8, **kw)
    return whole, [whole[a:a + n] for a, n in zip(offs, sizes)]


class _State:
    """What a program holds: a context (or server), its buffers and plan; released with the object."""

    def __init__(self, case):
        self.case = case
        self.ctx = self.server = self.batch = self.index = None

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.batch is not None:
                self.batch.free()
            if self.index is not None:
                pgz.pgz_index_free(self.index)
            if self.server is not None:
                self.server.close()
            if self.ctx is not None:
                pgz.pgz_destroy(self.ctx)
        except Exception:
            pass


def _context(**kw):
    return pgz.pgz_create(pgz.pgz_config_init(cuda_stream=torch.cuda.current_stream().cuda_stream, **kw))


def prepare(case, seed):
    kind = case["kind"]
    s = _State(case)
    if kind in ("noalloc", "file", "bgzf", "stream", "ranges", "at"):
        text = case.get("text", "fastq")
        data = _texts([(text, case["bytes"], case["read"], seed + 11)])[0]
        gz = _bgzf(data, case["level"]) if kind == "bgzf" else _gzips([data], [case["level"]])[0]
        s.n = len(data)
        if kind == "stream":
            s.gz = np.frombuffer(gz, dtype=np.uint8)
            s.out = np.zeros(len(data), dtype=np.uint8)
            s.ctx = _context()
            return s
        s.gz = _dev(gz)
        s.gz_len = len(gz)
        if kind == "at":
            s.bit = int(8 * len(gz) * case["from"])
            cap = int(len(data) * (1.0 - case["from"]) * 1.25) + MIB
            s.sym = torch.zeros(cap, dtype=torch.int16, device="cuda")
            s.out = torch.zeros(cap, dtype=torch.uint8, device="cuda")
            s.spans = torch.zeros((cap // case["read"] + 1024, 2), dtype=torch.int64, device="cuda")
            s.ctx = _context()
            return s
        if kind == "ranges":
            r = random.Random(case["bytes"] + case["count"])
            s.ranges = []
            for _ in range(case["count"]):
                n = min(case["bytes"], _logint(r, case["lo"], case["hi"]))
                s.ranges.append((r.randint(0, case["bytes"] - n), n))
            s.outs = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _, n in s.ranges]
            s.ctx = _context()
            s.index = pgz.pgz_index_build(s.ctx, s.gz.data_ptr(), s.gz_len)
            return s
        s.out = torch.zeros(len(data) + 64, dtype=torch.uint8, device="cuda")
        if kind == "file":
            s.ctx = _context(determined_tail=case["tail"], n_chunks=case["parts"])
        elif kind == "bgzf":
            s.ctx = _context()
        else:
            s.stream = torch.cuda.current_stream().cuda_stream
        return s
    if kind == "graph":
        datas = _texts([("fastq", case["bytes"], case["read"], seed + 17 + k) for k in range(2)])
        gzs = _gzips(datas, [1, 9])
        s.gzs = [_dev(g) for g in gzs]
        s.outs = [torch.zeros(len(d), dtype=torch.uint8, device="cuda") for d in datas]
        s.jobs = [(g.data_ptr(), len(b), o.data_ptr(), o.numel()) for g, b, o in zip(s.gzs, gzs, s.outs)]
        s.ctx = _context()
        _, chunk, _ = pgz.pgz_wave_chunk_bytes(s.ctx, s.jobs, 4, 1.0)
        pgz.pgz_set_tuning(s.ctx, max(chunk, 32768), 4, 0)
        s.batch = pgz.Batch(s.ctx, s.jobs)
        return s
    if kind in ("batch", "host"):
        specs, levels = _member_specs(case, seed)
        datas = _texts(specs)
        gzs = _gzips(datas, levels)
        s.out, s.outs = _arena([len(d) for d in datas], kind == "host")
        if kind == "batch":
            s.gzs = [_dev(g) for g in gzs]
            s.ctx = _context(chunk_bytes=case["chunk"], warps_per_block=case["wpb"], exec_pipelined=case["pipe"])
        else:
            s.gzs = []
            for g in gzs:
                t = torch.empty(len(g), dtype=torch.uint8, pin_memory=True)
                t.copy_(torch.from_numpy(np.frombuffer(g, dtype=np.uint8).copy()))
                s.gzs.append(t)
            s.ctx = _context(chunk_bytes=131072)
        s.jobs = [(g.data_ptr(), g.numel(), o.data_ptr(), o.numel()) for g, o in zip(s.gzs, s.outs)]
        return s
    # served: resident files; requests drawn once, 70 % whole members, 30 % byte ranges
    r = random.Random(case["files"] * 31 + case["requests"])
    sizes = [_logint(r, case["lo"], case["hi"]) for _ in range(case["files"])]
    datas = _texts([("fastq", n, 150, seed * 17 + k) for k, n in enumerate(sizes)])
    s.gzs = [_dev(g) for g in _gzips(datas, [(1, 6)[k & 1] for k in range(case["files"])])]
    torch.cuda.synchronize()
    s.server = pgz.Server(pgz.pgz_config_init(), slots=case["slots"], mem_budget=16 << 30)
    ids = [s.server.add_file(g.data_ptr(), g.numel()) for g in s.gzs]
    drawn = []
    for _ in range(case["requests"]):
        f = r.randrange(case["files"])
        if r.random() < 0.7:
            off, n = 0, None
        else:
            n = min(sizes[f], _logint(r, 4 * KIB, MIB))
            off = r.randint(0, sizes[f] - n)
        drawn.append((f, off, n))
    s.out, outs = _arena([sizes[f] if n is None else n for f, _, n in drawn], False)
    s.reqs = [(ids[f], off, n, o) for (f, off, n), o in zip(drawn, outs)]
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s.case["kind"]
    if kind == "noalloc":
        st, n = pgz.pgz_decompress_noalloc(s.gz.data_ptr(), s.gz_len, s.out.data_ptr(), s.out.numel(), s.stream)
        return {"status": st, "len": n, "out": s.out[:n]}
    if kind in ("file", "bgzf"):
        st, n, _ = pgz.pgz_decompress(s.ctx, s.gz.data_ptr(), s.gz_len, s.out.data_ptr(), s.out.numel())
        return {"status": st, "len": n, "out": s.out[:n]}
    if kind == "stream":
        out, pos = s.out, [0]

        def sink(view):
            k = len(view)
            out[pos[0]:pos[0] + k] = np.frombuffer(view, dtype=np.uint8)
            pos[0] += k
            return False

        st, n, _, _ = pgz.pgz_decompress_stream(s.ctx, s.gz, s.case["segment"], sink)
        return {"status": st, "len": n, "out": out[:n]}
    if kind == "ranges":
        st = [pgz.pgz_decompress_range(s.ctx, s.index, off, n, o.data_ptr()) for (off, n), o in zip(s.ranges, s.outs)]
        return {"status": max(st), "outs": s.outs}
    if kind == "at":
        st, n, bit, det = pgz.pgz_decompress_at(s.ctx, s.gz.data_ptr(), s.gz_len, s.bit, s.sym.data_ptr(),
                                                s.out.data_ptr(), ord("?"), s.out.numel())
        st2, found, und = pgz.pgz_extract_sequences(s.ctx, s.sym.data_ptr(), n, 40, s.spans.data_ptr(),
                                                    s.spans.shape[0])
        # the spans come in no particular order: sorted by their start (rows not written are zero)
        return {"status": max(st, st2), "len": n, "bit": bit, "determined": det, "found": found, "undetermined": und,
                "symbols": s.sym, "out": s.out, "spans": s.spans[torch.argsort(s.spans[:, 0], stable=True)]}
    if kind == "graph":
        st, per, _ = s.batch.run()
        return {"status": st, "lens": np.array([n for _, n in per]), "outs": s.outs}
    if kind in ("batch", "host"):
        call = pgz.pgz_decompress_batch if kind == "batch" else pgz.pgz_decompress_batch_host
        st, per, _ = call(s.ctx, s.jobs)
        return {"status": st, "lens": np.array([n for _, n in per]), "out": s.out}
    reqs = [s.server.submit(f, o.data_ptr(), o.numel(), off, n) for f, off, n, o in s.reqs]
    s.server.drain()
    return {"status": max(q.status for q in reqs), "lens": np.array([q.out_len for q in reqs]), "out": s.out}


def work(case):
    """Bytes one pass cannot do without: the compressed bytes read once and the output written once."""
    kind = case["kind"]
    if kind in ("noalloc", "file", "bgzf", "stream"):
        n = case["bytes"]
        b = n * (1.0 + _RATIO[(case.get("text", "fastq"), case["level"])])
    elif kind == "graph":
        b = case["bytes"] * (2.0 + _RATIO[("fastq", 1)] + _RATIO[("fastq", 9)])
    elif kind in ("batch", "host"):
        specs, levels = _member_specs(case, 0)
        b = sum(n * (1.0 + _RATIO[(k, lv)]) for (k, n, _, _), lv in zip(specs, levels))
    elif kind == "ranges":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        b = case["count"] * mean * (1.0 + _RATIO[("fastq", case["level"])])
    elif kind == "at":
        n = case["bytes"] * (1.0 - case["from"])
        b = n * (3.0 + _RATIO[("fastq", case["level"])])
    else:
        r = random.Random(case["files"] * 31 + case["requests"])
        sizes = [_logint(r, case["lo"], case["hi"]) for _ in range(case["files"])]
        b = 0.0
        for _ in range(case["requests"]):
            f = r.randrange(case["files"])
            if r.random() < 0.7:
                n = sizes[f]
            else:
                n = min(sizes[f], _logint(r, 4 * KIB, MIB))
                r.randint(0, sizes[f] - n)
            b += 1.5 * n
    return {"bytes": int(b), "flops": 0}


def exact(case, seed):
    """Every output is bytes and whole numbers, which stay equal; no computed real numbers."""
    return None
