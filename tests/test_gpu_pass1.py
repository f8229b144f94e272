"""Pass 1 at the edges of its kernels' tiles: passes of the copy-map executor and segments of the block decoder."""
import base64
import functools
import zlib

import numpy as np
import pytest

import deflate_writer as dw
import oracle
from gpu_util import Ctx, empty, to_device
from paper_1905_07224_gb300 import synth

pytestmark = pytest.mark.gpu

DISTS = [1, 2, 3, 7, 8, 9, 255, 256, 257, 2047, 2048, 4095, 4096, 4097, 8191, 8192, 8193, 16384, 24576, 32759, 32767,
         32768]


@functools.lru_cache(maxsize=None)
def _copies(n, seed):
    """A member of exactly n bytes of literals and copies whose distances lie around the executor's pass sizes (4096
    and 8192 positions), its 16-bit pointers' and the window's ends, overlapping copies included."""
    rng = np.random.default_rng(seed)
    tokens, size = [], 0
    while size < n:
        d = int(rng.choice(DISTS))
        if d > size or n - size < 3 or rng.random() < 0.2:
            tokens.append(("lit", int(rng.choice(list(b"ACGT\n")))))
            size += 1
        else:
            length = min(int(rng.choice([3, 4, 7, 8, 9, 31, 64, 257, 258])), n - size)
            tokens.append(("match", length, d))
            size += length
    w = dw.BitWriter()
    for a in range(0, len(tokens), 5000):
        dw.write_dynamic(w, tokens[a:a + 5000], a + 5000 >= len(tokens))
    text = dw.expand(tokens)
    assert len(text) == n
    return dw.gzip_wrap(w.tobytes(), text), text


@pytest.mark.parametrize("tail", [0, 1])
@pytest.mark.parametrize("members", [1, 160])
def test_copies_across_the_executors_passes(members, tail):
    """One member alone and many at once (the executor's block size depends on the number of parts)."""
    sizes = [1, 7, 8, 9, 4095, 4096, 4097, 8191, 8192, 8193, 32768, 40960, 40961, 90001]
    ctx = Ctx(determined_tail=tail)
    try:
        for n in sizes if members == 1 else [0]:
            made = [_copies(n, n)] if members == 1 else [_copies(sizes[k % len(sizes)], k // 14) for k in range(members)]
            gz = [to_device(g) for g, _ in made]
            out = [empty(len(t)) for _, t in made]
            st, per, _ = ctx.pgz.pgz_decompress_batch(
                ctx.h, [(d.data_ptr(), len(g), o.data_ptr(), len(t)) for d, o, (g, t) in zip(gz, out, made)])
            assert st == 0, (n, ctx.pgz.pgz_strerror(st))
            for (_, t), o, (s, k) in zip(made, out, per):
                assert s == 0 and k == len(t) and o[:k].cpu().numpy().tobytes() == t
    finally:
        ctx.close()


@functools.lru_cache(maxsize=None)
def _dense(kind):
    """Members whose blocks stress the block decoder's segments: tokens of very few bits, codes of one length (parses
    that start wrong stay wrong), fixed codes, and many small blocks."""
    rng = np.random.default_rng(len(kind))
    if kind == "runs":
        text = b"A" * 3_000_000 + b"AC" * 400_000
        c = zlib.compressobj(9, zlib.DEFLATED, 31)
    elif kind == "base64":
        text = base64.b64encode(rng.integers(0, 256, 400_000, dtype=np.uint8).tobytes())
        c = zlib.compressobj(6, zlib.DEFLATED, 31)
    elif kind == "one_length":
        text = rng.choice(np.frombuffer(bytes(range(33, 97)), dtype=np.uint8), 500_000).tobytes()
        c = zlib.compressobj(6, zlib.DEFLATED, 31, 8, zlib.Z_HUFFMAN_ONLY)
    elif kind == "two_literals":
        text = (rng.random(600_000) < 0.3).astype(np.uint8).tobytes().replace(b"\0", b"x").replace(b"\1", b"y")
        c = zlib.compressobj(6, zlib.DEFLATED, 31, 8, zlib.Z_HUFFMAN_ONLY)
    elif kind == "fixed":
        text = synth.fastq(700_000, 100, 0.001, 4)
        c = zlib.compressobj(6, zlib.DEFLATED, 31, 8, zlib.Z_FIXED)
    else:                                            # memLevel 1: blocks of 127 tokens
        text = synth.fastq(500_000, 100, 0.001, 5)
        c = zlib.compressobj(6, zlib.DEFLATED, 31, 1)
    return c.compress(text) + c.flush(), text


@pytest.mark.parametrize("wpb", [2, 4, 8])
@pytest.mark.parametrize("kind", ["runs", "base64", "one_length", "two_literals", "fixed", "small_blocks"])
def test_block_decoder_edges(kind, wpb):
    """Every team size (16 warps with few parts, the configured size with many), one part and many."""
    gz, text = _dense(kind)
    for n in [1, 5, 310, 700, 2500]:
        ctx = Ctx(n_chunks=n, warps_per_block=wpb, min_block=16)
        try:
            st, out, k, _ = ctx.decompress(gz, out_cap=len(text) + 1000)
            assert st == 0, (n, ctx.pgz.pgz_strerror(st))
            assert k == len(text) and out == text, n
        finally:
            ctx.close()


@pytest.mark.parametrize("chunk", [4096, 16384, 65536])
@pytest.mark.parametrize("kind", ["fastq", "markov", "runs", "tail"])
def test_decoding_from_an_offset_in_several_parts(kind, chunk):
    """pgz_decompress_at over one, two and many parts equals the oracle's one symbolic decode: symbols, bytes, block
    start, last placeholder; so do the inspection calls, which report one part."""
    import torch
    text = {"fastq": lambda: synth.fastq(900_001, 150, 0.001, 8), "markov": lambda: synth.markov(400_003, 9),
            "runs": lambda: (b"@ab\n" * 40_000 + synth.fastq(200_000, 100, 0.0, 3)) * 2,
            "tail": lambda: synth.fastq(150_000, 100, 0.0, 4)}[kind]()
    gz = synth.gzip_compress(text, 6)
    ctx = Ctx(chunk_bytes=chunk)
    try:
        d = to_device(gz)
        cap = len(text) + 1000
        for start in [0, 8 * len(gz) // 5, 8 * len(gz) // 2 + 3]:
            ref = oracle.decompress_at(gz, start, fill=ord("?"))
            sym, byt = torch.zeros(cap, dtype=torch.int16, device="cuda"), empty(cap)
            st, n, bb, fd = ctx.pgz.pgz_decompress_at(ctx.h, d.data_ptr(), len(gz), start, sym.data_ptr(),
                                                      byt.data_ptr(), ord("?"), cap)
            if ref["status"]:
                assert st != 0
                continue
            assert st == 0, ctx.pgz.pgz_strerror(st)
            assert (n, bb, fd) == (ref["sym"].size, ref["block_bit"], ref["first_determined"])
            assert np.array_equal(sym[:n].cpu().numpy().view(np.uint16), ref["sym"])
            assert byt[:n].cpu().numpy().tobytes() == ref["bytes"]
            sb, ns, nph = ctx.pgz.pgz_inspect_parts(ctx.h)
            assert list(sb) == [bb] and list(ns) == [n] and list(nph) == [int((ref["sym"] >= 0x8000).sum())]
            assert np.array_equal(ctx.pgz.pgz_inspect_symbols(ctx.h, 0), ref["sym"])
            st, n, _, _ = ctx.pgz.pgz_decompress_at(ctx.h, d.data_ptr(), len(gz), start, None, None, 0, n - 1)
            assert st == ctx.pgz.PGZ_E_CAPACITY and n == ref["sym"].size
    finally:
        ctx.close()


@pytest.mark.parametrize("chunk", [4096, 16384, 65536, 1 << 20])
def test_decoding_a_damaged_member_from_an_offset(chunk):
    """One block after another given the reserved type: whatever the parts (1 MiB: a single one), the verdict is the
    oracle's -- the start is refused if the damage lies in its window of six blocks, else the data is invalid -- and
    where it is success, so are the block start and the symbols."""
    import torch
    c = zlib.compressobj(6, zlib.DEFLATED, 31, 7)
    text = synth.fastq(800_000, 150, 0.001, 8)
    gz = c.compress(text) + c.flush()
    _, _, blocks, _ = oracle.gunzip(gz, max_blocks=1000)
    start = 8 * (len(gz) // 5)
    later = [int(b) for b in blocks if b >= start]
    ctx = Ctx(chunk_bytes=chunk)
    try:
        P = ctx.pgz
        verdicts = {0: 0, -3: P.PGZ_E_DATA, -13: P.PGZ_E_NOSYNC}
        seen = set()
        for b in later[:8] + later[8::5] + later[-1:]:
            bad = bytearray(gz)
            for k in (1, 2):
                bad[(b + k) // 8] |= 1 << (b + k) % 8
            ref = oracle.decompress_at(bytes(bad), start, fill=ord("?"), cap=len(text))
            sym, byt = torch.zeros(len(text), dtype=torch.int16, device="cuda"), empty(len(text))
            d = to_device(bytes(bad))
            st, n, bb, fd = P.pgz_decompress_at(ctx.h, d.data_ptr(), len(bad), start, sym.data_ptr(), byt.data_ptr(),
                                                ord("?"), len(text))
            assert st == verdicts[ref["status"]], (b, P.pgz_strerror(st))
            seen.add(st)
            if st == 0:
                assert (n, bb, fd) == (ref["sym"].size, ref["block_bit"], ref["first_determined"])
                assert np.array_equal(sym[:n].cpu().numpy().view(np.uint16), ref["sym"])
                assert byt[:n].cpu().numpy().tobytes() == ref["bytes"]
        assert {0, P.PGZ_E_DATA} <= seen
    finally:
        ctx.close()


def test_the_autotuner_runs_each_configuration_once():
    """Both execution forms are one: asked for, they are listed with the one time measured, for the same launches."""
    text = synth.fastq(300_000, 100, 0.001, 7)
    gz = synth.gzip_compress(text, 6)
    ctx = Ctx()
    try:
        P = ctx.pgz
        d, out = to_device(gz), empty(len(text))
        job = [(d.data_ptr(), len(gz), out.data_ptr(), len(text))]
        launches = []
        for sweep in (False, True):
            k = P.pgz_kernel_launches(ctx.h)
            st, entries, best = P.pgz_autotune(ctx.h, job, [16384, 65536], [4], 2, sweep_exec=sweep)
            launches.append(P.pgz_kernel_launches(ctx.h) - k)
            assert st == 0 and len(entries) == (4 if sweep else 2)
        assert launches[0] == launches[1]
        assert [e["exec_pipelined"] for e in entries] == [0, 1, 0, 1]
        assert [e["ms"] for e in entries[::2]] == [e["ms"] for e in entries[1::2]]
        assert best["ms"] == min(e["ms"] for e in entries)
    finally:
        ctx.close()


@pytest.mark.parametrize("chunk", [16384, 65536])
def test_errors_from_an_offset_are_decoded_once(chunk):
    """A buffer too small, no block start, invalid data past the first start's window: each is reported by the run in
    parts, with the launches of one run (and, for the length, its symbols put in order once more), and what the
    inspection calls report is what a run in one part leaves."""
    c = zlib.compressobj(6, zlib.DEFLATED, 31, 4)
    text = synth.fastq(600_000, 150, 0.001, 8)
    noise = np.random.default_rng(4).integers(0, 256, 300_000, dtype=np.uint8).tobytes()
    gz = c.compress(text + noise) + c.flush()
    _, _, blocks, _ = oracle.gunzip(gz, max_blocks=5000)
    start = 8 * (len(gz) // 20)
    after = [int(b) for b in blocks if b >= start]
    quiet = 8 * (len(gz) - 200_000)
    assert oracle.decompress_at(gz, quiet)["status"] == -13
    bad = bytearray(gz)
    for k in (1, 2):                                   # the 8th block from the start: past its window, in its part
        bad[(after[7] + k) // 8] |= 1 << (after[7] + k) % 8
    assert after[7] < start + 8 * chunk and oracle.decompress_at(bytes(bad), start)["status"] == -3
    cap = len(text) + len(noise)
    out = empty(cap)
    ctx = Ctx(chunk_bytes=chunk)
    try:
        P = ctx.pgz
        d, db = to_device(gz), to_device(bytes(bad))

        def at(dev, bit, cap):
            k = P.pgz_kernel_launches(ctx.h)
            r = P.pgz_decompress_at(ctx.h, dev.data_ptr(), len(gz), bit, None, out.data_ptr(), ord("?"), cap)
            return r[0], r[1], P.pgz_kernel_launches(ctx.h) - k

        ref = oracle.decompress_at(gz, start, cap=cap)
        st, n, once = at(d, start, cap)
        assert (st, n) == (0, ref["sym"].size)
        for small in (n - 1, 1000, 0):
            st, k, launches = at(d, start, small)
            assert (st, k) == (P.PGZ_E_CAPACITY, n) and launches < 2 * once
            sb, ns, nph = P.pgz_inspect_parts(ctx.h)
            assert list(sb) == [ref["block_bit"]] and list(ns) == [n]
            assert list(nph) == [int((ref["sym"] >= 0x8000).sum())]
            assert np.array_equal(P.pgz_inspect_symbols(ctx.h, 0), ref["sym"])
        for dev, bit, want in ((d, quiet, P.PGZ_E_NOSYNC), (db, start, P.PGZ_E_DATA)):
            st, k, launches = at(dev, bit, cap)
            assert (st, k) == (want, 0) and launches <= once
            sb, ns, nph = P.pgz_inspect_parts(ctx.h)
            assert list(sb) == [(1 << 64) - 1] and list(ns) == [0] and list(nph) == [0]
    finally:
        ctx.close()


def test_decoding_from_an_offset_shares_the_contexts_scratch():
    """After a file has been decoded, decoding it from an offset takes no more device memory than the symbols in order
    and the wider windows (32 KiB a part more), with a little room for the allocator's granularity."""
    import torch
    text = synth.fastq(8_000_000, 150, 0.001, 8)
    gz = synth.gzip_compress(text, 6)
    parts = len(gz) // 4096 + 1
    ctx = Ctx(chunk_bytes=4096)
    try:
        P = ctx.pgz
        d, out = to_device(gz), empty(len(text))
        torch.cuda.synchronize()
        assert P.pgz_decompress(ctx.h, d.data_ptr(), len(gz), out.data_ptr(), len(text), False)[:2] == (0, len(text))
        before = torch.cuda.mem_get_info()[0]
        st, n, bb, fd = P.pgz_decompress_at(ctx.h, d.data_ptr(), len(gz), 8 * (len(gz) // 10), None, out.data_ptr(),
                                            ord("?"), len(text))
        assert st == 0 and n < len(text)
        assert before - torch.cuda.mem_get_info()[0] <= 2 * len(text) + 33 * 1024 * parts + (32 << 20)
        # the context goes on with either call
        assert P.pgz_decompress(ctx.h, d.data_ptr(), len(gz), out.data_ptr(), len(text), False)[:2] == (0, len(text))
        assert out[:len(text)].cpu().numpy().tobytes() == text
    finally:
        ctx.close()


@pytest.mark.parametrize("together", [False, True])
def test_a_batch_reports_each_job_and_refuses_what_lies_outside_device_memory(together):
    """Members in allocations of their own or side by side in one: headers within the gathered 64 bytes, longer, and a
    member shorter than that; a length that runs out of device memory, one below a member's least, a pointer off the
    alignment.  Each job has its own status, the good ones their output, and the next call is not affected."""
    import torch
    text = synth.fastq(60_000, 100, 0.001, 6)
    raw = zlib.compressobj(6, zlib.DEFLATED, -15)
    body = raw.compress(text) + raw.flush()
    good = [(synth.gzip_compress(text, 6), text), (synth.gzip_compress(b"A", 6), b"A"),
            (dw.gzip_wrap(body, text, flags=8, name=b"n" * 40), text),
            (dw.gzip_wrap(body, text, flags=8, name=b"n" * 53), text),
            (dw.gzip_wrap(body, text, flags=2 | 4 | 8 | 16, name=b"n" * 5000, extra=b"e" * 300, comment=b"c"), text)]
    ctx = Ctx()
    try:
        P = ctx.pgz
        if together:
            offs = np.cumsum([0] + [(len(g) + 15) // 16 * 16 for g, _ in good])
            one = to_device(b"".join(g + b"\0" * (-len(g) % 16) for g, _ in good))
            ptrs = [one.data_ptr() + int(o) for o in offs[:-1]]
        else:
            dev = [to_device(g) for g, _ in good]
            ptrs = [d.data_ptr() for d in dev]
        outs = [empty(len(t)) for _, t in good]
        jobs = [(p, len(g), o.data_ptr(), len(t)) for p, o, (g, t) in zip(ptrs, outs, good)]
        bad = [((ptrs[0], 1 << 62, outs[0].data_ptr(), len(text)), P.PGZ_E_CUDA),
               ((ptrs[0], 17, outs[0].data_ptr(), len(text)), P.PGZ_E_HEADER),
               ((ptrs[0] + 1, 100, outs[0].data_ptr(), len(text)), P.PGZ_E_ARG)]
        for k, (job, want) in enumerate(bad):
            st, res, _ = P.pgz_decompress_batch(ctx.h, jobs[:k] + [job] + jobs[k:])
            assert st == want and res[k] == (want, 0)
            assert [r for i, r in enumerate(res) if i != k] == [(0, len(t)) for _, t in good]
            for o, (_, t) in zip(outs, good):
                assert o[:len(t)].cpu().numpy().tobytes() == t
                o.zero_()
            with pytest.raises(P.PgzError):
                P.Batch(ctx.h, jobs + [job])
        st, res, _ = P.pgz_decompress_batch(ctx.h, jobs)
        assert st == 0 and all(o[:len(t)].cpu().numpy().tobytes() == t for o, (_, t) in zip(outs, good))
        torch.cuda.synchronize()
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 8191, 8192, 8193, 70001])
def test_sequences_at_word_and_block_edges(n):
    """Runs over words of 32 symbols and over the kernels' blocks, ends of the array included, against the oracle."""
    import torch
    rng = np.random.default_rng(n)
    kinds = np.array([ord("A"), ord("C"), 0x8000 | 7, ord("\n"), ord("x")], dtype=np.uint16)
    ctx = Ctx()
    try:
        for weights in [[4, 4, 1, 1, 0.3], [50, 50, 30, 0.3, 0.02], [1, 1, 1, 1, 1], [1, 0, 0, 0, 0], [0, 0, 1, 0, 0]]:
            p = np.array(weights) / sum(weights)
            s = kinds[rng.choice(5, size=n, p=p)]
            d = torch.from_numpy(s.view(np.int16).copy()).cuda()
            spans = torch.zeros((n + 1, 2), dtype=torch.int64, device="cuda")
            for min_len in (0, 5):
                want = oracle.sequences(s, min_len)
                st, k, nu = ctx.pgz.pgz_extract_sequences(ctx.h, d.data_ptr(), n, min_len, spans.data_ptr(), n + 1)
                got = sorted((int(a), int(b) & (2**63 - 1), int(b) < 0) for a, b in spans[:k].cpu().tolist())
                assert st == 0 and got == want and nu == sum(u for _, _, u in want)
    finally:
        ctx.close()


@pytest.mark.parametrize("offset", [0, 1])
def test_crc_at_the_edges_of_pieces_segments_and_forms(offset):
    """CRC-32 of outputs around the sizes of a lane's piece, a warp's segment and the change of the lookup tables' form
    (9728 segments on 152 SMs), the output aligned or not: the right trailer is accepted, a wrong one is not."""
    line = np.random.default_rng(5).choice(np.frombuffer(b"ACGT\n", dtype=np.uint8), 1 << 20).tobytes()
    ctx = Ctx()
    try:
        for n in [0, 1, 31, 32, 33, 1023, 1024, 1025, 1056, 262143, 9728 * 1024, 9728 * 1024 + 1]:
            text = (line * (n // len(line) + 1))[:n]
            c = zlib.compressobj(1, zlib.DEFLATED, 31)
            gz = c.compress(text) + c.flush()
            bad = gz[:-8] + bytes([gz[-8] ^ 0x10]) + gz[-7:]
            out = empty(n + 16)
            for data, want in ((gz, 0), (bad, ctx.pgz.PGZ_E_CRC)):
                d = to_device(data)
                st, k, _ = ctx.pgz.pgz_decompress(ctx.h, d.data_ptr(), len(data), out.data_ptr() + offset, n, False)
                assert st == want, (n, ctx.pgz.pgz_strerror(st))
                if want == 0:
                    assert k == n and out[offset:offset + n].cpu().numpy().tobytes() == text
    finally:
        ctx.close()
