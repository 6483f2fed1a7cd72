"""Performance cases of the codec: what a user has it do, through its public calls.

``listed()`` names the cases, ``draw(rng)`` gives one more of the same
ranges, ``prepare(case, seed)`` makes the inputs and keeps what a user's
program keeps (buffers, plans, a server), ``run(state)`` is one pass,
``work(case)`` the bytes it cannot do without, and ``exact(case, seed)`` the
decoded bytes a decompressing pass has to give.

Inputs are made on the GPU from the seed: Zipf-word text, Zipf ASCII bytes,
uniform and geometric bytes and FPGA-bitstream-like data with the same shapes
as the generators in ``synth`` (which run on one host core and would take
seconds per case).
"""
from __future__ import annotations

import math
import random

import torch

import paper_2306_11070_gb300 as hg

KiB, MiB, GiB = 1 << 10, 1 << 20, 1 << 30
CHUNK = hg.DEFAULT_CHUNK_SYMBOLS
PIECE = 64 * MiB  # inputs are generated in pieces, which bounds the temporaries

# stream bytes per input byte, for work(): text 4.54 bits a byte, Zipf ASCII
# 5.2, uniform 8, geometric 2; LZSS bitstream 70%, Method 3 with move-to-front 40%
RATIO = {"text": 0.568, "zipf": 0.65, "uniform": 1.0, "geometric": 0.25}
LZSS_RATIO, M3_RATIO = 0.70, 0.40


def listed():
    return [
        # The shortest request the served workload knows, there and back, as a
        # program that sizes the output and reads the stream's size does it:
        # allocations, launches and reads back count.
        {"name": "roundtrip_4k", "op": "roundtrip", "n": 4 * KiB, "dist": "text"},
        # Config 2 at 64 MiB, the paper's corpus scale (its text is ~45 MB): a
        # corpus compressed and decompressed in one call each.
        {"name": "compress_64m", "op": "compress", "n": 64 * MiB, "dist": "text"},
        {"name": "decompress_64m", "op": "decompress", "n": 64 * MiB, "dist": "text"},
        # The headline size: one 1 GiB buffer.
        {"name": "compress_1g", "op": "compress", "n": GiB, "dist": "text"},
        {"name": "decompress_1g", "op": "decompress", "n": GiB, "dist": "text"},
        # Config 3: 4096 buffers of 1 KiB to 4 MiB, a codebook each, one launch.
        {"name": "batch_compress", "op": "batch_compress", "count": 4096, "lo": KiB, "hi": 4 * MiB,
         "sizes": 3},
        {"name": "batch_decompress", "op": "batch_decompress", "count": 4096, "lo": KiB,
         "hi": 4 * MiB, "sizes": 3},
        # Config 5's request mix as one burst: host buffers in and out, half
        # compress and half decompress, all submitted and then waited for.
        {"name": "served_burst", "op": "served", "count": 64, "lo": 4 * KiB, "hi": 16 * MiB,
         "sizes": 5},
        # Method 3: the block-sorting transform, move-to-front and per-segment
        # codebooks over a corpus, and back (1 MiB blocks, 64 KiB segments).
        {"name": "m3_compress", "op": "m3_compress", "n": 64 * MiB, "block": MiB,
         "segment": 64 * KiB, "mtf": True},
        {"name": "m3_decompress", "op": "m3_decompress", "n": 64 * MiB, "block": MiB,
         "segment": 64 * KiB, "mtf": True},
        # LZSS Method 2 with the paper's 1024/24/12/8 over bitstream data in
        # 64 KiB segments, and back.
        {"name": "lzss_compress", "op": "lzss_compress", "n": 64 * MiB, "segment": 64 * KiB,
         "window": 1024, "min_len": 12, "max_len": 24, "literal": 8, "dict": 2},
        {"name": "lzss_decompress", "op": "lzss_decompress", "n": 64 * MiB, "segment": 64 * KiB,
         "window": 1024, "min_len": 12, "max_len": 24, "literal": 8, "dict": 2},
    ]


def _log_uniform(rng, lo, hi):
    """A size spread over the logarithm; any residue, so mostly odd ones."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    op = rng.choice(["roundtrip", "compress", "decompress", "compress", "decompress",
                     "batch_compress", "batch_decompress", "served", "m3_compress",
                     "m3_decompress", "lzss_compress", "lzss_decompress"])
    if op == "roundtrip":
        return {"op": op, "n": _log_uniform(rng, 1 * KiB, 4 * MiB),
                "dist": rng.choice(["text", "zipf", "uniform", "geometric"])}
    if op in ("compress", "decompress"):
        dist = rng.choice(["text", "text", "zipf", "uniform", "geometric"])
        # geometric bytes need codes of about log2 n bits: below the 32-bit limit
        hi = {"text": GiB, "zipf": GiB, "uniform": 256 * MiB, "geometric": 64 * MiB}[dist]
        return {"op": op, "n": _log_uniform(rng, 256 * KiB, hi), "dist": dist}
    if op in ("batch_compress", "batch_decompress"):
        return {"op": op, "count": _log_uniform(rng, 16, 4096), "lo": KiB,
                "hi": rng.choice([64 * KiB, MiB, 4 * MiB]), "sizes": rng.randrange(1 << 20)}
    if op == "served":
        return {"op": op, "count": rng.randrange(1, 65), "lo": 4 * KiB,
                "hi": rng.choice([64 * KiB, MiB, 16 * MiB]), "sizes": rng.randrange(1 << 20)}
    if op in ("m3_compress", "m3_decompress"):
        return {"op": op, "n": _log_uniform(rng, MiB, 64 * MiB),
                "block": rng.choice([64 * KiB, 256 * KiB, MiB]),
                "segment": rng.choice([16 * KiB, 64 * KiB]), "mtf": rng.random() < 0.5}
    window = rng.choice([256, 512, 1024, 2048, 4096])
    lens = rng.choice([(12, 24, 8), (12, 24, 8), (16, 32, 8)])
    dictionary = rng.choice([1, 2, 2])
    # long segments only with the stored prefix and a window of the paper's
    # order: a segment is coded in order, so its length sets the shortest time
    short = dictionary == 1 or window > 2048
    return {"op": op, "n": _log_uniform(rng, MiB, 64 * MiB * min(1024, window) // window),
            "segment": 16 * KiB if short else rng.choice([16 * KiB, 32 * KiB, 64 * KiB]),
            "window": window, "min_len": lens[0], "max_len": lens[1], "literal": lens[2],
            "dict": dictionary}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _pieces(n, make):
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    for at in range(0, n, PIECE):
        out[at:at + PIECE] = make(min(PIECE, n - at))
    return out


def _text(n, seed):
    """Words of a 50,000-word vocabulary (random lowercase, length geometric
    with p = 0.3 up to 12), drawn Zipf(1.0), 5% followed by a punctuation
    mark, separated by spaces and a newline about every 80 characters."""
    g, words = _gen(seed), 50000
    u = torch.rand(words, generator=g, device="cuda", dtype=torch.float64).clamp_(min=1e-12)
    wlen = (1 + torch.floor(torch.log(u) / math.log(0.7))).clamp_(max=12).long()
    letters = torch.randint(97, 123, (words, 12), generator=g, device="cuda", dtype=torch.uint8)
    cdf = torch.cumsum(1.0 / torch.arange(1, words + 1, device="cuda", dtype=torch.float64), 0)
    cdf /= cdf[-1].clone()
    marks = torch.tensor(list(b".,;:!?"), dtype=torch.uint8, device="cuda")
    mean = float((torch.diff(cdf, prepend=cdf.new_zeros(1)) * wlen).sum()) + 1.05

    def make(m):
        k, total = int(m / mean * 1.05) + 64, 0
        while total < m:
            k *= 2 if total else 1
            w = torch.searchsorted(cdf, torch.rand(k, generator=g, device="cuda",
                                                   dtype=torch.float64)).clamp_(max=words - 1)
            mark = torch.rand(k, generator=g, device="cuda") < 0.05
            length = wlen[w] + mark + 1
            end = torch.cumsum(length, 0)
            total = int(end[-1])
        start = end - length
        sep = torch.where(end // 80 != start // 80, 10, 32).to(torch.uint8)
        of = torch.repeat_interleave(torch.arange(k, device="cuda"), length, output_size=total)[:m]
        off = torch.arange(m, device="cuda") - start[of]
        out = letters[w[of], off.clamp(max=11)]
        last = off == length[of] - 1
        out = torch.where(last, sep[of], out)
        return torch.where((off == wlen[w[of]]) & ~last, marks[of % 6], out)

    return _pieces(n, make)


def _bytes(n, dist, seed):
    if dist == "text":
        return _text(n, seed)
    g = _gen(seed)
    if dist == "uniform":
        return _pieces(n, lambda m: torch.randint(0, 256, (m,), generator=g, device="cuda",
                                                  dtype=torch.uint8))
    if dist == "zipf":  # i.i.d. Zipf(1.1) over the 96 codes from the space
        p = torch.arange(1, 97, device="cuda", dtype=torch.float64) ** -1.1
        cdf = torch.cumsum(p / p.sum(), 0)
        return _pieces(n, lambda m: (torch.searchsorted(cdf, torch.rand(
            m, generator=g, device="cuda", dtype=torch.float64)).clamp_(max=95) + 32).to(torch.uint8))
    # geometric: P(k) = 2^-(k + 1)
    return _pieces(n, lambda m: torch.floor(-torch.log2(1 - torch.rand(
        m, generator=g, device="cuda", dtype=torch.float64))).clamp_(max=255).to(torch.uint8))


def _bitstream(n, seed):
    """FPGA-configuration-like data: zero runs of 16 + Exp(500) bytes (55% of
    the records), copies of 16 random 32..255-byte templates with one to three
    bits flipped (30%), random stretches of 8 + Exp(64) bytes (15%)."""
    g = _gen(seed)
    tlen = torch.randint(32, 256, (16,), generator=g, device="cuda")
    tpl = torch.randint(0, 256, (16, 256), generator=g, device="cuda", dtype=torch.uint8)

    def make(m):
        k, total = m // 200 + 256, 0
        while total < m:
            k *= 2 if total else 1
            kind = torch.rand(k, generator=g, device="cuda")
            e = -torch.log(1 - torch.rand(k, generator=g, device="cuda"))
            t = torch.randint(0, 16, (k,), generator=g, device="cuda")
            length = torch.where(kind < 0.55, 16 + (500 * e).long(),
                                 torch.where(kind < 0.85, tlen[t], 8 + (64 * e).long()))
            end = torch.cumsum(length, 0)
            total = int(end[-1])
        start = end - length
        of = torch.repeat_interleave(torch.arange(k, device="cuda"), length, output_size=total)
        off = torch.arange(total, device="cuda") - start[of]
        rnd = torch.randint(0, 256, (total,), generator=g, device="cuda", dtype=torch.uint8)
        kd = kind[of]
        out = torch.where(kd < 0.55, torch.zeros_like(rnd),
                          torch.where(kd < 0.85, tpl[t[of], off.clamp(max=255)], rnd))
        copies = torch.nonzero((kind >= 0.55) & (kind < 0.85)).reshape(-1)
        flips = torch.randint(1, 4, (copies.numel(),), generator=g, device="cuda")
        for f in range(3):  # one bit each; a record's flips may meet
            use = copies[flips > f]
            bit = (torch.rand(use.numel(), generator=g, device="cuda", dtype=torch.float64)
                   * (8 * length[use])).long()
            at = start[use] + bit // 8
            out[at] ^= (128 >> (bit % 8)).to(torch.uint8)
        return out[:m]

    return _pieces(n, make)


def _sizes(case):
    r = random.Random(case["sizes"])
    return [_log_uniform(r, case["lo"], case["hi"]) for _ in range(case["count"])]


def _cut(sizes):
    """Starts of buffers laid one after the other at multiples of 256, and the end."""
    at, starts = 0, []
    for s in sizes:
        starts.append(at)
        at += (s + 255) // 256 * 256
    return starts, at


def _zeros(n, dtype=torch.uint8):
    return torch.zeros(max(int(n), 1), dtype=dtype, device="cuda")


def _input(case, seed):
    """The uncompressed bytes of a case."""
    op = case["op"]
    if op in ("roundtrip", "compress", "decompress"):
        return _bytes(case["n"], case["dist"], seed)
    if op.startswith("m3"):
        return _text(case["n"], seed)
    if op.startswith("lzss"):
        return _bitstream(case["n"], seed)
    return _text(_cut(_sizes(case))[1], seed)  # batch, served: buffers cut from one text


def _lzss_params(case):
    return (case["window"], case["min_len"], case["max_len"], case["literal"], case["dict"])


def _batch_streams(x, sizes, starts):
    """Every buffer's stream, made by a batch plan: (arena, streams, sizes)."""
    caps = [hg.huff_max_stream_size(s) for s in sizes]
    at, total = _cut(caps)
    arena = _zeros(total)
    outs = [arena[a:a + c] for a, c in zip(at, caps)]
    plan = hg.BatchPlan([x[a:a + s] for a, s in zip(starts, sizes)], outs, hg.HUFF_BATCH_COMPRESS)
    plan.run()
    torch.cuda.synchronize()
    return plan, arena, outs


def prepare(case, seed):
    op = case["op"]
    x = _input(case, seed)
    s = {"op": op, "case": case}
    if op == "roundtrip":
        s.update(x=x, out=_zeros(hg.huff_max_stream_size(case["n"])))
    elif op == "compress":
        n = case["n"]
        s.update(x=x, out=_zeros(hg.huff_max_stream_size(n)), bytes=_zeros(1, torch.int64),
                 ws=_zeros(hg.huff_workspace_size(n)), status=_zeros(1, torch.int32))
    elif op == "decompress":
        s.update(stream=hg.compress(x).clone(), out=_zeros(case["n"]), n=_zeros(1, torch.int64),
                 status=_zeros(1, torch.int32))
    elif op in ("batch_compress", "batch_decompress"):
        sizes = _sizes(case)
        starts, total = _cut(sizes)
        plan, arena, outs = _batch_streams(x, sizes, starts)
        s["arena"] = arena
        if op == "batch_decompress":
            got = plan.out_bytes.tolist()
            s["arena"] = _zeros(total)
            back = [s["arena"][a:a + m] for a, m in zip(starts, sizes)]
            plan.close()
            plan = hg.BatchPlan([o[:b] for o, b in zip(outs, got)], back, hg.HUFF_BATCH_DECOMPRESS)
        s["plan"] = plan
    elif op == "served":
        sizes = _sizes(case)
        starts, total = _cut(sizes)
        plan, arena, outs = _batch_streams(x, sizes, starts)
        got = plan.out_bytes.tolist()
        plan.close()
        # even requests compress their buffer, odd ones decompress its stream
        ins, caps = [], []
        for i, (a, m) in enumerate(zip(starts, sizes)):
            ins.append(outs[i][:got[i]] if i % 2 else x[a:a + m])
            caps.append(m if i % 2 else hg.huff_max_stream_size(m))
        at_in, total_in = _cut([t.numel() for t in ins])
        at_out, total_out = _cut(caps)
        h_in = torch.zeros(total_in, dtype=torch.uint8, pin_memory=True)
        h_out = torch.zeros(total_out, dtype=torch.uint8, pin_memory=True)
        s["requests"] = []
        for i, t in enumerate(ins):
            view = h_in[at_in[i]:at_in[i] + t.numel()]
            view.copy_(t)
            s["requests"].append((hg.HUFF_BATCH_DECOMPRESS if i % 2 else hg.HUFF_BATCH_COMPRESS,
                                  view, h_out[at_out[i]:at_out[i] + caps[i]]))
        cfg = hg.huff_server_default_config()
        cfg.device_budget = GiB
        s.update(h_in=h_in, h_out=h_out, server=hg.Server(cfg))
    elif op == "m3_compress":
        L, a = hg.lib(), (case["n"], case["block"], case["segment"], CHUNK)
        s.update(x=x, out=_zeros(L.huff_m3_max_size(*a)), ws=_zeros(L.huff_m3_workspace_size(*a)),
                 bytes=_zeros(1, torch.int64), status=_zeros(1, torch.int32))
    elif op == "m3_decompress":
        c, _ = hg.huff_m3_compress(x, case["block"], case["segment"],
                                   stages=hg.HUFF_M3_MTF if case["mtf"] else 0)
        s["c"] = c.clone()
    else:
        p = _lzss_params(case)
        L, n, seg = hg.lib(), case["n"], case["segment"]
        P = hg.LzssParams(*p)
        out = _zeros(L.huff_lzss_max_size(n, seg, P))
        ws = _zeros(L.huff_lzss_workspace_size(n, seg, P))
        ob, st = _zeros(1, torch.int64), _zeros(1, torch.int32)
        s.update(x=x, out=out, bytes=ob, ws=ws, status=st, params=p)
        if op == "lzss_decompress":
            hg.huff_lzss_compress(x, seg, p, d_out=out, d_out_bytes=ob, d_ws=ws, d_status=st)
            c = out[:int(ob.item())].clone()
            s = {"op": op, "c": c, "out": _zeros(n), "n": _zeros(1, torch.int64), "status": st,
                 "ws": _zeros(L.huff_lzss_decompress_workspace_size(c.numel()))}
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    op = s["op"]
    if op == "roundtrip":
        out, size, _ = hg.huff_compress(s["x"], d_out=s["out"])
        data, n, status = hg.huff_decode(out, int(size.item()))
        return {"stream": out, "bytes": size, "data": data, "n": n, "status": status}
    if op == "compress":
        hg.huff_compress(s["x"], CHUNK, d_out=s["out"], d_out_bytes=s["bytes"], d_ws=s["ws"],
                         d_status=s["status"])
        return {"stream": s["out"], "bytes": s["bytes"], "status": s["status"]}
    if op == "decompress":
        hg.huff_decode(s["stream"], d_out=s["out"], d_n=s["n"], d_status=s["status"])
        return {"data": s["out"], "n": s["n"], "status": s["status"]}
    if op in ("batch_compress", "batch_decompress"):
        s["plan"].run()
        return {"arena": s["arena"], "bytes": s["plan"].out_bytes, "status": s["plan"].status}
    if op == "served":
        srv = s["server"]
        tickets = [srv.submit(o, i, y) for o, i, y in s["requests"]]
        res = [srv.wait(t) for t in tickets]
        for t in tickets:
            srv.release(t)
        return {"arena": s["h_out"], "bytes": torch.tensor([r["out_bytes"] for r in res]),
                "status": torch.tensor([r["status"] for r in res])}
    if op == "m3_compress":
        c, x, out, ws = s["case"], s["x"], s["out"], s["ws"]
        got = hg.lib().huff_m3_compress(
            x.data_ptr(), x.numel(), c["block"], c["segment"], CHUNK,
            hg.HUFF_M3_MTF if c["mtf"] else 0, out.data_ptr(), out.numel(), s["bytes"].data_ptr(),
            ws.data_ptr(), ws.numel(), s["status"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        return {"container": out, "bytes": s["bytes"], "status": s["status"], "returned": got}
    if op == "m3_decompress":
        data, n, st = hg.huff_m3_decompress(s["c"])
        return {"data": data, "n": n, "status": st}
    if op == "lzss_compress":
        hg.huff_lzss_compress(s["x"], s["case"]["segment"], s["params"], d_out=s["out"],
                              d_out_bytes=s["bytes"], d_ws=s["ws"], d_status=s["status"])
        return {"container": s["out"], "bytes": s["bytes"], "status": s["status"]}
    hg.huff_lzss_decompress(s["c"], d_out=s["out"], d_n=s["n"], d_ws=s["ws"], d_status=s["status"])
    return {"data": s["out"], "n": s["n"], "status": s["status"]}


def work(case):
    """Input read once and output written once; integer work, no flops counted."""
    op = case["op"]
    if op in ("roundtrip", "compress", "decompress"):
        once = case["n"] * (1 + RATIO[case["dist"]])
        return {"bytes": (2 if op == "roundtrip" else 1) * once, "flops": 0}
    if op.startswith("m3"):
        return {"bytes": case["n"] * (1 + M3_RATIO), "flops": 0}
    if op.startswith("lzss"):
        return {"bytes": case["n"] * (1 + LZSS_RATIO), "flops": 0}
    return {"bytes": sum(_sizes(case)) * (1 + RATIO["text"]), "flops": 0}


def exact(case, seed):
    """What a decompressing pass gives: the bytes that were compressed.  The
    compressed forms have no value without a coder."""
    op = case["op"]
    if op == "roundtrip":
        return {"stream": None, "bytes": None, "data": _input(case, seed), "n": None,
                "status": None}
    if op in ("decompress", "m3_decompress", "lzss_decompress"):
        return {"data": _input(case, seed), "n": None, "status": None}
    return None
