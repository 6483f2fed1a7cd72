"""The encoder's steps where they can go wrong: every longest code length at
which the grouping of codes changes, groups that do not fit, inputs that end
just before, at and after a step or a unit, outputs that just hold the stream or
just do not, and bytes without a code.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_11070_gb300 as hg
from paper_2306_11070_gb300 import build as nvbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    nvbuild.build()
    hg.lib()


SIZES = (1, 31, 1023, 1024, 1025, 3000, 16383, 16384, 16385, 17408, 50000)
CHUNK = 4096


def _codebook(lengths):
    raw = np.zeros(hg.CODEBOOK_BYTES, np.uint8)
    raw[:256] = lengths
    raw[256:1280] = oracle.canonical_codes(lengths).astype("<u4").view(np.uint8)
    raw[1280:1284] = np.array([np.count_nonzero(lengths)], "<u4").view(np.uint8)
    raw[1284:1288] = np.array([lengths.max()], "<u4").view(np.uint8)
    return torch.from_numpy(raw).cuda()


def _encode(x, cb, cap):
    d = torch.from_numpy(x).cuda()
    out = torch.zeros(max(cap, 16), dtype=torch.uint8, device="cuda")
    nbytes = torch.zeros(1, dtype=torch.int64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(hg.huff_workspace_size(x.size, CHUNK), dtype=torch.uint8, device="cuda")
    rc = hg.lib().huff_encode(d.data_ptr(), x.size, cb.data_ptr(), CHUNK, out.data_ptr(), cap,
                              nbytes.data_ptr(), ws.data_ptr(), ws.numel(), status.data_ptr(), None)
    torch.cuda.synchronize()
    assert rc == 0
    return int(status), int(nbytes), out.cpu().numpy()


@pytest.mark.parametrize("longest", [1, 2, 3, 7, 8, 10, 11, 15, 16, 22, 23, 31, 32])
@pytest.mark.parametrize("skewed", [False, True])
def test_lengths_sizes_and_capacities(longest, skewed):
    lengths = np.zeros(256, np.uint8)
    lengths[: longest + 1] = list(range(1, longest + 1)) + [longest]
    cb = _codebook(lengths)
    rng = np.random.default_rng(longest)
    for n in SIZES:
        # skewed: as rare as the codes are long; else long codes in every group
        x = rng.geometric(0.5, n) - 1 if skewed else rng.integers(0, longest + 1, n)
        x = np.minimum(x, longest).astype(np.uint8)
        x[-1] = longest  # a long last code
        ost, ref, size = oracle.encode(x, lengths, CHUNK, 400 + 8 * n)
        assert ost == oracle.OK
        for cap in (size, size + 64):
            st, nbytes, out = _encode(x, cb, cap)
            assert (st, nbytes) == (0, size), (n, cap)
            assert np.array_equal(out[:size], ref[:size]), (n, cap)
        st, nbytes, _ = _encode(x, cb, size - 4)
        assert (st, nbytes) == (hg.HUFF_ERR_CAPACITY, size), n


@pytest.mark.parametrize("longest", [4, 8, 16])
def test_bytes_without_a_code_add_no_bits(longest):
    lengths = np.zeros(256, np.uint8)
    lengths[: longest + 1] = list(range(1, longest + 1)) + [longest]
    cb = _codebook(lengths)
    rng = np.random.default_rng(longest)
    for n in SIZES:
        if n > 16384:
            continue
        x = np.full(n, 200, np.uint8)  # no code
        some = rng.random(n) < rng.choice([0.0, 0.01, 0.3])
        x[some] = rng.integers(0, longest + 1, int(some.sum()))
        cap = 400 + 8 * n
        st, nbytes, out = _encode(x, cb, cap)
        kept = x[x != 200]
        words = np.zeros(0, np.uint8)
        if kept.size:
            _, ref, size = oracle.encode(kept, lengths, CHUNK, 400 + 8 * n)
            words = ref[272 + 8 * -(-kept.size // CHUNK) : size]
        head = 272 + 8 * -(-n // CHUNK)
        assert (st, nbytes) == (0, head + words.size), n
        assert np.array_equal(out[head : head + words.size], words), n


@pytest.mark.parametrize("n", [0, 5, 70000, 5 << 20])
def test_chained_launches_under_capture_and_back_to_back(n):
    rng = np.random.default_rng(n)
    xs = [np.minimum(rng.geometric(0.3, n) * k % 256, 255).astype(np.uint8) for k in (1, 3, 7)]
    refs = [oracle.compress(x)[1] for x in xs]
    d = torch.zeros(max(n, 1), dtype=torch.uint8, device="cuda")
    cap = hg.huff_max_stream_size(n)
    out = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    nbytes = torch.zeros(1, dtype=torch.int64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(hg.huff_workspace_size(n), dtype=torch.uint8, device="cuda")

    def run():
        hg.huff_compress(d[:n], d_out=out, d_out_bytes=nbytes, d_ws=ws, d_status=status)

    run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for go in (graph.replay, run):
        got = []
        for x in xs:  # one workspace, no synchronisation in between
            d[:n].copy_(torch.from_numpy(x))
            go()
            got.append((out.clone(), nbytes.clone(), status.clone()))
        torch.cuda.synchronize()
        for (o, b, s), ref in zip(got, refs):
            assert int(s) == 0 and int(b) == ref.size
            assert np.array_equal(o[: ref.size].cpu().numpy(), ref)


def test_batches_of_every_grouping():
    rng = np.random.default_rng(5)
    fib = [1, 1]
    while len(fib) < 33:
        fib.append(fib[-1] + fib[-2])
    xs = [np.repeat(np.arange(33, dtype=np.uint8), fib)]  # a 32-bit code
    for n in SIZES + (150000,):
        xs.append(np.full(n, 9, np.uint8))
        xs.append(rng.integers(0, 3, n).astype(np.uint8))
        xs.append(rng.integers(0, 60, n).astype(np.uint8))
        xs.append(rng.integers(0, 256, n).astype(np.uint8))
        xs.append(np.minimum(rng.geometric(0.5, n), 255).astype(np.uint8))
        xs.append(np.minimum(rng.geometric(0.04, n), 255).astype(np.uint8))
        x = np.minimum(rng.geometric(0.5, n), 255)
        x[n // 3 : n // 2] = rng.integers(0, 256, n // 2 - n // 3)  # groups that do not fit
        xs.append(x.astype(np.uint8))
    refs = [oracle.compress(x)[1] for x in xs]
    ins = [torch.from_numpy(x).cuda() for x in xs]
    outs = [torch.zeros(hg.huff_max_stream_size(x.size), dtype=torch.uint8, device="cuda") for x in xs]
    plan = hg.BatchPlan(ins, outs, hg.HUFF_BATCH_COMPRESS)
    plan.run()
    torch.cuda.synchronize()
    sizes = plan.out_bytes.cpu().numpy()
    for x, ref, out, size in zip(xs, refs, outs, sizes):
        assert int(size) == ref.size, x.size
        assert np.array_equal(out[: ref.size].cpu().numpy(), ref), x.size


@pytest.mark.parametrize("units", [1, 2, 3, 607, 608, 609, 1216, 1217, 1825])
def test_unit_histograms_counted_in_pairs(units):
    rng = np.random.default_rng(units)
    for n in (units * 16384 - 16383, units * 16384):
        x = rng.integers(0, 256, n, dtype=np.uint8)
        x[: 2 * 16384] = 255  # 16384 of one byte in both of a pair
        d = torch.from_numpy(x).cuda()
        hist = torch.zeros(256, dtype=torch.int64, device="cuda")
        uh = torch.zeros(hg.huff_unit_hist_size(n), dtype=torch.uint8, device="cuda")
        hg.huff_histogram_units(d, hist, uh)
        got = uh.cpu().numpy().view("<u2").reshape(units, 256)
        pad = np.zeros(units * 16384, np.int64)
        pad[:n] = x.astype(np.int64) + 1
        at = np.arange(units * 16384) // 16384 * 257 + pad
        ref = np.bincount(at, minlength=units * 257).reshape(units, 257)[:, 1:]
        assert np.array_equal(got, ref)
        assert np.array_equal(hist.cpu().numpy(), ref.sum(0))
