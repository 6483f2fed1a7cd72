"""Sub-segment decoding where its steps can go wrong: codes that never or
hardly resynchronise, sub-segments shorter than a window or than the list of
boundaries, and sizes that leave ragged last chunks and payloads.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2306_11070_gb300 as hg
from paper_2306_11070_gb300 import build as nvbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    nvbuild.build()
    hg.lib()


def _input(kind, n):
    if kind == "fixed8":  # 256 equally frequent bytes: every code has 8 bits
        return synth.shuffle(np.resize(np.arange(256, dtype=np.uint8), n), 1)
    if kind == "fixed3":
        return synth.shuffle(np.resize(np.arange(40, 48, dtype=np.uint8), n), 2)
    if kind == "near8":  # 7 to 9 bits: paths join after hundreds of bits
        return synth.uniform(n, n)
    if kind == "long":  # codes beyond the 12-bit table
        return synth.geometric(n, n)
    if kind == "one":
        return synth.single(n)
    return synth.text(n, n)


SIZES = (1, 33, 700, 4096, 16384, 16400, 40000, 131071, 700001)


@pytest.mark.parametrize("kind", ["fixed8", "fixed3", "near8", "long", "one", "text"])
def test_split_chunks_against_oracle(kind):
    for n in SIZES:
        x = _input(kind, n)
        ost, ref = oracle.compress(x)
        assert ost == oracle.OK
        back = hg.decompress(torch.from_numpy(ref).cuda())
        assert np.array_equal(back.cpu().numpy(), x), (kind, n)


@pytest.mark.parametrize("kind", ["fixed8", "near8", "text"])
@pytest.mark.parametrize("lanes", [1, 32, 65536])
def test_split_buffers_in_a_batch(kind, lanes):
    prm = hg.huff_batch_default_params()
    prm.decode_lanes = lanes
    xs = [_input(kind, n) for n in SIZES]
    refs = [oracle.compress(x)[1] for x in xs]
    ins = [torch.from_numpy(r).cuda() for r in refs]
    outs = [torch.zeros(x.size, dtype=torch.uint8, device="cuda") for x in xs]
    plan = hg.BatchPlan(ins, outs, hg.HUFF_BATCH_DECOMPRESS, prm)
    plan.run()
    torch.cuda.synchronize()
    assert plan.status.tolist() == [0] * len(xs)
    for x, y in zip(xs, outs):
        assert np.array_equal(y.cpu().numpy(), x), (kind, x.size)


def test_cut_short_payloads_report_corruption():
    """A payload that ends early: the oracle's status."""
    for kind in ("fixed8", "near8", "text"):
        x = _input(kind, 40000)
        ref = oracle.compress(x)[1]
        for cut in (4, 64, 9000):
            bad = ref[:-cut]
            ost = oracle.decode(bad, x.size)[0]
            out, n, st = hg.huff_decode(torch.from_numpy(bad.copy()).cuda(), d_out=torch.zeros(
                x.size, dtype=torch.uint8, device="cuda"))
            torch.cuda.synchronize()
            assert int(st.item()) == ost, (kind, cut)


@pytest.mark.parametrize("chunks", [1, 19, 33, 64, 100])
def test_batches_that_fill_the_chip(chunks):
    """Enough chunks that a buffer is split by what it costs, not by the lanes
    asked for; the sizes differ, so the largest go first."""
    cs = 4096  # (small chunks: the rule counts chunks)
    lanes = torch.cuda.get_device_properties(0).multi_processor_count * 2 * 256
    sizes = [cs * chunks - (37 * i) % cs for i in range(lanes // 2 // chunks + 200)]
    sizes[7] = 1
    x = torch.from_numpy(synth.text(2 * cs * chunks, 3)).cuda()
    ins = [x[16 * (i % 50):16 * (i % 50) + n] for i, n in enumerate(sizes)]
    prm = hg.huff_batch_default_params()
    prm.chunk_symbols = cs
    outs = [torch.zeros(hg.huff_max_stream_size(n, cs), dtype=torch.uint8, device="cuda")
            for n in sizes]
    plan = hg.BatchPlan(ins, outs, hg.HUFF_BATCH_COMPRESS, prm)
    plan.run()
    got = plan.out_bytes.tolist()
    assert not any(plan.status.tolist())
    back = [torch.zeros(n, dtype=torch.uint8, device="cuda") for n in sizes]
    plan = hg.BatchPlan([o[:g] for o, g in zip(outs, got)], back, hg.HUFF_BATCH_DECOMPRESS)
    plan.run()
    assert not any(plan.status.tolist()) and plan.out_bytes.tolist() == sizes
    assert all(torch.equal(a, b) for a, b in zip(ins, back))
    one = oracle.compress(ins[-1].cpu().numpy(), cs)[1]
    assert np.array_equal(outs[-1][:got[-1]].cpu().numpy(), one)
