"""Codes of 11 to 15 bits, written in pairs where groups of three or four do not
fit: single streams and batches against the oracle, and their time.
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


def _bytes(kind, n):
    rng = np.random.default_rng(n)
    if kind == "gauss":  # 7.4 bits on average: no group of three is sure
        return np.clip(rng.normal(128, 40, n), 0, 255).astype(np.uint8)
    if kind == "bursts":  # 2 bits on average, but for stretches of rare bytes
        x = np.minimum(rng.geometric(0.5, n) - 1, 6).astype(np.uint8)
        for at in range(0, n, 9000):
            x[at:at + 40] = rng.integers(7, 60, x[at:at + 40].size)
        return x
    x = synth.text(n, n)  # text with rare bytes strewn in
    x[rng.random(n) < 0.02] = 200
    x[rng.integers(0, n, n // 50 + 1)] = rng.integers(128, 256, n // 50 + 1)
    return x


@pytest.mark.parametrize("kind", ["gauss", "bursts", "strewn"])
def test_pairs_against_oracle(kind):
    xs = [_bytes(kind, n) for n in (70000, 300001, 16384 * 8, 16384 * 8 + 1023)]
    refs = [oracle.compress(x)[1] for x in xs]
    assert all(11 <= r[:256].max() <= 15 for r in refs), [int(r[:256].max()) for r in refs]
    ins = [torch.from_numpy(x).cuda() for x in xs]
    outs = [torch.zeros(hg.huff_max_stream_size(x.size), dtype=torch.uint8, device="cuda") for x in xs]
    plan = hg.BatchPlan(ins, outs, hg.HUFF_BATCH_COMPRESS)
    plan.run()
    got = plan.out_bytes.tolist()
    assert not any(plan.status.tolist())
    for d, o, g, ref in zip(ins, outs, got, refs):
        assert np.array_equal(o[:g].cpu().numpy(), ref)
        assert np.array_equal(hg.compress(d).cpu().numpy(), ref)


def test_codes_of_15_bits_take_little_longer_than_of_8():
    n, ms = 128 << 20, {}
    out = torch.zeros(hg.huff_max_stream_size(n), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(hg.huff_workspace_size(n), dtype=torch.uint8, device="cuda")
    size, st = torch.zeros(1, dtype=torch.int64, device="cuda"), hg.new_status()
    g = torch.Generator(device="cuda").manual_seed(1)
    for kind in ("uniform", "gauss"):
        x = (torch.randint(0, 256, (n,), generator=g, device="cuda") if kind == "uniform" else
             (128 + 40 * torch.randn(n, generator=g, device="cuda")).clamp_(0, 255)).to(torch.uint8)
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            hg.huff_compress(x, d_out=out, d_out_bytes=size, d_ws=ws, d_status=st)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        assert int(st.item()) == 0
        ms[kind] = sorted(times)[4]
    assert ms["gauss"] < 1.2 * ms["uniform"], ms
