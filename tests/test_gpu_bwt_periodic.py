"""Blocks that repeat a period: their walk closes after one, and the rest of the
block is copied from it, whatever the block's size.
"""
import numpy as np
import pytest
import torch

import synth
import paper_2306_11070_gb300 as hg
from paper_2306_11070_gb300 import build as nvbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    nvbuild.build()
    hg.lib()


# periods below, at and above a warp, a walk's kept bytes and a copied piece
@pytest.mark.parametrize("period", [1, 2, 31, 32, 33, 511, 513, 4095, 4097])
@pytest.mark.parametrize("about", [64, 4096, 9000, 70000])
def test_whole_periods(period, about):
    block = period * max(2, about // period)
    for n in (block, 3 * block, 2 * block + period, 2 * block + 1):
        x = np.resize(synth.uniform(period, period), n)
        d = torch.from_numpy(x).cuda()
        last, prim, st = hg.huff_bwt_forward(d, block)
        assert int(st.item()) == 0
        back, st = hg.huff_bwt_inverse(last, block, prim)
        torch.cuda.synchronize()
        assert int(st.item()) == 0 and torch.equal(back, d), (block, n)


def test_constant_block_takes_no_longer_than_text():
    """One block of 16 MiB (a CTA copied a block by itself, in three times the
    time of the whole transform of text)."""
    n, ms = 16 << 20, {}
    for kind in ("text", "constant"):
        x = torch.from_numpy(synth.text(n, 2) if kind == "text" else np.full(n, 9, np.uint8)).cuda()
        ws = torch.zeros(hg.lib().huff_bwt_workspace_size(n, n), dtype=torch.uint8, device="cuda")
        last, prim, st = hg.huff_bwt_forward(x, n, ws=ws)
        y, times = torch.zeros_like(x), []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            hg.huff_bwt_inverse(last, n, prim, y, ws)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        assert torch.equal(y, x)
        ms[kind] = sorted(times)[3]
    assert ms["constant"] < 1.25 * ms["text"], ms
