"""Move-to-front where its steps can go wrong: blocks around a whole number of
chained segment runs, short last blocks, lists that change in all 256 entries,
bytes deep in the list, and buffers that are not 16-byte aligned."""
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
    if kind == "uniform":
        return synth.uniform(n, n)
    if kind == "cycle":  # every byte comes from the end of the list
        return np.resize(np.arange(256, dtype=np.uint8), n)
    if kind == "late":  # most of the alphabet appears in the last segments only
        x = np.zeros(n, np.uint8)
        x[-300:] = synth.uniform(n, 5)[-300:]
        return x
    return synth.bitstream(n, n)


# 32 segments of 1 KiB are chained by one warp; more go in runs
@pytest.mark.parametrize("block", [1023, 32 << 10, (32 << 10) + 1, (33 << 10) - 16, 65 << 10,
                                   (96 << 10) + 7])
@pytest.mark.parametrize("kind", ["uniform", "cycle", "late", "bitstream"])
def test_runs_of_segments(block, kind):
    for n in (block, 2 * block + 1, 3 * block - 5):
        x = _input(kind, n)
        ref = oracle.mtf(x, block)
        for off in (0, 1):  # aligned and not
            d = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")[off:off + n]
            d.copy_(torch.from_numpy(x))
            y = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")[off:off + n]
            hg.huff_mtf_forward(d, block, d_out=y)
            assert np.array_equal(y.cpu().numpy(), ref), (n, off)
            hg.huff_mtf_inverse(y, block, d_out=y)  # in place
            assert torch.equal(y, d), (n, off)
