"""The block-sorting transform's first keys: alphabets of one byte value to
all 256, blocks shorter than a key, rotations that wrap inside it, and inputs
that do not start on a 16-byte boundary; and radix tiles that are not full."""
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


def _input(sigma, n):
    if sigma == "text":
        return synth.text(n, n)
    vals = np.linspace(0, 255, sigma).astype(np.uint8)
    return vals[synth.uniform(n, n).astype(np.int64) * sigma // 256]


@pytest.mark.parametrize("sigma", [1, 2, 3, 17, 256, "text"])
@pytest.mark.parametrize("block", [1, 7, 16, 300, 4096, 5000, 20000])
def test_first_keys_against_oracle(sigma, block):
    for n, off in ((9, 3), (15, 0), (4096, 0), (12289, 1), (20000, 15)):
        x = _input(sigma, n)
        d = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")[off:off + n]
        d.copy_(torch.from_numpy(x))
        ref_last, ref_prim = oracle.bwt(x, block)
        last, prim, st = hg.huff_bwt_forward(d, block)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        assert np.array_equal(last.cpu().numpy(), ref_last), (n, off)
        assert np.array_equal(prim.cpu().numpy().astype(np.uint32), ref_prim), (n, off)


# blocks sorted each by itself (from tiles 8/9 full) and all together, with a
# last block of any length
@pytest.mark.parametrize("sigma", [2, 34, 256])
@pytest.mark.parametrize("block", [3640, 3641, 4096, 4097, 8192, 8193, 14564, 65536])
def test_blocks_sorted_by_themselves(sigma, block):
    for n in (2 * block, 2 * block + 1, 9 * block - 1):
        x = _input(sigma, n)
        last, prim, st = hg.huff_bwt_forward(torch.from_numpy(x).cuda(), block)
        ref_last, ref_prim = oracle.bwt(x, block)
        assert int(st.item()) == 0
        assert np.array_equal(last.cpu().numpy(), ref_last), n
        assert np.array_equal(prim.cpu().numpy().astype(np.uint32), ref_prim), n


# LF by tiles (blocks from 4 KiB) and by sorting (below), samples every 32 rows
# ranked in shared memory (4 KiB..1 MiB) or every 64 by global jumps, walks of
# a few rows to a whole block (periodic and constant blocks), blocks that do
# not start at a sample
@pytest.mark.parametrize("block", [4095, 4096, 4097, 8192, 33333, 1 << 20, (1 << 20) + 1])
@pytest.mark.parametrize("kind", ["text", "constant", "periodic", "almost"])
def test_inverse_against_input(block, kind):
    n = 2 * block + 4100
    x = {"text": lambda: synth.text(n, 3), "constant": lambda: np.full(n, 7, np.uint8),
         "periodic": lambda: np.resize(np.frombuffer(b"abcab", np.uint8), n),
         "almost": lambda: np.resize(np.frombuffer(b"abcab", np.uint8), n)}[kind]().copy()
    if kind == "almost":
        x[::block] = ord("z")  # one byte breaks each block's period
    if n <= 70000:
        last, prim = oracle.bwt(x, block)
        L = torch.from_numpy(last).cuda()
        P = torch.from_numpy(prim.astype(np.int32)).cuda()
    else:  # (the oracle sorts a periodic block slowly)
        L, P, st = hg.huff_bwt_forward(torch.from_numpy(x).cuda(), block)
        assert int(st.item()) == 0
    back, st = hg.huff_bwt_inverse(L, block, P)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert np.array_equal(back.cpu().numpy(), x)


def test_blocks_beyond_16_mib():
    """LF words of 64 bits."""
    block = (1 << 24) + 33
    x = torch.from_numpy(synth.text(block + 5000, 9)).cuda()
    L, P, st = hg.huff_bwt_forward(x, block)
    assert int(st.item()) == 0
    back, st = hg.huff_bwt_inverse(L, block, P)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and torch.equal(back, x)
