"""LZSS decoders at the edges of their choice and of their steps: the CTA per
segment (two warps) and the thread per segment that very many segments take.
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


def _mixed(n, seed):
    """Zero runs, short periods and random bytes, a few tens of bytes each."""
    rng = np.random.default_rng(seed)
    parts, left = [], n
    while left > 0:
        k = min(left, int(rng.integers(1, 90)))
        kind = rng.integers(0, 3)
        if kind == 0:
            parts.append(np.zeros(k, np.uint8))
        elif kind == 1:
            parts.append(np.resize(rng.integers(0, 256, rng.integers(1, 6)).astype(np.uint8), k))
        else:
            parts.append(rng.integers(0, 256, k).astype(np.uint8))
        left -= k
    return np.concatenate(parts) if parts else np.zeros(0, np.uint8)


def _decode(c, n):
    y, got, st = hg.huff_lzss_decompress(c, out_cap=n)
    torch.cuda.synchronize()
    return y, got, int(st.item())


# stored prefix, windows of 32..2048 bits, literals up to 31 bits: a thread per
# segment from 320 segments per SM on; anything else a CTA per segment
@pytest.mark.parametrize("params", [(1024, 12, 24, 8, 2), (32, 3, 3, 1, 2), (2048, 1, 1, 16, 2),
                                    (256, 4, 32, 31, 2), (256, 4, 32, 32, 2), (64, 6, 9, 5, 1)])
@pytest.mark.parametrize("delta", [-1, 0])
def test_segment_count_at_the_choice(params, delta):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    seg = 48
    n = (320 * sms + delta) * seg - 5
    x = _mixed(n, 3)
    d = torch.from_numpy(x).cuda()
    c, st = hg.huff_lzss_compress(d, seg, params)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    y, got, s = _decode(c, n)
    assert s == 0 and got == n and torch.equal(y, d)
    bad = c.clone()
    bad[48:52] = torch.tensor([255, 255, 0, 0], dtype=torch.uint8)  # segment 0's length
    assert _decode(bad, n)[2] == hg.HUFF_ERR_CORRUPT_STREAM


# shortest tokens (two bits), 33-bit literals, runs of one distance far longer
# than a batch of 32 tokens, and distances beyond the copy warp's ring
@pytest.mark.parametrize("params", [(2, 1, 1, 1, 1), (2, 1, 1, 1, 2), (16, 1, 32, 32, 1),
                                    (8192, 12, 24, 8, 2), (1024, 12, 24, 8, 2)])
@pytest.mark.parametrize("n", [33, 260, 2600])
def test_batch_edges_against_oracle(params, n):
    for x in (np.zeros(n, np.uint8), np.resize(np.array([0xB6, 0xDB, 0x6D], np.uint8), n),
              _mixed(n, n)):
        ost, ref = oracle.lzss_segmented_compress(x, 4096, params)
        assert ost == oracle.OK
        y, got, s = _decode(torch.from_numpy(ref).cuda(), n)
        assert s == 0 and got == n and np.array_equal(y.cpu().numpy(), x)


def _period(n, k, seed):
    return np.resize(np.random.default_rng(seed).integers(0, 256, k).astype(np.uint8), n)


# segments of 8 KiB and more coded in parts whose token chains must meet: quickly
# (bitstream, random), at the end of a run, or never (constant data, a period
# that matches are cut from), and parts that a run covers whole
@pytest.mark.parametrize("params", [(256, 12, 24, 8, 2), (64, 9, 32, 16, 1), (512, 16, 16, 7, 2),
                                    (128, 2, 8, 3, 2)])
@pytest.mark.parametrize("seg", [16384, 32768, 65536])
def test_segments_in_parts_against_oracle(params, seg):
    n = seg + 9001
    runs = synth.bitstream(n, 3)
    runs[seg // 5:seg // 2] = 0
    runs[seg // 2:seg // 2 + 3000] = 0xFF
    for x in (runs, synth.uniform(n, 2), np.zeros(n, np.uint8), _period(n, 5, 1),
              _period(n, 61, 2)):
        ost, ref = oracle.lzss_segmented_compress(x, seg, params)
        assert ost == oracle.OK
        c, st = hg.huff_lzss_compress(torch.from_numpy(x).cuda(), seg, params)
        torch.cuda.synchronize()
        assert int(st.item()) == 0 and np.array_equal(c.cpu().numpy(), ref)
