"""LZSS compress with narrow windows, whose search takes a distance at a time:
both dictionaries, matches of one bit to 32, literals of one bit to 32, and
segments of 16 bytes to whole parts, against the oracle.
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


def _check(x, seg, params):
    ost, ref = oracle.lzss_segmented_compress(x, seg, params)
    assert ost == oracle.OK
    c, st = hg.huff_lzss_compress(torch.from_numpy(x).cuda(), seg, params)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and np.array_equal(c.cpu().numpy(), ref), (params, seg, x.size)


@pytest.mark.parametrize("dictionary", [1, 2])
@pytest.mark.parametrize("params", [(64, 1, 8, 1), (64, 1, 32, 32), (64, 20, 32, 8), (64, 32, 32, 7),
                                    (128, 1, 1, 1), (128, 2, 17, 16), (128, 11, 32, 31),
                                    (128, 12, 24, 8)])
@pytest.mark.parametrize("seg", [16, 48, 1024, 16384])
def test_narrow_windows_against_oracle(params, dictionary, seg):
    n = 3 * seg + 5
    period = np.resize(synth.uniform(9, 1), n)
    for x in (synth.uniform(n, 2), synth.text(n, 3), synth.bitstream(n, 4), period,
              np.zeros(n, np.uint8)):
        _check(x, seg, params + (dictionary,))


# 128- and 256-bit windows from 50 segments per SM on, and one fewer
@pytest.mark.parametrize("params", [(256, 1, 32, 8, 1), (256, 4, 11, 8, 2), (256, 7, 32, 16, 2),
                                    (128, 12, 24, 8, 1)])
def test_many_segments_against_oracle(params):
    seg = 48
    for count in (50 * torch.cuda.get_device_properties(0).multi_processor_count - 1,
                  50 * torch.cuda.get_device_properties(0).multi_processor_count):
        _check(synth.text(count * seg - 7, 1), seg, params)


def test_a_narrow_window_takes_no_longer_than_a_wide_one():
    """1 KiB segments of random bytes: a 64-bit window against 1024 bits (all
    distances at once took 1.7 times as long with the narrow one)."""
    n, seg, ms = 16 << 20, 1024, {}
    x, L = torch.from_numpy(synth.uniform(n, 1)).cuda(), hg.lib()
    for window in (64, 1024):
        params = (window, 4, 11, 8, 2)
        P = hg._lzss_params(params)
        out = torch.empty(L.huff_lzss_max_size(n, seg, P), dtype=torch.uint8, device="cuda")
        ws = torch.empty(L.huff_lzss_workspace_size(n, seg, P), dtype=torch.uint8, device="cuda")
        size, st, times = torch.zeros(1, dtype=torch.int64, device="cuda"), hg.new_status(), []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            hg.huff_lzss_compress(x, seg, params, d_out=out, d_out_bytes=size, d_ws=ws, d_status=st)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        assert int(st.item()) == 0
        ms[window] = sorted(times)[2]
    assert ms[64] < ms[1024], ms
