"""LZSS segments coded in parts, with the counting dictionary (the first part
starts at bit 0 and matches reach before the segment) and windows of several
search passes (whose stored prefix is most of the first part's head start):
against the oracle, with last segments of 16 bytes, shorter than the window,
and nearly whole.
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


def _compress(x, seg, params):
    """(container, first segment's slot of the workspace)"""
    L, P, n = hg.lib(), hg._lzss_params(params), x.size
    new = lambda k, t=torch.uint8: torch.zeros(max(k, 1), dtype=t, device="cuda")
    out, ws = new(L.huff_lzss_max_size(n, seg, P)), new(L.huff_lzss_workspace_size(n, seg, P))
    size, st = new(1, torch.int64), new(1, torch.int32)
    hg.huff_lzss_compress(torch.from_numpy(x).cuda(), seg, params, d_out=out, d_out_bytes=size,
                          d_ws=ws, d_status=st)
    assert int(st.item()) == 0
    return out[:int(size.item())].cpu().numpy(), ws[:16].cpu().numpy()


@pytest.mark.parametrize("params,seg", [((1024, 12, 24, 8, 1), 16384), ((1024, 12, 24, 8, 1), 65536),
                                        ((256, 12, 32, 8, 1), 16384), ((2048, 12, 24, 8, 2), 16384),
                                        ((2048, 12, 24, 8, 2), 65536), ((4096, 16, 32, 8, 2), 16384),
                                        ((4096, 12, 24, 8, 1), 16384),
                                        ((16384, 16, 32, 8, 1), 16384)])
def test_parts_against_oracle(params, seg):
    # the slot of a segment in parts starts with {end, bits, 0, 0}: not so the
    # code of random bytes
    _, slot = _compress(synth.uniform(2 * seg, 1), seg, params)
    assert not slot[8:].any(), "these parameters no longer code in parts"
    window = params[0]
    lasts = (16,) if window > 4096 else (16, window // 16 + 1, seg - 1)
    for last in lasts:
        n = seg + last
        mixed = synth.bitstream(n, 3)
        mixed[seg // 5:seg // 2] = 0
        xs = [mixed]
        if last == 16 and window <= 4096:
            xs += [synth.uniform(n, last), np.resize(synth.uniform(61, 2), n)]
        for x in xs:
            ost, ref = oracle.lzss_segmented_compress(x, seg, params)
            assert ost == oracle.OK
            got, _ = _compress(x, seg, params)
            assert np.array_equal(got, ref), (params, seg, last)
