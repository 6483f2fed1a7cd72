"""The lanes a caller asks a buffer's decoding to be spread over count in a
batch that fills the chip too; the default leaves them to what costs least.
"""
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


def _median_ms(plan):
    plan.run()
    times = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        plan.run()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times)[3]


def test_own_lanes_in_a_batch_that_fills_the_chip():
    # 16 chunks a buffer, 65536 in all: one lane asks for whole chunks, which
    # leave half of a warp and three of an item's four warps idle
    count, size, cs = 4096, 1 << 16, 4096
    x = torch.from_numpy(synth.text(64 * size, 5)).cuda()
    ins = [x[size * (i % 64):size * (i % 64 + 1)] for i in range(count)]
    prm = hg.huff_batch_default_params()
    prm.chunk_symbols = cs
    cap = hg.huff_max_stream_size(size, cs) + 255 & ~255
    arena = torch.zeros(count * cap, dtype=torch.uint8, device="cuda")
    plan = hg.BatchPlan(ins, [arena[i * cap:(i + 1) * cap] for i in range(count)],
                        hg.HUFF_BATCH_COMPRESS, prm)
    plan.run()
    got = plan.out_bytes.tolist()
    back = torch.zeros(count * size, dtype=torch.uint8, device="cuda")
    ms = {}
    for lanes in (1, 32, 128, 256):
        prm.decode_lanes = lanes
        plan = hg.BatchPlan([arena[i * cap:i * cap + g] for i, g in enumerate(got)],
                            [back[i * size:(i + 1) * size] for i in range(count)],
                            hg.HUFF_BATCH_DECOMPRESS, prm)
        ms[lanes] = _median_ms(plan)
        assert not any(plan.status.tolist()) and torch.equal(back, x.repeat(count // 64))
        back.zero_()
    assert ms[1] > 1.25 * ms[128], ms
    assert ms[32] > 1.1 * ms[128], ms
