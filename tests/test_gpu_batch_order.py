"""Batches whose buffers are taken in another order than they are given in, and
those that keep it: every buffer's result goes where it belongs.
"""
import ctypes
import time

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


@pytest.mark.parametrize("sizes", [[0, 5, 70000, 16, 16384, 1, 300000, 9, 0], [1000] * 5, [7, 8, 15, 14, 16],
                                   [40000, 20000, 30000], [2000, 999, 1999, 4000]])
def test_results_follow_their_buffers(sizes):
    xs = [synth.text(max(n, 1), i)[:n] for i, n in enumerate(sizes)]
    refs = [oracle.compress(x)[1] for x in xs]
    ins = [torch.from_numpy(x).cuda() for x in xs]
    outs = [torch.zeros(hg.huff_max_stream_size(n), dtype=torch.uint8, device="cuda") for n in sizes]
    plan = hg.BatchPlan(ins, outs, hg.HUFF_BATCH_COMPRESS)
    plan.run()
    got = plan.out_bytes.tolist()
    assert not any(plan.status.tolist()) and got == [r.size for r in refs]
    streams = [o[:g].clone() for o, g in zip(outs, got)]
    assert all(np.array_equal(s.cpu().numpy(), r) for s, r in zip(streams, refs))
    streams[1] = streams[1][:200]  # one that is cut short
    back = [torch.zeros(max(n, 1), dtype=torch.uint8, device="cuda") for n in sizes]
    plan = hg.BatchPlan(streams, back, hg.HUFF_BATCH_DECOMPRESS)
    plan.run()
    st = plan.status.tolist()
    assert st[1] == hg.HUFF_ERR_CORRUPT_STREAM and not any(st[:1] + st[2:])
    assert all(np.array_equal(b[:n].cpu().numpy(), x)
               for i, (b, n, x) in enumerate(zip(back, sizes, xs)) if i != 1)


def test_segments_need_no_second_plan():
    """16384 segments of 1 KiB against a plan over as many buffers and its run:
    the container's call also lays out and moves the streams."""
    n, seg, cs = 16 << 20, 1024, hg.DEFAULT_CHUNK_SYMBOLS
    L, count = hg.lib(), n // seg
    new = lambda k, t=torch.uint8: torch.zeros(k, dtype=t, device="cuda")
    x = new(n)
    cap, wsb = L.huff_segmented_max_size(n, seg, cs), L.huff_segmented_workspace_size(n, seg, cs)
    out, ws, size, st = new(cap), new(wsb), new(1, torch.int64), hg.new_status()
    slot = (hg.huff_max_stream_size(seg) + 15) // 16 * 16
    outs, sizes, sts = new(slot * count), new(count, torch.int64), new(count, torch.int32)
    descs = (hg.BatchDesc * count)(*[
        hg.BatchDesc(x.data_ptr() + i * seg, seg, outs.data_ptr() + i * slot, slot,
                     sizes.data_ptr() + 8 * i, sts.data_ptr() + 4 * i) for i in range(count)])
    prm = hg.huff_batch_default_params()
    prm.use_graph = 0

    def container():
        return L.huff_segmented_compress(x.data_ptr(), n, seg, cs, out.data_ptr(), cap, size.data_ptr(),
                                         ws.data_ptr(), wsb, st.data_ptr(), None)

    def planned():
        h = ctypes.c_void_p(0)
        r = L.huff_batch_plan(descs, count, hg.HUFF_BATCH_COMPRESS, ctypes.byref(prm), ctypes.byref(h))
        r = r or L.huff_batch_run(h, None)
        torch.cuda.synchronize()
        L.huff_batch_destroy(h)
        return r

    times = {f.__name__: [] for f in (container, planned)}
    for _ in range(40):  # in turn, and the least of each: the host's own noise
        for f in (container, planned):
            t0 = time.perf_counter()
            assert f() == 0
            torch.cuda.synchronize()
            times[f.__name__].append(time.perf_counter() - t0)
    least = {k: min(v) for k, v in times.items()}
    assert least["container"] < 1.2 * least["planned"], least
