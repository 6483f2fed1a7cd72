"""The decoder that very many short segments take, a thread each, for every
kind of parameters: at the segment counts from which it is chosen, against the
decoder of two warps per segment and the input, and its time on tiny segments.
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


def _data(n, seed):
    x = synth.bitstream(n, seed)
    x[n // 3:n // 2] = 0
    x[n // 2:n // 2 + n // 8] = np.resize(np.array([0xB6, 0xDB, 0x6D], np.uint8), n // 8)
    return x


def _container(x, seg, params):
    c, st = hg.huff_lzss_compress(torch.from_numpy(x).cuda(), seg, params)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    return c


# (parameters, segment bytes, segments per SM from which a thread each decodes):
# windows below a word, in the thread's ring and read back from the output; both
# dictionaries; segments shorter than the stored prefix; 32-bit literals
@pytest.mark.parametrize("params,seg,per_sm", [
    ((2, 1, 1, 1, 1), 16, 100), ((16, 3, 10, 4, 1), 64, 100), ((16, 3, 10, 4, 2), 80, 200),
    ((64, 4, 11, 8, 1), 128, 200), ((64, 4, 11, 8, 2), 80, 100), ((256, 4, 32, 32, 2), 48, 100),
    ((256, 12, 24, 32, 2), 64, 200), ((1024, 12, 24, 8, 1), 32, 100),
    ((2048, 16, 32, 8, 1), 128, 320), ((4096, 12, 24, 8, 1), 48, 200),
    ((4096, 16, 32, 8, 2), 128, 320), ((65536, 24, 32, 8, 1), 16, 100)])
def test_every_kind_at_the_choice(params, seg, per_sm):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for count in (per_sm * sms - 1, per_sm * sms):
        n = count * seg - 5
        x = _data(n, seg)
        c = _container(x, seg, params)
        y, got, st = hg.huff_lzss_decompress(c, out_cap=n)
        torch.cuda.synchronize()
        assert int(st.item()) == 0 and got == n
        assert np.array_equal(y.cpu().numpy(), x), count
        for at in (48, 48 + 4 * (count // 2)):  # a segment's length one bit too long
            bad = c.clone()
            bad[at] = bad[at] ^ 1
            y, got, st = hg.huff_lzss_decompress(bad, out_cap=n)
            torch.cuda.synchronize()
            assert int(st.item()) == hg.HUFF_ERR_CORRUPT_STREAM


@pytest.mark.parametrize("params", [(16, 3, 10, 4, 1), (256, 4, 32, 32, 2), (4096, 12, 24, 8, 1),
                                    (4096, 16, 32, 8, 2), (65536, 24, 32, 8, 1)])
def test_few_segments_of_many_against_oracle(params):
    """The oracle's container, its segments repeated until a thread each decodes."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    seg, kinds = 48, 64
    x = _data(seg * kinds, 5)
    reps = (200 * sms + kinds - 1) // kinds
    ost, ref = oracle.lzss_segmented_compress(np.tile(x, reps)[:seg * kinds * 2], seg, params)
    assert ost == oracle.OK
    head = ref[48:48 + 4 * kinds]
    start = (48 + 4 * kinds * 2 + 15) // 16 * 16
    bits = head.view(np.uint32).astype(np.int64)
    size = int((((bits + 7) // 8 + 15) // 16).sum()) * 16
    codes = ref[start:start + size]
    count = reps * kinds
    table = np.tile(head, reps)
    hdr = ref[:48].copy()
    hdr[:8] = np.frombuffer(np.uint64(count * seg).tobytes(), np.uint8)
    hdr[40:48] = np.frombuffer(np.uint64(count).tobytes(), np.uint8)
    pad = np.zeros((48 + table.size + 15) // 16 * 16 - 48 - table.size, np.uint8)
    c = torch.from_numpy(np.concatenate([hdr, table, pad, np.tile(codes, reps)])).cuda()
    y, got, st = hg.huff_lzss_decompress(c, out_cap=count * seg)
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and got == count * seg
    assert np.array_equal(y.cpu().numpy(), np.tile(x, reps))


def test_tiny_segments_take_no_longer_with_the_dictionary():
    """A million 16-byte segments: the counting dictionary, which has tokens to
    decode, against the stored prefix, which has none, within twice its time
    (a CTA per segment took 3.6 times)."""
    n = 16 << 20
    x, ms = _data(n, 1), {}
    for dictionary in (1, 2):
        c = _container(x, 16, (1024, 12, 24, 8, dictionary))
        out, dn = torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
        ws = torch.zeros(hg.lib().huff_lzss_decompress_workspace_size(c.numel()), dtype=torch.uint8, device="cuda")
        st, times = hg.new_status(), []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            hg.huff_lzss_decompress(c, d_out=out, d_n=dn, d_ws=ws, d_status=st)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        ms[dictionary] = sorted(times)[4]
    assert ms[1] < 2 * ms[2], ms
