"""The batched encoder's code table lies at a fixed address of shared memory: a
build whose static shared memory leaves no place there refuses the batch when
it is planned, and says so, instead of failing every buffer of every run.
"""
import ctypes
import os
import subprocess

import pytest
import torch

import paper_2306_11070_gb300 as hg
from paper_2306_11070_gb300 import build as nvbuild

pytestmark = pytest.mark.gpu


def test_a_build_without_room_for_the_table(tmp_path):
    nvbuild.build()
    hg.lib()
    src = os.path.join(nvbuild.CSRC, "batch.cu")
    obj, so = str(tmp_path / "batch.o"), str(tmp_path / "libhuff_moved.so")
    subprocess.run([nvbuild.nvcc()] + nvbuild.ARCH + nvbuild.NVCC_FLAGS +
                   ["-DHUFF_BATCH_TABLE_AT=2048", "-c", src, "-o", obj], check=True)
    others = [os.path.join(nvbuild.BUILD, os.path.basename(s)[:-3] + ".o")
              for s in nvbuild.sources() if s != src]
    subprocess.run([nvbuild.nvcc()] + nvbuild.ARCH + ["-shared", "-cudart", "shared", "-o", so, obj] + others,
                   check=True)
    moved = ctypes.CDLL(so)
    x = torch.zeros(1000, dtype=torch.uint8, device="cuda")
    out = torch.zeros(hg.huff_max_stream_size(1000), dtype=torch.uint8, device="cuda")
    size, st = torch.zeros(1, dtype=torch.int64, device="cuda"), hg.new_status()
    desc = hg.BatchDesc(x.data_ptr(), 1000, out.data_ptr(), out.numel(), size.data_ptr(), st.data_ptr())
    for lib, want in ((hg.lib(), hg.HUFF_OK), (moved, hg.HUFF_ERR_UNSUPPORTED)):
        plan = ctypes.c_void_p(0)
        got = lib.huff_batch_plan(ctypes.byref(desc), 1, hg.HUFF_BATCH_COMPRESS, None, ctypes.byref(plan))
        assert ctypes.c_int32(got).value == want
        assert bool(plan.value) == (want == hg.HUFF_OK)
        lib.huff_batch_destroy(plan)
