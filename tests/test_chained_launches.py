"""Kernels launched behind one another (launch_chained) start while the ones
before them still run: each waits at its top level, before anything else that
could touch global memory, and reads nothing through the read-only path.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2306_11070_gb300", "csrc")


def _text(path):
    text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _matching(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def _chained():
    """(file, kernel) -> (parameters, body) of every kernel given to launch_chained."""
    files = {p: _text(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))}
    names = set()
    for text in files.values():
        for m in re.finditer(r"launch_chained\(([^,]*),", text):
            names.update(re.findall(r"\bk_\w+", m.group(1)))
    found = {}
    for path, text in files.items():
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            if m.group(1) in names:
                close = _matching(text, m.end() - 1, "()")
                start = text.index("{", close)
                found[os.path.basename(path), m.group(1)] = (
                    text[m.end():close], text[start + 1:_matching(text, start, "{}")])
    assert names and names == {k for _, k in found}
    return found


CHAINED = _chained()


@pytest.mark.parametrize("where", sorted(CHAINED))
def test_waits_before_it_touches_memory(where):
    params, body = CHAINED[where]
    head, wait, _ = body.partition("chain_wait();")
    assert wait, "no wait"
    assert head.count("{") == head.count("}") and "return" not in head, "not on every path"
    for p in params.split(","):
        name = re.search(r"(\w+)\s*$", p).group(1)
        assert not re.search(rf"\b{name}\b", head), f"{name} is used before the wait"
    assert "__restrict__" not in params


def test_their_routines_have_no_read_only_pointers():
    """The device routines that chained kernels pass their pointers to."""
    for name in ("codebook_impl.cuh", "hist_impl.cuh", "encode_impl.cuh", "sort_impl.cuh"):
        assert "__restrict__" not in _text(os.path.join(CSRC, name)), name
