"""The codebook's merge in rounds and step by step: alphabets around the size
that parts them, and weights that tie, spread evenly or grow like powers."""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_11070_gb300 as hg
from paper_2306_11070_gb300 import build as nvbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    nvbuild.build()
    hg.lib()


@pytest.mark.parametrize("values", [2, 63, 64, 65, 66, 97, 128, 255, 256])
@pytest.mark.parametrize("kind", ["equal", "few", "even", "powers", "golden", "heavy"])
def test_lengths_and_codes_against_oracle(values, kind):
    rng = np.random.default_rng(values)
    k = np.arange(values)
    w = {"equal": lambda: np.full(values, 5), "few": lambda: rng.integers(1, 4, values),
         "even": lambda: rng.integers(1, 100000, values), "powers": lambda: 1 << rng.integers(0, 30, values),
         "golden": lambda: (1.618 ** np.minimum(k, 20)).astype(np.int64),
         "heavy": lambda: rng.integers(1, 1 << 47, values)}[kind]()
    hist = np.zeros(256, np.int64)
    hist[rng.permutation(256)[:values]] = w
    ost, lengths = oracle.code_lengths(hist)
    cb, st = hg.huff_build_codebook(torch.from_numpy(hist).cuda())
    raw = cb.cpu().numpy()
    assert int(st.item()) == ost  # (one of the inputs needs a code of 33 bits)
    if ost != oracle.OK:
        assert not raw.any()
        return
    assert np.array_equal(raw[:256], lengths)
    assert np.array_equal(raw[256:1280].view("<u4"), oracle.canonical_codes(lengths))
