"""Offsets of the centroid rows where one CTA adds them up (two turns at most)
and where they are scanned: rows of different lengths, empty ones among them."""
from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_harness import gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["dense", "sort"])
@pytest.mark.parametrize("k", [1, 2, 4095, 4096, 4097, 8191, 8192, 8193, 20_001])
def test_offsets_on_both_sides_of_the_line(k, mode):
    from synth.corpus import Corpus
    n, D = k + 700, 40
    lens = np.arange(n) % 7  # documents without terms too
    row_ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    idx = np.concatenate([np.arange(m) + 5 * (i % 6) for i, m in enumerate(lens)]).astype(np.int32)
    val = np.repeat(1 / np.sqrt(np.maximum(lens, 1)), lens).astype(np.float32)
    c = Corpus(N=n, D=D, row_ptr=row_ptr, idx=idx, val=val)
    g = gpu_instance(c, k, np.arange(k), update_mode=mode)
    try:
        for shift in (0, 3):
            lab = ((np.arange(n) + shift) % k).astype(np.int32)
            g.set_labels(lab)
            g.update()
            doc = np.repeat(np.arange(n), lens)
            cells = np.unique(lab[doc].astype(np.int64) * D + idx)
            off, term, _ = g.centroids()
            want = np.concatenate([[0], np.cumsum(np.bincount(cells // D, minlength=k))])
            assert np.array_equal(off, want) and np.array_equal(term, cells % D)
    finally:
        g.close()
