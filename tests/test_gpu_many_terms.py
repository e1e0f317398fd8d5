"""Vocabularies of millions of terms: the offsets of the inverted file where its
tiles (1024 terms) are added up by every block and where they are scanned first,
and an update's time that does not grow faster than the vocabulary."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import Oracle
from tests.gpu_harness import gpu_instance

pytestmark = pytest.mark.gpu


def _corpus(D, n=400, common=8, rare=12):
    """Documents of most of a few common terms (dense rows) and some rare ones,
    both spread over the whole vocabulary, its last terms among them."""
    from synth.corpus import Corpus
    rng = np.random.default_rng(D)
    head = (np.arange(common, dtype=np.int64) * (D - 1) // (common - 1))
    rows = []
    for _ in range(n):
        t = np.concatenate([rng.choice(head, common - 2, replace=False), rng.integers(0, D, rare),
                            D - 1 - rng.integers(0, 3_000, 2)])
        rows.append(np.unique(t))
    lens = np.array([len(r) for r in rows])
    val = rng.random(lens.sum()) + 0.1
    row_ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    norm = np.sqrt(np.add.reduceat(val * val, row_ptr[:-1]))
    return Corpus(N=n, D=D, row_ptr=row_ptr, idx=np.concatenate(rows).astype(np.int32),
                  val=(val / np.repeat(norm, lens)).astype(np.float32))


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("D", [4096 * 1024 - 1, 4096 * 1024, 4096 * 1024 + 1, 4100 * 1024 + 777, 9_000_001])
def test_offsets_on_both_sides_of_the_line(D, precision):
    c = _corpus(D)
    k = 160
    ini = np.arange(k, dtype=np.int32) * 2
    g = gpu_instance(c, k, ini, precision=precision, update_mode="sort")
    o = Oracle(c, k, ini, icp=True)
    try:
        for _ in range(3):
            g.assign(), o.assign()
            g.set_labels(o.labels())
            g.update(), o.update()
            off, mf0, cid, u = g.inverted_file()
            o_off, o_mf0, o_cid, o_u = o.inverted_file()
            assert np.array_equal(off, o_off) and np.array_equal(mf0, o_mf0) and np.array_equal(cid, o_cid)
            np.testing.assert_allclose(u, o_u, rtol=1e-5, atol=0)
        assert g.stats()["dense_terms"] > 0
        # the scan copy is addressed through the same offsets: exact scores, exact labels
        g.assign(), o.assign()
        best, second, _ = o.scores()
        diff = np.nonzero(g.labels() != o.labels())[0]
        assert np.all(best[diff] - second[diff] < 1e-6)
    finally:
        g.close()


def test_time_grows_with_the_vocabulary_not_faster():
    """Eight times the terms, at most eight times the device time of an update
    (every block adding up every earlier tile took thirteen times as long)."""
    ms = []
    for D in (16_000_000, 128_000_000):
        c = _corpus(D)
        g = gpu_instance(c, 50, np.arange(50), update_mode="sort", dense_max_bytes=1 << 20)
        lab = np.arange(c.N, dtype=np.int32) % 50
        t = []
        for r in range(8):
            g.set_labels(np.roll(lab, r))
            g.update()
            t.append(g.stats()["ms_update"])
        g.close()
        ms.append(min(t[2:]))
    assert ms[1] <= 8 * ms[0], ms
