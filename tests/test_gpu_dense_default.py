"""The default line from which a list becomes a dense row is a quarter of k for
every precision: shorter lists keep their exact integer sums unless the caller
asks for rows."""
from __future__ import annotations

import pytest

from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_default_is_a_quarter(precision):
    w = CONFIGS["c1"].scaled(N=3_000, D=2_000, k=200)
    c, ini = corpus_for(w, seed=4)
    seen = {}
    for frac in (0.0, 0.25, 0.17):
        g = gpu_instance(c, w.k, ini, precision=precision, dense_min_fraction=frac)
        for _ in range(3):
            g.assign()
            g.update()
        st = g.stats()
        seen[frac] = (st["dense_terms"], st["dense_row_entries"], st["dense_entries"], st["dense_postings"])
        g.close()
    assert seen[0.0] == seen[0.25]
    assert seen[0.17][0] > seen[0.25][0]  # the corpus has lists between the two
