"""<s_j, mu_j> of an update where the previous centroid's value is too small for
the unit of the exact sum: 1000 members of one term, whose value in the seed's
row is far below 1, and nothing else in common. One product per cluster, so that
it holds to the rounding of FP64 (2^-52 with the sum over the members), with
either part of the row passes."""
from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_harness import gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["dense", "sort"])
@pytest.mark.parametrize("D", [3, 5_000])
@pytest.mark.parametrize("small", [2.0**-20, 2.0**-40, 2.0**-41, 2.0**-55, 2.0**-62, 2.0**-64, 2.0**-100, 2.0**-126, 2.0**-140])
def test_objective_of_small_previous_values(small, D, mode):
    from synth.corpus import Corpus
    n = 1_000
    u = np.float32(small * 1.2345678)  # bits all the way down, except where subnormal
    # document 0: terms 0 and 1, document 1: term 2, the others: term 1 alone
    idx = np.concatenate([[0, 1, 2], np.ones(n)]).astype(np.int32)
    val = np.concatenate([[1.0, u, 1.0], np.ones(n)]).astype(np.float32)
    row_ptr = np.concatenate([[0, 2, 3], 3 + np.arange(1, n + 1)]).astype(np.int64)
    c = Corpus(N=n + 2, D=D, row_ptr=row_ptr, idx=idx, val=val)
    g = gpu_instance(c, 2, np.array([0, 1]), update_mode=mode)
    try:
        lab = np.zeros(c.N, np.int32)
        lab[0] = 1  # document 0 away from its seed's cluster, which the others join
        g.set_labels(lab)
        g.update()
        want = n * float(u)
        assert abs(g.stats()["objective_assign"] - want) <= 4e-16 * want
    finally:
        g.close()
