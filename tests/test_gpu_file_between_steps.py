"""sivf_get_inverted_file between an assignment (or sivf_set_labels) and the
update: lambda has changed, the file has not, and the getter gives the file of the
last update whether or not it was asked before."""
from __future__ import annotations

import numpy as np
import pytest

from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("icp", [1, 0, "cbicp"])
@pytest.mark.parametrize("step", ["assign", "set_labels"])
def test_file_of_the_last_update(step, icp):
    w = CONFIGS["c1"].scaled(N=900, D=1_500, k=30)
    c, ini = corpus_for(w, seed=6)
    g, h = (gpu_instance(c, w.k, ini, icp=icp) for _ in range(2))
    try:
        for _ in range(2):
            for x in (g, h):
                x.assign()
                x.update()
        want = g.inverted_file()
        lam = h.lam()
        other = g.labels()
        other[:50] = (other[:50] + 1) % w.k
        for x in (g, h):
            x.assign() if step == "assign" else x.set_labels(other)
        assert (h.lam() != lam).any()
        for x in (g, h):
            assert all(np.array_equal(a, b) for a, b in zip(x.inverted_file(), want))
    finally:
        g.close()
        h.close()
