"""Checked mode looks at every object's offsets and terms, also at the filtered
objects of a converged run, which no kernel scores any more."""
from __future__ import annotations

import pytest

from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flaw", ["term_eq_D", "term_negative", "row_ptr"])
@pytest.mark.parametrize("light_max_moving", [0, -1])
@pytest.mark.parametrize("icp", [1, "relaxed", "cbicp"])
def test_a_change_after_convergence_is_caught(icp, light_max_moving, flaw):
    from paper_2103_16141_gb300 import sivf as S
    w = CONFIGS["c1"].scaled(N=400, D=1_500, k=12)
    c, ini = corpus_for(w, seed=3)
    g = gpu_instance(c, w.k, ini, icp=icp, checked=True, light_max_moving=light_max_moving)
    try:
        for _ in range(40):
            n = g.assign()
            g.update()
            if n == 0:
                break
        assert n == 0 and g.stats()["n_moving"] == 0
        assert g.assign() == 0  # every object filtered, nothing wrong
        assert g.stats()["filtered"] == c.N
        g.update()
        if flaw == "row_ptr":
            g.row_ptr[9] = int(c.row_ptr[-1]) + 100
        else:
            g.idx[int(c.row_ptr[8]) - 1] = w.D if flaw == "term_eq_D" else -1
        with pytest.raises(S.SivfError) as ex:
            g.assign()
        assert ex.value.status == S.SIVF_ERR_STATE and "device-side check" in g.last_error()
    finally:
        g.close()
