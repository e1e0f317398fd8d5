"""sivf_reseed over a borrowed CSR whose offsets changed after sivf_init: seed
rows that lie outside the CSR, or do not fit the centroid buffers, are not read;
the call reports SIVF_ERR_OOM and the context is latched."""
from __future__ import annotations

import numpy as np
import pytest

from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["dense", "sort"])
@pytest.mark.parametrize("offsets", ["beyond_nnz", "descending", "negative", "overlapping"])
def test_changed_offsets_are_refused(offsets, mode):
    from paper_2103_16141_gb300 import sivf as S
    w = CONFIGS["c1"].scaled(N=400, D=1_500, k=12)
    c, ini = corpus_for(w, seed=3)
    nnz = int(c.row_ptr[-1])
    g = gpu_instance(c, w.k, ini, update_mode=mode)
    try:
        g.run(3)
        ini = np.arange(0, 2 * w.k, 2, dtype=np.int32)
        if offsets == "beyond_nnz":
            g.row_ptr[1] = nnz + 100
        elif offsets == "descending":
            g.row_ptr[2] = int(c.row_ptr[4])
        elif offsets == "negative":
            g.row_ptr[0] = -4
        else:  # every seed's row inside the CSR, together more than 2 nnz + 1024 entries
            g.row_ptr[0:2 * w.k:2] = 0
            g.row_ptr[1:2 * w.k:2] = nnz
        with pytest.raises(S.SivfError) as ex:
            g.reseed(ini)
        assert ex.value.status == S.SIVF_ERR_OOM
        with pytest.raises(S.SivfError) as ex:
            g.run(1)
        assert ex.value.status == S.SIVF_ERR_STATE
    finally:
        g.close()
