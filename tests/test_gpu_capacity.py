"""Centroids that outgrow their buffers (2 nnz + 1024 entries: empty clusters
keep their rows, so labels set by a caller can get there). The new rows are then
not written, nothing is built from them, and the call reports SIVF_ERR_OOM: after
an update, and from inside the device loop, which ends with it."""
from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_harness import gpu_instance

pytestmark = pytest.mark.gpu

TOPICS, DOCS, CORE, OWN = 20, 20, 10, 20


def _topics():
    """400 documents in 20 topics: 10 terms of the topic and 20 of its own each.
    The means of a topic are near its documents, the mean of all is not."""
    from synth.corpus import Corpus
    n = TOPICS * DOCS
    idx = np.concatenate([np.concatenate([np.arange(CORE) + CORE * (i // DOCS),
                                          TOPICS * CORE + OWN * i + np.arange(OWN)]) for i in range(n)])
    val = np.tile(np.concatenate([np.full(CORE, np.sqrt(0.7 / CORE)), np.full(OWN, np.sqrt(0.3 / OWN))]), n)
    return Corpus(N=n, D=TOPICS * CORE + n * OWN, row_ptr=np.arange(n + 1, dtype=np.int64) * (CORE + OWN),
                  idx=idx.astype(np.int32), val=val.astype(np.float32))


def _outgrown(g, call):
    from paper_2103_16141_gb300 import sivf as S
    with pytest.raises(S.SivfError) as ex:
        call()
    assert ex.value.status == S.SIVF_ERR_OOM and "outgrew" in g.last_error()
    for later in (g.assign, g.update, g.labels):
        with pytest.raises(S.SivfError) as ex:
            later()
        assert ex.value.status == S.SIVF_ERR_STATE


@pytest.mark.parametrize("mode", ["dense", "sort"])
def test_one_cluster_after_another(mode):
    c = _topics()
    k, cap = 23, 2 * len(c.idx) + 1024
    g = gpu_instance(c, k, np.arange(k) * (c.N // k), update_mode=mode)
    try:
        full = (cap - (k - 3) * (CORE + OWN)) // c.D  # rows of all D terms that fit beside the seeds' rows
        for j in range(full):
            g.set_labels(np.full(c.N, j, np.int32))
            g.update()
            assert g.stats()["centroid_nnz"] == (j + 1) * c.D + (k - 1 - j) * (CORE + OWN)
        g.set_labels(np.full(c.N, full, np.int32))
        _outgrown(g, g.update)
    finally:
        g.close()


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("mode", ["dense", "sort"])
def test_in_the_middle_of_a_run(mode, use_graph):
    c = _topics()
    topic = np.arange(c.N) // DOCS
    first = np.arange(TOPICS) * DOCS
    ini = np.concatenate([first, [1, 2, 3]])
    g = gpu_instance(c, TOPICS + 3, ini, update_mode=mode, use_graph=use_graph)
    try:
        for _ in range(2):
            g.assign()
            g.update()
        one = np.full(c.N, TOPICS, np.int32)
        ones = one.copy()
        ones[first] = topic[first]  # a document of each topic in a cluster of its own
        half = one.copy()
        half[:c.N // 2] = TOPICS + 1
        for lab in (ones, half, one, one + 2):
            g.set_labels(lab)
            g.update()
        # rows of one document per topic, two of all terms, one of half of the documents
        small = TOPICS * (CORE + OWN) + 2 * c.D
        half_row = TOPICS // 2 * (CORE + OWN * DOCS)
        assert g.stats()["centroid_nnz"] == small + half_row <= 2 * len(c.idx) + 1024
        assert 3 * c.D + half_row > 2 * len(c.idx) + 1024  # every topic back in its cluster, the rest kept
        _outgrown(g, lambda: g.run(5))
    finally:
        g.close()
