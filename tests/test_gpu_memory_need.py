"""What a context needs of its memory cap where the vocabulary is nearly as large
as the corpus, so that most lists are a posting or two and are padded most: no
more than with lists padded as a whole, in the sort form of the update, whose
buffers for the tuples are the larger ones. The getters' file lies in the spare
centroid buffer and leaves the run alone."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import Oracle
from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k, precision, need", [(100, "fp32", 295_195_840), (50_000, "fp32", 297940340)])
def test_large_vocabulary_fits_its_cap(k, precision, need):
    """140,000 documents of 7 terms out of 1,000,000."""
    from synth.corpus import Corpus
    n, D, L = 140_000, 1_000_000, 7
    idx = np.arange(n)[:, None] * 7 % (D // L) + np.arange(L)[None, :] * (D // L)
    c = Corpus(N=n, D=D, row_ptr=np.arange(n + 1, dtype=np.int64) * L, idx=idx.astype(np.int32).reshape(-1),
               val=np.full(n * L, 1 / np.sqrt(L), np.float32))
    g = gpu_instance(c, k, np.arange(k), precision=precision, update_mode="sort", mem_cap_bytes=need)
    try:
        g.set_labels(np.arange(n, dtype=np.int32) % k)
        g.update()
        assert g.stats()["centroid_nnz"] <= n * L
    finally:
        g.close()


@pytest.mark.parametrize("mode", ["dense", "sort"])
@pytest.mark.parametrize("use_graph", [False, True])
def test_file_between_the_steps(mode, use_graph):
    """The canonical file after every update, and a run that does not notice."""
    w = CONFIGS["c1"].scaled(N=900, D=1_500, k=30)
    c, ini = corpus_for(w, seed=6)
    g = gpu_instance(c, w.k, ini, update_mode=mode, use_graph=use_graph)
    h = gpu_instance(c, w.k, ini, update_mode=mode, use_graph=use_graph)
    o = Oracle(c, w.k, ini, icp=True)
    try:
        for _ in range(3):
            g.assign(), h.assign(), o.assign()
            for x in (g, h):
                x.set_labels(o.labels())
                x.update()
            o.update()
            off, mf0, cid, u = g.inverted_file()
            o_off, o_mf0, o_cid, o_u = o.inverted_file()
            assert np.array_equal(off, o_off) and np.array_equal(mf0, o_mf0) and np.array_equal(cid, o_cid)
            np.testing.assert_allclose(u, o_u, rtol=1e-5, atol=0)
            assert all(np.array_equal(a, b) for a, b in zip(g.centroids(), h.centroids()))
        assert g.run(10) == h.run(10)
        assert np.array_equal(g.labels(), h.labels())
        g.set_labels(g.labels()), h.set_labels(h.labels())
        g.update(), h.update()
        assert all(np.array_equal(a, b) for a, b in zip(g.inverted_file(), h.inverted_file()))
        assert all(np.array_equal(a, b) for a, b in zip(g.centroids(), h.centroids()))
    finally:
        g.close()
        h.close()


@pytest.mark.parametrize("k", [3, 60])
def test_more_clusters_than_terms_in_the_corpus(k):
    """Documents without terms: the sort form's table of clusters has k entries
    where its tuples are three."""
    from synth.corpus import Corpus
    n = 200
    row_ptr = np.zeros(n + 1, np.int64)
    row_ptr[150:] = 1
    row_ptr[160:] = 2
    row_ptr[170:] = 3
    c = Corpus(N=n, D=9, row_ptr=row_ptr, idx=np.array([4, 4, 8], np.int32), val=np.ones(3, np.float32))
    g = gpu_instance(c, k, np.arange(k), update_mode="sort")
    try:
        lab = np.arange(n, dtype=np.int32) % k
        g.set_labels(lab)
        g.update()
        off, term, u = g.centroids()
        want = {int(lab[149]): 4, int(lab[159]): 4, int(lab[169]): 8}  # k = 3 and 60: three clusters
        assert len(want) == 3 and np.array_equal(u, np.ones(3, np.float32))
        assert {j: int(term[off[j]]) for j in range(k) if off[j + 1] > off[j]} == want
    finally:
        g.close()
