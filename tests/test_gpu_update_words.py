"""The words of non-zero entries that the update's first row pass leaves for
the second, where rows are too full for the occupancy map (the words lie in
scratch) or one row of a mapped accumulator is (they lie in the map). Sparsity
patterns are the oracle's; with the words or without them the centroids are the
same, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance, lockstep

pytestmark = pytest.mark.gpu


# one word, its edges, odd rows, one turn of the first pass (2048 entries) and more, eight stretches of one word and of two
@pytest.mark.parametrize("D", [31, 32, 33, 63, 65, 255, 257, 2_047, 2_049, 9_001])
def test_full_rows_at_the_edges(D):
    w = CONFIGS["c1"].scaled(N=700, D=D, k=5, mu=3.0, lo=2, hi=min(D, 60))
    c, ini = corpus_for(w, seed=9)
    assert c.row_ptr[-1] * 16 // 3 > 5 * D  # no map
    lockstep(c, w.k, ini, 5, update_mode="dense")


def test_full_row_of_a_mapped_accumulator():
    """All objects in one cluster of 300, then spread: that cluster's row is read
    whole and leaves its words in the map, which the later steps read."""
    w = CONFIGS["c1"].scaled(N=1_500, D=4_001, k=300)
    c, ini = corpus_for(w, seed=10)
    spread = (np.arange(c.N) * 11 % w.k).astype(np.int32)
    out = []
    for mode in ("dense", "sort"):
        g = gpu_instance(c, w.k, ini, update_mode=mode)
        for lab in (spread, np.zeros(c.N, np.int32), spread, spread[::-1].copy()):
            g.set_labels(lab)
            g.update()
        out.append(g.centroids())
        g.close()
    (o0, t0, u0), (o1, t1, u1) = out
    assert np.array_equal(o0, o1) and np.array_equal(t0, t1)
    np.testing.assert_allclose(u0.astype(np.float64), u1, rtol=5e-7, atol=0)  # FP32 rounding of either form


def test_no_room_for_map_or_words():
    """Rows nearly empty and a memory cap that leaves no map; the workspace is
    then too small for the words as well, and rows are read whole twice."""
    from paper_2103_16141_gb300 import SivfError
    w = CONFIGS["c1"].scaled(N=600, D=20_001, k=500, mu=1.0, lo=2, hi=4)
    c, ini = corpus_for(w, seed=11)

    def run(**kw):
        g = gpu_instance(c, w.k, ini, update_mode="dense", **kw)
        for _ in range(4):
            g.assign()
            g.update()
        r = (g.labels(), *g.centroids(), g.stats()["objective_update"])
        g.close()
        return r

    want = run()
    lo, hi = 0, 1 << 29
    while hi - lo > 256:
        mid = (lo + hi) // 2
        try:
            gpu_instance(c, w.k, ini, update_mode="dense", mem_cap_bytes=mid).close()
            hi = mid
        except SivfError:
            lo = mid
    assert all(np.array_equal(x, y) for x, y in zip(want, run(mem_cap_bytes=hi)))


@pytest.mark.parametrize("D", [33, 2_049, 9_001, 20_000])
def test_objective_of_the_previous_centroids(D):
    """<s_j, mu_j> summed over the clusters whose members changed, taken in
    stretches of 8192 entries and exactly, against the exact sum over the objects.
    The accumulator's entries are rounded up by less than 2^-52 each: 4e-12 in all
    for 17,000 values; the sums per cluster are added in FP64."""
    from math import fsum
    w = CONFIGS["c1"].scaled(N=700, D=D, k=5, mu=3.0, lo=2, hi=min(D, 60))
    c, ini = corpus_for(w, seed=12)
    g = gpu_instance(c, w.k, ini, update_mode="dense")
    obj = np.repeat(np.arange(c.N), np.diff(c.row_ptr))
    rng = np.random.default_rng(D)
    for step in range(3):
        off, term, u = g.centroids()
        mu = np.zeros((w.k, D))
        for j in range(w.k):
            mu[j, term[off[j]:off[j + 1]]] = u[off[j]:off[j + 1]]
        lab = rng.integers(0, w.k, c.N).astype(np.int32)
        g.set_labels(lab)
        g.update()
        want = fsum(c.val.astype(np.float64) * mu[lab[obj], c.idx])
        assert abs(g.stats()["objective_assign"] - want) <= 1e-11 + 1e-14 * want, step
    g.close()
