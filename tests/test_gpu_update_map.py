"""The occupancy map of the update step's accumulator.

Where rows are mostly empty, the dense update reads them through a map of the
entries that may be non-zero. The map is dropped when the memory cap has no
room for it (whole rows are then read), and a restart empties the accumulator
through it. Either way the centroids are the same, bit for bit.
"""
from __future__ import annotations

import numpy as np
import pytest

from synth import CONFIGS
from tests.gpu_harness import corpus_for, gpu_instance, lockstep

pytestmark = pytest.mark.gpu


def _run(g, iters=8):
    for _ in range(iters):
        g.assign()
        g.update()
    return (g.labels(), *g.centroids(), g.stats()["objective_update"], g.stats()["objective_assign"])


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("D", [31, 32, 33, 5_000])
def test_rows_at_the_edges_of_map_words(D):
    w = CONFIGS["c1"].scaled(N=60, D=D, k=50, mu=1.0, lo=2, hi=4)  # rows nearly empty: the map is in use
    c, ini = corpus_for(w, seed=5)
    lockstep(c, w.k, ini, 6, update_mode="dense")


def test_without_room_for_the_map():
    from paper_2103_16141_gb300 import SivfError
    w = CONFIGS["c1"].scaled(N=1_500, D=4_001, k=300)
    c, ini = corpus_for(w, seed=6)
    g = gpu_instance(c, w.k, ini, update_mode="dense")
    want = _run(g)
    g.close()
    lo, hi = 0, 1 << 28  # the smallest cap that the context fits in: nothing is left for the map
    while hi - lo > 256:
        mid = (lo + hi) // 2
        try:
            gpu_instance(c, w.k, ini, update_mode="dense", mem_cap_bytes=mid).close()
            hi = mid
        except SivfError:
            lo = mid
    g = gpu_instance(c, w.k, ini, update_mode="dense", mem_cap_bytes=hi)
    assert _same(want, _run(g))
    g.reseed(ini)
    assert _same(want, _run(g))
    g.close()


def test_restart_leaves_nothing_behind():
    w = CONFIGS["c1"].scaled(N=1_500, D=4_001, k=300)
    c, ini = corpus_for(w, seed=7)
    other = ini[::-1].copy()
    g = gpu_instance(c, w.k, ini, update_mode="dense")
    want = _run(g)
    g.reseed(other)
    _run(g, 3)
    g.reseed(ini)
    assert _same(want, _run(g))
    g.close()


def test_entries_that_empty_and_fill_again():
    """Labels that empty half of the clusters, and back: the map follows, as
    the sort form (which has no accumulator) shows. Its sums are FP64 in member
    order, the values agree to the FP32 rounding of either form (2.4e-7)."""
    w = CONFIGS["c1"].scaled(N=1_500, D=4_001, k=300)
    c, ini = corpus_for(w, seed=8)
    lab = (np.arange(c.N) * 7 % w.k).astype(np.int32)
    merged = np.where(lab < 150, 0, lab).astype(np.int32)  # one full row (read whole), 149 emptied
    rows = []
    for mode in ("dense", "sort"):
        g = gpu_instance(c, w.k, ini, update_mode=mode)
        for x in (lab, merged, lab):
            g.set_labels(x)
            g.update()
        rows.append(g.centroids())
        g.close()
    (o0, t0, u0), (o1, t1, u1) = rows
    assert np.array_equal(o0, o1) and np.array_equal(t0, t1)
    np.testing.assert_allclose(u0.astype(np.float64), u1, rtol=5e-7, atol=0)
