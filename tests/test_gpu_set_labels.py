"""Labels replaced in the middle of a run: after the update the centroids and
the objective are those of the labels set, whatever the labels before them were,
and the run goes on like the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import Oracle
from synth import CONFIGS
from tests.gpu_harness import OBJECTIVE_RTOL, compare_centroids, compare_labels, corpus_for, gpu_instance, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["dense", "sort"])
@pytest.mark.parametrize("seq", ["previous", "there_and_back", "twice_before_the_update", "same"])
def test_centroids_belong_to_the_labels_set(mode, seq):
    w = CONFIGS["c1"].scaled(N=700, D=1_500, k=14)
    c, ini = corpus_for(w, seed=21)
    g = gpu_instance(c, w.k, ini, update_mode=mode)
    o, ou = Oracle(c, w.k, ini, icp=True), Oracle(c, w.k, ini, icp=False)  # the unfiltered twin gives the margins
    last = prev = None

    def push(*labels):
        for lab in labels:
            g.set_labels(lab)
            o.set_labels(lab)
            ou.set_labels(lab)
        g.update()
        u = o.update()
        ou.update()
        assert np.array_equal(g.labels(), labels[-1])
        assert rel(g.stats()["objective_update"], u.objective) <= OBJECTIVE_RTOL
        compare_centroids(g, o)

    def iterate():
        g.assign(), o.assign(), ou.assign()
        best, second, _ = ou.scores()
        compare_labels(g.labels(), ou.labels(), best, second)
        push(ou.labels())
        return ou.labels()

    try:
        for _ in range(2):
            prev, last = last, iterate()
        assert (last != prev).any()
        other = last.copy()
        other[::5] = (other[::5] + 1) % w.k  # a fifth of the objects elsewhere
        for step in {"previous": [(prev,)], "there_and_back": [(other,), (last,), (prev,)], "same": [(last,)],
                     "twice_before_the_update": [(other, prev), (last, other, last)]}[seq]:
            push(*step)
        for _ in range(3):
            iterate()
    finally:
        g.close()
