"""The assignment kernels at the edges of their tiles, against the oracle.

A CTA covers 8 x threads score positions per pass of the dense rows, four at a
time, and finds the winner with 16-byte reads of the scores: numbers of
clusters around those widths, with every posting precision, thread count and
score buffer, on rows that include empty ones. Labels are exact (near ties
below an FP64 margin of 1e-6 excepted), counts equal the oracle's.
"""
from __future__ import annotations

import numpy as np
import pytest

from synth import CONFIGS, Corpus, generate, init_ids
from tests.gpu_harness import lockstep

pytestmark = pytest.mark.gpu


def _corpus_with_empty_rows(N, D, seed):
    """A generated corpus with every 97th row emptied."""
    w = CONFIGS["c2"].scaled(N=N, D=D)
    c = generate(w.N, w.D, w.zipf_s, 3.6, 0.7, 5, 400, seed)
    lens = np.diff(c.row_ptr)
    row = np.repeat(np.arange(N), lens)
    keep = row % 97 != 5
    lens[np.arange(N) % 97 == 5] = 0
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    return Corpus(N=N, D=D, row_ptr=rp, idx=np.ascontiguousarray(c.idx[keep]), val=np.ascontiguousarray(c.val[keep]))


def _seeds(c, k, seed):
    """k distinct non-empty documents."""
    full = np.nonzero(np.diff(c.row_ptr) > 0)[0]
    return np.ascontiguousarray(full[init_ids(len(full), k, seed)].astype(np.int32))


@pytest.mark.parametrize("k,threads,precision,buf", [
    (1, 32, "fp32", "shared"), (3, 64, "bf16", "shared"), (4, 32, "fp16", "global"), (5, 512, "fp32", "shared"),
    (8, 64, "fp32", "global"), (9, 32, "bf16", "shared"), (129, 32, "fp32", "shared"), (255, 32, "bf16", "global"),
    (256, 32, "fp32", "shared"), (257, 32, "fp32", "shared"), (258, 32, "fp16", "shared"),
    (511, 64, "fp32", "shared"), (513, 64, "bf16", "shared"), (515, 128, "fp32", "global"),
])
def test_cluster_counts_around_the_tiles(k, threads, precision, buf):
    c = _corpus_with_empty_rows(1_300, 2_500, 900 + k)
    recs = lockstep(c, k, _seeds(c, k, 17), 5, precision=precision, threads=threads, score_buffer=buf,
                    dense_min_fraction=0.05)
    assert any(r["stats"]["dense_entries"] > 0 for r in recs) or k < 32


@pytest.mark.parametrize("icp", [False, "cbicp", "relaxed"])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_other_modes_with_empty_rows(icp, precision):
    c = _corpus_with_empty_rows(1_300, 2_500, 31)
    lockstep(c, 130, _seeds(c, 130, 5), 8, precision=precision, icp=icp, dense_min_fraction=0.05)


def test_contexts_of_different_k_take_turns():
    """Two live contexts whose score vectors differ in size, stepped in turn."""
    from tests.gpu_harness import gpu_instance
    c = _corpus_with_empty_rows(1_300, 2_500, 77)
    runs = {}
    for turns in (False, True):
        a, b = (gpu_instance(c, k, _seeds(c, k, 5), threads=64) for k in (900, 33))
        try:
            for _ in range(3):
                a.assign(), a.update()
                if turns:
                    b.assign(), b.update()
            if not turns:
                for _ in range(3):
                    b.assign(), b.update()
            runs[turns] = (a.labels(), b.labels())
        finally:
            a.close()
            b.close()
    assert all(np.array_equal(x, y) for x, y in zip(runs[False], runs[True]))


@pytest.mark.parametrize("threads", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("buf", ["shared", "global"])
def test_every_kernel_form(threads, precision, buf):
    """All block sizes, precisions and score buffers, with and without dense
    rows, over numbers of clusters that leave warps without tiles or rows."""
    for k, frac in ((3, 1.0), (40, 0.05), (300, 1.0), (300, 0.05)):
        c = _corpus_with_empty_rows(700, 1_500, 40 + k)
        lockstep(c, k, _seeds(c, k, 9), 3, precision=precision, threads=threads, score_buffer=buf,
                 dense_min_fraction=frac)
