"""k around the largest score vector that a CTA's shared memory holds beside its
staging and static arrays: the automatic score buffer turns to global memory
before the launch would fail, at every block size and for a kernel of one
configuration, and the labels are the global buffer's."""
from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_harness import gpu_instance

pytestmark = pytest.mark.gpu


def _corpus(n, D=512):
    """Two terms per document, pairs spread over the terms (most repeated often)."""
    from synth.corpus import Corpus
    i = np.arange(n, dtype=np.int64)
    a, b = i % D, (i * 7 + i // D * 13 + 1) % D
    b = np.where(a == b, (b + 1) % D, b)
    w = 0.3 + 0.4 * ((i * 31) % 97) / 97.0
    idx = np.stack([np.minimum(a, b), np.maximum(a, b)], 1).astype(np.int32)
    val = np.stack([np.sqrt(w), np.sqrt(1.0 - w)], 1).astype(np.float32)
    return Corpus(N=n, D=D, row_ptr=np.arange(n + 1, dtype=np.int64) * 2, idx=idx.reshape(-1), val=val.reshape(-1))


def _optin():
    import torch
    return getattr(torch.cuda.get_device_properties(0), "shared_memory_per_block_optin", 227 << 10)


@pytest.mark.parametrize("threads", [0, 64])
@pytest.mark.parametrize("below", [-64, 0, 24, 72, 520, 640, 1200])  # bytes left by staging and scores
def test_either_side_of_the_limit(threads, below):
    k = (_optin() - 24 * (threads or 512) - below) // 4 // 8 * 8
    c = _corpus(k + 40)
    ini = np.arange(k)
    out = []
    for buf in ("auto", "global"):
        g = gpu_instance(c, k, ini, score_buffer=buf, threads=threads, update_mode="sort")
        try:
            g.assign()
            out.append(g.labels())
            st = g.stats()
            if buf == "auto":
                assert st["assign_global"] == int(below < st["assign_threads"] + 128)
        finally:
            g.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("below", [0, 100, 190, 256, 400])
def test_ivf_cbicp_is_refused_at_init_or_runs(below):
    """k (33/8 bytes each) whose scores and bits leave `below` bytes or little more."""
    from paper_2103_16141_gb300 import SivfError, sivf as S
    k = (_optin() - 24 * 128 - below) * 8 // 33 // 32 * 32
    c = _corpus(k + 8)
    try:
        g = gpu_instance(c, k, np.arange(k), icp="cbicp", update_mode="sort")
    except SivfError as ex:
        assert ex.status == S.SIVF_ERR_INVALID_ARG
        return
    try:
        g.assign()
    finally:
        g.close()
