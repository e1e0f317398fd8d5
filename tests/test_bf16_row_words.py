"""The library's own encoding of the BF16 dense rows' words, compiled from its
source for the host, and the scan that reads them on a GPU."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_16141_gb300", "csrc")


@pytest.fixture(scope="module")
def odd_upper_half(tmp_path_factory):
    d = tmp_path_factory.mktemp("bf16")
    src, so = d / "w.cpp", d / "w.so"
    src.write_text('#include "bf16_rows.cuh"\n'
                   'extern "C" void run(long n, const uint32_t *u, const uint16_t *low, uint16_t *out) {\n'
                   "    for (long i = 0; i < n; ++i) out[i] = sivf::odd_upper_half(u[i], low[i]);\n}\n")
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)])
    lib = ctypes.CDLL(str(so))

    def call(u, low):
        u, low = np.ascontiguousarray(u, np.float32), np.ascontiguousarray(low, np.uint16)
        out = np.empty(len(u), np.uint16)
        lib.run(ctypes.c_long(len(u)), u.ctypes.data_as(ctypes.c_void_p), low.ctypes.data_as(ctypes.c_void_p),
                out.ctypes.data_as(ctypes.c_void_p))
        return out
    return call


def bf16_bits(u):
    """BF16, to nearest even, of positive FP32 values."""
    b = np.ascontiguousarray(u, np.float32).view(np.uint32).astype(np.uint64)
    return ((b + 0x7FFF + ((b >> 16) & 1)) >> 16).astype(np.uint16)


def word(high, low):
    return ((high.astype(np.uint32) << 16) | low.astype(np.uint32)).view(np.float32)


@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e-12, 1e-36])
def test_word_is_the_nearest_with_its_lower_half(odd_upper_half, scale):
    rng = np.random.default_rng(5)
    u = np.concatenate([(rng.random(100_000) * scale).astype(np.float32), np.float32(2) ** -np.arange(0, 120, 7)])
    u = u[u >= np.float32(2) ** -120].astype(np.float32)
    low = rng.integers(0, 65536, len(u)).astype(np.uint16)
    low[::5], low[1::5] = 0, 65535
    high = odd_upper_half(u, low)
    w = word(high, low)
    # words with this lower half lie 2^16 apart in the order of FP32 bits
    assert np.all(np.abs(w.view(np.uint32).astype(np.int64) - u.view(np.uint32).astype(np.int64)) <= 1 << 15)
    assert np.all(np.abs(w.astype(np.float64) - u) <= 2.0**-8 * u)


def test_smallest_values(odd_upper_half):
    """Values at and below the smallest normal: what is read (subnormals count as
    0) is within 2^-125."""
    u = np.array([1, 1 << 22, (1 << 23) - 1, 1 << 23, (1 << 23) + 1], np.uint32).view(np.float32)
    for l in (0, 1, 0x7FFF, 0x8000, 65535):
        low = np.full(len(u), l, np.uint16)
        w = word(odd_upper_half(u, low), low).astype(np.float64)
        assert np.all(np.abs(np.where(w < 2.0**-126, 0.0, w) - u) <= 2.0**-125)


def one_term_rows(parity, k=64, T=1_000):
    """Centroid values (k, T), 0 where a centroid lacks the term: the two largest
    of a term at even or odd positions, their gap around twice the bound, and the
    odd ones' bits on the edge of rounding up beside the lower half that their
    word has (that of an even neighbour, or 0 where that lacks the term)."""
    rng = np.random.default_rng(7 + parity)
    u = (rng.random((k, T)) * 0.004 + 0.004).astype(np.float32)
    u[0::2][rng.random((k // 2, T)) < 0.25] = 0.0
    for t in range(T):
        a, b = rng.choice(np.arange(parity, k, 2), 2, replace=False)
        top = 0.02 + 0.015 * rng.random()
        for j, v in ((a, top), (b, top * (1 - 2.0**-7 * (0.5 + rng.random())))):
            u[j, t] = v
            if parity:
                low = int(bf16_bits(u[j - 1, t:t + 1])[0])
                bits = (int(u[j, t:t + 1].view(np.uint32)[0]) & 0xFFFF0000) + ((low + 0x8000 - int(rng.integers(2))) & 0xFFFF)
                u[j, t] = np.array([bits], np.uint32).view(np.float32)[0]
    return u


def expected_rescore(u, odd_upper_half):
    """Which one-term documents are re-scored, and how many candidates in all,
    from the words' values: a score is the value's fixed-point ceil, the bound
    that of one term in one dense row, without an absolute error of the value."""
    k, T = u.shape
    low = bf16_bits(u[0::2].reshape(-1))
    stored = np.empty((k, T))
    stored[0::2] = (low.astype(np.uint32) << 16).view(np.float32).reshape(k // 2, T)
    stored[1::2] = word(odd_upper_half(u[1::2].reshape(-1), low), low).reshape(k // 2, T)
    eps, quantum, ur = 2.0**-8, 2.0**-31, 2.0**-24
    q = np.ceil(stored / quantum)
    best, second = np.sort(q, axis=0)[:-3:-1]
    c = eps + (1 + eps) * (ur / (1 - ur))
    E = (c * best * quantum + 2 * quantum) / (1 - c) * (1 + 1e-12)
    flagged = (best - second) * quantum <= 2 * E
    thr = best - np.ceil(2 * E / quantum)
    return flagged, int((q[:, flagged] >= thr[flagged]).sum())


def test_the_rows_are_sensitive(odd_upper_half):
    """A rounding constant off by one, no lower half, the wrong neighbour's: other counts."""
    u = one_term_rows(1)

    def planted(constant=0x8000, low_of=lambda low: low):
        def f(v, low):
            b = np.maximum(np.ascontiguousarray(v, np.float32).view(np.uint32), 0x00800000).astype(np.int64)
            return (((b - low_of(low).astype(np.int64) + constant) >> 16) & 0xFFFF).astype(np.uint16)
        return f

    def counts(f):
        flagged, cands = expected_rescore(u, f)
        return int(flagged.sum()), cands

    want = counts(odd_upper_half)
    assert counts(planted()) == want
    for f in (planted(0x8001), planted(0x7FFF), planted(0), planted(low_of=np.zeros_like),
              planted(low_of=lambda low: np.roll(low, -1))):
        assert counts(f) != want


@pytest.mark.gpu
@pytest.mark.parametrize("parity", [0, 1])
def test_scan_reads_the_words(odd_upper_half, parity):
    """Documents of one term over its dense row: a score is the stored value
    itself, so that the re-scored documents and candidates follow from the words."""
    from synth.corpus import Corpus
    from tests.gpu_harness import gpu_instance
    u = one_term_rows(parity)
    k, T = u.shape
    flagged, cands = expected_rescore(u, odd_upper_half)
    assert 100 < flagged.sum() < T - 100
    norm2 = (u.astype(np.float64) ** 2).sum(axis=1)
    assert norm2.max() < 0.5  # a seed's own score of 1 is clear of the others'
    idx, val = [], []
    for j in range(k):  # the seeds: their terms, and one of their own that makes them unit rows
        t = np.nonzero(u[j])[0]
        idx += [t, [T + j]]
        val += [u[j, t], [np.sqrt(1.0 - norm2[j])]]
    lens = [int((u[j] > 0).sum()) + 1 for j in range(k)] + [1] * T
    c = Corpus(N=k + T, D=T + k, row_ptr=np.concatenate([[0], np.cumsum(lens)]).astype(np.int64),
               idx=np.concatenate(idx + [np.arange(T)]).astype(np.int32),
               val=np.concatenate(val + [np.ones(T)]).astype(np.float32))
    g = gpu_instance(c, k, np.arange(k), precision="bf16")
    try:
        g.assign()
        st = g.stats()
        assert st["dense_terms"] == T
        assert (st["rescored"], st["rescore_cands"]) == (int(flagged.sum()), cands)
        assert np.array_equal(g.labels(), np.concatenate([np.arange(k), np.argmax(u, axis=0)]))
    finally:
        g.close()
