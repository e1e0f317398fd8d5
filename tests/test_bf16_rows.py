"""The BF16 dense rows' odd entries, in a model of their arithmetic (CPU).

A 32-bit word of a row holds the even entry's BF16 bits below and the odd
entry's above, and the scan reads the whole word as FP32 for the odd entry.
The build chooses the upper half so that this is within 2^-8 of the value
(the error bound's eps of BF16, as for rounding to nearest), whatever the
lower half is; a word without an odd entry is subnormal.
"""
from __future__ import annotations

import numpy as np
import pytest


def upper_half(u: np.ndarray, low: np.ndarray) -> np.ndarray:
    bits = np.maximum(u.view(np.uint32), np.uint32(0x00800000)).astype(np.uint64)
    return ((bits - low + 0x8000) & 0xFFFFFFFF) >> 16


def as_read(high: np.ndarray, low: np.ndarray) -> np.ndarray:
    return ((high << 16) | low).astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e-12, 1e-36])
def test_error_of_the_word_as_fp32(scale):
    rng = np.random.default_rng(3)
    u = (rng.random(400_000) * scale).astype(np.float32)
    u[:4] = [1.0, np.float32(scale), np.nextafter(np.float32(1), np.float32(0)), np.float32(2) ** -20]
    u = u[u >= np.float32(2) ** -126]
    low = rng.integers(0, 65536, len(u)).astype(np.uint64)
    low[:100] = 0
    low[100:200] = 65535
    word = as_read(upper_half(u, low), low).astype(np.float64)
    ref = u.astype(np.float64)
    # a value next to the smallest normal may be read as a subnormal, which counts as 0
    err = np.abs(np.where(word < 2.0**-126, 0.0, word) - ref)
    assert np.all(err <= 2.0**-8 * ref + np.where(ref < 2.0**-125, 2.0**-125, 0.0))


def test_words_without_an_odd_entry_are_subnormal():
    low = np.arange(65536, dtype=np.uint64)
    assert np.all(as_read(np.zeros_like(low), low) < np.float32(2) ** -126)
