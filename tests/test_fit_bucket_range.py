"""The numbers of the fit's buckets (Buckets::rank_of of csrc/kmq_fit.cu), restated in numpy: they never decrease with the value, a
bucket lies inside one octave unless it is at zero or the last, and rows with outliers or with many values next to zero stay within
the numbers of members that keep a row off the sorting path."""
import os
import re

import numpy as np
import pytest

from paper_2602_15563_b200 import build as kb

SOURCE = open(os.path.join(kb.CSRC, "kmq_fit.cu")).read()


def constant(name):
    return int(re.search(rf"constexpr int {name} = (\d+);", SOURCE).group(1))


def mantissa(K):
    return max(10, int(np.ceil(np.log2(K)))) - 5


def ranks(magnitude, ec, m):
    """Bucket numbers inside a sign; c = 2^(ec - 127)."""
    c = np.array(ec << 23, dtype=np.uint32).view(np.float32).astype(np.float64)
    exact = magnitude.astype(np.float64) + c
    with np.errstate(over="ignore"):
        f = exact.astype(np.float32)
    f = np.where(f.astype(np.float64) > exact, np.nextafter(f, np.float32(0)), f)         # rounded towards zero
    t = (f.view(np.uint32) >> (23 - m)).astype(np.int64) - (ec << m)
    u = (magnitude.view(np.uint32) >> (26 - m)).astype(np.int64) + (9 << (m - 2)) - ((ec + 2) << (m - 3))
    return np.maximum(np.minimum(np.minimum(t, u), (3 << m) - 1), 0)


def test_the_source_is_what_is_restated():
    for line in ("t = (int)(__float_as_uint(__fadd_rz(magnitude, c)) >> shift) - base;",
                 "u = (int)(__float_as_uint(magnitude) >> (shift + 3)) + far;", "return __vimin3_s32_relu(t, u, half - 1);",
                 "bk.shift = 23 - m;", "bk.base = ec << m;", "bk.half = 3 << m;", "bk.fine = 9 << (m - 2);",
                 "bk.far = bk.fine - ((ec + 2) << (m - 3));"):
        assert line in SOURCE
    assert constant("kAboveTypical") == 2


@pytest.mark.parametrize("ec", (32, 120, 248))
@pytest.mark.parametrize("m", (5, 6, 7, 8, 9, 10))
def test_order_and_octaves(m, ec):
    rng = np.random.default_rng(m + ec)
    c = float(np.array(ec << 23, dtype=np.uint32).view(np.float32))
    top = min(2.0 ** 10 * c, float(np.finfo(np.float32).max))
    v = np.concatenate([[0.0, 1e-45], c * 2.0 ** rng.uniform(-24, 2, 40000), rng.uniform(0, 8 * c, 40000),
                        2.0 ** rng.uniform(np.log2(c), np.log2(top), 40000), c * np.arange(1, 16 << m) / (1 << m)])
    v = np.minimum(v, top).astype(np.float32)
    v = np.unique(np.concatenate([v, np.nextafter(v, np.float32(0)), np.nextafter(v, np.float32(top))]))
    r = ranks(v, ec, m)
    assert np.all(np.diff(r) >= 0) and r[0] == 0
    octave = v.view(np.uint32) >> 23
    for b in np.unique(r):
        if 0 < b < (3 << m) - 1:
            assert np.unique(octave[r == b]).size == 1
    if top > 300 * c:
        assert r[np.searchsorted(v, np.float32(255.9 * c)) - 1] == (3 << m) - 1
        assert r[np.searchsorted(v, np.float32(223 * c))] < (3 << m) - 1
    # what u adds changes no number below 4 c
    low = v[v < 4 * c]
    t = ranks(low, ec, m)
    plain = np.floor((low.astype(np.float64) + c) / c * (1 << m)).astype(np.int64) - (1 << m)
    assert np.array_equal(t[low < c], plain[low < c])


ROWS = {
    "a tenth at 8 sigma": lambda g, s: g.standard_normal(s) * np.where(g.random(s) < 0.1, 8, 1),
    "a fifth at 20 sigma": lambda g, s: g.standard_normal(s) * np.where(g.random(s) < 0.2, 20, 1),
    "1 in 50 at 100 sigma": lambda g, s: g.standard_normal(s) * np.where(g.random(s) < 0.02, 100, 1),
    "Cauchy": lambda g, s: g.standard_cauchy(s),
    "Student, 2 degrees": lambda g, s: g.standard_t(2, s),
    "products of normals": lambda g, s: g.standard_normal(s) * g.standard_normal(s),
    "three of ten a hundredth": lambda g, s: g.standard_normal(s) * np.where(g.random(s) < 0.3, 0.01, 1),
}


@pytest.mark.parametrize("kind", sorted(ROWS))
@pytest.mark.parametrize("K", (1024, 4096, 8192, 28672, 32768))
def test_rows_that_stay_off_the_sorting_path(K, kind):
    W = (ROWS[kind](np.random.default_rng(K), (8, K)) * 0.02).astype(np.float32)
    m = mantissa(K)
    for row in W:
        e = (row[:min(K, (1 << (m + 5)) // 8)].view(np.uint32) >> 23) & 255
        e = e[e > 0].astype(np.int64)
        r = ranks(np.abs(row), int(np.clip(e.sum() // e.size + 2, 32, 248)), m)
        for sign in (row < 0, row >= 0):
            n = np.bincount(r[sign], minlength=3 << m)
            assert max(n[0], n[-1]) <= constant("kMaxMixed") and n[1:-1].max() <= constant("kMaxMembers")
