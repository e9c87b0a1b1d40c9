"""Weighted counts whose pairs all fall into one bin of a large histogram: the
integer weight records of few lane copies fill and are flushed all the time by
single warps while the others add.  Weights just below the top of their scale;
the sums are known in closed form."""

import math

import numpy as np
import pytest

P = pytest.importorskip("paper_2301_12557_gb300")

pytestmark = pytest.mark.gpu
L = 100.0


def _clump(n, mode, rng):
    """Points whose pairs all lie in one bin of 40 x 40 (sigma, pi) or 40 x 100
    (s, mu) bins of width 0.75: a small clump, or a line of mu = 0.995."""
    if mode == "sigpi":
        return 50.0 + rng.uniform(-0.25, 0.25, (n, 3))
    t = rng.uniform(0.0, 0.7, n)
    d = np.array([math.sqrt(1.0 - 0.995 ** 2), 0.0, 0.995])
    return 50.0 + t[:, None] * d


@pytest.mark.parametrize("wtype", ["f32", "f64"])
@pytest.mark.parametrize("mode,nb", [("sigpi", 40), ("smu", 100)])
@pytest.mark.parametrize("form", ["count", "count_tree"])
def test_all_pairs_in_one_bin(form, mode, nb, wtype):
    rng = np.random.default_rng(7)
    n = 20011
    x = _clump(n, mode, rng)
    w = 0.9999 + 0.0001 * rng.random(n)
    if wtype == "f32":
        w = w.astype(np.float32)
    v = w.astype(np.longdouble)
    eb = np.linspace(0.0, 30.0 if mode == "sigpi" else 1.0, nb + 1)
    got, gotw = getattr(P, form)(x, w1=w, box=L, periodic=True, mode=mode, edges_a=np.linspace(0.0, 30.0, 41),
                                 edges_b=eb)
    b = int(np.argmax(got))
    assert b == (0 if mode == "sigpi" else nb - 1)
    assert got[b] == n * (n - 1) // 2 and got.sum() == got[b]
    want = float((v.sum() ** 2 - (v * v).sum()) / 2)
    # products truncated below 2^-34 of their value each
    assert abs(gotw[b] - want) <= 2.0 ** -34 * want
    assert np.count_nonzero(gotw) == 1
