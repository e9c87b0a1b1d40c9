"""Counts of the default precision in any unit of length, against the oracle: a
catalogue, its box and its edges scaled by powers of two.  Where binary32 squares of
the separations would overflow the grid path counts in binary64, and the k-d tree
path, which has no binary64 kernel, refuses."""

import numpy as np
import pytest

oracle = pytest.importorskip("oracle")
P = pytest.importorskip("paper_2301_12557_gb300")

SCALES = [-300, -140, -76, -60, -40, -31, -22, -20, 0, 19, 21, 22, 30, 45, 56, 58, 60, 62, 66, 100, 300]
CASES = [("s", "z"), ("smu", "z"), ("sigpi", "z"), ("smu", "mid"), ("sigpi", "mid")]
L = 100.0


def _edges(mode, f):
    eb = {"s": None, "smu": np.linspace(0.0, 1.0, 11), "sigpi": np.linspace(0.0, 20.0, 11) * f}[mode]
    return np.linspace(0.0, 30.0, 16) * f, eb


def test_the_plan_knows_where_squares_overflow():
    for e in SCALES:
        f = 2.0 ** e
        k = P.pc_fp32_bands(P.Bins("s", "z", *_edges("s", f)), 30.0 * f, np.zeros(3), np.full(3, L * f),
                            np.full(3, L * f), True)
        assert k["fp32_ok"] == (30.0 * f < 1.7e19), e


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["count", "count_tree"])
@pytest.mark.parametrize("mode,los", CASES)
def test_counts_in_any_unit(mode, los, form):
    rng = np.random.default_rng(11)
    x = rng.random((3001, 3)) * L
    if los == "mid":
        x[:, 0] += 3.0 * L
    reach = 30.0 if mode != "sigpi" else np.hypot(30.0, 20.0)
    # the largest binary32 square: of the reach, along the midpoint of x_i + x_j
    top = reach if los == "z" else 4.0 * x.max() + reach
    for e in SCALES:
        f = 2.0 ** e
        ea, eb = _edges(mode, f)
        kw = dict(mode=mode, los=los, edges_a=ea, edges_b=eb)
        if los == "z":
            kw.update(box=L * f, periodic=True)
        if form == "count_tree" and not top * f < 1.7e19:
            with pytest.raises(P.PairCountError):
                P.count_tree(x * f, **kw)
            continue
        want, _ = oracle.count(x * f, None, method="brute", **kw)
        got, _ = getattr(P, form)(x * f, **kw)
        np.testing.assert_array_equal(got, want, err_msg=f"2^{e}")
