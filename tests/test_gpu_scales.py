"""Binary64 counts in any unit of length: a catalogue, its box and its edges
scaled by powers of two against the oracle's binary64 definition, also where the
binary32 box tests overflow or underflow (and, along the midpoint line of sight,
where the definition's own fourth powers do)."""

import numpy as np
import pytest

oracle = pytest.importorskip("oracle")
P = pytest.importorskip("paper_2301_12557_gb300")

pytestmark = pytest.mark.gpu
SCALES = [-300, -140, -100, -76, -73, -70, -60, 58, 60, 62, 64, 66, 100, 127, 140, 300]


@pytest.mark.parametrize("mode,los", [("s", "z"), ("smu", "z"), ("sigpi", "z"), ("smu", "mid"), ("sigpi", "mid")])
def test_counts_in_any_unit(mode, los):
    rng = np.random.default_rng(3)
    L = 100.0
    x, y = rng.random((3001, 3)) * L, rng.random((700, 3)) * L
    w, v = 0.5 + rng.random(3001), 0.5 + rng.random(700)
    if los == "mid":
        x[:, 0] += 3.0 * L
        y[:, 0] += 3.0 * L

    for other in (False, True):
        for e in SCALES:
            f = 2.0 ** e
            eb = {"s": None, "smu": np.linspace(0.0, 1.0, 11), "sigpi": np.linspace(0.0, 20.0, 11) * f}[mode]
            kw = dict(w1=w, w2=v if other else None, mode=mode, los=los, edges_a=np.linspace(0.0, 30.0, 16) * f,
                      edges_b=eb)
            if los == "z":
                kw.update(box=L * f, periodic=True)
            y_f = y * f if other else None
            want, wantw = oracle.count(x * f, y_f, method="brute", **kw)
            got, gotw = P.count(x * f, y_f, prec="f64", **kw)
            np.testing.assert_array_equal(got, want, err_msg=f"2^{e}")
            np.testing.assert_allclose(gotw, wantw, rtol=1e-12, err_msg=f"2^{e}")
