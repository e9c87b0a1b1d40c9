"""The FP32 pair kernel at the edges of its pieces (GPU against the oracle):
i-blocks of 64 points and octs of eight around their sizes, the bin counts
where the fixed-point floors (at most 126 bins an axis, edges from zero) hand
over to the packed ones, cross counts either way round (the denser catalogue
gives the i-points), catalogues whose points coincide, and not-a-number
coordinates in a periodic box (no pair)."""

import numpy as np
import pytest

import synth

oracle = pytest.importorskip("oracle")
P = pytest.importorskip("paper_2301_12557_gb300")

pytestmark = pytest.mark.gpu
L = 100.0


def _points(n, seed, clump=0.3):
    rng = np.random.default_rng(seed)
    k = int(n * clump)
    x = rng.random((n, 3)) * L
    x[:k] = 40.0 + rng.normal(0.0, 2.0, (k, 3))      # one dense clump
    return np.ascontiguousarray(np.mod(x, L))


def _check(x, y=None, w=None, v=None, **kw):
    want, wantw = oracle.count(x, y, w1=w, w2=v, box=L, periodic=True, method="grid", **kw)
    for f in (P.count, P.count_tree):
        got, gotw = f(x, y, w1=w, w2=v, box=L, periodic=True, **kw)
        np.testing.assert_array_equal(got, want, err_msg=f.__name__)
        if w is not None:
            np.testing.assert_allclose(gotw, wantw, rtol=1e-10, atol=0.0, err_msg=f.__name__)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 63, 64, 65, 127, 129, 257, 1000, 4099])
def test_block_and_oct_sizes(n):
    x = _points(n, n)
    w = synth.lognormal_weights(n, 0.3, n + 1)
    _check(x, w=w, mode="s", edges_a=np.linspace(0.0, 30.0, 16))
    _check(x, mode="smu", edges_a=np.linspace(0.0, 30.0, 16), edges_b=np.linspace(0.0, 1.0, 11))


@pytest.mark.parametrize("na,nb", [(1, 1), (125, 3), (126, 126), (127, 5), (128, 4), (3, 127), (200, 120)])
@pytest.mark.parametrize("mode", ["s", "smu", "sigpi"])
@pytest.mark.parametrize("weights", [None, "f32", "f64"])
def test_bin_counts_around_the_fixed_point_limit(mode, na, nb, weights):
    x = _points(3000, 11)
    ea = np.linspace(0.0, 25.0, na + 1)
    eb = {"s": None, "smu": np.linspace(0.0, 1.0, nb + 1), "sigpi": np.linspace(0.0, 20.0, nb + 1)}[mode]
    w = None
    if weights == "f32":
        w = synth.lognormal_weights(x.shape[0], 0.3, 12)
    elif weights == "f64":
        w = 0.3 + 0.7 * np.random.default_rng(13).random(x.shape[0])
    _check(x, w=w, mode=mode, edges_a=ea, edges_b=eb)


@pytest.mark.parametrize("na", [1, 7, 125, 126])
@pytest.mark.parametrize("e0,spacing", [(3.0, "even"), (24.0, "even"), (0.004, "log"), (0.5, "log"), (20.0, "log")])
@pytest.mark.parametrize("mode,los", [("s", "z"), ("smu", "z"), ("sigpi", "z"), ("smu", "mid"), ("sigpi", "mid")])
def test_first_edges_above_zero(mode, los, e0, spacing, na):
    """Offset and logarithmic first axes (also sigma), about their limit of 125
    bins, from one bin over orders of magnitude to narrow ones far out."""
    rng = np.random.default_rng(na + 41)
    ea = np.linspace(e0, 25.0, na + 1) if spacing == "even" else np.geomspace(e0, 25.0, na + 1)
    eb = {"s": None, "smu": np.linspace(0.0, 1.0, 13), "sigpi": np.linspace(0.0, 20.0, 21)}[mode]
    x = _points(2500, 42)
    box = dict(box=L, periodic=True)
    if los == "mid":
        x, box = x + 400.0, {}
    w = 0.3 + 0.7 * rng.random(x.shape[0])
    want, wantw = oracle.count(x, w1=w, mode=mode, los=los, edges_a=ea, edges_b=eb, method="brute", **box)
    for f in (P.count, P.count_tree):
        for v in (None, w, w.astype(np.float32)):
            got, gotw = f(x, w1=v, mode=mode, los=los, edges_a=ea, edges_b=eb, **box)
            np.testing.assert_array_equal(got, want, err_msg=f.__name__)
            if v is w:
                np.testing.assert_allclose(gotw, wantw, rtol=1e-10, atol=0.0, err_msg=f.__name__)


@pytest.mark.parametrize("wtype", ["f32", "f64"])
@pytest.mark.parametrize("mode", ["s", "smu"])
def test_weight_records_that_fill(mode, wtype):
    """All pairs in one or a few bins, weights just below the scale's top: the
    integer weight records are flushed long before a piece or count overflows."""
    n = 5003
    rng = np.random.default_rng(51)
    x = 50.0 + rng.normal(0.0, 0.2, (n, 3))
    w = 1.0 - 1e-6 * rng.random(n)
    if wtype == "f32":
        w = w.astype(np.float32)
    kw = dict(mode=mode, edges_a=np.linspace(0.0, 25.0, 6))
    if mode == "smu":
        kw["edges_b"] = np.linspace(0.0, 1.0, 3)
    want, wantw = oracle.count(x, w1=w.astype(np.float64), box=L, periodic=True, method="grid", **kw)
    for f in (P.count, P.count_tree):
        got, gotw = f(x, w1=w, box=L, periodic=True, **kw)
        np.testing.assert_array_equal(got, want, err_msg=f.__name__)
        np.testing.assert_allclose(gotw, wantw, rtol=1e-10, atol=0.0, err_msg=f.__name__)


@pytest.mark.parametrize("n1,n2", [(40, 5000), (5000, 40), (1, 300), (300, 1)])
def test_cross_counts_either_way_round(n1, n2):
    x, y = _points(n1, 21), _points(n2, 22)
    w = 0.3 + 0.7 * np.random.default_rng(23).random(n1)
    v = 0.3 + 0.7 * np.random.default_rng(24).random(n2)
    _check(x, y, w, v, mode="smu", edges_a=np.linspace(0.0, 25.0, 11), edges_b=np.linspace(0.0, 1.0, 9))
    _check(x, y, w, v, mode="sigpi", edges_a=np.linspace(0.0, 20.0, 41), edges_b=np.linspace(0.0, 20.0, 41))


def test_shell_smu_midpoint():
    """(s, mu) floors along the midpoint line of sight, auto and cross."""
    d = synth.survey_shell(3000, True, 31)
    r = synth.survey_shell(9000, False, 32)
    wd, wr = synth.fkp_weights(d, 3000), synth.fkp_weights(r, 3000)
    kw = dict(mode="smu", los="mid", edges_a=np.linspace(0.0, 200.0, 41), edges_b=np.linspace(0.0, 1.0, 101))
    for y, v in ((None, None), (r, wr)):
        want, wantw = oracle.count(d, y, w1=wd, w2=v, method="brute", **kw)
        for f in (P.count, P.count_tree):
            got, gotw = f(d, y, w1=wd, w2=v, **kw)
            np.testing.assert_array_equal(got, want)
            np.testing.assert_allclose(gotw, wantw, rtol=1e-10, atol=0.0)


@pytest.mark.parametrize("mode,na,nb", [("s", 20, 1), ("smu", 20, 10), ("sigpi", 20, 10), ("smu", 130, 10)])
def test_coincident_points_and_not_a_number(mode, na, nb):
    rng = np.random.default_rng(41)
    x = np.repeat(_points(150, 42), 3, axis=0)        # every point three times: s = 0 pairs
    eb = {"s": None, "smu": np.linspace(0.0, 1.0, nb + 1), "sigpi": np.linspace(0.0, 20.0, nb + 1)}[mode]
    ea = np.linspace(0.0, 20.0, na + 1)
    _check(x, mode=mode, edges_a=ea, edges_b=eb)
    bad = x.copy()
    rows = rng.choice(x.shape[0], 20, replace=False)
    bad[rows, rng.integers(0, 3, 20)] = np.nan
    keep = np.delete(x, rows, axis=0)
    want, _ = oracle.count(keep, box=L, periodic=True, method="grid", mode=mode, edges_a=ea, edges_b=eb)
    got, _ = P.count(bad, box=L, periodic=True, mode=mode, edges_a=ea, edges_b=eb)
    np.testing.assert_array_equal(got, want)
