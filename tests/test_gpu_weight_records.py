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


def _unit_product(w, wtype):
    """A pair's integer product of two weights w in [0.5, 1), in units of 2^-48."""
    a = int(w * 2.0 ** 32)                                 # the packed 32 bits
    if wtype == "f32":
        return (a * a) >> 16
    b = int((w * 2.0 ** 32 - a) * 2.0 ** 31)               # and the next 31
    t = ((((a >> 1) * b) >> 32) + ((((a & 1) << 30 | b >> 1) * a) >> 32) + 0x2000) * 2
    return (t + (a >> 1) * a) >> 15


@pytest.mark.parametrize("wtype", ["f32", "f64"])
@pytest.mark.parametrize("mode", ["s", "sigpi"])
def test_sums_are_exact_but_for_one_conversion_a_cta(mode, wtype):
    """5.0e9 pairs of equal weights in one bin: every product is the same integer,
    so their exact sum is known.  A CTA's part is exact until it is converted (two
    roundings) and added (one): at most three halves of 2^-52 of the sum a CTA."""
    torch = pytest.importorskip("torch")
    n, w = 100003, float(np.float32(0.7853981))
    if wtype == "f64":
        w += 1.23e-10
    x = 50.0 + np.random.default_rng(1).uniform(-0.25, 0.25, (n, 3))
    weights = np.full(n, w, np.float32 if wtype == "f32" else np.float64)
    eb = np.linspace(0.0, 30.0, 41) if mode == "sigpi" else None
    bins = P.Bins(mode, "z", np.linspace(0.0, 30.0, 31 if mode == "s" else 41), eb)
    g = P.pc_build_grid(x, weights, box=P.make_box(L, True), r_max=bins.r_max)
    got, gotw, st = P.pc_count_auto(g, bins, opts=P.make_opts(grid_ctas_per_sm=1), weighted=True)
    assert st.wsum == (2 if wtype == "f32" else 3)
    assert got[0] == n * (n - 1) // 2
    want = int(got[0]) * _unit_product(w, wtype) / 2 ** 48
    ctas = torch.cuda.get_device_properties(0).multi_processor_count
    assert abs(gotw[0] - want) <= 3 * ctas * 2.0 ** -53 * want


@pytest.mark.parametrize("capacity", [0, 1 << 20])
@pytest.mark.parametrize("wtype", ["f32", "f64"])
@pytest.mark.parametrize("mode", ["s", "smu", "sigpi"])
def test_pairs_taken_out_of_a_bin_leave_nothing(mode, wtype, capacity):
    """90,000 pairs 1e-9 (relative) below an edge are counted past it in binary32
    and put right: a bin without pairs has a weighted sum of exactly zero."""
    rng = np.random.default_rng(2)
    n = 300
    a = np.array([20.0, 30.0, 40.0]) + 1e-10 * rng.random((n, 3))
    d = {"s": [3.0, 0.0, 4.0], "smu": [3.0, 0.0, 4.0], "sigpi": [3.0, 4.0, 2.0]}[mode]   # s or sigma = 5
    x = np.concatenate([a, a + np.array(d) * (1.0 - 1e-9)])
    w = 0.5 + 0.5 * rng.random(2 * n)
    v = w.astype(np.float32) if wtype == "f32" else w
    eb = {"s": None, "smu": np.linspace(0.0, 1.0, 101), "sigpi": np.linspace(0.0, 30.0, 41)}[mode]
    bins = P.Bins(mode, "z", np.linspace(0.0, 25.0, 6), eb)
    g = P.pc_build_grid(x, v, box=P.make_box(L, True), r_max=bins.r_max)
    got, gotw, st = P.pc_count_auto(g, bins, opts=P.make_opts(rescue_capacity=capacity), weighted=True)
    assert st.wsum == (2 if wtype == "f32" else 3) and st.rescued >= n * n
    row = got.reshape(5, -1).sum(1)
    assert row[1] == 0 and got.sum() == n * (2 * n - 1)
    assert not np.any(gotw[got == 0])
    y = v.astype(np.longdouble)
    want = float((y.sum() ** 2 - (y * y).sum()) / 2)
    assert abs(gotw.sum() - want) <= 2.0 ** -34 * want


@pytest.mark.parametrize("wtype", ["f32", "f64"])
@pytest.mark.parametrize("mode", ["s", "sigpi", "smu"])
@pytest.mark.parametrize("form", ["grid", "tree"])
def test_no_product_is_lost_while_others_fill(form, mode, wtype):
    """1.8e9 pairs of equal weights in a clump, bins from crowded ones, for which the
    records are flushed all the time, to rare ones: every bin's sum is its count
    times one product, to the conversions of the CTAs (three halves of 2^-52 each) and
    to a unit of 2^-48 for each pair that its binary64 check moved."""
    torch = pytest.importorskip("torch")
    n, w = 60001, float(np.float32(0.7853981))
    if wtype == "f64":
        w += 1.23e-10
    x = 50.0 + np.random.default_rng(4).normal(0.0, 0.5, (n, 3))
    weights = np.full(n, w, np.float32 if wtype == "f32" else np.float64)
    eb = {"s": None, "sigpi": np.linspace(0.0, 30.0, 41), "smu": np.linspace(0.0, 1.0, 101)}[mode]
    bins = P.Bins(mode, "z", np.linspace(0.0, 30.0, 41), eb)
    box, v = P.make_box(L, True), _unit_product(w, wtype)
    if form == "grid":
        g = P.pc_build_grid(x, weights, box=box, r_max=bins.r_max)
        got, gotw, st = P.pc_count_auto(g, bins, weighted=True)
    else:
        t = P.pc_build_tree(x, weights, box=box)
        got, gotw, st = P.pc_count_tree(t, None, bins, weighted=True)
    assert st.wsum == (2 if wtype == "f32" else 3) and got.sum() == n * (n - 1) // 2
    want = np.array([int(c) * v / 2 ** 48 for c in got])
    ctas = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    np.testing.assert_array_less(np.abs(gotw - want), want * (3 * ctas * 2.0 ** -53) + got * 2.0 ** -48 + 1e-300)
