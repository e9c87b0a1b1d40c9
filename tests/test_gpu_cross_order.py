"""Cross counts of a sparse and a dense catalogue: whichever gives the i-points, and in
either order of the arguments, the counts are the oracle's; a catalogue of less than
two points a cell gives them (its runs of eight points are mostly other cells')."""

import numpy as np
import pytest

oracle = pytest.importorskip("oracle")
P = pytest.importorskip("paper_2301_12557_gb300")

pytestmark = pytest.mark.gpu
L, CELL, NCELL = 100.0, 10.0, 1000


@pytest.mark.parametrize("mode,los,weighted", [("s", "z", False), ("smu", "z", True), ("sigpi", "z", False),
                                               ("smu", "mid", True), ("sigpi", "mid", True)])
@pytest.mark.parametrize("n", [0, 1, 33, 2 * NCELL - 1, 2 * NCELL])
def test_either_order(n, mode, los, weighted):
    rng = np.random.default_rng(n + len(mode))
    few, many = rng.random((n, 3)) * L, rng.random((20_011, 3)) * L
    wf, wm = (0.5 + rng.random(n), 0.5 + rng.random(20_011)) if weighted else (None, None)
    lo, hi = np.zeros(3), np.full(3, L)
    if los == "mid":
        few, many, lo, hi = (a + np.array([300.0, 0.0, 0.0]) for a in (few, many, lo, hi))
    eb = {"s": None, "smu": np.linspace(0.0, 1.0, 11), "sigpi": np.linspace(0.0, 20.0, 11)}[mode]
    bins = P.Bins(mode, los, np.linspace(0.0, 25.0, 16), eb)
    box = P.make_box(L, periodic=True) if los == "z" else P.make_box(lo=lo, hi=hi)
    want, wantw = oracle.count(few, many, w1=wf, w2=wm, mode=mode, los=los, edges_a=bins.ea, method="brute",
                               edges_b=eb, **(dict(box=L, periodic=True) if los == "z" else {}))
    grids = [P.pc_build_grid(x, w, box=box, r_max=bins.r_max, opts=P.make_opts(cell_size=CELL))
             for x, w in ((few, wf), (many, wm))]
    for a, b in (grids, grids[::-1]):
        got, gotw, st = P.pc_count_cross(a, b, bins, weighted=weighted)
        np.testing.assert_array_equal(got, want)
        if weighted:
            np.testing.assert_allclose(gotw, wantw, rtol=1e-10)
        if los == "z":   # (a box without periods may have more cells)
            assert st.blocks <= n if n < 2 * NCELL else st.blocks == NCELL   # 20 points a cell
    for g in grids:
        P.pc_free_grid(g)
