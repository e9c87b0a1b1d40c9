"""Default grids of periodic boxes: catalogues of different sizes for which the
cost model gives one cell side are laid on one grid, so that cross counts and
batches take them without a given side."""

import numpy as np
import pytest

oracle = pytest.importorskip("oracle")
P = pytest.importorskip("paper_2301_12557_gb300")

pytestmark = pytest.mark.gpu
L = 100.0


def _classes(r_max, lo, hi):
    """{model side: sizes with that side} over sizes lo .. hi."""
    out = {}
    for n in np.unique(np.geomspace(lo, hi, 60).astype(int)):
        out.setdefault(P.pc_suggest_cell_size(int(n), L ** 3, r_max), []).append(int(n))
    return out


@pytest.mark.parametrize("r_max", [8.0, 20.0, 45.0])
def test_one_default_grid_per_model_side(r_max):
    box, rng = P.make_box(L, True), np.random.default_rng(5)
    bins = P.Bins("s", "z", np.linspace(0.0, r_max, 11))
    crossed = 0
    for sizes in _classes(r_max, 20, 300_000).values():
        grids = [P.pc_build_grid(rng.random((n, 3)) * L, box=box, r_max=r_max) for n in sizes]
        assert len({g.cell_size for g in grids}) == 1
        if len(sizes) > 1:
            P.pc_count_cross(grids[0], grids[-1], bins)
            P.pc_count_batch(grids, bins)
            crossed += 1
    assert crossed > 1


def test_counts_of_default_grids():
    r_max, rng = 45.0, np.random.default_rng(6)
    sizes = max(_classes(r_max, 100, 12_000).values(), key=len)
    x, y = (rng.random((n, 3)) * L for n in (sizes[0], sizes[-1]))
    box, bins = P.make_box(L, True), P.Bins("smu", "z", np.linspace(0.0, r_max, 11), np.linspace(0.0, 1.0, 9))
    g, h = (P.pc_build_grid(v, box=box, r_max=r_max) for v in (x, y))
    kw = dict(box=L, periodic=True, mode="smu", edges_a=bins.ea, edges_b=bins.eb, method="grid")
    np.testing.assert_array_equal(P.pc_count_cross(g, h, bins)[0], oracle.count(x, y, **kw)[0])
    got = P.pc_count_batch([g, h], bins)[0].reshape(2, -1)
    for row, v in zip(got, (x, y)):
        np.testing.assert_array_equal(row, oracle.count(v, **kw)[0])
