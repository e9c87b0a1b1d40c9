"""(s, mu) counts whose reach is small against the cells or list nodes (a k-d tree's
nodes of 250 points around pairs a few units apart): pairs close enough to be near
an edge whatever their mu must stay few, since each is checked in binary64, and the
fixed-point floors must still decide the others as the oracle does (CPU, emulated
with the constants that the kernel receives)."""

import importlib.util
import os

import numpy as np
import pytest

_spec = importlib.util.spec_from_file_location(
    "kernel_floors", os.path.join(os.path.dirname(__file__), "test_kernel_floors.py"))
kf = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(kf)
P = kf.P


@pytest.mark.parametrize("R", [5.0, 8.0, 20.0])
def test_small_reach_decides_as_the_oracle(R, monkeypatch):
    monkeypatch.setitem(kf.EVEN, "smu", (np.linspace(0.0, R, 11), np.linspace(0.0, 1.0, 21)))
    # cells of 62.5; asserts too that a quarter of the pairs at least are binned without a check
    kf.test_fixed_point_floors_decide_as_the_oracle("smu", "z", "even", 1000.0, 16)


@pytest.mark.parametrize("los", ["z", "mid"])
@pytest.mark.parametrize("nb", [1, 20, 120])
@pytest.mark.parametrize("ratio", [0.05, 0.5, 1.0, 2.0, 5.0, 20.0, 80.0])
def test_few_pairs_are_near_for_their_separation_alone(ratio, nb, los):
    """Uniform pairs: the share (s / R)^3 below 1/500."""
    R = 10.0
    lo, hi = (np.zeros(3), np.full(3, 1e4)) if los == "z" else (np.full(3, 1e3), np.full(3, 5e3))
    k = P.pc_fp32_floors(P.Bins("smu", los, np.linspace(0.0, R, 41), np.linspace(0.0, 1.0, nb + 1)), ratio * R, lo, hi,
                         np.full(3, 1e4) if los == "z" else None, los == "z", 0.0 if los == "z" else 1700.0)
    if int(k["fix"]):
        assert (np.sqrt(k["mu_s2"]) / R) ** 3 < 1.0 / 500.0
    else:
        assert los == "mid"
    # clusters tighter than the cells: never beyond the separation whose band is 1/2048
    # of a bin (mu_A: its band times s, in units of 2^-16), or a 64th of the cell
    if int(k["fix"]):
        assert np.sqrt(k["mu_s2"]) < 1.01 * max(ratio * R / 64.0, 1e-3 * R, 2048.0 * k["mu_A"] / 65536.0)
