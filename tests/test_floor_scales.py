"""(sigma, pi) along the midpoint line of sight in any unit of length (CPU,
emulated): sigma^2 |l|^2 = |d x l|^2 is a fourth power of the lengths, so its
binary32 value overflows, or falls below the constant that the fixed-point floors
add to squares, long before the squares do.  A survey shell, its grid and its edges
are scaled by powers of two, which changes no bin; wherever the library chooses
fixed-point floors, with the constants that it exports, every pair not near an
edge must keep the bin of the binary64 definition."""

import importlib.util
import os

import numpy as np
import pytest

_spec = importlib.util.spec_from_file_location(
    "kernel_floors", os.path.join(os.path.dirname(__file__), "test_kernel_floors.py"))
kf = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(kf)
P, fb, F32 = kf.P, kf.fb, kf.F32


@pytest.mark.parametrize("kind", ["even", "log"])
def test_sigma_along_the_midpoint_in_any_unit(kind):
    rng = np.random.default_rng(5)
    ea, eb = kf.EVEN["sigpi"]
    if kind == "log":
        ea = np.geomspace(0.5, ea[-1], 21)
    xi, xj, dd, c, lo, hi, _, rmin = kf._geometry(rng, "mid", "sigpi", ea, eb, None, 0)
    _, sig, _ = kf._exact_values(xi, xj, None, "mid")
    # outside the first axis: discarded rows, before it (logarithms) and past it
    n_exact = np.digitize(sig, ea) - 1
    inside = (n_exact >= 0) & (n_exact < ea.size - 1)
    fixed = []
    for e in range(-60, 61):
        f = 2.0 ** e
        k = P.pc_fp32_floors(P.Bins("sigpi", "mid", ea * f, eb * f), c * f, lo * f, hi * f, None, False, rmin * f)
        if int(k["fix"]) == 0:
            continue
        fixed.append(e)
        with np.errstate(all="ignore"):
            v = kf._separations(dd * F32(f), F32(2.0 * f) * xi.astype(F32), k, "mid")
            assert np.isfinite(v["cc"][inside]).all(), f"2^{e}"
            b = kf._bands("sigpi", "mid", k, v["s2"], 0.0 * v["q"])
            for rl in fb._rsqrt_ends(v["ll"]):
                if kind == "log":
                    ts = [kf.fma32(g, kf._full(k["inv"], g), b["cfs"]) for g in fb._lg2_ends((v["cc"] * rl) * rl)]
                else:
                    ts = [kf.fma32(v["cc"], r * (rl * F32(k["inv"])), b["cfs"]) for r in fb._rsqrt_ends(v["cc"])]
                for t in ts:
                    if kind == "log":
                        t = np.fmax(t, F32(128.5))
                    bits = np.fmin(t, F32(k["max_a"])).view(np.uint32)
                    n = ((bits >> 16) & 0x7F).astype(np.int64) - (1 if kind == "log" else 0)
                    fast = inside & ((bits & 0xFFFF) >= b["ts2"])
                    bad = int(np.sum(n[fast] != n_exact[fast]))
                    assert bad == 0, f"2^{e}: {bad} of {int(fast.sum())}"
    # the units that catalogues come in (Gpc to pc)
    assert set(range(-11, 21)) <= set(fixed), fixed
