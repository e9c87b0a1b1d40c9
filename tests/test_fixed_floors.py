"""The pair kernel's fixed-point floors (CPU, emulated): for bins evenly spaced
from zero a scaled value t is summed once in binary32 onto 128 + B 2^-16 (a grid
of 2^-16; offset and logarithmic edges: 129 + B 2^-16 less the first edge's t),
the bin is the sum's third byte and the pair is near an edge iff its low half is
below 2 B.  On the kernel's own binary32 separations (cell-relative
coordinates, both ends of the reciprocal root's error) every pair that is not
near must sit in the bin of its binary64 value, for s (band of the whole count)
and mu (band at a lower bound of the pair's separation), with the bands as the
library forms them; halving a band must break it."""

import importlib.util
import os

import numpy as np
import pytest

_spec = importlib.util.spec_from_file_location(
    "fp32_bands", os.path.join(os.path.dirname(__file__), "test_fp32_bands.py"))
fb = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(fb)
F32, F64, U = fb.F32, fb.F64, fb.U


def _fixed(v, rv, band):
    """(bin, fraction) of RN(v rv + 128 + band 2^-16), v and rv binary32."""
    c = F32(128.0 + band / 65536.0)
    t = fb.fma32(v, rv, np.full(v.shape, c)).view(np.uint32)
    return ((t >> 16) & 0x7F).astype(np.int64), t & 0xFFFF


@pytest.mark.parametrize("L,ng,lo,R,periodic", fb.GEOMETRIES)
@pytest.mark.parametrize("na,nb", [(40, 100), (126, 126), (7, 3)])
def test_fixed_floors_decide_like_binary64(L, ng, lo, R, periodic, na, nb):
    rng = np.random.default_rng(na + ng)
    c, xi, xj, idi, idj, dxc = fb._pairs(rng, 200_000, L, ng, lo, R, periodic)
    o = fb._oracle_values(xi, xj, L, periodic)
    D = R / na
    X, Lm = max(abs(lo), abs(lo + ng * c)), L if periodic else 0.0
    tiny = 2.0 ** -48 * (X + Lm + R)
    eps_s = (1.25 * U * (4.34 * c + 8.7 * R) + tiny) / D + 1e-9
    bs = int(np.ceil(eps_s * 65536.0 + 0.5))
    mA = nb * (1.25 * 6.9 * U * c + tiny) * 65536.0 * 1.02
    mB = nb * (1.25 * 10.7 * U + 2.0 ** -46) * 65536.0 * 1.02 + 1.0
    keep = (o["s"] < R) & (o["s"] > c / 16.0)
    low = o["s"] * rng.choice([1.0, 0.7], o["s"].shape)     # a batch's smallest separation
    bm = np.ceil(mA / low + mB).astype(np.int64)
    inv_d = F32(na / R)
    k_true = np.floor(o["s"] / D).astype(np.int64)
    j_true = np.minimum(np.floor(o["mu"] * nb).astype(np.int64), nb - 1)
    seen = 0
    with np.errstate(all="ignore"):
        values = fb._kernel_values(c, lo, xi, xj, idi, idj, dxc)
    for kv in values:
        n, frac = _fixed(kv["s2"], kv["rs"] * inv_d, bs)
        far = keep & (frac >= 2 * bs)
        assert np.array_equal(n[far], k_true[far])
        dz = kv["pi"]
        cm = (128.0 + bm / 65536.0).astype(F32)
        t = fb.fma32(dz, kv["rs"] * F32(nb), cm).view(np.uint32)
        m, frac = ((t >> 16) & 0x7F).astype(np.int64), (t & 0xFFFF).astype(np.int64)
        far = keep & (frac >= 2 * bm)
        assert np.array_equal(m[far], j_true[far])
        seen += int(far.sum())
    assert seen > 0


@pytest.mark.parametrize("L,ng,lo,R,periodic", fb.GEOMETRIES)
@pytest.mark.parametrize("e0,na,log", [(0.3, 125, False), (0.02, 7, False), (1e-3, 40, True), (0.2, 125, True),
                                       (0.02, 1, True)])
def test_offset_and_log_floors_decide_like_binary64(L, ng, lo, R, periodic, e0, na, log):
    """First edge e0 R: bins below (row 0) and past the last are discarded."""
    rng = np.random.default_rng(na + ng)
    c, xi, xj, idi, idj, dxc = fb._pairs(rng, 200_000, L, ng, lo, R, periodic)
    o = fb._oracle_values(xi, xj, L, periodic)
    e0 = e0 * R
    X, Lm = max(abs(lo), abs(lo + ng * c)), L if periodic else 0.0
    tiny = 2.0 ** -48 * (X + Lm + R)
    s = o["s"]
    low = np.maximum(s * rng.choice([1.0, 0.7], s.shape), 0.5 * e0)   # a batch's smallest separation
    if log:
        lq = np.log2(R / e0) / na
        A, B = 0.5 / lq, -np.log2(e0) / lq
        Lmax = max(abs(np.log2(R * R)), abs(np.log2(0.25 * e0 * e0)))
        C = 129.0 + B
        common = (A * 2.0 ** -21 * max(1.0, Lmax) + U * (A * Lmax + abs(B) + na + 130.0) * 2.0 + 1e-6 + A * 2.0 ** -45)
        sC = 2.0 * (A * 9.0 * U / np.log(2.0) * 1.01 + common) * 65536.0 + 2.0
        sA = 4.0 * A * (4.4 * U * c + 2.0 ** -51 * (X + Lm + R)) / np.log(2.0) * 1.01 * 65536.0
        if not (abs(C) < 250.0 and sA / (0.5 * e0) + sC < 8192.0 and
                2.0 * U * (4.4 * c + 10.5 * R) + tiny < 0.05 * e0):
            pytest.skip("the library keeps the tables here")
        b = np.ceil(sA / low + sC)
        t = np.log2(s / e0) / lq
        inv = F32(A)
    else:
        D = (R - e0) / na
        C = 129.0 - e0 / D
        if abs(C) >= 250.0:
            pytest.skip("the library keeps the packed floors here")
        b = np.full(s.shape, np.ceil(((1.25 * U * (4.34 * c + 8.7 * R) + tiny) / D + 1e-9) * 65536.0 + 1.5))
        t = (s - e0) / D
        inv = F32(1.0 / D)
    k_true = np.where(s < e0, -1, np.minimum(np.floor(t), na)).astype(np.int64)
    cst = (F32(C) + (b / 65536.0).astype(F32)).astype(F32)
    seen = 0
    with np.errstate(all="ignore"):
        values = fb._kernel_values(c, lo, xi, xj, idi, idj, dxc)
    for kv in values:
        s2 = kv["s2"]
        for v, r in ([(lg, np.full(s2.shape, inv)) for lg in fb._lg2_ends(np.maximum(s2, F32(1e-30)))] if log
                     else [(s2, kv["rs"] * inv)]):
            T = fb.fma32(v, r, cst)
            T = np.clip(np.where(np.isnan(T), F32(128.5), T), F32(128.5), F32(129.5 + na)).view(np.uint32)
            far = (T & 0xFFFF) >= 2 * b
            assert np.array_equal(((T >> 16) & 0x7F).astype(np.int64)[far] - 1, k_true[far])
            seen += int(far.sum())
    assert seen > 0


def test_fixed_floors_need_their_band():
    """Pairs planted within the band of an s edge: with a band of zero some land
    in the wrong bin without being near."""
    L, ng, R, na = 1000.0, 11, 200.0, 40
    rng = np.random.default_rng(3)
    c, xi, xj, idi, idj, dxc = fb._pairs(rng, 400_000, L, ng, 0.0, R, True)
    d = xj - xi
    d = np.where(d > L / 2, d - L, np.where(d < -L / 2, d + L, d))
    s = np.sqrt((d * d).sum(1))
    edge = np.maximum(np.round(s / 5.0), 1.0) * 5.0
    xj = xi + d * (edge * (1.0 + rng.choice([-1, 1], s.size) * 1e-8) / s)[:, None]
    shift = np.floor(xj / L)
    xj = xj - shift * L
    idj = np.minimum(np.floor(xj / c).astype(np.int64), ng - 1)
    dxc = idj - idi + (shift * ng).astype(np.int64)
    o = fb._oracle_values(xi, xj, L, True)
    with np.errstate(all="ignore"):
        kv = fb._kernel_values(c, 0.0, xi, xj, idi, idj, dxc)[0]
    k_true = np.floor(o["s"] / 5.0).astype(np.int64)
    keep = o["s"] < R
    n, _ = _fixed(kv["s2"], kv["rs"] * F32(0.2), 0)
    assert np.any(n[keep] != k_true[keep])
    n, frac = _fixed(kv["s2"], kv["rs"] * F32(0.2), 3)
    assert np.all((frac < 6)[keep])       # every planted pair is near
