"""The FP32 kernel's bin decisions with the constants that it receives (CPU,
emulated): pc_fp32_floors exports them, so a changed factor in the library's plan
shows here.

  * Fixed-point floors (at most 126 bins an axis): s, (s, mu) and (sigma, pi) along
    z and the midpoint, edges even from zero, even from any edge and logarithmic.
    Every pair that is not near an edge must lie in its binary64 bin, on random
    pairs and pairs planted about edges, at both ends of the reciprocal roots' and
    the logarithm's errors, with the growing bands at a lower bound of the pair's
    separation; and the sums stray from their binary64 values by no more than the
    band (the check that sees a band cut short although no planted pair does).
  * Packed floors of mu along the midpoint (more than 126 bins).
  * The box tests: no pair in range is dropped, whatever box of eight and half of
    the i-points it is in.
  * Points that are not there: near an edge no more often than others."""

import importlib.util
import os

import numpy as np
import pytest

_spec = importlib.util.spec_from_file_location(
    "fp32_bands", os.path.join(os.path.dirname(__file__), "test_fp32_bands.py"))
fb = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(fb)
P, F32, F64, U, fma32 = fb.P, fb.F32, fb.F64, fb.U, fb.fma32
FIX, FIXOFF, FIXLOG = 5, 6, 7


@pytest.fixture(scope="module", autouse=True)
def lib():
    P.build()
    return P.lib()


def _full(v, like):
    return np.full(like.shape, F32(v))


def _planted(rng, n, L, ea, mode, eb):
    """Pairs along z whose first value lies about an edge, and half of them their
    second one."""
    x = rng.uniform(0.0, L, (n, 3))
    delta = rng.choice([0.0, 1e-7, -1e-7, 1e-6, -1e-6, 1e-5, -1e-5], n)
    a = np.maximum(ea[rng.integers(0, ea.size, n)] * (1.0 + delta), 1e-3 * ea[-1])
    phi, b = rng.uniform(0.0, 2.0 * np.pi, n), rng.random(n)
    if eb is not None:
        h = n // 2
        b[:h] = eb[rng.integers(0, eb.size, h)] / eb[-1] * (1.0 + rng.choice([0.0, 1e-6, -1e-6], h))
    b = np.clip(b, 0.0, 1.0)
    dz, dt = (a * b, a * np.sqrt(1.0 - b * b)) if mode != "sigpi" else (b * eb[-1], a)
    return x, x + np.stack([dt * np.cos(phi), dt * np.sin(phi), dz * rng.choice([-1.0, 1.0], n)], axis=1)


def _geometry(rng, los, mode, ea, eb, periodic_L, ng):
    """(xi, xj, dd, c, lo, hi, L or None, rmin): positions and the kernel's binary32
    separations."""
    R = float(ea[-1] if mode != "sigpi" else np.hypot(ea[-1], eb[-1]))
    if los == "z":
        L = periodic_L
        c, xi, xj, idi, idj, dxc = fb._pairs(rng, 120_000, L, ng, 0.0, R, True)
        xp, xq = _planted(rng, 120_000, L, ea, mode, eb)
        xq = np.mod(xq, L)
        xq = np.where(xq >= L, 0.0, xq)
        idp, idq = (np.minimum(np.floor(v / c).astype(np.int64), ng - 1) for v in (xp, xq))
        dq = idq - idp + (np.round((xp - xq) / L) * ng).astype(np.int64)
        xi, xj = np.vstack([xi, xp]), np.vstack([xj, xq])
        idi, idj, dxc = np.vstack([idi, idp]), np.vstack([idj, idq]), np.vstack([dxc, dq])
        lo, hi, rmin = np.zeros(3), np.full(3, L), 0.0
    else:
        L, c, rmin = None, 81.0, 1000.0
        xi, xj, idi, idj, lo, hi = fb._shell_pairs(rng, 300_000, rmin, 2000.0, c, R)
        dxc = idj - idi
    reli, relj = (xi - (lo + (idi + 0.5) * c)).astype(F32), (xj - (lo + (idj + 0.5) * c)).astype(F32)
    dd = fma32(dxc.astype(F32), np.full(dxc.shape, F32(c)), relj) - reli
    return xi, xj, dd, c, lo, hi, L, rmin


def _separations(dd, two_x, k, los):
    """s2, q, |d.l| and |d x l|^2 as the kernel forms them (two_x: 2 x_i)."""
    dx, dy, dz = dd[:, 0], dd[:, 1], dd[:, 2]
    tiny = _full(k["tiny"], dx)
    q = fma32(dy, dy, fma32(dx, dx, tiny))
    out = dict(q=q, s2=fma32(dz, dz, q), pz=np.abs(dz))
    if los == "mid":
        lx, ly, lz = (two_x[:, a] + dd[:, a] for a in range(3))
        out["pz"] = np.abs(fma32(dz, lz, fma32(dy, ly, dx * lx)))
        out["ll"] = fma32(lz, lz, fma32(ly, ly, fma32(lx, lx, tiny)))
        cx, cy, cz = fma32(dy, lz, -dz * ly), fma32(dz, lx, -dx * lz), fma32(dx, ly, -dy * lx)
        out["cc"] = fma32(cz, cz, fma32(cy, cy, fma32(cx, cx, tiny)))
    return out


def _sums(mode, los, k, v, bands):
    """(T, M) of every combination of the functions' error ends; M None for s."""
    fix = int(k["fix"])
    inv, inv_b = F32(k["inv"]), F32(k["inv_b"])
    cfs, cfm = bands["cfs"], bands["cfm"]
    rls = fb._rsqrt_ends(v["ll"]) if los == "mid" else (None,)
    for rl in rls:
        if mode == "sigpi":
            w = v["cc"] if los == "mid" else v["q"]
            m = fma32(v["pz"], _full(inv_b, w) if rl is None else rl * inv_b, cfm)
            m = np.minimum(m, F32(k["max_b"]))
            if fix == FIXLOG:
                w = w if rl is None else (w * rl) * rl
                first = [(lg, _full(inv, w)) for lg in fb._lg2_ends(w)]
            else:
                first = [(w, r * (inv if rl is None else rl * inv)) for r in fb._rsqrt_ends(w)]
            seconds = [m]
        else:
            rs_ends = fb._rsqrt_ends(v["s2"])
            first = ([(lg, _full(inv, v["s2"])) for lg in fb._lg2_ends(v["s2"])] if fix == FIXLOG
                     else [(v["s2"], rs * inv) for rs in rs_ends])
            seconds = [None] if mode == "s" else [
                fma32(v["pz"], rs * inv_b if rl is None else (rl * rs) * inv_b, cfm) for rs in rs_ends]
        for a, r in first:
            t = fma32(a, r, cfs)
            if fix != FIX:
                t = np.maximum(t, F32(128.5))
            for m in seconds:
                yield np.minimum(t, F32(k["max_a"])), m


def _bands(mode, los, k, s2, q):
    """The batch's bands at lower bounds (16-bit) of the separations given."""
    key = lambda x: (np.maximum(x, 0.0).astype(F32).view(np.uint32) & np.uint32(0xFFFF0000)).view(F32)
    s2m = key(s2 if mode != "sigpi" else (q if los == "z" else 0.0 * q))
    up = lambda a, r2, floor, b: np.ceil(fma32(_full(a, r2), fb._rsqrt_ends(np.maximum(r2, F32(floor)))[0],
                                               _full(b, r2))).astype(F32)
    out = dict(cfs=_full(k["c_a"], s2m), ts2=np.full(s2m.shape, k["near_a"]),
               cfm=_full(k["c_pi"], s2m), tm2=np.full(s2m.shape, k["near_pi"]))
    if int(k["fix"]) == FIXLOG:
        n = up(k["log_A"], s2m, k["log_s2"], k["log_C"])
        out.update(cfs=fma32(n, _full(2.0 ** -16, n), _full(k["c_a"], n)), ts2=2.0 * n.astype(F64))
    if mode == "smu":
        n = up(k["mu_A"], s2m, k["mu_s2"], k["mu_B"])
        out.update(cfm=fma32(n, _full(2.0 ** -16, n), _full(128.0, n)), tm2=2.0 * n.astype(F64))
    out["close"] = (k["close"] + out["ts2"] / 65536.0) if mode == "smu" else np.zeros(s2m.shape)
    return out


def _exact_values(xi, xj, L, los):
    d = xj - xi
    if L:
        d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
    s2 = (d * d).sum(1)
    p = np.abs(d[:, 2])
    if los == "mid":
        l = xi + xj
        p = np.abs((d * l).sum(1)) / np.sqrt((l * l).sum(1))
    sig = np.sqrt(np.maximum(s2 - p * p, 0.0))
    if los == "z":
        sig = np.sqrt(d[:, 0] ** 2 + d[:, 1] ** 2)
    return np.sqrt(s2), sig, p


EVEN = {"s": (np.linspace(0.0, 200.0, 41), None), "smu": (np.linspace(0.0, 200.0, 41), np.linspace(0.0, 1.0, 101)),
        "sigpi": (np.linspace(0.0, 140.0, 41), np.linspace(0.0, 140.0, 41))}
CASES = [(mode, los, "even") for mode in EVEN for los in ("z", "mid") if (mode, los) != ("s", "mid")]
CASES += [(mode, los, kind) for mode in EVEN for los in ("z", "mid") for kind in ("offset", "log")
          if (mode, los) != ("s", "mid") and (mode, kind) != ("sigpi", "offset")]


@pytest.mark.parametrize("mode,los,kind", CASES)
@pytest.mark.parametrize("L,ng", [(1000.0, 11), (3000.0, 59)])
def test_fixed_point_floors_decide_as_the_oracle(mode, los, kind, L, ng):
    if los == "mid" and ng == 59:
        pytest.skip("the shell has one geometry")
    rng = np.random.default_rng(len(mode) + ng + len(kind))
    ea, eb = EVEN[mode]
    if kind == "offset":
        ea = np.linspace(20.0, ea[-1], 121)
    elif kind == "log":
        ea = np.geomspace(0.5, ea[-1], 21)
    xi, xj, dd, c, lo, hi, box, rmin = _geometry(rng, los, mode, ea, eb, L, ng)
    bins = P.Bins(mode, los, ea, eb)
    args = (bins, c, lo, hi, None if box is None else np.full(3, box), box is not None, rmin)
    k = P.pc_fp32_floors(*args)
    assert int(k["fix"]) == {"even": FIX, "offset": FIXOFF, "log": FIXLOG}[kind]
    bp = P.pc_fp32_bands(*args)
    want = fb._oracle_bins(mode, los, xi, xj, box or 0.0, box is not None, ea, eb)
    na, nb = ea.size - 1, 1 if eb is None else eb.size - 1
    s, sig, pi = _exact_values(xi, xj, box, los)
    first = sig if mode == "sigpi" else s
    # exact sums: first axis and, where finite, second
    with np.errstate(divide="ignore", invalid="ignore", over="ignore"):
        D = (ea[-1] - ea[0]) / na
        t_exact = (np.log2(first / ea[0]) / (np.log2(ea[-1] / ea[0]) / na) if kind == "log" else (first - ea[0]) / D)
        m_exact = pi / s * nb if mode == "smu" else pi / ((eb[-1] if eb is not None else 1.0) / nb)
        v = _separations(dd, F32(2.0) * xi.astype(F32), k, los)
        low = rng.choice([1.0, 0.7], s.shape)
        b = _bands(mode, los, k, (s * low) ** 2 * (1 - 1e-6), (sig * low) ** 2 * (1 - 1e-6))
        base = 0.0 if kind == "even" else 1.0
        binned, worst = 0, 0.0
        for t, m in _sums(mode, los, k, v, b):
            bits = t.view(np.uint32)
            near = (bits & 0xFFFF) < b["ts2"]
            n = ((bits >> 16) & 0x7F).astype(np.int64) - int(base)
            j = np.zeros_like(n)
            if m is not None:
                mb = m.view(np.uint32)
                near |= (mb & 0xFFFF) < b["tm2"]
                j = ((mb >> 16) & 0x7F).astype(np.int64)
            if mode == "smu":
                near |= t < b["close"]
            got = np.where((n >= 0) & (n < na) & (j < nb), n * nb + j, -1)
            reach = v["s2"] < F32(bp["r2cut"])
            fast = ~near & reach
            assert np.array_equal(got[fast], want[fast]), int(np.sum(got[fast] != want[fast]))
            binned = max(binned, int(np.sum(fast & (want >= 0))))
            # the sums' errors, in units of the band (pairs inside the clamps, and
            # separations at which the growing bands hold)
            ok = reach & (t > 128.6 if kind != "even" else t > 0) & (t < F32(k["max_a"]) - 0.6) & (s > c / 16.0)
            if kind == "log":
                ok &= first > ea[0]
            err = np.abs(t.astype(F64) - 128.0 - base - t_exact - b["ts2"] / 131072.0)[ok] / (b["ts2"][ok] / 131072.0)
            worst = max(worst, float(err.max()))
            if m is not None:
                ok = reach & (m < F32(k["max_b"]) - 0.6) & (s > c / 16.0) & (s > np.sqrt(k["mu_s2"]))
                err = np.abs(m.astype(F64) - 128.0 - m_exact - b["tm2"] / 131072.0)[ok] / (b["tm2"][ok] / 131072.0)
                worst = max(worst, float(err.max()))
    assert worst <= 1.0 and worst > 0.05, worst          # it does see the rounding
    assert binned > 0.25 * np.sum(want >= 0)          # planted pairs are near by design


@pytest.mark.parametrize("L,ng,lo,R,periodic", fb.GEOMETRIES)
def test_bands_along_z_are_the_derived_ones(L, ng, lo, R, periodic):
    """Per axis u (2.5 c + 3 |d|): s errs by u (4.33 c + 8.7 s), mu by u (6.9 c / s +
    10.7), each taken 1.25 times (a band changed in the library without this
    derivation shows here)."""
    c, n_mu = L / ng, 100
    k = P.pc_fp32_floors(P.Bins("smu", "z", np.linspace(0.0, R, 41), np.linspace(0.0, 1.0, n_mu + 1)), c,
                         np.full(3, lo), np.full(3, lo + ng * c), np.full(3, L) if periodic else None, periodic)
    assert int(k["fix"]) == FIX and k["inv"] == F32(40 / R) and k["inv_b"] == n_mu
    Rb, tiny = R * (1 + 1e-6) + 1e-6 * c, 2.0 ** -48 * (max(abs(lo), abs(lo + ng * c)) + (L if periodic else 0.0) + R)
    eps = (1.25 * U * (4.34 * c + 8.7 * Rb) + tiny) * 40 / R + 1e-9
    assert k["near_a"] == 2 * np.ceil(eps * 65536.0 + 0.5)
    assert k["c_a"] == F32(128.0 + k["near_a"] / 131072.0)
    assert k["mu_A"] == pytest.approx(n_mu * (1.25 * 6.9 * U * c + tiny) * 65536.0 * 1.001, rel=1e-5)
    assert k["mu_B"] == pytest.approx(n_mu * (1.25 * 10.7 * U + 2.0 ** -46) * 65536.0 * 1.001 + 1.0, rel=1e-5)
    # sigma, even and logarithmic (bands of 1.12 / (sigma ln q)), and pi
    r, Rb = R / np.sqrt(2.0) * (1.0 - 1e-12), R * (1 - 1e-12) * (1 + 1e-6) + 1e-6 * c
    eps_z, eps_sig = 2 * U * (2.5 * c + 4 * Rb) + tiny, 2 * U * (3.6 * c + 11.5 * Rb) + Rb * 2.0 ** -25 + tiny
    eb = np.linspace(0.0, r, 121)
    for ea in (np.linspace(0.0, r, 41), np.geomspace(0.01 * R, r, 41)):
        k = P.pc_fp32_floors(P.Bins("sigpi", "z", ea, eb), c, np.full(3, lo), np.full(3, lo + ng * c),
                             np.full(3, L) if periodic else None, periodic)
        assert k["near_pi"] == 2 * np.ceil((eps_z * 120 / r + 1e-9 + 4 * U * 120) * 65536.0 + 0.5)
        if ea[0] == 0.0:
            assert int(k["fix"]) == FIX
            assert k["near_a"] == 2 * np.ceil(np.ceil((eps_sig * 40 / r + 1e-9 + 4 * U * 40) * 65536.0 + 0.5))
        else:
            lq = np.log2(ea[-1] / ea[0]) / 40
            assert int(k["fix"]) == FIXLOG
            assert k["log_A"] == pytest.approx(1.12 * 1.001 * eps_sig / (lq * np.log(2.0)) * 65536.0, rel=1e-5)
            most = max(abs(np.log2(R * R)), abs(np.log2(0.25 * ea[0] ** 2))) * 0.5 / lq
            assert k["log_C"] > 2.0 * (0.5 / lq * 2.0 ** -21 + 2 * U * most) * 65536.0


@pytest.mark.parametrize("e0,log", [(0.0, False), (20.0, False), (0.5, True)])
def test_packed_floors_along_the_midpoint(e0, log):
    """(s, mu) with 130 mu bins along the midpoint: pc_fp32_bands reports the tables
    there, the kernel runs floors."""
    rng = np.random.default_rng(17)
    ea = np.geomspace(e0, 200.0, 41) if log else np.linspace(e0, 200.0, 41)
    eb = np.linspace(0.0, 1.0, 131)
    xi, xj, dd, c, lo, hi, _, rmin = _geometry(rng, "mid", "smu", ea, eb, 0.0, 0)
    args = (P.Bins("smu", "mid", ea, eb), c, lo, hi, None, False, rmin)
    k, bp = P.pc_fp32_floors(*args), P.pc_fp32_bands(*args)
    assert int(k["fix"]) == 0 and int(k["path"]) == (3 if log else (2 if e0 else 1)) and bp["lin"] == 0.0
    want = fb._oracle_bins("smu", "mid", xi, xj, 0.0, False, ea, eb)
    na, nb = 40, 130
    dx, dy, dz = dd[:, 0], dd[:, 1], dd[:, 2]
    lx, ly, lz = (F32(2.0) * xi[:, a].astype(F32) + dd[:, a] for a in range(3))
    sl = np.abs(fma32(dz, lz, fma32(dy, ly, dx * lx)))
    ll = fma32(lz, lz, fma32(ly, ly, lx * lx))
    s2 = fma32(dz, dz, fma32(dy, dy, dx * dx))
    C23, H = F32(2.0 ** 23), F32(2.0 ** 23 - 0.5)
    off = 0 if int(k["path"]) == 1 else 1
    binned = 0
    with np.errstate(divide="ignore", invalid="ignore"):
        for rl in fb._rsqrt_ends(ll):
            for rs in fb._rsqrt_ends(s2):
                if log:
                    ts = [fma32(lg, _full(k["lin_invA"], s2), _full(k["lin_offA"], s2)) for lg in fb._lg2_ends(s2)]
                elif off:
                    ts = [fma32(s2, rs * F32(k["lin_invA"]), _full(k["lin_offA"], s2))]
                else:
                    ts = [None]
                for t in ts:
                    if t is None:                           # one fused step each
                        p = s2.astype(F64) * (rs * F32(k["lin_invA"])).astype(F64)
                        f = np.floor(p)
                        d = fma32(s2, rs * F32(k["lin_invA"]), -(f + 0.5).astype(F32))
                    else:
                        f = fb._rd32(t.astype(F64) + F64(C23)).astype(F64) - 2.0 ** 23
                        d = t - (f + 0.5).astype(F32)
                    th = fma32(_full(-k["lin_mS"], rs), rs, _full(k["lin_thrA"], rs)) if log else _full(k["lin_thrA"], rs)
                    near = ~(np.abs(d) < th)
                    rm = (rl * rs) * F32(k["lin_nB"])
                    fm = np.floor(sl.astype(F64) * rm.astype(F64))
                    dm = fma32(sl, rm, -(fm + 0.5).astype(F32))
                    near |= ~(np.abs(dm) < fma32(_full(-k["lin_mA"], rs), rs, _full(k["lin_cB"], rs)))
                    n, j = f.astype(np.int64) - off, fm.astype(np.int64)
                    got = np.where((n >= 0) & (n < na), n * nb + j, -1)
                    fast = ~near & (s2 < F32(bp["r2cut"]))
                    assert np.all(j[fast] < nb)
                    assert np.array_equal(got[fast], want[fast])
                    binned = max(binned, int(np.sum(fast & (want >= 0))))
    assert binned > 0.25 * np.sum(want >= 0)          # planted pairs are near by design
    assert H == C23 - F32(0.5)


def _rd(x):
    return fb._rd32(x)


def _ru(x):
    return -fb._rd32(-x)


@pytest.mark.parametrize("mode", ["s", "sigpi"])
@pytest.mark.parametrize("L,ng,lo,R,periodic", fb.GEOMETRIES)
def test_box_tests_keep_every_pair_in_range(mode, L, ng, lo, R, periodic):
    """Boxes of eight j-points (relative to their grid's origin, rounded outward)
    against the box of up to 32 i-points, at distances about the reach and across
    the periodic boundary."""
    rng = np.random.default_rng(ng)
    c = L / ng
    ra, rb = (R, None) if mode == "s" else (0.6 * R, 0.5 * R)
    ea = np.linspace(0.0, ra, 11)
    bins = P.Bins(mode, "z", ea, None if rb is None else np.linspace(0.0, rb, 11))
    k = P.pc_fp32_floors(bins, c, np.full(3, lo), np.full(3, lo + ng * c), np.full(3, L) if periodic else None, periodic)
    B, NI, NJ = 6000, 16, 8
    w = np.minimum(rng.choice([1e-4, 0.05, 0.4], (B, 1, 1)) * c, 0.2 * R)
    xi = lo + rng.uniform(0.0, ng * c, (B, 1, 3)) + rng.uniform(-1.0, 1.0, (B, NI, 3)) * w
    off = rng.normal(size=(B, 1, 3))
    off /= np.linalg.norm(off, axis=2, keepdims=True)
    off[: B // 3] = np.eye(3)[rng.integers(0, 3, B // 3)][:, None, :]
    if mode == "sigpi":                                        # about the cylinder's mantle and its ends
        t = rng.uniform(0.0, 2.0 * np.pi, (B, 1))
        mantle = rng.random((B, 1)) < 0.5
        off[:, :, 0], off[:, :, 1] = (np.where(mantle, ra, ra * rng.random((B, 1))) * f(t) for f in (np.cos, np.sin))
        off[:, :, 2] = np.where(mantle, rb * rng.uniform(-1, 1, (B, 1)), rb * rng.choice([-1.0, 1.0], (B, 1)))
    else:
        off *= ra
    xj = xi[:, :1] + off * rng.choice([0.9, 1.0 - 1e-9, 1.0, 1.02], (B, 1, 1)) + rng.uniform(-1.0, 1.0, (B, NJ, 3)) * w
    lo_b, hi_b = lo, lo + ng * c
    if periodic:
        xi = np.mod(xi, L)                                     # halves that straddle the boundary are wide boxes
        img = np.floor(xj[:, :1] / L)                          # one image a box
        xj = xj - img * L
        keep = np.all((xj >= 0) & (xj < L), axis=(1, 2)) & (np.ptp(xi, axis=1).max(1) < 0.5 * L)
        xi, xj, img = xi[keep], xj[keep], img[keep][:, 0]
    else:
        keep = np.all((xi >= lo_b) & (xi < hi_b), axis=(1, 2)) & np.all((xj >= lo_b) & (xj < hi_b), axis=(1, 2))
        xi, xj, img = xi[keep], xj[keep], np.zeros((int(keep.sum()), 3))
    assert xi.shape[0] > 1500
    li, hi_i = _rd((xi - lo).min(1)), _ru((xi - lo).max(1))
    lj, hj = _rd((xj - lo).min(1)), _ru((xj - lo).max(1))
    if periodic:
        sh = img.astype(F32) * F32(L)
        lj, hj = lj + sh, hj + sh
    g = np.maximum(np.maximum(lj - hi_i, li - hj), F32(0.0))
    gq = fma32(g[:, 1], g[:, 1], g[:, 0] * g[:, 0])
    g2 = fma32(g[:, 2], g[:, 2], gq)
    kept = g2 <= F32(k["gap2"])
    if mode == "sigpi":
        kept &= (gq <= F32(k["gap2_across"])) & (g[:, 2] <= F32(k["gap_along"]))
    d = xj[:, None] + (img * L)[:, None, None] - xi[:, :, None]
    s2, q2 = (d * d).sum(-1), d[..., 0] ** 2 + d[..., 1] ** 2
    inside = s2 < ra * ra if mode == "s" else (q2 < ra * ra) & (d[..., 2] ** 2 < rb * rb)
    inside = inside.reshape(inside.shape[0], -1)
    assert not np.any(inside.any(1) & ~kept)
    assert 0.02 < np.mean(~kept) < 0.98                        # the test does drop boxes
    # the bound of the separations that the growing bands take: never above a pair's
    root = np.maximum(np.sqrt((gq if mode == "sigpi" else g2).astype(F64)) * (1 - 2.0 ** -21) - k["gap_error"], 0.0)
    least = np.sqrt((q2 if mode == "sigpi" else s2).reshape(s2.shape[0], -1).min(1))
    assert np.all(root <= least)


@pytest.mark.parametrize("mode", ["smu", "sigpi"])
def test_absent_points_are_seldom_near_an_edge(mode):
    """An i-point that is not there stands at x = -far with 2 x_i = (0, far, 0) along
    the midpoint: l is not parallel to d, so sigma and pi lie past the last edge and
    mu is near one as often as any value, 2 B 2^-16.  (With 2 x_i = 0, l = d: mu = 1
    and sigma = 0, always near.)"""
    rng = np.random.default_rng(9)
    ea, eb = EVEN[mode]
    c = 200.0
    k = P.pc_fp32_floors(P.Bins(mode, "mid", ea, eb), c, np.full(3, -2000.0), np.full(3, 2000.0), None, False, 1000.0)
    assert int(k["fix"]) == FIX
    far, n = F32(k["far"]), 100_000
    xj = rng.uniform(-400.0, 400.0, (n, 3)).astype(F32)
    dd = xj - np.array([-far, 0, 0], F32)
    for y in (far, F32(0.0)):
        v = _separations(dd, np.tile(np.array([0, y, 0], F32), (n, 1)), k, "mid")
        with np.errstate(divide="ignore", invalid="ignore"):
            b = _bands(mode, "mid", k, np.zeros(n), np.zeros(n))
            for t, m in _sums(mode, "mid", k, v, b):
                near = ((t.view(np.uint32) & 0xFFFF) < b["ts2"]) | ((m.view(np.uint32) & 0xFFFF) < b["tm2"])
                usual = (b["ts2"][0] + b["tm2"][0]) / 65536.0
                assert near.mean() < 1.5 * usual if y else near.mean() > 0.99
