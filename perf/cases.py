"""The calls that users of the pair counter make, as measurable cases.

A case is one call (or one build-and-count sequence) through the package's
public functions on a seeded catalogue held in device memory, the way an
analysis script holds it.  The catalogues follow the repository's workloads:
uniform and Neyman-Scott clustered points in a periodic cube of side 1000, the
half-uniform half-clustered cube with binary32 lognormal weights, the survey
shell (1000 <= r < 2000, 60 x 60 degrees, FKP-like binary64 weights, midpoint
line of sight), and batches of uneven mocks.

Case fields:
  call     count      paircount's one-call grid form (build, count, free)
           tree       the same through the k-d tree
           held       a grid the program keeps, one auto count of it
           batch      the grids of `mocks` catalogues and one batched count
           tree_batch the same through the batched k-d trees
  points   uniform, clustered, mixed (periodic) or survey
  n, n2    points of the catalogue, and of the second one of a cross count
           (n2 = 0: auto count); for batches n and n2 bound the mocks' sizes
  mode, los, bins, na, nb, ra, rb
           the histogram: bins linear, log or wp (logarithmic sigma from 0.5,
           linear pi); na x nb bins up to ra (and rb for pi)
  weights  none, f32 (lognormal) or f64 (FKP)
  prec     f32 (binary32 separations, binary64 near the edges) or f64
"""

import math

import numpy as np
import torch

import paper_2301_12557_gb300 as P

L = 1000.0                       # side of the periodic cubes
SIGMA = 5.0                      # cluster width
CHILDREN = 10                    # mean points per cluster
R_LO, R_HI = 1000.0, 2000.0      # survey shell
N_SURVEY = 1_000_000             # data points the FKP weights' density refers to
P0 = 1.0e4


def _case(name, call, points, n, n2=0, mode="s", los="z", bins="linear", na=40, nb=1, ra=200.0,
          rb=0.0, weights="none", prec="f32", mocks=1):
    c = dict(call=call, points=points, n=n, n2=n2, mode=mode, los=los, bins=bins, na=na, nb=nb,
             ra=ra, rb=rb, weights=weights, prec=prec, mocks=mocks)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest whole call: a small box, where fixed costs count
        _case("uniform_20k_s", "count", "uniform", 20_000),
        # the plain binary64 method on a small box (a user's cross-check)
        _case("uniform_50k_s_f64", "count", "uniform", 50_001, prec="f64"),
        # the (s, mu) count of one clustered simulation box, grid and tree
        _case("clustered_2m_smu", "count", "clustered", 2_000_000, mode="smu", nb=100),
        _case("clustered_2m_smu_tree", "tree", "clustered", 2_000_000, mode="smu", nb=100),
        # the weighted isotropic count of a dense box (1/27 of the 100M-point cube)
        _case("mixed_3700k_s_w32", "count", "mixed", 3_703_704, weights="f32"),
        # logarithmic s bins down to small scales, one mock-sized catalogue
        _case("clustered_300k_logsmu", "count", "clustered", 312_345, mode="smu", bins="log", nb=100),
        # the paper's large histogram: 200 s bins x 120 mu bins
        _case("clustered_1m_200x120", "count", "clustered", 1_000_003, mode="smu", na=200, nb=120),
        # projected correlation function: log sigma x linear pi in a periodic box
        _case("clustered_1m_wp", "count", "clustered", 1_000_000, mode="sigpi", bins="wp", na=20,
              nb=60, ra=60.0, rb=60.0),
        # a survey's data-random count in (sigma, pi), midpoint line of sight, FKP weights
        _case("survey_dr_sigpi_w64", "count", "survey", 100_000, 2_000_000, mode="sigpi", los="mid",
              nb=40, rb=200.0, weights="f64"),
        # a survey's random-random count in (s, mu) for multipoles, on a kept grid
        _case("survey_rr_smu_w64", "held", "survey", 500_000, mode="smu", los="mid", nb=100,
              weights="f64"),
        # covariance mocks of uneven sizes, one batched count: grids and trees
        _case("mocks_12_smu", "batch", "clustered", 200_000, 800_000, mode="smu", nb=100, mocks=12),
        _case("mocks_12_smu_tree", "tree_batch", "clustered", 200_000, 800_000, mode="smu", nb=100,
              mocks=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1


def draw(rng):
    kind = rng.randrange(8)
    if kind == 0:      # small boxes, either precision
        prec = rng.choice(("f32", "f32", "f64"))
        return _case(None, "count", "uniform", _log_int(rng, 2_000, 60_000), na=rng.randrange(10, 61),
                     ra=float(rng.randrange(80, 221)), prec=prec)
    if kind == 1:      # simulation boxes in (s, mu), grid or tree, linear or log s
        return _case(None, rng.choice(("count", "tree")), "clustered", _log_int(rng, 30_000, 2_000_000),
                     mode="smu", bins=rng.choice(("linear", "linear", "log")),
                     na=rng.randrange(20, 61), nb=rng.randrange(20, 121),
                     ra=float(rng.randrange(100, 201)))
    if kind == 2:      # isotropic weighted boxes
        return _case(None, rng.choice(("count", "count", "tree")), rng.choice(("mixed", "clustered")),
                     _log_int(rng, 100_000, 3_000_000), na=rng.randrange(20, 61),
                     ra=float(rng.randrange(120, 201)), weights=rng.choice(("f32", "none")))
    if kind == 3:      # large histograms
        return _case(None, "count", "clustered", _log_int(rng, 100_000, 1_200_000), mode="smu",
                     na=rng.randrange(120, 201), nb=rng.randrange(100, 121),
                     ra=float(rng.randrange(150, 201)))
    if kind == 4:      # projected correlation functions
        return _case(None, rng.choice(("count", "tree")), "clustered", _log_int(rng, 100_000, 2_000_000),
                     mode="sigpi", bins="wp", na=rng.randrange(10, 31), nb=rng.randrange(30, 81),
                     ra=float(rng.randrange(30, 81)), rb=float(rng.randrange(40, 101)))
    if kind == 5:      # survey cross counts
        return _case(None, rng.choice(("count", "tree")), "survey", _log_int(rng, 10_000, 120_000),
                     _log_int(rng, 100_000, 2_000_000), mode=rng.choice(("sigpi", "smu")), los="mid",
                     na=40, nb=rng.choice((20, 40, 60)), rb=200.0, weights=rng.choice(("f64", "none")))
    if kind == 6:      # survey auto counts on a kept grid
        return _case(None, "held", "survey", _log_int(rng, 30_000, 600_000),
                     mode=rng.choice(("smu", "sigpi", "s")), los="mid", na=40,
                     nb=rng.choice((20, 40, 100)), ra=float(rng.randrange(120, 201)), rb=150.0,
                     weights=rng.choice(("f64", "none")))
    hi = _log_int(rng, 100_000, 800_000)
    return _case(None, rng.choice(("batch", "tree_batch")), "clustered", hi // 4, hi, mode="smu",
                 na=rng.randrange(20, 51), nb=rng.randrange(20, 101),
                 ra=float(rng.randrange(120, 201)), mocks=rng.randrange(3, 15))


# ---------------------------------------------------------------------------
# catalogues
# ---------------------------------------------------------------------------
def _edges(case):
    na, nb, ra, rb = case["na"], case["nb"], case["ra"], case["rb"]
    if case["bins"] == "log":
        ea = np.geomspace(0.1, ra, na + 1)
    elif case["bins"] == "wp":
        ea = np.geomspace(0.5, ra, na + 1)
    else:
        ea = np.linspace(0.0, ra, na + 1)
    if case["mode"] == "smu":
        return ea, np.linspace(0.0, 1.0, nb + 1)
    if case["mode"] == "sigpi":
        return ea, np.linspace(0.0, rb, nb + 1)
    return ea, None


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _fold(x):
    x = torch.remainder(x, L)
    return torch.where(x >= L, torch.zeros_like(x), x)


def _uniform(g, n):
    return _fold(_rand(g, n, 3) * L)


def _clustered(g, n, sigma=SIGMA):
    parents = _rand(g, max(1, n // CHILDREN), 3) * L
    which = torch.randint(parents.shape[0], (n,), generator=g, device="cuda")
    return _fold(parents[which] + sigma * _randn(g, n, 3))


def _selection(r):
    return torch.exp(-((r - 1500.0) / 500.0) ** 2)


def _shell(g, m):
    r = (R_LO ** 3 + _rand(g, m) * (R_HI ** 3 - R_LO ** 3)) ** (1.0 / 3.0)
    ra = _rand(g, m) * (math.pi / 3.0)
    sd = 2.0 * _rand(g, m) * 0.5 - 0.5
    cd = torch.sqrt(1.0 - sd * sd)
    return torch.stack([r * cd * torch.cos(ra), r * cd * torch.sin(ra), r * sd], dim=1)


def _survey(g, n, clustered):
    m = 3 * n + 1000
    if clustered:
        parents = _shell(g, max(1, m // CHILDREN))
        which = torch.randint(parents.shape[0], (m,), generator=g, device="cuda")
        x = parents[which] + SIGMA * _randn(g, m, 3)
    else:
        x = _shell(g, m)
    r = x.norm(dim=1)
    ra, sd = torch.atan2(x[:, 1], x[:, 0]), x[:, 2] / r
    ok = (r >= R_LO) & (r < R_HI) & (ra >= 0) & (ra < math.pi / 3) & (sd.abs() <= 0.5)
    ok &= _rand(g, m) < _selection(r)
    return x[ok][:n].contiguous()


def _fkp(x):
    rr = np.linspace(R_LO, R_HI, 20001)
    f = np.exp(-((rr - 1500.0) / 500.0) ** 2) * rr * rr
    volume = (math.pi / 3.0) * float(np.sum(0.5 * (f[1:] + f[:-1]) * np.diff(rr)))
    return (1.0 / (1.0 + N_SURVEY * _selection(x.norm(dim=1)) / volume * P0)).contiguous()


def _points(case, g, n, second=False, sigma=SIGMA):
    kind = case["points"]
    if kind == "uniform":
        return _uniform(g, n)
    if kind == "clustered":
        return _clustered(g, n, sigma)
    if kind == "mixed":
        return torch.cat([_uniform(g, n // 2), _clustered(g, n - n // 2)]).contiguous()
    # survey: the first catalogue of a cross count is data, the others randoms
    return _survey(g, n, clustered=case["n2"] > 0 and not second)


def _weights(case, g, x):
    if case["weights"] == "none":
        return None
    if case["weights"] == "f64":
        return _fkp(x)
    return torch.exp(0.3 * _randn(g, x.shape[0]) - 0.045).to(torch.float32)


def _mock_sizes(case, seed):
    r = np.random.RandomState(int(seed) % (1 << 31))
    return [int(v) for v in r.randint(case["n"], case["n2"] + 1, case["mocks"])]


def _catalogues(case, seed):
    """[(points, weights)] of the case's call, on the device."""
    g = _gen(seed)
    out = []
    if case["call"] in ("batch", "tree_batch"):
        for n in _mock_sizes(case, seed):
            sigma = 3.0 + 5.0 * float(torch.rand(1, generator=g, device="cuda"))
            out.append((_points(case, g, n, sigma=sigma), None))
        return out
    for k, n in enumerate([case["n"]] + ([case["n2"]] if case["n2"] else [])):
        x = _points(case, g, n, second=k > 0)
        out.append((x, _weights(case, g, x)))
    return out


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    cats = _catalogues(case, seed)
    ea, eb = _edges(case)
    s = {"case": case, "cats": cats, "ea": ea, "eb": eb}
    if case["call"] in ("held", "batch", "tree_batch"):
        s["bins"] = P.Bins(case["mode"], case["los"], ea, eb)
        periodic = case["points"] != "survey"
        s["box"] = P.make_box(L if periodic else None, periodic)
    if case["call"] == "held":
        x, w = cats[0]
        s["grid"] = P.pc_build_grid(x, w, box=s["box"], r_max=s["bins"].r_max)
    return s


def run(s):
    case, cats = s["case"], s["cats"]
    weighted = case["weights"] != "none"
    if case["call"] == "held":
        c, w, _ = P.pc_count_auto(s["grid"], s["bins"], weighted=weighted)
    elif case["call"] == "batch":
        cell = 0.0
        grids = []
        for x, _ in cats:    # one cell size for all: the first mock's
            grids.append(P.pc_build_grid(x, box=s["box"], r_max=s["bins"].r_max,
                                         opts=P.make_opts(cell_size=cell)))
            cell = cell or grids[0].cell_size
        c, w, _ = P.pc_count_batch(grids, s["bins"])
        for g in grids:
            P.pc_free_grid(g)
    elif case["call"] == "tree_batch":
        trees = P.pc_build_tree_batch([x for x, _ in cats], box=s["box"])
        c, w, _ = P.pc_count_tree_batch(trees, s["bins"])
        for t in trees:
            P.pc_free_tree(t)
    else:
        x1, w1 = cats[0]
        x2, w2 = cats[1] if len(cats) > 1 else (None, None)
        periodic = case["points"] != "survey"
        kw = dict(w1=w1, w2=w2, box=L if periodic else None, periodic=periodic, mode=case["mode"],
                  los=case["los"], edges_a=s["ea"], edges_b=s["eb"])
        if case["call"] == "tree":
            c, w = P.count_tree(x1, x2, **kw)
        else:
            c, w = P.count(x1, x2, prec=case["prec"], **kw)
    return [c, w] if weighted else [c]


# ---------------------------------------------------------------------------
# what a pass cannot do without, and what it should return
# ---------------------------------------------------------------------------
def _reach_volume(case):
    if case["mode"] == "sigpi":
        return 2.0 * math.pi * case["ra"] ** 2 * case["rb"]
    return 4.0 / 3.0 * math.pi * case["ra"] ** 3


def _in_range(case, n1, n2):
    """Expected in-range pairs of n1 x n2 points (boundaries of the shell not
    taken off)."""
    if case["points"] == "survey":
        rr = np.linspace(R_LO, R_HI, 2001)
        p = np.exp(-((rr - 1500.0) / 500.0) ** 2)
        dr = rr[1] - rr[0]
        volume = (math.pi / 3.0) * float((p * rr * rr).sum() * dr) ** 2 / float((p * p * rr * rr).sum() * dr)
    else:
        volume = L ** 3
    return float(n1) * float(n2) * _reach_volume(case) / volume


def work(case):
    """Inputs read and histograms written once; 8 binary operations for the
    squared separation of each in-range pair and 6 for its bin, 2 more for a
    weighted sum."""
    nbins = case["na"] * case["nb"]
    per = 14 + (2 if case["weights"] != "none" else 0)
    wb = {"none": 0, "f32": 4, "f64": 8}[case["weights"]]
    if case["call"] in ("batch", "tree_batch"):
        mean = 0.5 * (case["n"] + case["n2"])
        square = (case["n"] ** 2 + case["n"] * case["n2"] + case["n2"] ** 2) / 3.0
        pairs = 0.5 * case["mocks"] * _in_range(case, 1.0, 1.0) * square
        return {"bytes": 24.0 * mean * case["mocks"] + 8.0 * nbins * case["mocks"],
                "flops": per * pairs}
    if case["n2"]:
        pairs, points = _in_range(case, case["n"], case["n2"]), case["n"] + case["n2"]
    else:
        pairs, points = 0.5 * _in_range(case, case["n"], case["n"]), case["n"]
    out = 8.0 * nbins * (2 if case["weights"] != "none" else 1)
    return {"bytes": (24.0 + wb) * points + out, "flops": per * pairs}


def _histogram(case, x1, w1, x2, w2, ea, eb):
    """Counts and weighted sums by brute force over all pairs, in binary64."""
    dev = x1.device
    Ea = torch.from_numpy(ea * ea).to(dev)
    Eb = torch.from_numpy(eb * eb).to(dev) if eb is not None else None
    na, nb = case["na"], case["nb"] if eb is not None else 1
    auto = x2 is None
    xj, wj = (x1, w1) if auto else (x2, w2)
    periodic = case["points"] != "survey"
    counts = torch.zeros(na * nb, dtype=torch.int64, device=dev)
    sums = torch.zeros(na * nb, dtype=torch.float64, device=dev)
    reach2 = float(Ea[-1]) + (float(Eb[-1]) if case["mode"] == "sigpi" else 0.0)
    step = max(1, (1 << 26) // xj.shape[0])
    for a in range(0, x1.shape[0], step):
        b = min(a + step, x1.shape[0])
        j0 = a if auto else 0
        s2 = torch.zeros(b - a, xj.shape[0] - j0, dtype=torch.float64, device=dev)
        for k in range(3):
            d = xj[None, j0:, k] - x1[a:b, None, k]
            if periodic:
                d = torch.where(d > 0.5 * L, d - L, torch.where(d < -0.5 * L, d + L, d))
            s2 += d * d
        near = s2 < reach2 * (1.0 + 1e-9)
        if auto:
            near &= torch.ones_like(near).triu_(1)
        i, j = near.nonzero(as_tuple=True)
        s2 = s2[i, j]
        i, j = i + a, j + j0
        ia = torch.bucketize(s2, Ea, right=True) - 1
        ok = (ia >= 0) & (ia < na)
        idx = ia
        if case["mode"] != "s":
            d = xj[j] - x1[i]
            if periodic:
                d = torch.where(d > 0.5 * L, d - L, torch.where(d < -0.5 * L, d + L, d))
            if case["los"] == "z":
                p2 = d[:, 2] * d[:, 2]
            else:
                l = x1[i] + xj[j]
                p2 = (d * l).sum(1) ** 2 / (l * l).sum(1)
            if case["mode"] == "smu":
                ib = (torch.bucketize(p2 / s2, Eb, right=True) - 1).clamp(0, nb - 1)
            else:
                ia = torch.bucketize((s2 - p2).clamp(min=0.0), Ea, right=True) - 1
                ib = torch.bucketize(p2, Eb, right=True) - 1
                ok = (ia >= 0) & (ia < na) & (ib >= 0) & (ib < nb)
            idx = ia * nb + ib
        idx = idx[ok]
        counts += torch.bincount(idx, minlength=na * nb)
        if w1 is not None:
            p = (w1[i].double() * wj[j].double())[ok]
            sums += torch.bincount(idx, weights=p, minlength=na * nb)
    return counts.cpu().numpy(), sums.cpu().numpy() if w1 is not None else None


def exact(case, seed):
    if case["call"] in ("batch", "tree_batch"):
        pairs = case["mocks"] * 0.5 * case["n2"] ** 2
    else:
        pairs = case["n"] * float(case["n2"]) if case["n2"] else 0.5 * case["n"] ** 2
    if pairs > 2.0e11:      # brute force over more would take over 20 seconds
        return None
    cats = _catalogues(case, seed)
    ea, eb = _edges(case)
    if case["call"] in ("batch", "tree_batch"):
        return [np.concatenate([_histogram(case, x, None, None, None, ea, eb)[0] for x, _ in cats])]
    x1, w1 = cats[0]
    x2, w2 = cats[1] if len(cats) > 1 else (None, None)
    c, w = _histogram(case, x1, w1, x2, w2, ea, eb)
    return [c, w] if case["weights"] != "none" else [c]
