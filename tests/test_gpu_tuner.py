"""The tuners time each option once: no two trials run the same code on the same
structure, where noise would decide between them."""

import numpy as np
import pytest

P = pytest.importorskip("paper_2301_12557_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weights", [False, True])
def test_no_option_is_timed_twice(weights):
    rng = np.random.default_rng(8)
    x, L = rng.random((20_000, 3)) * 100.0, 100.0
    w = (0.5 + rng.random(x.shape[0])).astype(np.float32) if weights else None
    box, bins = P.make_box(L, True), P.Bins("s", "z", np.linspace(0.0, 20.0, 21))
    opts, trials = P.pc_tune(x, w, box=box, bins=bins)
    keys = [(c, ipt, priv if weights else 0) for c, ipt, priv, _ in trials]
    assert len(keys) == len(set(keys)) and (1 in [k[2] for k in keys]) == weights
    assert opts.rescue_capacity == 0 and (weights or opts.priv == 0)
    opts, cap, trials = P.pc_tune_tree(x, w, box=box, bins=bins)
    keys = [(c, ipt) for c, ipt, *_ in trials]
    assert len(keys) == len(set(keys)) and opts.rescue_capacity == 0
