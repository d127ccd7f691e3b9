"""Graph replay of the FP64 reference step (lattices that launch every step):
the fields are bitwise those of plain launches and of the oracle, over whole
periods and ragged remainders, and the diagnostics agree, taken once per
replayed period."""
import numpy as np
import pytest

import lbm_inputs
import oracle
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu

BASE = dict(R=1000.0, omega_g=0.6, omega_l=120.0 / 67.0, omega_alpha=1.5, drag_model=1, kappa_I=2.4e-4,
            g_hat=1e-6 / 999.0, gamma=1.0, n_gamma=7, spalding_mode=2)


@pytest.mark.parametrize("lat, dims, p", [
    ("D2Q9", (70, 37), dict(g_axis=1, bc_lo=(0, 1, 0), bc_hi=(0, 1, 0), diag_every=20)),
    ("D2Q9", (33, 30), dict(R=20.0, drag_model=0, kappa_I=1e-2, kappa_W=2e-3, g_axis=1, g_hat=1e-5, spalding_mode=1,
                            n_gamma=1, bc_lo=(1, 1, 0), bc_hi=(1, 3, 0), diag_every=0)),
    ("D1Q3", (6000,), dict(g_axis=0, kappa_W=2.4e-4, bc_lo=(1, 0, 0), bc_hi=(1, 0, 0), diag_every=35)),
    ("D1Q3", (4257,), dict(g_axis=0, bc_lo=(0, 0, 0), bc_hi=(0, 0, 0), diag_every=0)),
    ("D3Q19", (12, 10, 11), dict(g_axis=2, bc_lo=(1, 0, 1), bc_hi=(1, 0, 1), diag_every=6))])
def test_fp64_graph_replay_is_bitwise_plain_launches(lat, dims, p):
    D = lbm.LATTICE[lat]
    long = 280 if p["diag_every"] == 20 else 150  # (periods of 140, 2, 70, 14 and 42 steps)
    f = lbm_inputs.fields_random(D, dims, seed=9, alpha=(0.05, 0.6), u_amp=2e-3, pk_amp=1e-5)
    runs = []
    for graph in (True, False):
        s = lbm.Simulation(lat, dims, {**BASE, **p, "precision": "fp64"})
        s.set_graph(graph)
        s.init(**f)
        for n in (1, 3, long, 29):
            s.step(n)
        runs.append((s.moments(), s.diag(), s.launches, s.t))
    (mg, dg, lg, tg), (mp, dp, lp, tp) = runs
    assert tg == tp == 33 + long
    # (a launch per step, at the least)
    assert lp >= tp and (lg == lp if p["diag_every"] == 0 else tp <= lg < lp)
    po = {k: v for k, v in {**BASE, **p}.items() if k != "diag_every"}
    o = oracle.Oracle(lat, tuple(dims) + (1,) * (3 - D), po, threads=8)
    o.init(**f)
    o.step(tp)
    ref = o.moments()
    for k in mg:
        assert np.isfinite(mg[k]).all() and np.array_equal(mg[k], mp[k]), k
        assert np.array_equal(mg[k], np.asarray(ref[k]).reshape(mg[k].shape)), k
    assert np.array_equal(dg, dp)
