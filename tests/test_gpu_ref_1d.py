"""Several steps per launch of short FP64 1D lattices: launches split at due
diagnostics against the oracle, and velocities whose square leaves the range
of doubles against the step of one launch, bit for bit."""
import numpy as np
import pytest

import lbm_inputs
import oracle
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu

PER, WALL, INLET, OUTLET = 0, 1, 2, 3


def _pair(n, p, f):
    o = oracle.Oracle("D1Q3", (n, 1, 1), p, threads=4)
    o.init(**f)
    s = lbm.Simulation("D1Q3", (n,), dict(p, precision="fp64"))
    s.init(**f)
    return s, o


@pytest.mark.parametrize("n, case", [(300, "walls"), (512, "periodic"), (203, "tube"), (2433, "walls")])
@pytest.mark.parametrize("diag_every, n_gamma", [(1, 3), (5, 1), (9, 4), (13, 2)])
def test_steps_split_at_diagnostics(n, case, diag_every, n_gamma):
    bc = {"walls": (WALL, WALL), "periodic": (PER, PER), "tube": (INLET, OUTLET)}[case]
    p = dict(R=30.0, omega_g=0.6, omega_l=1.2, omega_alpha=1.7, drag_model=1, kappa_I=1e-3, kappa_W=1e-3, psi_g=0.1,
             psi_l=0.2, g_hat=1e-6, g_axis=0, gamma=0.5, n_gamma=n_gamma, spalding_mode=2, bc_lo=(bc[0], 0, 0),
             bc_hi=(bc[1], 0, 0), in_alpha=(0.3, 0.5), in_ug=(1e-3, 5e-3), in_ul=(0.0, 1e-3), ramp_nt=20,
             diag_every=diag_every)
    f = lbm_inputs.fields_random(1, (n,), seed=n, alpha=(0.2, 0.6), u_amp=1e-3, pk_amp=1e-6)
    s, o = _pair(n, p, f)
    for steps in (1, 8, 3, 30, 41):
        o.step(steps)
        s.step(steps)
        got, ref = s.moments(), o.moments()
        for k in ("alpha_g", "u_g", "u_l", "p_k", "S_g", "S_l"):
            assert np.array_equal(got[k], np.asarray(ref[k]).reshape(got[k].shape)), (k, s.t)
        d = s.diag()
        pops = [np.asarray(o.pops(sch)).reshape(3, -1) for sch in range(4)]
        assert d[0] == pytest.approx(pops[2].sum(), rel=1e-13 * n) and d[1] == pytest.approx(pops[3].sum(), rel=1e-13 * n)
        assert d[2] == pytest.approx(ref["alpha_g"].sum(), rel=1e-13 * n)
        u = max(np.abs(ref["u_g"]).max(), np.abs(ref["u_l"]).max())
        assert d[4] == pytest.approx(u, rel=1e-15) and d[5] == 0


@pytest.mark.parametrize("phase", ["u_g", "u_l"])
@pytest.mark.parametrize("exponent", [480, 488, 499, 500, 503, 506, 509, 511])
@pytest.mark.parametrize("kappa", [0.0, 1e-3])
def test_overflowing_velocities(phase, exponent, kappa):
    """One phase starts at velocities of 2^exponent: within a few steps they
    pass 2^512 and 2^1000, where u u is infinite and the formulas' |u| =
    sqrt(u u) with it.  The short lattice's populations, the non-finite ones
    among them, are those of the step of one launch, which a periodic lattice
    of 100 copies of it takes, being too long for the other."""
    n, copies = 64, 100
    p = dict(R=30.0, omega_g=0.6, omega_l=1.2, omega_alpha=1.7, drag_model=0, kappa_I=kappa, kappa_W=kappa, g_hat=0.0,
             g_axis=0, gamma=0.0, n_gamma=1, spalding_mode=2, bc_lo=(PER, 0, 0), bc_hi=(PER, 0, 0), precision="fp64")
    f = lbm_inputs.fields_random(1, (n,), seed=1, alpha=(0.2, 0.6), u_amp=1e-3, pk_amp=1e-6)
    # different sizes from node to node, and nodes at rest among them
    f[phase] = np.ldexp(1.0 + np.arange(n) % 7 / 8.0, exponent)[None, :] * (np.arange(n) % 5 != 0)
    short, long = lbm.Simulation("D1Q3", (n,), p), lbm.Simulation("D1Q3", (n * copies,), p)
    short.init(**f)
    long.init(**{k: np.ascontiguousarray(np.tile(v, copies)) for k, v in f.items()})
    seen = set()
    for t in range(6):
        for sch in range(6):
            a, b = short.populations(sch), long.populations(sch)
            assert np.array_equal(np.tile(a, (1, copies)), b, equal_nan=True), (sch, t)
            seen.add(bool(np.isfinite(a).all()))
        short.step(1)
        long.step(1)
    assert seen == {True, False}
