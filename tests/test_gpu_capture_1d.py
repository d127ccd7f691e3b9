"""A caller's own capture of lbm_step on a short FP64 1D lattice (several steps
per launch, two copies of the store): once captured, a lattice's calls leave the
state where the capture read it, so a captured call can be replayed, between
plain calls too, whether the steps of a call divide by the steps of a launch or
not, and from whichever copy the capture started.  Against the same steps taken
by plain calls, bit for bit."""
import numpy as np
import pytest

import lbm_inputs
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu

PER, WALL, INLET, OUTLET = 0, 1, 2, 3
BC = {"walls": (WALL, WALL), "periodic": (PER, PER), "tube": (INLET, OUTLET)}


def _sim(n, case, n_gamma, stream=None):
    p = dict(R=30.0, omega_g=0.6, omega_l=1.2, omega_alpha=1.7, drag_model=0, kappa_I=1e-3, kappa_W=1e-3, g_hat=1e-6,
             g_axis=0, gamma=0.5, n_gamma=n_gamma, spalding_mode=2, bc_lo=(BC[case][0], 0, 0),
             bc_hi=(BC[case][1], 0, 0), in_alpha=(0.3, 0.3), in_ug=(1e-3, 1e-3), in_ul=(1e-4, 1e-4), ramp_nt=0)
    s = lbm.Simulation("D1Q3", (n,), dict(p, precision="fp64"))
    s.set_graph(False)
    if stream is not None:
        s.set_stream(stream)
    s.init(**lbm_inputs.fields_random(1, (n,), seed=n, alpha=(0.2, 0.5), u_amp=1e-3, pk_amp=1e-6))
    return s


@pytest.mark.parametrize("n, case", [(64, "walls"), (300, "periodic"), (201, "tube"), (512, "walls"), (3000, "walls"),
                                     (4257, "periodic")])
@pytest.mark.parametrize("before", [False, True])
@pytest.mark.parametrize("calls", [(2,), (1, 1), (6,), (7, 1), (10,), (200,), (3, 15)])
def test_captured_calls_replay(n, case, calls, before):
    import torch
    period = sum(calls)  # even, and a whole number of latches
    n_gamma = period if period in (2, 10, 200) else 2
    stream = torch.cuda.Stream()
    a, b = _sim(n, case, n_gamma, stream), _sim(n, case, n_gamma)
    a.step(period)
    if before:  # other numbers of launches before the capture
        for _ in range(period):
            a.step(1)
        a.step(period)
        a.step(period)
    stream.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for k in calls:
            a.step(k)
    with torch.cuda.stream(stream):
        for _ in range(3):
            g.replay()
        a.step(2 * period)  # plain steps between replays
        for _ in range(2):
            g.replay()
    stream.synchronize()
    b.step((1 + 3 * before) * period + 3 * period + 2 * period + 2 * period)
    ma, mb = a.moments(), b.moments()
    for k in mb:
        assert np.isfinite(mb[k]).all(), k
        assert np.array_equal(ma[k], mb[k]), k
