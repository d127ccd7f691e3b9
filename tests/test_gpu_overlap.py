"""Steps launched while the step before still runs (programmatic dependent
launch) against steps taken one at a time with the GPU idle in between: the
same bits, over hundreds of steps of lattices of several waves of blocks, from
plain launches and from graph replay, for every store and for the batch."""
import numpy as np
import pytest

import lbm_inputs
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu

BASE = dict(R=1000.0, omega_g=0.6, omega_l=120.0 / 67.0, omega_alpha=1.5, drag_model=1, kappa_I=2.4e-4,
            g_hat=1e-6 / 999.0, gamma=1.0, n_gamma=7, spalding_mode=2)
WALLS2 = dict(g_axis=1, bc_lo=(0, 1, 0), bc_hi=(0, 1, 0))
STRIP2 = dict(g_axis=1, bc_lo=(0, 2, 0), bc_hi=(0, 1, 0), inlet_lo=40, inlet_hi=90, in_alpha=(0.01, 0.3),
              in_ug=(4.3e-4, 4.3e-3), ramp_nt=60, inlet_ul_mode=1)
WALLS3 = dict(g_axis=2, bc_lo=(1, 1, 0), bc_hi=(1, 1, 0))


def _fields(D, dims, seed=4):
    return lbm_inputs.fields_random(D, dims, seed=seed, alpha=(0.05, 0.6), u_amp=2e-3, pk_amp=1e-5)


@pytest.mark.parametrize("lat, dims, prec, p, steps", [
    ("D2Q9", (256, 1024), "fp32", WALLS2, 200), ("D2Q9", (256, 1024), "fp16dev", WALLS2, 200),
    ("D2Q9", (256, 1024), "fp16ab", WALLS2, 200), ("D2Q9", (131, 513), "fp32", STRIP2, 200),
    ("D2Q9", (131, 513), "fp16ab", STRIP2, 200), ("D2Q9", (256, 512), "fp64dev", WALLS2, 60),
    ("D2Q9", (256, 512), "fp32", dict(WALLS2, beta_stencil=1), 200),
    ("D2Q9", (256, 512), "fp16dev", dict(WALLS2, beta_stencil=1), 200),
    ("D3Q19", (65, 63, 64), "fp32", WALLS3, 100), ("D3Q19", (65, 63, 64), "fp16dev", WALLS3, 100),
    ("D3Q19", (65, 63, 64), "fp16ab", WALLS3, 100), ("D1Q3", (40000,), "fp32", dict(g_axis=0, bc_lo=(1, 0, 0), bc_hi=(1, 0, 0)), 200),
])
def test_overlapped_steps_are_bitwise_serial_steps(lat, dims, prec, p, steps):
    import torch
    f = _fields(lbm.LATTICE[lat], dims)
    runs = []
    for graph, serial in ((False, True), (False, False), (True, False)):
        s = lbm.Simulation(lat, dims, dict(BASE, precision=prec, **p))
        s.set_graph(graph)
        s.init(**f)
        for _ in range(steps if serial else 1):
            s.step(1 if serial else steps)
            if serial:
                torch.cuda.synchronize()
        runs.append(s.moments())
        s.close()
    for k in runs[0]:
        assert np.isfinite(runs[0][k]).all(), k
        for r in runs[1:]:
            assert np.array_equal(r[k], runs[0][k]), k


@pytest.mark.parametrize("prec", ["fp32", "fp16dev"])
def test_overlapped_batch_steps_are_bitwise_serial_steps(prec):
    import torch
    dims = [(257, 300), (64, 256), (190, 411)]
    params = [dict(BASE, precision=prec, **WALLS2) for _ in dims]
    runs = []
    for graph, serial in ((False, True), (False, False), (True, False)):
        b = lbm.Batch("D2Q9", dims, params)
        b.set_graph(graph)
        for i, d in enumerate(dims):
            b.init(i, **_fields(2, d, seed=10 + i))
        for _ in range(200 if serial else 1):
            b.step(1 if serial else 200)
            if serial:
                torch.cuda.synchronize()
        runs.append([b.moments(i) for i in range(len(dims))])
        b.close()
    for i in range(len(dims)):
        for k in runs[0][i]:
            assert np.isfinite(runs[0][i][k]).all(), (i, k)
            for r in runs[1:]:
                assert np.array_equal(r[i][k], runs[0][i][k]), (i, k)
