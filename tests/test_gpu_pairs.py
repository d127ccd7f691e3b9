"""The FP32 step of D2Q9 and D3Q19 with the two phases in packed pairs
(lbm_pairs.cuh): against the FP64 oracle at the 1e-5 bar of the FP32 path, on
sizes where warps are full, ragged and split between interior and face nodes,
and bitwise the same over tiles (interior and general path)."""
import numpy as np
import pytest

import lbm_inputs
import oracle
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu

P = dict(R=100.0, omega_g=0.6, omega_l=1.5, omega_alpha=1.5, drag_model=1, kappa_I=2e-4, kappa_W=1e-4, g_hat=1e-8,
         gamma=1.0, n_gamma=4, psi_g=0.1, psi_l=0.05)


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("lat, dims, bc", [
    ("D2Q9", (1, 5), ((0, 1), (0, 1))), ("D2Q9", (64, 2), ((0, 0), (0, 0))), ("D2Q9", (130, 9), ((1, 0), (1, 0))),
    ("D2Q9", (65, 34), ((0, 2), (0, 3))), ("D3Q19", (16, 8, 1), ((0, 0, 0), (0, 0, 0))),
    ("D3Q19", (33, 9, 5), ((1, 1, 0), (1, 1, 0))), ("D3Q19", (17, 10, 6), ((0, 1, 2), (0, 1, 3)))])
def test_paired_fp32_step(lat, dims, bc, mode):
    D = len(dims)
    lo, hi = (tuple(v) + (0,) * (3 - D) for v in bc)
    p = dict(P, g_axis=D - 1, spalding_mode=mode, bc_lo=lo, bc_hi=hi, inlet_lo=3, inlet_hi=12, in_alpha=(0.1, 0.3),
             in_ug=(1e-3, 3e-3), in_ul=(0.0, 2e-4), ramp_nt=10)
    f = lbm_inputs.fields_random(D, dims, seed=5, alpha=(0.1, 0.6), u_amp=2e-3, pk_amp=1e-5)
    o = oracle.Oracle(lat, tuple(dims) + (1,) * (3 - D), p, threads=4)
    o.init(**f)
    o.step(9)
    ref = o.moments()
    runs = []
    for tile in ((64, 2, 1), (32, 1, 1)) if D == 2 and 2 not in lo else (None,) if D == 2 else (None, (8, 4, 2)):
        s = lbm.Simulation(lat, dims, dict(p, precision="fp32"))
        if tile:
            s.set_tile(*tile)
        s.init(**f)
        s.step(9)
        runs.append(s.moments())
        s.close()
    for k in ("alpha_g", "u_g", "u_l", "p_k"):
        a, b = runs[0][k].reshape(-1), np.asarray(ref[k]).reshape(-1)
        scale = max(np.linalg.norm(b), np.linalg.norm(ref["u_g"]) / p["R"] if k == "u_l" else 0.0)
        assert np.linalg.norm(a - b) <= 1e-5 * scale, k
        assert all(np.array_equal(r[k], runs[0][k]) for r in runs[1:]), k
