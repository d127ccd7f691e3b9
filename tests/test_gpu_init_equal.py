"""The same initial fields from the host and from the device give the same
lattice, bit for bit, in every store: alpha_g is summed (the deviation
reference) in one order whatever the side it comes from."""
import numpy as np
import pytest

import lbm_inputs
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat, dims", [("D1Q3", (777,)), ("D2Q9", (16, 16)), ("D2Q9", (257, 1)), ("D2Q9", (300, 1000)),
                                       ("D2Q9", (1030, 513)), ("D3Q19", (33, 21, 40))])
@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "fp16ab", "fp64dev", "fp64"])
def test_host_and_device_fields_give_the_same_lattice(lat, dims, precision):
    import torch
    D = lbm.LATTICE[lat]
    f = lbm_inputs.fields_random(D, dims, seed=6, alpha=(0.05, 0.6), u_amp=2e-3, pk_amp=1e-5)
    dev = {k: torch.tensor(v, device="cuda") for k, v in f.items()}
    p = dict(R=10.0, omega_g=0.6, omega_l=1.2, precision=precision)
    a, b = lbm.Simulation(lat, dims, p), lbm.Simulation(lat, dims, p)
    a.init(**f)
    b.init(**dev)
    for sch in range(6):
        assert np.array_equal(a.populations(sch), b.populations(sch)), sch
    a.step(20)
    b.step(20)
    ma, mb = a.moments(), b.moments()
    for k in ma:
        assert np.isfinite(ma[k]).all() and np.array_equal(ma[k], mb[k]), k


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_bad_host_alpha_is_reported_and_changes_nothing(precision):
    dims = (300, 200)
    f = lbm_inputs.fields_random(2, dims, seed=2, alpha=(0.0, 1.0))
    s = lbm.Simulation("D2Q9", dims, dict(R=10.0, precision=precision))
    s.init(**f)
    s.step(3)
    before = s.moments()
    n = dims[0] * dims[1]
    bad = {k: v.copy() for k, v in f.items()}
    for i, v in ((n - 1, 1.5), (n // 2, -1e-3), (7, float("inf")), (0, float("nan"))):
        bad["alpha_g"][i] = v
        with pytest.raises(lbm.LBMError, match=r"alpha_g\[%d\]" % i):
            s.init(**bad)
    after = s.moments()
    assert s.t == 3 and all(np.array_equal(before[k], after[k]) for k in before)
