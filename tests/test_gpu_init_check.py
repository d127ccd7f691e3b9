"""lbm_init's check and sum of a device alpha_g: sizes about the check's blocks,
the first bad value reported wherever it lies, and the same lattice as from host
fields."""
import numpy as np
import pytest

import lbm_inputs
import paper_2409_10399_gb300 as lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 3), (16, 16), (257, 1), (300, 1000), (1030, 513)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_device_alpha_check(dims, precision):
    import torch
    f = lbm_inputs.fields_random(2, dims, seed=2, alpha=(0.0, 1.0))
    dev = {k: torch.tensor(v, device="cuda") for k, v in f.items()}
    p = dict(R=10.0, precision=precision)
    a, b = lbm.Simulation("D2Q9", dims, p), lbm.Simulation("D2Q9", dims, p)
    a.init(**f)
    b.init(**dev)
    a.step(3)
    b.step(3)
    ma, mb = a.moments(), b.moments()
    for k in ma:
        scale = np.abs(ma[k]).max()
        assert np.abs(ma[k] - mb[k]).max() <= (1e-6 if precision == "fp32" else 0.0) * scale, k
    n = dims[0] * dims[1]
    before = b.moments()
    for i, v in ((n - 1, 1.5), (n // 2, -1e-3), (0, float("nan"))):
        dev["alpha_g"][i] = v
        with pytest.raises(lbm.LBMError, match=r"alpha_g\[%d\]" % i):
            b.init(**dev)
    after = b.moments()
    assert all(np.array_equal(before[k], after[k]) for k in before)
