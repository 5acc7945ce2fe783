"""Small boxes on a device (or a part of one) that cannot place the one-launch form's blocks together: the
steps are launched one by one, with the same result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fl():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_16486_gb300 as fl

    return fl


@pytest.mark.parametrize("lattice,dims", [(0, (64, 64, 1)), (1, (11, 12, 13)), (2, (8, 8, 8)), (3, (9, 5, 7))])
@pytest.mark.parametrize("kbt", [1e-4, 0.0])
def test_steps_without_the_one_launch_form(fl, lattice, dims, kbt):
    q = (9, 27, 27, 19)[lattice]
    lam = np.ones(q)
    lam[[4, 5] if lattice == 0 else [7, 8, 9]] = 1.6
    out = []
    for refused in (False, True):
        with fl.Lattice(lattice, dims, lam, kbt, 1.0, 5) as lat:
            fl.flbm_test_cluster_refused(lat.ctx, refused)
            lat.init_uniform((0.03, 0.01, 0.0), 1e-3, 2)
            lat.step(21)
            lat.step(12)
            assert lat.step_count == 33
            out.append(lat.populations())
    assert np.array_equal(out[0], out[1])
