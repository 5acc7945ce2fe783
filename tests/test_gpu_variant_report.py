"""flbm_get_step_variant: what it reports, set again, is what was there (no other kernel is launched)."""
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


@pytest.mark.parametrize("lattice,dims,storage,default", [
    (0, (64, 64, 1), 0, 7), (0, (65, 63, 1), 0, 7), (0, (64, 130, 1), 0, 5), (0, (64, 64, 1), 1, 5),
    (1, (25, 10, 8), 0, 7), (1, (25, 50, 10), 0, 5), (1, (64, 9, 8), 0, 5), (2, (9, 9, 9), 2, 5), (3, (8, 8, 8), 0, 7)])
def test_reported_variant_is_the_choice(fl, lattice, dims, storage, default):
    q = (9, 27, 27, 19)[lattice]
    with fl.Lattice(lattice, dims, np.ones(q), 1e-4, 1.0, 1, storage) as lat:
        assert lat.variant == default
        for v in range(1, 9):
            lat.variant = v
            assert lat.variant == v
        lat.variant = 0
        assert lat.variant == default
        chosen = lat.autotune(4)
        assert lat.variant == chosen


def test_raw_collision_reports_the_choice(fl):
    with fl.Lattice(1, (64, 9, 8), np.ones(27), 1e-4, 1.0, 1) as lat:
        lat.collision = fl.FLBM_COLLISION_RAW
        assert lat.variant == 5
        lat.variant = 5
        assert lat.variant == 5
