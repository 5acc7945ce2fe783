"""Where the normals of an FP32 step lie about the generator's definition.

One step from rest leaves f* = w + (response of the collision to the normals), so the normals the GPU
used follow from the populations by the oracle's collision, which is linear in them. Each Box-Muller pair
is then a vector whose angle is compared with the oracle's. The definition takes the middle of the 2^9
words that share their top 23 bits; an angle formed from the whole word is off by up to half that
interval, 2 pi 2^-24 = 3.7e-7, to either side, and by nothing on average. An angle that is taken from an
interval's end is off by half an interval on average. The bound is a quarter of that; the roundings of
the populations (2^-24 of each, as often up as down) average out over more than 10^4 pairs.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOUND = 0.25 * 2.0 * np.pi * 2.0 ** -24


@pytest.fixture(scope="module")
def fl():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_16486_gb300 as fl

    return fl


@pytest.mark.parametrize("lattice,dims", [(0, (64, 64, 1)), (1, (16, 16, 16)), (3, (15, 16, 17))])
@pytest.mark.parametrize("variant", [1, 5])
def test_angles_lie_about_the_definition(fl, oracle_mod, lattice, dims, variant):
    q, first = ((9, 3), (27, 4), (27, 4), (19, 4))[lattice]
    lam, kbt, seed = np.ones(q), 1e-4, 91
    c, w, _ = oracle_mod.tables(lattice)
    with fl.Lattice(lattice, dims, lam, kbt, 1.0, seed) as lat:
        lat.variant = variant
        lat.step(1)
        f = lat.populations().reshape(q, dims[2], dims[1], dims[0])
    star = np.stack([np.roll(f[i], (-c[i, 2], -c[i, 1], -c[i, 0]), (0, 1, 2)).ravel() - w[i] for i in range(q)])
    base = oracle_mod.collide_site(lattice, w, lam, kbt, np.zeros(q))[0]
    response = np.stack([oracle_mod.collide_site(lattice, w, lam, kbt, np.eye(q)[v])[0] - base
                         for v in range(first, q)], 1)
    got = np.linalg.lstsq(response, star - (base - w)[:, None], rcond=None)[0]
    want = np.stack([oracle_mod.site_eta(lattice, seed, 0, s)[first:] for s in range(star.shape[1])], 1)
    pairs = (q - first) // 2
    a, b = want[0:2 * pairs:2] + 1j * want[1:2 * pairs:2], got[0:2 * pairs:2] + 1j * got[1:2 * pairs:2]
    turn = (np.conj(a) * b).sum()
    assert abs(np.angle(turn)) <= BOUND, (np.angle(turn), BOUND)
