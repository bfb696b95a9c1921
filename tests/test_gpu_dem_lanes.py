"""Spheres share eight lanes of the DEM sub-step each, or two where there are many. The order of the
sums does not depend on it: a bed of spheres on a wall (more contacts than two lanes take in a pass,
walls on one to three axes) moves by the same bits alone and beside 50000 spheres far from it."""
import numpy as np
import pytest

import paper_1901_09745_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [(0, 0, 1), (1, 0, 1), (1, 1, 1)])
@pytest.mark.parametrize("adhesive", [0, 1])
def test_same_bits_with_two_and_eight_lanes(walls, adhesive):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    rng = np.random.default_rng(2)
    n = (192, 192, 160)
    k = np.arange(343)
    # close enough that diagonal neighbours touch, too
    X = np.stack([1.4 + 2.4 * (k % 7), 1.4 + 2.4 * (k // 7 % 7), 1.4 + 2.4 * (k // 49)], 1) + rng.uniform(-0.1, 0.1, (343, 3))
    U, Om, r = rng.normal(0, 1e-3, (343, 3)), rng.normal(0, 1e-3, (343, 3)), rng.uniform(1.5, 1.95, 343)
    m = np.arange(50000)
    far = np.stack([40 + 2.5 * (m % 50), 40 + 2.5 * (m // 50 % 50), 40 + 2.5 * (m // 2500)], 1)

    def run(X, U, Om, r):
        ctx = P.lbm_create(19, *n, bc=walls, storage="f16")
        P.lbm_set_particles(ctx, X, U, Om, r)
        dem = P.dem_create(ctx, dt_dem=0.05, adhesive=adhesive, E=20.0, poisson=0.3, gamma=2e-3, density=3.0, skin=0.5)
        P.dem_step(dem, 3)
        P.dem_step(dem, 4)
        out = [np.array(v)[:343] for v in P.dem_get_particles(dem)]
        P.dem_destroy(dem)
        P.lbm_destroy(ctx)
        return out

    alone = run(X, U, Om, r)
    many = run(np.concatenate([X, far]), np.concatenate([U, np.zeros_like(far)]), np.concatenate([Om, np.zeros_like(far)]),
               np.concatenate([r, np.full(50000, 1.0)]))
    for a, b in zip(alone, many):
        assert np.array_equal(a, b)
    assert not np.array_equal(alone[1], U)
