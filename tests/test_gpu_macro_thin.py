"""Velocity of cells whose density is far from 1 (0.016 to 60): as close to the quotient of the exact
moments as a division in FP64 is. The populations' deviations lie within a factor of 2^8 of each other, so
that the kernel's split sums are exact, and what is left is the rounding of the density, of the momentum
with half the body force, and of the quotient: at most 2^-53 of the result each, with one more
2^-53 for what the corrected quotient may miss."""
from fractions import Fraction

import numpy as np
import pytest

import paper_1901_09745_gb300 as P
from test_gpu_macro import pull, stored

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,n", [(9, (33, 9, 1)), (19, (34, 9, 3)), (19, (97, 5, 3))])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("density", [0.0165, 0.02, 0.05, 0.1, 0.3, 3.0, 10.0, 28.0, 50.0])
def test_velocity(lattice, n, storage, density):
    if storage == "f16" and density > 30:
        pytest.skip("beyond the storage format's range")
    F = (1e-4, -3e-5, 0.0)
    ctx = P.lbm_create(lattice, *n, tau=0.8, body_force=F, storage=storage)
    w = P.lbm_lattice_tables(lattice)[1][:, None, None, None]
    rng = np.random.default_rng(7)
    f = density * w * (1 + rng.uniform(-0.04, 0.04, (lattice,) + n[::-1]))
    P.lbm_set_populations(ctx, f)
    u = P.lbm_get_macro(ctx)[1].reshape(-1, 3)
    e, d = pull(ctx, stored(ctx, storage), (0, 0, 0))
    d = d.reshape(lattice, -1)
    assert np.abs(d).max() < 256 * np.abs(d).min()
    Ff = [Fraction(float(np.float32(v))) for v in F]
    for c in range(d.shape[1]):
        v = [Fraction(float(x)) for x in d[:, c]]
        rho = 1 + sum(v)
        for a in range(2 if lattice == 9 else 3):
            want = (sum(int(e[i][a]) * v[i] for i in range(lattice)) + Ff[a] / 2) / rho
            assert abs(Fraction(float(u[c, a])) - want) <= abs(want) * 4 / 2**53, (c, a, float(rho), float(want), u[c, a])
