"""The step's kernels at the edges of their tiles and dispatch: row lengths around the tile widths
(32 and 64 cells), even and odd, one tile, rows shorter than a tile, periodic and walled x, moving
and fixed particles (which take different visits), more candidates than a lane keeps fractions of,
against the FP64 oracle with the parity protocol's tolerances; and the same rows stepped by the
kernel without particles and by the one with, bit for bit."""
import numpy as np
import pytest

from parity_utils import compare, perturbed_state, run_gpu, run_oracle

import paper_1901_09745_gb300 as P

pytestmark = pytest.mark.gpu


def case(lattice, n, bc, moving, count=4, seed=5):
    rng = np.random.default_rng(seed)
    dim = 2 if lattice == 9 else 3
    X = np.zeros((count, 3))
    X[:, :dim] = rng.uniform(0, 1, (count, dim)) * np.array(n[:dim])
    r = rng.uniform(1.5, 2.4, count)
    U, Om = np.zeros((count, 3)), np.zeros((count, 3))
    if moving:
        U[:, :dim] = rng.normal(0, 2e-3, (count, dim))
        Om[:, (2 if dim == 2 else 0):] = rng.normal(0, 5e-4, (count, 1 if dim == 2 else 3))
    return dict(lattice=lattice, n=n, bc=bc, tau=0.7, body_force=(1e-5, 2e-6, 0.0), X=X, U=U, Om=Om, r=r, psc=0)


SHAPES = [(9, (w, 19, 1), (bx, 1 - bx, 0)) for w in (11, 31, 32, 33, 64, 65, 130) for bx in (0, 1)]
SHAPES += [(19, (w, 11, 9), (bx, 0, 1 - bx)) for w in (11, 32, 63, 64, 65, 66, 130) for bx in (0, 1)]
SHAPES += [(19, (w, 11, 9), (bx, 0, 1 - bx)) for w in (97, 127, 128, 198) for bx in (0, 1)]     # wide tiles


@pytest.mark.parametrize("lattice,n,bc", SHAPES)
@pytest.mark.parametrize("moving", [False, True])
def test_row_lengths(lattice, n, bc, moving):
    c = case(lattice, n, bc, moving)
    f0 = perturbed_state(c, 3)
    e = compare(run_gpu(P, c, f0, 4), run_oracle(c, f0, 4), 2 if lattice == 9 else 3)
    assert e["u"] <= 1e-5 and e["rho"] <= 1e-5 and e["F"] <= 1e-4 and e["T"] <= 1e-4, e


@pytest.mark.parametrize("lattice,n", [(9, (32, 24, 1)), (19, (64, 12, 8))])
@pytest.mark.parametrize("count", [9, 31, 40])
def test_many_candidates(lattice, n, count):
    """More candidates in a tile than fractions are kept (4) or than a tile may have here (32)."""
    c = case(lattice, n, (0, 0, 0), True, count=count)
    f0 = perturbed_state(c, 4)
    for storage, tol in (("f32", (1e-5, 1e-4)), ("f64", (1e-10, 1e-10))):
        e = compare(run_gpu(P, c, f0, 2, storage=storage), run_oracle(c, f0, 2), 2 if lattice == 9 else 3)
        assert e["u"] <= tol[0] and e["rho"] <= tol[0] and e["F"] <= tol[1] and e["T"] <= tol[1], (storage, e)


@pytest.mark.parametrize("lattice,n,bc", [(9, (160, 40, 1), (0, 1, 0)), (9, (97, 40, 1), (0, 0, 0)),
                                          (19, (128, 20, 18), (0, 0, 1)), (19, (65, 20, 18), (0, 0, 0))])
@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_same_bits_with_and_without_particles(lattice, n, bc, storage):
    c = case(lattice, n, bc, False, count=1)
    c["X"][0, : 2 if lattice == 9 else 3] = 6.0
    f0 = perturbed_state(c, 7)
    a = run_gpu(P, c, f0, 1, storage=storage)["f"]
    b = run_gpu(P, dict(c, X=c["X"][:0], U=c["U"][:0], Om=c["Om"][:0], r=c["r"][:0]), f0, 1, storage=storage)["f"]
    same = a == b
    same[:, :16, :16, :16] = True            # the particle and what streamed out of it
    assert same.all(), np.argwhere(~same)[:5]
