"""The adjoint steps FP32 lattices on tiles and kernels of its own: between plain steps of one context
(rows that are cut into wide and into narrow tiles, 2D and 3D, periodic and walled, with and without
particles) it leaves the forces of its last forward step, the lists and the state as an FP64 context
has them, with the tolerances of the parity protocol (forces 1e-4, gradient 1e-3)."""
import numpy as np
import pytest

import paper_1901_09745_gb300 as P
from parity_utils import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,n,bc", [(19, (128, 20, 18), (0, 0, 1)), (19, (198, 11, 12), (0, 0, 0)),
                                          (19, (40, 20, 18), (1, 0, 0)), (9, (97, 40, 1), (0, 1, 0))])
@pytest.mark.parametrize("count", [0, 5, 40])
def test_adjoint_between_steps(lattice, n, bc, count):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    rng = np.random.default_rng(4)
    dim = 2 if lattice == 9 else 3
    X = np.zeros((count, 3))
    X[:, :dim] = rng.uniform(0, 1, (count, dim)) * np.array(n[:dim])
    zero, r = np.zeros((count, 3)), rng.uniform(1.5, 2.4, count)

    def run(storage):
        ctx = P.lbm_create(lattice, *n, bc=bc, tau=0.7, body_force=(1e-5, 2e-6, 0.0), storage=storage, tile_cap=64)
        if count:
            P.lbm_set_particles(ctx, X, zero, zero, r)
        out = []
        P.lbm_step(ctx, 3)
        for _ in range(2):
            J, dX, dF = P.lbm_adjoint_drag(ctx, 5, 2)
            F = np.array(P.lbm_get_forces(ctx)[0]) if count else np.zeros((0, 3))
            P.lbm_step(ctx, 3)
            G = np.array(P.lbm_get_forces(ctx)[0]) if count else np.zeros((0, 3))
            out.append((np.array([J]), np.array(dF), np.array(dX), F, G, np.array(P.lbm_get_macro(ctx)[1])))
        P.lbm_destroy(ctx)
        return out

    for a, b in zip(run("f32"), run("f64")):
        if count:
            assert rel_l2(a[0], b[0]) <= 1e-3 and rel_l2(a[1], b[1]) <= 1e-3 and rel_l2(a[2], b[2]) <= 1e-3
            assert rel_l2(a[3], b[3]) <= 1e-4 and rel_l2(a[4], b[4]) <= 1e-4
        assert rel_l2(a[5], b[5]) <= 1e-5
