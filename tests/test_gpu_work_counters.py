"""The work counters that the step's kernel draws its tiles from are cleared by each step, in a
kernel before, and by no launch for its successor: whatever they hold before a call (here values far
above the number of tiles, with which no tile would be stepped), its state has the same bits. Both
launches of a coupled step, steps that bin and steps that keep their lists, with and without tiles that
overflow, replayed steps, the adjoint's FP64 steps, the step on a caller's buffers, and a lattice
without particles, which draws from none."""
import ctypes as C

import numpy as np
import pytest

import paper_1901_09745_gb300 as P
from parity_utils import perturbed_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


def fill(ctx, on):
    if on:
        lib = C.CDLL(P.library_path())
        lib.psc_test_fill_work.argtypes, lib.psc_test_fill_work.restype = [C.c_void_p, C.c_int], C.c_int
        assert lib.psc_test_fill_work(ctx.handle if ctx is not None else None, 1) == 0


def case(lattice, n, count):
    rng = np.random.default_rng(3)
    dim = 2 if lattice == 9 else 3
    X = np.zeros((count, 3))
    X[:, :dim] = rng.uniform(0, 1, (count, dim)) * np.array(n[:dim])
    U = np.zeros((count, 3))
    U[:, :dim] = rng.normal(0, 1e-3, (count, dim))
    return dict(lattice=lattice, n=n, bc=(0, 0, 0), tau=0.7, body_force=(1e-5, 0, 0), X=X, U=U, Om=np.zeros((count, 3)),
                r=rng.uniform(1.5, 2.4, count))


def create(c, storage, tile_cap=0):
    ctx = P.lbm_create(c["lattice"], *c["n"], bc=c["bc"], tau=c["tau"], body_force=c["body_force"], storage=storage,
                       tile_cap=tile_cap)
    P.lbm_set_populations(ctx, perturbed_state(c, 3))
    if len(c["r"]):
        P.lbm_set_particles(ctx, c["X"], c["U"], c["Om"], c["r"])
    return ctx


@pytest.mark.parametrize("lattice,n", [(9, (97, 40, 1)), (19, (128, 12, 10)), (19, (40, 12, 10))])
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("count,cap", [(0, 0), (3, 0), (40, 2)])
def test_steps(torch, lattice, n, storage, count, cap):
    def run(on):
        ctx = create(case(lattice, n, count), storage, cap)
        for _ in range(4):       # binned, kept lists, and both replayed
            fill(ctx, on)
            P.lbm_step(ctx, 1)
        out = P.lbm_get_populations(ctx).copy(), P.lbm_get_forces(ctx)[0].copy()
        P.lbm_destroy(ctx)
        return out

    (f, F), (g, G) = run(False), run(True)
    assert np.array_equal(f, g)
    assert np.allclose(F, G, rtol=1e-12, atol=1e-15)        # sums of atomic additions, FP64


def test_coupled_step(torch):
    def run(on):
        c = case(9, (160, 120, 1), 0)
        k = np.arange(12)
        c.update(X=np.stack([20.0 + 30 * (k % 4), 20.0 + 30 * (k // 4), 0 * k], 1), U=np.zeros((12, 3)),
                 Om=np.zeros((12, 3)), r=np.full(12, 4.0))
        ctx = create(c, "f32")
        dem = P.dem_create(ctx, dt_dem=0.1, E=2.0, poisson=0.3, gamma=2e-4, density=3.0)
        for _ in range(3):
            fill(ctx, on)
            P.lbm_coupled_step(ctx, dem, 1, 10)
        f = P.lbm_get_populations(ctx).copy()
        P.dem_destroy(dem)
        P.lbm_destroy(ctx)
        return f

    # (the discs' positions carry the rounding of atomic sums into the fractions)
    assert np.allclose(run(False), run(True), rtol=0, atol=1e-6 / 36)


def test_adjoint_f64(torch):
    def run(on):
        c = case(19, (34, 12, 10), 3)
        c["U"][:] = 0
        ctx = create(c, "f64")
        J, token = P.lbm_adjoint_forward(ctx, 5, 3)
        fill(ctx, on)
        dX, dF = P.lbm_adjoint_backward(ctx, token)
        P.lbm_destroy(ctx)
        return J, dX, dF

    for a, b in zip(run(False), run(True)):
        assert np.allclose(a, b, rtol=1e-10, atol=1e-14)


@pytest.mark.parametrize("lattice,n", [(9, (97, 40, 1)), (19, (128, 12, 10))])
@pytest.mark.parametrize("count", [0, 20])
def test_callers_buffers(torch, lattice, n, count):
    c = case(lattice, n, count)
    params = P.LbmParams()
    params.lattice, params.nx, params.ny, params.nz = lattice, *n
    params.tau, params.storage, params.stream = 0.7, P.LBM_F32, torch.cuda.current_stream().cuda_stream
    w = P.lbm_lattice_tables(lattice)[1]
    f = torch.as_tensor(perturbed_state(c, 3) - w[:, None, None, None], device="cuda").float().contiguous()
    particles = [torch.as_tensor(np.ascontiguousarray(c[k]), device="cuda") for k in ("X", "U", "Om", "r")]
    F, T = (torch.zeros((count, 3), dtype=torch.float64, device="cuda") for _ in range(2))
    args = particles + [F, T] if count else []
    want, got = torch.empty_like(f), torch.empty_like(f)
    P.lbm_psc_step_noalloc(params, f, want, *args)
    fill(None, True)
    P.lbm_psc_step_noalloc(params, f, got, *args)
    torch.cuda.synchronize()
    assert torch.equal(want, got) and not torch.equal(got, f)
