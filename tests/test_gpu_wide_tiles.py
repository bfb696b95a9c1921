"""FP32 lattices in 3D whose rows are cut into tiles 64 cells wide (positions in records count from the
tile's middle): tiles with 9 to 40 candidates (more than 32 take the exact path over all particles),
both schemes, a minimum image per cell along x, the field read-out, the step on a caller's buffers with
more than its 16 candidates, slabs, and all of it in the bounds-checked build. Against the FP64
oracle with the parity protocol's tolerances."""
import ctypes as C
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_1901_09745_gb300 as P
import test_gpu_macro as M
from parity_utils import compare, perturbed_state, ragged_case3d, rel_l2, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

TOL = dict(u=1e-5, rho=1e-5, F=1e-4, T=1e-4)


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return t


def check(case, steps, **kw):
    f0 = perturbed_state(case, 4)
    g = run_gpu(P, case, f0, steps, **kw)
    e = compare(g, run_oracle(case, f0, steps), 3)
    assert all(e[k] <= v for k, v in TOL.items() if k in e), e
    return g


def cluster(n, bc, count, x=(65.0, 95.0)):
    """count moving spheres about one tile, many overlapping (the fractions sum above one)."""
    rng = np.random.default_rng(5)
    X = np.stack([rng.uniform(*x, count), rng.uniform(3.0, 7.0, count), rng.uniform(2.0, 6.0, count)], 1)
    return dict(lattice=19, n=n, bc=bc, tau=0.7, body_force=(1e-5, 2e-6, 0.0), X=X, U=rng.normal(0, 2e-3, (count, 3)),
                Om=rng.normal(0, 5e-4, (count, 3)), r=rng.uniform(1.5, 2.4, count), psc=0)


@pytest.mark.parametrize("n,bc", [((97, 12, 8), (0, 0, 0)), ((128, 12, 8), (1, 0, 0)), ((198, 11, 9), (0, 1, 0))])
@pytest.mark.parametrize("count", [9, 31, 40])
def test_many_candidates(n, bc, count):
    g = check(cluster(n, bc, count), 3)
    assert g["info"]["max_tile_candidates"] > {9: 4, 31: 16, 40: 32}[count]


@pytest.mark.parametrize("psc", [0, 1])
@pytest.mark.parametrize("bc,nx", [((0, 0, 1), 97), ((1, 0, 0), 128)])
def test_both_schemes(psc, bc, nx):
    check(ragged_case3d(psc=psc, bc=bc, n=(nx, 29, 24)), 6)


@pytest.mark.parametrize("tile_cap", [1, 4])
def test_overflow(tile_cap):
    check(ragged_case3d(bc=(0, 0, 1), n=(97, 29, 24)), 3, tile_cap=tile_cap)


@pytest.mark.parametrize("x", [3.3, 48.6, 94.2])
def test_minimum_image_per_cell(x):
    """A period of 97 cells is less than a tile, the reach of the larger sphere on both sides and two;
    the smaller one needs no image."""
    X = np.array([[x, 20.4, 17.7], [(x + 46.0) % 97.0, 9.1, 8.3]])
    check(dict(lattice=19, n=(97, 40, 36), bc=(0, 0, 1), tau=0.62, body_force=(1e-5, 0, 0), X=X,
               U=np.array([[1e-3, -5e-4, 2e-4], [0, 0, 0]]), Om=np.array([[2e-4, 1e-4, -1e-4], [0, 0, 0]]),
               r=np.array([15.6, 4.2]), psc=0), 4)


@pytest.mark.parametrize("n,bc", [((97, 9, 5), (0, 0, 1)), ((130, 5, 4), (0, 0, 0)), ((128, 4, 4), (1, 0, 0))])
@pytest.mark.parametrize("spread", [0, 12])
def test_macro(n, bc, spread):
    M.test_moments(19, n, bc, "f32", spread)


@pytest.mark.parametrize("count", [9, 20])
@pytest.mark.parametrize("x", [(20.0, 42.0), (90.0, 103.0)])
def test_callers_buffers(torch, count, x):
    """As test_zz_no_alloc compares the two paths: its bounds."""
    c = cluster((97, 12, 8), (0, 0, 0), count, x)
    ctx = P.lbm_create(19, *c["n"], tau=c["tau"], body_force=c["body_force"], storage="f32")
    P.lbm_set_populations(ctx, perturbed_state(c, 12))
    P.lbm_set_particles(ctx, c["X"], c["U"], c["Om"], c["r"])
    size = 19 * int(np.prod(c["n"])) * 4
    raw = lambda: np.frombuffer(P.lbm_save_state(ctx), dtype=np.float32, count=size // 4, offset=64).copy()
    f = torch.as_tensor(raw(), device="cuda")
    P.lbm_step(ctx, 1)
    F, T = (np.array(v) for v in P.lbm_get_forces(ctx))
    want, params = raw(), ctx.params
    P.lbm_destroy(ctx)
    dev = [torch.as_tensor(np.ascontiguousarray(c[k]), device="cuda") for k in ("X", "U", "Om", "r")]
    G, S = (torch.zeros((count, 3), dtype=torch.float64, device="cuda") for _ in range(2))
    out = torch.empty_like(f)
    params.stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    P.lbm_psc_step_noalloc(params, f, out, *dev, G, S)
    assert rel_l2(out.cpu().numpy(), want) <= 1e-6
    assert rel_l2(G.cpu().numpy(), F) <= 1e-6 and rel_l2(S.cpu().numpy(), T) <= 1e-6


def test_slabs():
    case = ragged_case3d(bc=(0, 0, 1), n=(97, 29, 32))
    kw = dict(bc=case["bc"], tau=case["tau"], body_force=case["body_force"], storage="f32")
    parts = (case["X"], case["U"], case["Om"], case["r"])
    ctx, d = P.lbm_create(19, *case["n"], **kw), P.lbm_decomp_create(19, *case["n"], 2, **kw)
    P.lbm_set_particles(ctx, *parts)
    P.lbm_decomp_set_particles(d, *parts)
    P.lbm_step(ctx, 4)
    P.lbm_decomp_step(d, 4)
    whole, slabs = P.lbm_get_populations(ctx).copy(), P.lbm_decomp_get_populations(d).copy()
    P.lbm_decomp_destroy(d)
    P.lbm_destroy(ctx)
    assert np.array_equal(whole, slabs)


def run_all(torch):
    """Every case above, in the bounds-checked library."""
    assert P.lbm_checked_build()
    P.lbm_check_violations()
    for count in (9, 31, 40):
        test_many_candidates((97, 12, 8), (0, 0, 0), count)
        test_many_candidates((198, 11, 9), (0, 1, 0), count)
    for psc in (0, 1):
        test_both_schemes(psc, (0, 0, 1), 97)
    test_overflow(1)
    test_minimum_image_per_cell(94.2)
    test_macro((97, 9, 5), (0, 0, 1), 0)
    test_callers_buffers(torch, 20, (90.0, 103.0))
    test_slabs()
    plain = cluster((97, 12, 8), (0, 1, 0), 0)        # no particles
    check(plain, 3)
    return P.lbm_check_violations()


def test_checked_build(torch):
    from paper_1901_09745_gb300 import build
    build.build(checked=True)
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PSC_LBM_CHECKED="1", PYTHONPATH=os.pathsep.join(
        [os.path.dirname(here), here] + [v for v in [os.environ.get("PYTHONPATH")] if v]))
    code = "import json, torch, test_gpu_wide_tiles as t; print(json.dumps(t.run_all(torch)))"
    r = subprocess.run([sys.executable, "-c", code], env=env, cwd=here, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    assert json.loads(r.stdout.strip().splitlines()[-1]) == 0
