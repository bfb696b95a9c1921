"""lbm_get_macro against the moments of the stored populations added exactly (math.fsum): the
density and velocity of FP32 and 16-bit lattices are as accurate as FP64 sums of the stored
values, on ragged tiles, with walls, with values of very different size in a cell, at rest
and where a population is not finite."""
import math

import numpy as np
import pytest

import paper_1901_09745_gb300 as P

pytestmark = pytest.mark.gpu


def stored(ctx, storage):
    """Post-collision deviations as stored, FP64 (exact for every storage type)."""
    raw = P.lbm_save_state(ctx)
    n = ctx.q * int(np.prod(ctx.shape))
    t = {"f64": np.float64, "f32": np.float32, "f16": np.float16, "bf16": np.uint16}[storage]
    v = np.frombuffer(raw, dtype=t, count=n, offset=64).reshape((ctx.q,) + ctx.shape)
    if storage == "bf16":
        v = (v.astype(np.uint32) << 16).view(np.float32)
    return v.astype(np.float64) / (4096.0 if storage == "f16" else 1.0)


def pull(ctx, g, bc):
    e, w, o = P.lbm_lattice_tables(ctx.q)
    n = ctx.shape[::-1]
    f = np.empty_like(g)
    for i in range(ctx.q):
        f[i] = np.roll(g[i], tuple(e[i][::-1]), axis=(0, 1, 2))
        for a in range(3):
            if bc[a] and e[i][a]:
                at = [slice(None)] * 3
                at[2 - a] = 0 if e[i][a] > 0 else n[a] - 1
                f[i][tuple(at)] = g[o[i]][tuple(at)]
    return e, f


@pytest.mark.parametrize("lattice,n,bc", [(9, (33, 9, 1), (0, 1, 0)), (9, (65, 17, 1), (0, 0, 0)),
                                          (19, (34, 9, 5), (0, 0, 1)), (19, (70, 13, 9), (0, 0, 0))])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("spread", [0, 12])
def test_moments(lattice, n, bc, storage, spread):
    F = (1e-4, -3e-5, 0.0)
    ctx = P.lbm_create(lattice, *n, bc=bc, tau=0.8, body_force=F, storage=storage)
    rng = np.random.default_rng(7)
    e, w, _ = P.lbm_lattice_tables(lattice)
    d = rng.uniform(-0.02, 0.02, (lattice, n[2], n[1], n[0]))
    if spread:      # values of a cell spread over decades, some of them zero
        d *= 10.0 ** -rng.uniform(0, spread, d.shape) * (rng.random(d.shape) < 0.9)
    P.lbm_set_populations(ctx, d + w[:, None, None, None])
    rho, u = P.lbm_get_macro(ctx)
    e, f = pull(ctx, stored(ctx, storage), bc)
    flat = f.reshape(lattice, -1)
    Ff = [float(np.float32(v)) if storage != "f64" else v for v in F]
    eps = 2.0 ** -52
    for c in range(flat.shape[1]):
        v = [float(x) for x in flat[:, c]]
        r = math.fsum([1.0] + v)
        # FP64 sums of Q values and one division: Q roundings of at most sum |d| each
        tol = eps * lattice * sum(abs(x) for x in v)
        assert abs(rho.reshape(-1)[c] - r) <= tol + eps
        for a in range(3):
            j = math.fsum([e[i][a] * v[i] for i in range(lattice)] + [0.5 * Ff[a]])
            got = u.reshape(-1, 3)[c, a]
            assert abs(got - j / r) <= (tol + 2 * eps * abs(j)) / r + tol * abs(j) / r ** 2, (c, a)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_rest_and_not_finite(storage):
    ctx = P.lbm_create(19, 40, 6, 5, tau=0.8, storage=storage)
    rho, u = P.lbm_get_macro(ctx)
    assert np.all(rho == 1.0) and np.all(u == 0.0)
    w = P.lbm_lattice_tables(19)[1]
    f = np.broadcast_to(w[:, None, None, None], (19, 5, 6, 40)).copy()
    f[1, 2, 3, 20] = np.nan
    f[3, 1, 1, 7] = np.inf
    f[:, 4, 4, 33] = w + 1e-30      # far below the values the split sums take
    P.lbm_set_populations(ctx, f)
    rho, u = P.lbm_get_macro(ctx)
    assert np.isnan(rho[2, 3, 20]) and np.isnan(u[2, 3, 20, 0])
    assert rho[1, 1, 7] == np.inf
    ok = np.isfinite(rho)
    assert ok.sum() == rho.size - 2 and np.all(np.abs(rho[ok] - 1.0) < 1e-15)
