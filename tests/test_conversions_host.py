"""The DEM kernels' integer forms of double -> float (to nearest, ties to even) and float -> double
(compiled for the host) give the conversions' bits: random values of every exponent, exact ties and
their neighbours, the ends of the normal range, subnormals, zeros, infinities and NaN."""
import ctypes as C

import numpy as np

from host_entries import H  # noqa: F401  (fixture)


def test_conversions(H):  # noqa: F811
    H.psc_test_to_f32.argtypes, H.psc_test_to_f32.restype = [C.c_double], C.c_float
    H.psc_test_to_f64.argtypes, H.psc_test_to_f64.restype = [C.c_float], C.c_double
    rng = np.random.default_rng(1)
    bits = rng.integers(0, 1 << 64, 40000, dtype=np.uint64)
    v = np.concatenate([bits.view(np.float64), np.ldexp(rng.uniform(-2, 2, 60000), rng.integers(-160, 140, 60000))])
    f = rng.integers(0, 1 << 32, 20000, dtype=np.uint64).astype(np.uint32).view(np.float32)
    f = f[np.isfinite(f)]
    mid = f.astype(np.float64) + np.spacing(np.abs(f)).astype(np.float64) / 2
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0**-126, 2.0**-149, 2.0**-150, 2.0**127, 3.4028235677973366e38])
    v = np.concatenate([v, mid, np.nextafter(mid, np.inf), np.nextafter(mid, -np.inf), edge, -edge])
    with np.errstate(all="ignore"):
        want, ends = v.astype(np.float32), edge.astype(np.float32)
    got = np.array([H.psc_test_to_f32(x) for x in v], np.float32)
    nan = np.isnan(want)
    assert np.isnan(got[nan]).all() and (got.view(np.uint32) == want.view(np.uint32))[~nan].all()
    f = np.concatenate([f, ends])
    back = np.array([H.psc_test_to_f64(x) for x in f], np.float64)
    nan = np.isnan(f)
    assert (back.view(np.uint64) == f.astype(np.float64).view(np.uint64))[~nan].all() and np.isnan(back[nan]).all()
