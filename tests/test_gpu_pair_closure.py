"""Closure-form sweep with two patches per thread: group edges.

The sizes give colours of one patch, odd counts (a lone last patch), one group
and several, in both dimensions and at every degree.  FP64: the reference is
the coarse-level kernel (one output per thread, itself held to the oracle);
both compute in double-float arithmetic, so 1e-12 covers two sweeps' rounding.
FP32: the reference is the FP64 sweep, at 1e-5 per sweep, the bound that FP32
sweeps are held to against the oracle.
"""
import numpy as np
import pytest

from paper_2407_02100_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg():
    from paper_2407_02100_gb300 import build, gmg as g
    build.build()
    return g


def sweep(gmg, dim, k, n, precision, small, reverse):
    P = gmg.Problem(dim, k, n, n_levels=1, precision=precision, small_sweep=small)
    gmg.gmg_set_shared_faces(P.h, False)
    u = P.to_device(inputs.random_nodal(dim, k, n, 31 + k))
    b = P.to_device(inputs.random_nodal(dim, k, n, 77 + n))
    gmg.gmg_smooth(P.h, 0, u, b, 2, reverse)
    out = P.from_device(u)
    P.close()
    return np.asarray(out, dtype=np.float64)


@pytest.mark.parametrize("dim,k,n", [
    (2, 1, 2), (2, 1, 41), (2, 2, 37), (2, 3, 33), (2, 4, 19), (2, 5, 11), (2, 6, 13), (2, 7, 7), (2, 8, 9),
    (3, 1, 11), (3, 2, 2), (3, 2, 9), (3, 3, 8), (3, 4, 7), (3, 5, 5), (3, 6, 4), (3, 7, 4), (3, 8, 4)])
def test_groups(gmg, dim, k, n):
    a = sweep(gmg, dim, k, n, gmg.GMG_FP64, 0, n % 2 == 1)
    c = sweep(gmg, dim, k, n, gmg.GMG_FP64, 1 << 20, n % 2 == 1)
    assert np.linalg.norm(a - c) <= 1e-12 * np.linalg.norm(c)
    s = sweep(gmg, dim, k, n, gmg.GMG_FP32, 0, n % 2 == 1)
    assert np.linalg.norm(s - a) <= 2e-5 * np.linalg.norm(a)
