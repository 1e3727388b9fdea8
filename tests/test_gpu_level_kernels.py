"""Kernels of the multigrid levels at the edges of their tiles and rules:
transfers, coarsest solve, operators, mid-size colours, variable coefficients.

Tolerances: 1e-12 where FP64 results differ by rounding order alone (each form
errs below 1e-13); FP32 transfers 5e-6 (three passes of up to 4k - 1 terms at
2^-24); FP32 sweeps 1e-5 and the FP64 solve of an FP32 right-hand side 3e-7, the bounds that FP32 results are held to elsewhere.
"""
import numpy as np
import pytest

from oracle.mesh import Mesh
from oracle.multigrid import prolongation
from oracle.varcoef import VarPatchSmoother
from paper_2407_02100_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg():
    from paper_2407_02100_gb300 import build, gmg as g
    build.build()
    return g


def rel(a, b):
    return np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dim,k,nc", [(2, 1, 2), (2, 2, 5), (2, 5, 3), (2, 8, 2), (3, 1, 3), (3, 2, 2), (3, 3, 2),
                                      (3, 4, 1)])
def test_fp32_transfers(gmg, dim, k, nc):
    Pm = prolongation(Mesh(dim, k, nc), Mesh(dim, k, 2 * nc), sparse=True)
    P = gmg.Problem(dim, k, 2 * nc, n_levels=2, precision=gmg.GMG_FP32)
    r = inputs.random_nodal(dim, k, 2 * nc, 3)
    e = inputs.random_nodal(dim, k, nc, 4)
    c, f = P.zeros(0), P.to_device(r)
    gmg.gmg_restrict(P.h, 1, f, c)
    gmg.gmg_prolongate_add(P.h, 0, P.to_device(e, 0), f)
    assert rel(P.from_device(c, 0), Pm.T @ r) < 5e-6
    assert rel(P.from_device(f), r + Pm @ e) < 5e-6


# unknowns per direction n k - 1: one launch up to 21 in 2D and 9 in 3D, axis passes above
@pytest.mark.parametrize("dim,k,n", [(2, 1, 2), (2, 2, 11), (2, 3, 8), (3, 1, 2), (3, 5, 2), (3, 2, 5), (3, 3, 4)])
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 3e-7)])
def test_coarsest_solve(gmg, dim, k, n, precision, tol):
    import scipy.sparse.linalg as sla
    m = Mesh(dim, k, n)
    P = gmg.Problem(dim, k, n, n_levels=1, precision=precision)
    b = inputs.random_nodal(dim, k, n, 5).astype(np.float32).astype(np.float64)
    x = P.to_device(inputs.random_nodal(dim, k, n, 6))
    gmg.gmg_coarse_solve(P.h, P.to_device(b), x)
    i = np.flatnonzero(~m.boundary_mask())
    ref = np.zeros(m.n_nodes)
    ref[i] = sla.spsolve(m.assemble()[i][:, i].tocsc(), b[i])
    assert rel(P.from_device(x), ref) < tol


# 3D: rows of 64 / k cells and 4 cells per tile; 2D: full and quarter tiles
@pytest.mark.parametrize("dim,k,n", [(3, 3, 21), (3, 3, 22), (3, 4, 17), (3, 5, 5), (3, 6, 11), (3, 7, 3), (3, 8, 9)])
def test_operator_tiles(gmg, dim, k, n):
    P = gmg.Problem(dim, k, n, n_levels=1)
    x = P.to_device(inputs.random_nodal(dim, k, n, 7))
    y, z = P.zeros(), P.zeros()
    gmg.gmg_apply_operator(P.h, 0, x, y)
    gmg.gmg_set_three_pass_operator(P.h, False)
    gmg.gmg_apply_operator(P.h, 0, x, z)
    assert rel(P.from_device(y), P.from_device(z)) < 1e-12


@pytest.mark.parametrize("k,n", [(1, 5), (1, 193), (2, 33), (2, 97), (3, 4), (3, 49), (5, 9), (8, 3), (8, 25)])
def test_operator_2d(gmg, k, n):
    m = Mesh(2, k, n)
    P = gmg.Problem(2, k, n, n_levels=1)
    x = inputs.random_nodal(2, k, n, 8)
    y = P.zeros()
    gmg.gmg_apply_operator(P.h, 0, P.to_device(x), y)
    assert rel(P.from_device(y), m.assemble() @ x) < 1e-12


# colours on both sides of the coarse-level kernel's line (1536 patches at k = 3, 640 at k = 4, 128
# above)
@pytest.mark.parametrize("k,n", [(3, 13), (3, 24), (4, 14), (4, 18), (5, 4), (6, 11), (7, 5), (8, 3)])
def test_mid_size_colours(gmg, k, n):
    out = []
    for kw in ({}, {"small_sweep": 0}):
        P = gmg.Problem(3, k, n, n_levels=1, **kw)
        u = P.to_device(inputs.random_nodal(3, k, n, 9))
        gmg.gmg_smooth(P.h, 0, u, P.to_device(inputs.random_nodal(3, k, n, 10)), 1, k == 4)
        out.append(P.from_device(u))
    assert rel(out[0], out[1]) < 1e-12


# a lone patch, odd colours, one group of pairs and several (the coarsest level
# of a variable coefficient is a dense inverse: as many levels as n allows)
@pytest.mark.parametrize("dim,k,n", [(2, 1, 21), (2, 2, 26), (2, 3, 24), (3, 1, 11), (3, 2, 8), (3, 3, 2), (3, 3, 6)])
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
def test_variable_coefficient_groups(gmg, dim, k, n, precision, tol):
    m = Mesh(dim, k, n)
    coef = inputs.lognormal_coefficient(dim, n, 13)
    P = gmg.Problem(dim, k, n, n_levels=0, precision=precision)
    gmg.gmg_set_coefficient(P.h, coef)
    u, b = inputs.random_nodal(dim, k, n, 14), inputs.random_nodal(dim, k, n, 15)
    ud = P.to_device(u)
    gmg.gmg_smooth(P.h, P.finest, ud, P.to_device(b), 1, n % 2 == 1)
    assert rel(P.from_device(ud), VarPatchSmoother(m, coef, "fd_mean").sweep(u, b, n % 2 == 1)) < tol
