"""Closure-form sweep on both sides of the lines between its kernels.

A launch of few patches takes one patch per thread (FP64) or more threads per
pair (FP32), a large one two patches per thread.  Every patch is to come out the
same bit for bit, whichever kernel takes it: the sizes are whole colours above
the line, the same sweep by slabs of one vertex row stays below it, and a slab
schedule gives each patch exactly the values that the whole colours give it.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle.mesh import Mesh
from oracle.multigrid import prolongation
from oracle.varcoef import VarPatchSmoother
from paper_2407_02100_gb300 import inputs

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def gmg():
    from paper_2407_02100_gb300 import build, gmg as g
    build.build()
    return g


def sweep(gmg, dim, k, n, precision, slab, reverse):
    P = gmg.Problem(dim, k, n, precision=precision, small_sweep=0)
    gmg.gmg_set_shared_faces(P.h, False)
    gmg.gmg_set_slab_width(P.h, slab)
    assert gmg.gmg_slab_width(P.h, P.finest) == slab
    u = P.to_device(inputs.random_nodal(dim, k, n, 51 + k))
    gmg.gmg_smooth(P.h, P.finest, u, P.to_device(inputs.random_nodal(dim, k, n, 52 + n)), 1, reverse)
    out = P.from_device(u)
    P.close()
    return out


@pytest.mark.parametrize("dim,k,n,precision", [
    (3, 2, 46, 0), (3, 3, 48, 0), (3, 4, 26, 0), (3, 5, 18, 0), (3, 6, 22, 0), (3, 7, 12, 0), (3, 8, 26, 0),
    (2, 7, 256, 0), (2, 8, 112, 0),
    (3, 5, 14, 1), (3, 6, 14, 1), (3, 7, 14, 1), (3, 8, 14, 1), (2, 2, 84, 1), (2, 4, 84, 1), (2, 7, 84, 1), (2, 8, 84, 1)])
def test_whole_colours_and_slabs_agree_bit_for_bit(gmg, dim, k, n, precision):
    whole = sweep(gmg, dim, k, n, precision, 0, k % 2 == 1)
    assert np.array_equal(whole, sweep(gmg, dim, k, n, precision, 1, k % 2 == 1))
    assert np.isfinite(whole).all()


def var_sweep(gmg, dim, k, n, precision):
    coef = inputs.lognormal_coefficient(dim, n, 13)
    P = gmg.Problem(dim, k, n, precision=precision)
    gmg.gmg_set_coefficient(P.h, coef)
    u, b = inputs.random_nodal(dim, k, n, 14), inputs.random_nodal(dim, k, n, 15)
    ud = P.to_device(u)
    gmg.gmg_smooth(P.h, P.finest, ud, P.to_device(b), 1, n % 2 == 1)
    out = P.from_device(ud)
    P.close()
    return out, coef, u, b


# variable coefficient, FP64 3D: up to 152 patches one per CTA, above one per
# thread, from 8000 on in larger groups.  Against the oracle at 1e-12 (FP64) and
# 1e-5 (FP32, whose small colours take another shape), as elsewhere
@pytest.mark.parametrize("dim,k,n", [(3, 1, 12), (3, 2, 8), (3, 2, 12), (3, 3, 8), (3, 3, 12), (2, 3, 24), (2, 3, 32)])
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
def test_variable_coefficient(gmg, dim, k, n, precision, tol):
    out, coef, u, b = var_sweep(gmg, dim, k, n, precision)
    ref = VarPatchSmoother(Mesh(dim, k, n), coef, "fd_mean").sweep(u, b, n % 2 == 1)
    assert np.linalg.norm(out - ref) <= tol * np.linalg.norm(ref)


# the largest groups: the FP64 sweep is the reference of the FP32 one, 1e-5
@pytest.mark.parametrize("k", [1, 2, 3])
def test_variable_coefficient_large_colours(gmg, k):
    ref = var_sweep(gmg, 3, k, 48, gmg.GMG_FP64)[0]
    out = var_sweep(gmg, 3, k, 48, gmg.GMG_FP32)[0]
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)


# FP32 prolongation on both sides of its lines, 240,000 fine nodes in 2D and 60,000 in 3D: three
# passes of up to k + 1 terms at 2^-24 each stay below 5e-6
@pytest.mark.parametrize("dim,k,nc", [(2, 3, 81), (2, 3, 82), (2, 8, 30), (2, 8, 31), (3, 2, 9), (3, 2, 10), (3, 4, 4), (3, 4, 5)])
def test_fp32_prolongation(gmg, dim, k, nc):
    Pm = prolongation(Mesh(dim, k, nc), Mesh(dim, k, 2 * nc), sparse=True)
    P = gmg.Problem(dim, k, 2 * nc, n_levels=2, precision=gmg.GMG_FP32)
    e, u = inputs.random_nodal(dim, k, nc, 16), inputs.random_nodal(dim, k, 2 * nc, 17)
    f = P.to_device(u)
    gmg.gmg_prolongate_add(P.h, 0, P.to_device(e, 0), f)
    ref = u + Pm @ e
    assert np.linalg.norm(P.from_device(f) - ref) <= 5e-6 * np.linalg.norm(ref)
    P.close()


# the limit of the coarse-level kernel: what is read can be given back, whichever
# rule set it, and levels that the kernel sweeps keep no slabs
@pytest.mark.parametrize("k,n,limit", [(2, 16, 256), (3, 20, 1536), (4, 16, 640), (5, 8, 0), (7, 6, 0)])
def test_limit_that_was_read_can_be_given_back(gmg, k, n, limit):
    u0, b = inputs.random_nodal(3, k, n, 18), inputs.random_nodal(3, k, n, 19)

    def run(P):
        u, launches = P.to_device(u0), gmg.gmg_kernel_launch_count()
        gmg.gmg_smooth(P.h, P.finest, u, P.to_device(b), 1, False)
        return P.from_device(u), gmg.gmg_kernel_launch_count() - launches

    P = gmg.Problem(3, k, n)
    ref, launches = run(P)
    assert gmg.gmg_small_sweep(P.h) == limit
    gmg.gmg_set_small_sweep(P.h, 0)
    off, _ = run(P)
    assert gmg.gmg_small_sweep(P.h) == 0
    gmg.gmg_set_small_sweep(P.h, limit)
    again, count = run(P)
    assert np.array_equal(again, ref) and count == launches
    assert np.linalg.norm(off - ref) <= 1e-12 * np.linalg.norm(ref)
    P.close()


@pytest.mark.parametrize("k,n", [(3, 20), (4, 16)])
def test_levels_of_the_raised_limit_keep_no_slabs(gmg, k, n):
    P = gmg.Problem(3, k, n)  # 1000 and 512 patches in the largest colour
    gmg.gmg_set_slab_width(P.h, 2)
    assert gmg.gmg_slab_width(P.h, P.finest) == 0
    gmg.gmg_set_shared_faces(P.h, False)  # the closure form, whose limit is 256
    assert gmg.gmg_small_sweep(P.h) == 256 and gmg.gmg_slab_width(P.h, P.finest) == 2
    gmg.gmg_set_shared_faces(P.h, True)
    assert gmg.gmg_slab_width(P.h, P.finest) == 0
    P.close()


# degrees 5 to 7 hand colours of up to 128 patches to the coarse-level kernel (one launch a
# colour), degree 8 keeps the shared-face form's two, whose error is smaller there
@pytest.mark.parametrize("k,n,launches", [(5, 10, 8), (6, 4, 8), (7, 4, 8), (8, 4, 16), (8, 6, 16)])
def test_few_patches_of_the_shared_face_form(gmg, k, n, launches):
    P = gmg.Problem(3, k, n)
    u, b = P.to_device(inputs.random_nodal(3, k, n, 20)), P.to_device(inputs.random_nodal(3, k, n, 21))
    u2, before = u.clone(), gmg.gmg_kernel_launch_count()
    gmg.gmg_smooth(P.h, P.finest, u, b, 1, False)
    assert gmg.gmg_kernel_launch_count() - before == launches
    gmg.gmg_set_shared_faces(P.h, False)
    gmg.gmg_smooth(P.h, P.finest, u2, b, 1, False)
    assert float((u - u2).norm() / u2.norm()) <= 1e-12
    P.close()


# gmg_smooth_noalloc after its first call at a degree: the kernel of another mesh size is loaded
# already, so that the call neither allocates nor waits for the legacy stream, which a bounded
# sleep of about 0.7 s keeps busy.  In a process of its own, where no other test has loaded the
# kernels; the sizes lie on both sides of the lines of degree 6 (1000 patches) and 7 (152)
NOALLOC = """
import torch
from paper_2407_02100_gb300 import gmg
for k, first, later in ((6, 6, 22), (7, 13, 6)):
    vecs = {}
    for n in (first, later):
        N = n * k + 1
        vecs[n] = [torch.zeros(N * N * ((N + 3) // 4 * 4), dtype=torch.float64, device="cuda") for _ in range(2)]
    side = torch.cuda.Stream()
    gmg.gmg_smooth_noalloc(3, k, first, *vecs[first], stream=side.cuda_stream)
    torch.cuda._sleep(1000)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    torch.cuda._sleep(int(1.5e9))
    gmg.gmg_smooth_noalloc(3, k, later, *vecs[later], stream=side.cuda_stream)
    side.synchronize()
    assert not torch.cuda.default_stream().query(), "the sweep waited for the legacy stream"
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
print("ok")
"""


def test_noalloc_at_another_mesh_size(gmg):
    res = subprocess.run([sys.executable, "-c", NOALLOC], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.endswith("ok\n"), res.stderr[-2000:]
