"""Shared-face FP64 sweep with two patches per thread: group edges.

Groups hold 2 PP patches (10 at k <= 4, 6 at k = 5, 2 above) and are handed
out to persistent CTAs as they become free.  The sizes give colours of one
patch, odd counts (a lone last patch), counts one off a multiple of the group
and, at the largest, more groups than CTAs.  The reference is the closure
form of the same sweep (an independent kernel, itself held to the oracle);
both compute in double-float arithmetic, so 1e-12 covers two sweeps' rounding
(measured below 4e-14 per form against 64 bits at k <= 7).
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


def sweep(gmg, k, n, shared, damping, reverse):
    P = gmg.Problem(3, k, n, n_levels=1, damping=damping, small_sweep=0)
    gmg.gmg_set_shared_faces(P.h, shared)
    u = P.to_device(inputs.random_nodal(3, k, n, 31 + k))
    b = P.to_device(inputs.random_nodal(3, k, n, 77 + n))
    gmg.gmg_smooth(P.h, 0, u, b, 2, reverse)
    out = P.from_device(u)
    P.close()
    return out


# colours: n = 2: one patch; 3: 1 and 2^a; 7: 27; 11: 125 and 5 * 5 * 4 ...; 43: 9261
@pytest.mark.parametrize("k,n,damping,reverse", [
    (3, 2, 1.0, False), (3, 7, 0.8, True), (3, 43, 1.0, False), (4, 3, 1.0, True), (4, 11, 0.7, False),
    (5, 7, 1.0, False), (6, 5, 1.0, True), (7, 7, 0.9, False), (8, 4, 1.0, True)])
def test_groups_agree_with_closure_form(gmg, k, n, damping, reverse):
    a = sweep(gmg, k, n, True, damping, reverse)
    c = sweep(gmg, k, n, False, damping, reverse)
    assert np.linalg.norm(a - c) <= 1e-12 * np.linalg.norm(c)
    # whichever CTA takes a group, its patches come out bit for bit the same
    assert np.array_equal(a, sweep(gmg, k, n, True, damping, reverse))


# more groups than resident CTAs (at most 304; 4 an SM at k = 6) at every degree: a CTA takes
# further groups, flips the phase of its barrier, refills the face blocks during the transforms
# and reuses the slots of b; the first colours have odd counts, so that a lone last patch
# follows full groups.  Largest colours: 3375, 2197, 1331, 729 and 729 patches, in groups of 10,
# 6, 2, 2 and 2
@pytest.mark.parametrize("k,n,damping,reverse", [
    (4, 31, 0.9, True), (5, 27, 1.0, False), (6, 23, 1.0, True), (7, 19, 0.8, False), (8, 19, 1.0, False)])
def test_persistent_groups_agree_with_closure_form(gmg, k, n, damping, reverse):
    a = sweep(gmg, k, n, True, damping, reverse)
    c = sweep(gmg, k, n, False, damping, reverse)
    assert np.linalg.norm(a - c) <= 1e-12 * np.linalg.norm(c)
    assert np.array_equal(a, sweep(gmg, k, n, True, damping, reverse))
