"""Near part of the far-field passes over lists of uneven length (images on some contacts), its sources in the
parts its rule gives: data on one sphere at a time, compared at the spheres near it with the all-pairs pass
operator, whose strengths are the same.

Tolerance: both sum the same terms in another order, each to 1e-13 of the absolute sum of the terms (as at the
tile edges), so 2e-13 of it, from the oracle's blocks and the strengths.
"""
import numpy as np
import pytest

from oracle import geometry, solve
from paper_2407_03343_gb300 import mfs
from tests import test_gpu_farfield as far_tests
from tests.layout import lib_to_oracle

pytestmark = pytest.mark.gpu


# near spheres of each: 0 to 2, and 2 to 5
@pytest.mark.parametrize("far_dist,most", [(5.0, 2), (6.5, 5)])
@pytest.mark.parametrize("n_proxy,m_basic", [(31, 65), (96, 129), (150, 300)])
def test_near_sums_of_uneven_lists(n_proxy, m_basic, far_dist, most):
    kw = dict(n_proxy=n_proxy, r_proxy=0.63, m_basic=m_basic)
    centres = far_tests.CENTRES
    P = len(centres)
    d = geometry.build(centres, 1.0, geometry.Params(**kw))
    dist = np.linalg.norm(centres[:, None] - centres[None], axis=2)
    near = (dist < far_dist) & ~np.eye(P, dtype=bool)
    assert near.sum(1).max() == most
    with mfs.Context(0) as far, mfs.Context(0) as full:
        for ctx, extra in ((far, dict(far_tests.FAR, far_dist=far_dist)), (full, {})):
            ctx.set_spheres(centres)
            ctx.build(**kw, **extra)
        owner = np.repeat(full.collocation()[2], 3)
        rng = np.random.default_rng(n_proxy)
        for j in range(P):
            v, w = np.zeros((P, 3)), np.zeros((P, 3))
            v[j], w[j] = rng.normal(size=3), rng.normal(size=3)
            full.set_rigid_velocities(v, w)
            mu = full.rhs()
            lam = np.abs(lib_to_oracle(d, full.apply_precond(mu, mfs.MIXED_PASS))[j])
            diff = np.abs(far.apply_operator(mu, mfs.MIXED_PASS) - full.apply_operator(mu, mfs.MIXED_PASS))
            for k in np.flatnonzero(near[j]):
                bound = np.abs(solve.scaled_block(d, k, j)) @ lam
                assert np.all(diff[owner == k] <= 2e-13 * bound)
