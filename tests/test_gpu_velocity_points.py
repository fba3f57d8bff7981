"""Flow at points (native FP64, 32 points a CTA, sources split over its warps and over CTAs) for point
counts around those sizes, against the direct sum over the library's own strengths.

Tolerance: FP64 sums of ~1e3 terms in another order, 1e-13 of the absolute sum of the terms.
"""
import numpy as np
import pytest

from oracle import kernels
from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[(2, 0.05, 95), (3, 0.4, 130)])
def solved(request):
    P, gap, N = request.param
    centres = workloads.cluster(P, gap, seed=4)
    ctx = mfs.Context(0)
    ctx.set_spheres(centres)
    ctx.build(n_proxy=N, r_proxy=0.63, m_basic=2 * N)
    rng = np.random.default_rng(5)
    ctx.set_rigid_velocities(rng.normal(size=(P, 3)), rng.normal(size=(P, 3)))
    ctx.solve(precision="mixed", tol=1e-6)
    lam, pos, typ = ctx.strengths(with_positions=True)
    yield ctx, centres, lam.reshape(-1, 3), pos, typ
    ctx.close()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 129, 1000])
def test_velocity_at_points(solved, n):
    ctx, centres, lam, pos, typ = solved
    rng = np.random.default_rng(n)
    d = rng.normal(size=(n, 3))
    x = centres[rng.integers(0, len(centres), n)] + 1.5 * d / np.linalg.norm(d, axis=1)[:, None]
    ref, bound = np.zeros((n, 3)), np.zeros((n, 3))
    for t, f in ((0, kernels.stokeslet), (1, kernels.rotlet), (2, kernels.dipole)):
        sel = typ == t
        r = x[:, None] - pos[sel][None]
        ref += np.einsum("ijab,jb->ia", f(r), lam[sel])
        bound += np.einsum("ijab,jb->ia", np.abs(f(r)), np.abs(lam[sel]))
    assert np.all(np.abs(ctx.eval_velocity(x) - ref) <= 1e-13 * bound)
