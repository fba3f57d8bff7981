"""Single solves that take several GMRES cycles, so that every cycle starts from a fresh residual and a
fresh double-float split of it: resistance and mobility, FP64 and MIXED.

Tolerance as in the parity tests: 1e-5 at a GMRES tolerance of 1e-8 against the oracle's dense solve.
"""
import numpy as np
import pytest

from oracle import geometry, solve
from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu


def error(a, b):
    return max(np.abs(x - y).max() for x, y in zip(a, b)) / max(np.abs(y).max() for y in b)


@pytest.mark.parametrize("restart", [5, 9])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_several_cycles(restart, precision):
    centres = workloads.two_spheres(0.4)
    kw = dict(n_proxy=60, r_proxy=0.63, m_basic=171)
    d = geometry.build(centres, 1.0, geometry.Params(**kw))
    rng = np.random.default_rng(restart)
    v, w = rng.normal(size=(2, 3)), rng.normal(size=(2, 3))
    ref = solve.forces_torques(d, solve.solve_o2(d, v, w).lam)
    opts = dict(precision=precision, tol=1e-8, restart=restart, max_iter=2000, max_refine=200)
    with mfs.Context(0) as ctx:
        ctx.set_spheres(centres)
        ctx.build(**kw)
        ctx.set_rigid_velocities(v, w)
        info = ctx.solve(**opts)
        assert info.iters > restart
        assert error(ctx.forces_torques(), ref) <= 1e-5
        ctx.set_forces_torques(*ref)
        info = ctx.solve(**opts)
        assert info.iters > restart
        assert error(ctx.rigid_velocities(), (v, w)) <= 1e-5
