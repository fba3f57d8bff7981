"""Single solves on both sides of 64 chunks of 1024 elements, where they change from the segmented vector
kernels to the unsegmented ones, resistance and mobility, against the same problem as a batch of one, which
keeps the segmented kernels.

Tolerance: both reach a residual of 1e-9 and the spheres are a diameter apart, so forces and torques follow
it to well below 1e-6 of the largest.
"""
import numpy as np
import pytest

from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu

G = np.arange(4) * 4.0
CENTRES = np.array([[x, y, 0.0] for x in G for y in G])


def error(a, b):
    return max(np.abs(x - y).max() for x, y in zip(a, b)) / max(np.abs(y).max() for y in b)


# 48 m_basic rows, 96 more with the mobility border: 65,520 / 65,616 (64 and 65 chunks), 65,568 / 65,664 (65)
@pytest.mark.parametrize("m_basic", [1363, 1365, 1366])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_single_solves_across_the_kernel_change(m_basic, precision):
    v, w = workloads.rigid_velocities(len(CENTRES), seed=m_basic)
    with mfs.Context(0) as ctx:
        ctx.set_spheres(CENTRES)
        ctx.build(n_proxy=24, r_proxy=0.63, m_basic=m_basic)
        ctx.set_rigid_velocities(v, w)
        mfs.batch_solve([ctx], precision=precision, tol=1e-9)
        ref = ctx.forces_torques()
        ctx.solve(precision=precision, tol=1e-9)
        assert error(ctx.forces_torques(), ref) <= 1e-6
        ctx.set_forces_torques(*ref)
        ctx.solve(precision=precision, tol=1e-9)
        assert error(ctx.rigid_velocities(), (v, w)) <= 1e-6
