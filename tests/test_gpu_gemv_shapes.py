"""Step 1 of one context over the range in which its double-float GEMVs choose how many right-hand sides of a
shared factor an item takes (one, two or four) and whether four warps share a row group's columns or a warp
takes a group: both sides of each line, odd numbers of spheres, rows and columns.

Tolerances as for the row-paired factors: 1e-12 of the norm for double-float factors against native FP64;
1e-6 of the operator's largest value on rigid-motion data with the FP32 factor.
"""
import numpy as np
import pytest

from paper_2407_03343_gb300 import mfs, workloads
from tests.test_gpu_gemv_paired import build, row_of_spheres

pytestmark = pytest.mark.gpu


# row pairs of all spheres: 1,379 / 1,576 (up to one wave and above it), 4,088 / 9,928 / 10,074 with short
# columns, 1,773 / 4,925 / 5,910 with more than 640, and 78,800 (a warp a row group by their number)
@pytest.mark.parametrize("P,n_proxy,m_basic", [(7, 131, 201), (8, 131, 201), (9, 131, 201), (11, 131, 201), (28, 97, 151),
                                               (68, 97, 151), (69, 97, 151), (71, 97, 151), (8, 131, 215),
                                               (9, 131, 215), (25, 131, 215), (30, 131, 215), (31, 131, 215),
                                               (400, 131, 215)])
def test_shared_factor_over_the_dispatch(P, n_proxy, m_basic):
    ctx = build(row_of_spheres(P), n_proxy=n_proxy, m_basic=m_basic)
    mu = np.random.default_rng(P).normal(size=3 * m_basic * P)
    ref = ctx.apply_precond(mu, mfs.FP64).reshape(P, -1)
    out = ctx.apply_precond(mu, mfs.MIXED).reshape(P, -1)
    assert np.all(np.linalg.norm(out - ref, axis=1) <= 1e-12 * np.linalg.norm(ref, axis=1))
    if P < 100:
        ctx.set_rigid_velocities(*workloads.rigid_velocities(P, seed=P))
        mu = ctx.rhs()
        ref = ctx.apply_operator(mu, mfs.FP64)
        out = ctx.apply_operator(mu, mfs.MIXED_PASS)
        assert np.abs(out - ref).max() <= 1e-6 * np.abs(ref).max()
    ctx.close()
