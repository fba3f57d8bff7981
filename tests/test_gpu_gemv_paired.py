"""Step 1 over factors stored in row pairs: FP32 pairs (inner GMRES passes and the FP32 mode) at odd row and
column counts against native FP64, and the double-float kernel where a warp takes a row group of its own
(from 9,728 row groups of several right-hand sides on).

Tolerances.  FP32 pairs in double-float arithmetic: on rigid-motion data the operator keeps the rounding of
the matrix entries, 6e-8 each over ~1e3 terms of either sign, so 1e-6 of its largest value.  FP32 mode: the
data, the factors and the strengths are rounded to 6e-8, amplified by the truncation 1e-3 used here, and the
sums run over ~600 terms: 1e-3 of the largest value (a row or column left out or taken twice is O(1) there).
Double-float: 1e-12 of the norm, as at the other edges.
"""
import numpy as np
import pytest

from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu


def row_of_spheres(P):
    return np.array([[4.0 * i, 0.3 * (i % 2), 0.0] for i in range(P)])


def build(centres, **kw):
    ctx = mfs.Context(0)
    ctx.set_spheres(centres)
    ctx.build(r_proxy=0.63, tensor_step1=0, **kw)
    return ctx


@pytest.mark.parametrize("P", [2, 3, 5])
@pytest.mark.parametrize("n_proxy,m_basic", [(5, 11), (33, 51), (57, 91), (64, 97), (131, 201)])
def test_fp32_pairs_against_fp64(P, n_proxy, m_basic):
    ctx = build(row_of_spheres(P), n_proxy=n_proxy, m_basic=m_basic)
    ctx.set_rigid_velocities(*workloads.rigid_velocities(P, seed=P))
    mu = ctx.rhs()
    ref = ctx.apply_operator(mu, mfs.FP64)
    out = ctx.apply_operator(mu, mfs.MIXED_PASS)
    ctx.close()
    assert np.abs(out - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("P", [1, 3])
@pytest.mark.parametrize("n_proxy,m_basic", [(5, 11), (33, 51), (57, 91), (131, 201)])
def test_fp32_mode_against_fp64(P, n_proxy, m_basic):
    ctx = build(row_of_spheres(P), n_proxy=n_proxy, m_basic=m_basic, eps_trunc=1e-3)
    mu = np.random.default_rng(n_proxy).normal(size=3 * m_basic * P)
    ref = ctx.apply_precond(mu, mfs.FP64)
    out = ctx.apply_precond(mu, mfs.FP32)
    ctx.close()
    assert np.abs(out - ref).max() <= 1e-3 * np.abs(ref).max()


@pytest.mark.parametrize("P", [400, 401])
def test_row_group_a_warp(P):
    # 100 or 101 groups of right-hand sides x 99 row groups
    n_proxy, m_basic = 131, 201
    ctx = build(row_of_spheres(P), n_proxy=n_proxy, m_basic=m_basic)
    mu = np.random.default_rng(P).normal(size=3 * m_basic * P)
    ref = ctx.apply_precond(mu, mfs.FP64).reshape(P, -1)
    out = ctx.apply_precond(mu, mfs.MIXED).reshape(P, -1)
    ctx.close()
    assert np.all(np.linalg.norm(out - ref, axis=1) <= 1e-12 * np.linalg.norm(ref, axis=1))
