"""Step 1 at the edges of its GEMV kernels: odd and even row and column counts, few rows, and spheres
that share a factor in groups of one to nine (right-hand sides are taken four at a time).

Reference: the native FP64 factors' product is compared with the double-float one to 1e-12 of the
strengths' norm (both factors' entries and sums carry ~2^-46 = 1.4e-14 relative to the row's absolute
sum, over ~1e3 terms), and each sphere of a group with the same sphere solved alone.
"""
import numpy as np
import pytest

from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu


def build(centres, **kw):
    ctx = mfs.Context(0)
    ctx.set_spheres(centres)
    ctx.build(r_proxy=0.63, **kw)
    return ctx


@pytest.mark.parametrize("P", [1, 2, 3, 4, 5, 9])
@pytest.mark.parametrize("n_proxy,m_basic", [(5, 11), (33, 50), (64, 97), (131, 200)])
def test_shared_factor_groups(P, n_proxy, m_basic):
    # far apart: one shared factor, with odd 3 m_basic for odd m_basic
    centres = np.array([[4.0 * i, 0.3 * (i % 2), 0.0] for i in range(P)])
    ctx = build(centres, n_proxy=n_proxy, m_basic=m_basic, tensor_step1=0)
    one = build(centres[:1], n_proxy=n_proxy, m_basic=m_basic, tensor_step1=0)
    mu = np.random.default_rng(P).normal(size=(P, 3 * m_basic))
    out = {p: ctx.apply_precond(mu.ravel(), p).reshape(P, -1) for p in (mfs.FP64, mfs.MIXED, mfs.MIXED_PASS)}
    for k in range(P):
        for p, tol in ((mfs.FP64, 1e-13), (mfs.MIXED, 1e-13), (mfs.MIXED_PASS, 1e-11)):
            alone = one.apply_precond(mu[k], p)
            assert np.abs(out[p][k] - alone).max() <= tol * np.abs(alone).max()
        ref = out[mfs.FP64][k]
        assert np.linalg.norm(out[mfs.MIXED][k] - ref) <= 1e-12 * np.linalg.norm(ref)
    ctx.close()
    one.close()


@pytest.mark.parametrize("nim", [1, 2])
def test_mixed_factors(nim):
    # two spheres with images of their own and five sharing the basic factor, in mixed order
    centres = np.array([[0.0, 0, 0], [2.05, 0, 0], [6.0, 0, 0], [10.0, 0, 0], [0, 6.0, 0], [0, 10.0, 0], [0, 0, 7.0]])
    centres = centres[[2, 0, 3, 4, 1, 5, 6]]
    ctx = build(centres, n_proxy=57, m_basic=91, nim_fixed=nim)
    mu = np.random.default_rng(7).normal(size=3 * ctx.sizes().n_colloc)
    ref = ctx.apply_precond(mu, mfs.FP64)
    out = ctx.apply_precond(mu, mfs.MIXED)
    assert np.linalg.norm(out - ref) <= 1e-12 * np.linalg.norm(ref)
    ctx.close()
