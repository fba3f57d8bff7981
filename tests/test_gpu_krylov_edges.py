"""GMRES vector kernels at the edges of their 1024-element chunks and 128-element pieces: systems of one
element short of, at and past them, resistance and mobility, alone and as a batch.

Force and torque tolerance as in the parity tests: 1e-5 at a GMRES tolerance of 1e-8 against the
oracle's dense solve.
"""
import numpy as np
import pytest

from oracle import geometry, solve
from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu


def error(a, b):
    return max(np.abs(x - y).max() for x, y in zip(a, b)) / max(np.abs(y).max() for y in b)


# system length 6 m_basic (+ 12 with the mobility border): 510, 1014 / 1026, 1020 / 1032, 1026, 2046 / 2058
@pytest.mark.parametrize("m_basic", [85, 169, 170, 171, 341])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solves_at_chunk_edges(m_basic, precision):
    centres = workloads.two_spheres(0.4)
    kw = dict(n_proxy=60, r_proxy=0.63, m_basic=m_basic)
    d = geometry.build(centres, 1.0, geometry.Params(**kw))
    rng = np.random.default_rng(m_basic)
    v, w = rng.normal(size=(2, 3)), rng.normal(size=(2, 3))
    ref = solve.forces_torques(d, solve.solve_o2(d, v, w).lam)
    ctxs = [mfs.Context(0) for _ in range(2)]
    for c in ctxs:
        c.set_spheres(centres)
        c.build(**kw)
        c.set_rigid_velocities(v, w)
    ctxs[0].solve(precision=precision, tol=1e-8)
    assert error(ctxs[0].forces_torques(), ref) <= 1e-5
    # the mobility problem driven by those forces gives back the velocities, alone and in a batch
    ctxs[0].set_forces_torques(*ref)
    ctxs[0].solve(precision=precision, tol=1e-8)
    assert error(ctxs[0].rigid_velocities(), (v, w)) <= 1e-5
    ctxs[0].set_forces_torques(*ref)
    mfs.batch_solve(ctxs, precision=precision, tol=1e-8)
    assert error(ctxs[0].rigid_velocities(), (v, w)) <= 1e-5
    assert error(ctxs[1].forces_torques(), ref) <= 1e-5
    for c in ctxs:
        c.close()
