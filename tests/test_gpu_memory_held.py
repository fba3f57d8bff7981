"""Device memory that a context holds, which a caller's cap has to cover: within 1 % of the bytes stated with
each size (discretisation, factors in their copies and work vectors).
"""
import numpy as np
import pytest

from paper_2407_03343_gb300 import mfs, workloads

pytestmark = pytest.mark.gpu


def lattice(n):
    g = np.arange(n) * 3.0
    return np.array([[x, y, z] for x in g for y in g for z in g])


@pytest.mark.parametrize("centres,kw,held", [
    (workloads.two_spheres(0.5), dict(n_proxy=24, m_basic=50), 417608),
    (lattice(4), dict(n_proxy=100, m_basic=200), 17622212),
    (lattice(5), dict(n_proxy=10, m_basic=600), 52000132),
    (lattice(5), dict(n_proxy=100, m_basic=200, build_factors=0), 16510188)])
def test_context_holds_no_more(centres, kw, held):
    with mfs.Context(0) as ctx:
        ctx.set_spheres(centres)
        ctx.build(r_proxy=0.63, **kw)
        assert ctx.memory_in_use() <= 1.01 * held
