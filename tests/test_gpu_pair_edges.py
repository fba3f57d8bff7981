"""Pair sums at the edges of their tiles and rounds: target tiles of 128 and 512 nodes in warps of
32, source rounds of up to 256 proxies and 64 image nodes of one sphere, two sources a lane pair.

Tolerance: 1e-13 of the absolute sum of the terms (double-float terms and sums are accurate to
~2^-44 = 5.7e-14 of it), as in the parity test of amplified strengths.
"""
import numpy as np
import pytest

from oracle import geometry, solve
from paper_2407_03343_gb300 import mfs, workloads
from tests.layout import oracle_to_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_proxy,m_basic,nim,P", [(1, 33, 0, 2), (31, 127, 1, 2), (32, 128, 2, 3), (33, 129, 3, 2),
                                                   (255, 511, 20, 2), (256, 512, 0, 3), (257, 513, 65, 2),
                                                   (513, 97, 0, 5)])
@pytest.mark.parametrize("prec", [mfs.MIXED, mfs.FP64])
def test_pair_sums_at_tile_edges(n_proxy, m_basic, nim, P, prec):
    centres = workloads.cluster(P, 0.05, seed=2)
    kw = dict(n_proxy=n_proxy, r_proxy=0.63, m_basic=m_basic, nim_fixed=nim, nim_max=max(20, nim))
    d = geometry.build(centres, 1.0, geometry.Params(**kw))
    rng = np.random.default_rng(3)
    lam = [rng.normal(size=solve.n_unknowns(d, k)) * 10.0 ** rng.uniform(0, 6) for k in range(P)]
    mu = rng.normal(size=sum(solve.n_rows(d, k) for k in range(P)))
    ref, bound = [], []
    for k in range(P):
        blocks = [(solve.scaled_block(d, k, q), lam[q]) for q in range(P) if q != k]
        ref.append(sum(b @ l for b, l in blocks))
        bound.append(sum(np.abs(b) @ np.abs(l) for b, l in blocks))
    ref, bound = np.concatenate(ref) + mu, np.concatenate(bound)
    with mfs.Context(0) as ctx:
        ctx.set_spheres(centres)
        ctx.build(build_factors=0, **kw)
        out = ctx.apply_pairs(oracle_to_lib(d, lam), mu, prec)
    assert np.all(np.abs(out - ref) <= 1e-13 * bound + 1e-15 * np.abs(mu))
