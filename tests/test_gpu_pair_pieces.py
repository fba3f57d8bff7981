"""Double-float pair sums at the edges of their work items: pieces of 64 targets (half a 128-node tile,
the second one empty, short or full) and source splits from one part to sixteen, 32 sources a part at
least, against the oracle's blocks.

Tolerance: that of the tile edges, 1e-13 of the absolute sum of the terms.
"""
import pytest

from paper_2407_03343_gb300 import mfs
from tests.test_gpu_pair_edges import test_pair_sums_at_tile_edges as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_proxy,m_basic", [(31, 63), (32, 64), (63, 65), (64, 96), (65, 191), (96, 192), (97, 193),
                                             (511, 255), (512, 256), (545, 257)])
@pytest.mark.parametrize("P", [2, 5])
def test_pair_sums_at_piece_edges(n_proxy, m_basic, P):
    check(n_proxy, m_basic, 2, P, mfs.MIXED)
