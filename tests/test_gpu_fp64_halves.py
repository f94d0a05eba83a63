"""binary64 strips of half the columns (few CTAs for the SMs) against exact integer
products: blocks that end in either half, flat grids and clusters, both layouts."""
import numpy as np
import pytest

from tests.gpu_util import lib_ready, pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,P,Q,G", [
    (1, 1, 1, 1, 1, 1),
    (33, 64, 40, 1, 1, 1),          # the second half empty
    (130, 65, 100, 1, 1, 1),        # one column in it, a second row tile
    (200, 254, 150, 2, 2, 4),       # blocks of 127 columns, flat
    (200, 254, 150, 2, 2, 1),       # 2 x 2 cluster
    (256, 512, 200, 4, 4, 4),
    (300, 260, 90, 4, 2, 2),        # 4 x 1 and 2 x 2 clusters
    (330, 200, 90, 5, 3, 1),        # 5 x 3 cluster: whole strips
    (700, 900, 300, 6, 8, 48),
])
@pytest.mark.parametrize("layout", ["block", "cyclic"])
def test_half_strips_integers_exact(M, N, K, P, Q, G, layout):
    hs = lib_ready()
    A, B, dA, dB = pair(M, N, K, 61, "smallint")
    C = hs.gemm(dA, dB, P=P, Q=Q, G=G, b=16, Bouter=32, layout=layout)
    hs.sync()
    assert np.array_equal(C.cpu().numpy(), A @ B)
