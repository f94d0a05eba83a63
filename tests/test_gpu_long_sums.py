"""Split products with as many terms as the product kernel's 64-bit sums admit."""
from fractions import Fraction

import pytest

from tests.gpu_util import lib_ready, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [4, 6])
def test_longest_sums_of_chunks_past_the_quick_conversion(S):
    # every entry has the digits 255, -255, 0, ..: a chunk of the pairs (1, 2) and
    # (2, 1) sums to -256 255^2, which the drain's quick conversion reads as about
    # +2^31 until the difference is added, while the sum of the whole tile (more tiles
    # than clusters: one cluster takes all of k) grows to 2^62 less 2 %.  The largest
    # K, a multiple of 64, with 2^16 K (2^27 + 2 2^18 + 3 2^9 + 4) < 4.5e18
    hs, torch = lib_ready(), torch_cuda()
    M, N, K = 2048, 1280, 509568
    x = 255 / 512 - 255 / 512 ** 2
    A = torch.full((M, K), x, dtype=torch.float64, device="cuda")
    B = torch.full((K, N), x, dtype=torch.float64, device="cuda")
    A[1::2] *= -1.0
    C = hs.gemm(A, B, P=8, Q=10, G=80, b=64, Bouter=256, kind="bf16", slices=S)
    hs.sync()
    want = float(K * Fraction(x) ** 2)
    assert torch.all(C[::2] == want) and torch.all(C[1::2] == -want)
    del A, B
    torch.cuda.empty_cache()
