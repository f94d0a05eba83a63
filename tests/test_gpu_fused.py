"""The split products that recombine in the product kernel (CTA pairs, the
default), against the oracle bit for bit: tile edges, odd panel counts, one and
several parts of a tile, every slice count, both layouts, and digits that reach
the bounds of exact fp32 sums; and against the separate steps (pair kernel off)
where the oracle would take long."""
import numpy as np
import pytest

import workloads
from oracle import split
from tests.gpu_util import lib_ready, pair, torch_cuda

pytestmark = pytest.mark.gpu


def gemm(hs, dA, dB, kind, S, P, Q, G, layout="block"):
    b = 64 if kind == "bf16" else 128
    C = hs.gemm(dA, dB, P=P, Q=Q, G=G, b=b, Bouter=4 * b, kind=kind, slices=S, layout=layout)
    hs.sync()
    return C


@pytest.mark.parametrize("kind,S", [("bf16", s) for s in range(1, 8)]
                         + [("int8", s) for s in range(1, 9)])
def test_every_slice_count(kind, S):
    hs = lib_ready()
    A, B, dA, dB = pair(257, 390, 321, 40 + S, "wide")      # short tiles, an odd panel count
    C = gemm(hs, dA, dB, kind, S, 3, 2, 6)
    assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, S, kind))


@pytest.mark.parametrize("M,N,K,P,Q,layout", [
    (1, 1, 1, 1, 1, "block"),
    (128, 128, 64, 1, 1, "block"),        # one row tile: the pair's second half is empty
    (129, 127, 65, 1, 1, "cyclic"),
    (256, 129, 128, 2, 1, "block"),
    (255, 257, 192, 1, 2, "block"),
    (384, 640, 1000, 5, 3, "block"),      # blocks of 77 rows, an empty last processor row
    (384, 640, 1000, 5, 3, "cyclic"),
    (70, 1030, 1500, 2, 5, "block"),      # few tiles, each cut along k
    (200, 200, 4133, 2, 1, "block"),
])
@pytest.mark.parametrize("kind,S", [("bf16", 4), ("bf16", 5), ("int8", 6)])
def test_tile_edges_and_parts(M, N, K, P, Q, layout, kind, S):
    hs = lib_ready()
    A, B, dA, dB = pair(M, N, K, 71, "uniform", "wide")
    C = gemm(hs, dA, dB, kind, S, P, Q, 1, layout)
    assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, S, kind))


def _digits(values, S, w):
    """x with all S digits equal to `values` (0 < value < 2^(w-1))."""
    return sum(values * 2.0 ** (-w * s) for s in range(1, S + 1))


@pytest.mark.parametrize("S", [2, 4, 5, 6])
@pytest.mark.parametrize("digit", [181, 182, 255])
def test_digits_at_the_chunk_bounds(S, digit):
    # every digit of every entry equal and positive: with 181 the windows of 128
    # squares stay at their bound (128 * 181^2 <= 2^22 < 128 * 182^2) and chunks
    # of 512 products run up to 2^24; above it, chunks of 256.  Sums beyond 2^22
    # take the drain's second conversion.  One entry of 1/4 fixes the exponents
    # at 2^0.
    hs = lib_ready()
    torch = torch_cuda()
    M, N, K = 256, 256, 1024
    x = float(_digits(np.float64(digit), S, 9))
    assert 0.25 < x < 0.5
    A = np.full((M, K), x)
    B = np.full((K, N), x)
    A[::3] *= -1.0
    B[5:9, 7] = 0.25
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = gemm(hs, dA, dB, "bf16", S, 2, 1, 1)
    assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, S, "bf16"))


@pytest.mark.parametrize("M,N,K,P,Q,G,kind,S", [
    (2560, 2560, 512, 20, 10, 100, "bf16", 4),     # 200 tile pairs: whole rounds and parts
    (1300, 3000, 1111, 11, 12, 132, "bf16", 6),    # odd P, ragged
    (2000, 1900, 777, 16, 15, 1, "int8", 8),
    (300, 700, 40000, 3, 3, 9, "bf16", 7),
])
def test_same_bits_as_the_separate_steps(M, N, K, P, Q, G, kind, S):
    hs = lib_ready()
    torch = torch_cuda()
    dA = workloads.matrix_torch(M, K, 81, "wide", device="cuda")
    dB = workloads.matrix_torch(K, N, 82, "uniform", device="cuda")
    C = gemm(hs, dA, dB, kind, S, P, Q, G)
    again = gemm(hs, dA, dB, kind, S, P, Q, G)     # the partial sums were left at zero
    was = hs.pair_kernel(False)
    try:
        D = gemm(hs, dA, dB, kind, S, P, Q, G)
    finally:
        hs.pair_kernel(was)
    assert torch.equal(C, D) and torch.equal(again, D)


@pytest.mark.parametrize("kind,S", [("bf16", 3), ("bf16", 6), ("int8", 8)])
@pytest.mark.parametrize("ea,eb", [(-520, -500), (-560, -520), (500, 460), (520, 500)])
def test_results_at_the_ends_of_the_exponent_range(kind, S, ea, eb):
    # subnormal, zero, largest and infinite entries beside ordinary ones: columns
    # go from 2^eb to 2^(eb + 60), so one tile holds both of the kernel's roundings
    hs = lib_ready()
    torch = torch_cuda()
    A, B, _, _ = pair(130, 203, 150, 91, "uniform", "uniform")
    A = np.ldexp(A, ea)
    B = np.ldexp(B, eb + (np.arange(203) * 60) // 202)
    C = gemm(hs, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), kind, S, 2, 1, 1)
    with np.errstate(over="ignore", under="ignore"):
        assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, S, kind))


@pytest.mark.parametrize("K", [1, 63, 129, 257, 900, 2049, 4300])
@pytest.mark.parametrize("kind,S", [("bf16", 4), ("bf16", 7), ("int8", 8)])
def test_exponents_and_digits(K, kind, S):
    # one to several steps a warp and windows a CTA; operands that start off 16
    # bytes with odd leading dimensions; rows and columns of zeros, of subnormals,
    # of few bits (ties at the digits' rounding), of values far below their largest
    hs = lib_ready()
    torch = torch_cuda()
    M, N = 37, 41
    A, B = workloads.matrix(M, K, 17, "wide"), workloads.matrix(K, N, 18, "wide")
    for X in (A, B.T):
        X[0] = 0.0
        X[1] *= 2.0 ** -1060
        X[2] = 5e-324
        X[3] = np.ldexp(np.rint(X[3] * 8), -3)
        X[4, ::2] *= 2.0 ** -300
        X[5, 1:] = np.ldexp(1.0, -(np.arange(K - 1) % 70))
        X[6, 0] = 1e300
    buf = torch.zeros(M * (K + 2) + 1, dtype=torch.float64, device="cuda")
    dA = buf[1:].as_strided((M, K), (K + 2 - K % 2, 1))
    dA.copy_(torch.from_numpy(A))
    buf = torch.zeros(K * (N + 2) + 1, dtype=torch.float64, device="cuda")
    dB = buf[1:].as_strided((K, N), (N + 2, 1))
    dB.copy_(torch.from_numpy(B))
    C = gemm(hs, dA, dB, kind, S, 1, 1, 1)
    with np.errstate(over="ignore", under="ignore"):
        assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, S, kind))


@pytest.mark.parametrize("M,N,K,P,Q,layout", [
    (300, 63, 200, 2, 1, "block"),        # one narrow column tile, short
    (256, 65, 128, 1, 1, "block"),        # a second one of one column
    (511, 700, 130, 4, 3, "block"),       # blocks of 234 columns: 3 x 64 + 42
    (511, 700, 130, 4, 3, "cyclic"),
    (260, 1290, 64, 1, 1, "block"),       # tiles for the whole device but a few
])
@pytest.mark.parametrize("kind,S", [("bf16", 3), ("bf16", 6), ("int8", 8)])
def test_narrow_tiles_against_wide_and_separate(M, N, K, P, Q, layout, kind, S):
    # small products take tiles of 64 columns; the same rows 64 times over take
    # tiles of 128
    hs = lib_ready()
    torch = torch_cuda()
    A, B, dA, dB = pair(M, N, K, 51, "wide", "uniform")
    C = gemm(hs, dA, dB, kind, S, P, Q, 1, layout)
    assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, S, kind))
    wide = gemm(hs, dA.repeat(64, 1), dB, kind, S, 64 * P, Q, 1, layout)
    assert torch.equal(wide[:M], C) and torch.equal(wide[-M:], C)


@pytest.mark.parametrize("rows", [1, 40])
def test_large_chunks_after_products_of_the_other_tile_width(rows):
    # two-pass products leave their low words in the kernel's buffer; what large
    # chunks add (digits of 255, one sign) has to find its own part of it at zero,
    # whichever width (64 columns with rows = 1, 128 with 40) ran before
    hs = lib_ready()
    torch = torch_cuda()
    other = 41 - rows
    _, _, dA, dB = pair(256 * other, 700, 300, 95, "uniform")
    gemm(hs, dA, dB, "bf16", 6, 2 * other, 3, 1)
    x = float(_digits(np.float64(255), 2, 9))
    A, B = np.full((256, 1024), x), np.full((1024, 700), x)
    A[::3] *= -1.0
    C = gemm(hs, torch.from_numpy(A).cuda().repeat(rows, 1), torch.from_numpy(B).cuda(), "bf16", 2,
             2 * rows, 3, 1)
    want = torch.from_numpy(split.split_gemm(A, B, 2, "bf16")).cuda()
    assert torch.equal(C, want.repeat(rows, 1))
