"""Split products whose digits are too large for the long chunks, beside other calls
(on another stream, before and after), bit for bit against the oracle."""
import ctypes

import numpy as np
import pytest

from oracle import split
from tests.gpu_util import lib_ready, pair, torch_cuda

pytestmark = pytest.mark.gpu

CFG = dict(P=2, Q=2, G=4, b=64, Bouter=256, kind="bf16", slices=4)


def large_digits(M, N, K):
    """Operands whose every digit is 255, rows of either sign, and their device copies."""
    torch = torch_cuda()
    x = sum(255 * 2.0 ** (-9 * s) for s in range(1, 5))
    A, B = np.full((M, K), x), np.full((K, N), x)
    A[::3] *= -1.0
    return A, B, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()


def test_calls_on_another_stream_leave_the_chunks_alone():
    # binary64 products, products of no terms and diagonal sums clear the counters on
    # their own stream whenever they come; sums of 512 products of 255^2 instead of
    # 256 would not be exact
    hs, torch = lib_ready(), torch_cuda()
    A, B, dA, dB = large_digits(256, 256, 1024)
    want = torch.from_numpy(split.split_gemm(A, B, 4, "bf16")).cuda()
    fA, fB, dfA, dfB = pair(64, 64, 64, 3, "smallint")
    e, f = hs.split_exponents(dfA, dfB)
    As, Bs = hs.split_slices(dfA, dfB, e, f, "bf16", 2)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    out = [torch.empty_like(want) for _ in range(60)]
    small = torch.empty(64, 64, dtype=torch.float64, device="cuda")
    zero = torch.empty_like(small)
    hs.gemm(dA, dB, out=out[0], **CFG)               # the workspace is there
    torch.cuda.synchronize()
    for C in out:
        hs.gemm(dA, dB, out=C, stream=s1, **CFG)
        for _ in range(3):
            hs.gemm(dfA, dfB, out=small, P=1, Q=1, G=1, b=32, Bouter=64, stream=s2)
            hs.gemm(dfA[:, :0], dfB[:0], out=zero, stream=s2, **CFG)
        hs.split_diagonals(As, Bs, 64, 64, 64, "bf16", 2, P=1, Q=1, G=1, b=64, Bouter=64, stream=s2)
    hs.sync(s1)
    hs.sync(s2)
    assert all(torch.equal(C, want) for C in out)
    assert np.array_equal(small.cpu().numpy(), fA @ fB) and torch.all(zero == 0)


def test_a_host_product_leaves_no_short_chunks_behind():
    # large digits cost the product that has them chunks of half the length (a sixth
    # of its rate), and no other: a product after a host-buffer product of such digits
    # takes as long as after one of ordinary digits
    hs, torch = lib_ready(), torch_cuda()
    n = 6144
    dA, dB = (torch.rand(n, n, dtype=torch.float64, device="cuda") - 0.5 for _ in range(2))
    C = torch.empty_like(dA)
    host = [[torch.from_numpy(x).pin_memory() for x in operands] for operands in
            (large_digits(1024, 1024, 512)[:2], pair(1024, 1024, 512, 5)[:2])]
    hC = torch.empty(1024, 1024, dtype=torch.float64).pin_memory()
    ms = [[], []]
    for i in range(14):
        which = i % 2
        hs.gemm_host(*host[which], hC, P=4, Q=2, G=4, b=64, Bouter=256, kind="bf16", slices=4)
        assert len(hs.host_row_blocks()) > 1                 # block by block
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        hs.gemm(dA, dB, out=C, P=48, Q=24, G=576, b=64, Bouter=512, kind="bf16", slices=4)
        t1.record()
        hs.sync()
        ms[which].append(t0.elapsed_time(t1))
    large, ordinary = (np.median(m[1:]) for m in ms)
    assert large < 1.06 * ordinary, (large, ordinary)


def test_a_product_that_gave_up_is_cleared_up_after_another_error():
    # hsumma_sync, with the first error a non-finite input and the words as a product
    # that gave up leaves them: the arrival counts end in the words before "finished"
    # and "large digits", "gave up" is the one behind
    hs, torch = lib_ready(), torch_cuda()
    A, B, dA, dB = pair(256, 256, 192, 7)
    bad = dA.clone()
    bad[3, 5] = float("nan")
    hs.gemm(bad, dB, **CFG)
    torch.cuda.synchronize()
    word = hs.lib()._ZN2hs16fused_big_digitsEv
    word.restype = ctypes.c_void_p
    view = type("words", (), {"__cuda_array_interface__": dict(
        shape=(6,), typestr="<i4", data=(word() - 16, False), version=2)})
    words = torch.as_tensor(view(), device="cuda")
    try:
        assert torch.all(words == 0)
        words[[0, 2, 5]] = torch.tensor([1, 3, 1], dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        with pytest.raises(hs.HsummaError) as error:
            hs.sync()
        assert error.value.status == -6
        assert torch.all(words == 0)
    finally:
        words.zero_()
    C = hs.gemm(dA, dB, **CFG)
    hs.sync()
    assert np.array_equal(C.cpu().numpy(), split.split_gemm(A, B, 4, "bf16"))
