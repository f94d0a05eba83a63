"""Split products in CUDA graphs, and what the library may allocate and free around
them, against the oracle bit for bit."""
import ctypes

import numpy as np
import pytest

from oracle import split
from tests.gpu_util import lib_ready, pair, torch_cuda

pytestmark = pytest.mark.gpu

CFG = dict(P=4, Q=2, G=4, b=64, Bouter=256, kind="bf16", slices=4)


def fresh():
    """The library as after its first hsumma_init: nothing allocated yet."""
    hs = lib_ready()
    hs.sync(None)
    hs.finalize()
    return lib_ready()


def capture(hs, torch, dA, dB, C):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="thread_local"):
        hs.gemm(dA, dB, out=C, **CFG)
    return graph


def replayed(torch, graph, C):
    C.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    return C.cpu().numpy()


def test_first_product_in_a_capture_beside_a_workspace():
    # the workspace comes from the separate steps, the product kernel's buffer is not
    # there and can't be had inside a capture
    hs, torch = fresh(), torch_cuda()
    A, B, dA, dB = pair(500, 390, 321, 21, "wide")
    want = split.split_gemm(A, B, 4, "bf16")
    C = torch.empty(500, 390, dtype=torch.float64, device="cuda")
    hs.pair_kernel(False)
    hs.gemm(dA, dB, out=C, **CFG)
    hs.sync()
    hs.pair_kernel(True)
    graph = capture(hs, torch, dA, dB, C)
    assert np.array_equal(replayed(torch, graph, C), want)
    hs.gemm(dA, dB, out=C, **CFG)              # outside, with the buffer
    hs.sync()
    assert np.array_equal(C.cpu().numpy(), want)
    dA *= -2.0                                 # and new inputs in the graph
    assert np.array_equal(replayed(torch, graph, C), -2.0 * want)


def too_large_for_any_device(hs):
    """A host product whose staging buffers (8 TiB) no device has: refused before any
    pointer is followed."""
    n = 1 << 20
    page = (ctypes.c_double * 8)()
    rc = hs.lib().hsumma_gemm_host(n, 8, n, page, n, page, 8, page, 8, 1, 1, 1, 64, 64,
                                   hs.mode_code("bf16", 4), None)
    assert rc == -3 and "host staging" in hs.last_error()
    with pytest.raises(hs.HsummaError):
        hs.sync(None)                          # the CUDA error, once
    hs.sync(None)


def buffer_word(hs):
    word = hs.lib()._ZN2hs16fused_big_digitsEv      # an address in the buffer of sums
    word.restype = ctypes.c_size_t
    return word()


def test_an_allocation_that_fails_leaves_a_graph_its_buffer():
    hs, torch = fresh(), torch_cuda()
    A, B, dA, dB = pair(300, 520, 700, 23, "uniform")
    want = split.split_gemm(A, B, 4, "bf16")
    C = hs.gemm(dA, dB, **CFG)
    hs.sync()
    graph = capture(hs, torch, dA, dB, C)
    before = buffer_word(hs)
    too_large_for_any_device(hs)
    assert buffer_word(hs) == before
    assert np.array_equal(replayed(torch, graph, C), want)
