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


def test_the_buffer_of_sums_is_given_up_and_had_again():
    hs, torch = fresh(), torch_cuda()
    A, B, dA, dB = pair(300, 520, 700, 25, "uniform")
    want = split.split_gemm(A, B, 4, "bf16")
    for _ in range(2):
        C = hs.gemm(dA, dB, **CFG)
        hs.sync()
        assert np.array_equal(C.cpu().numpy(), want)
        assert buffer_word(hs) > 1 << 32
        too_large_for_any_device(hs)
        assert buffer_word(hs) < 1 << 32       # an offset: the buffer is gone


@pytest.mark.parametrize("kind,S", [("bf16", 5), ("int8", 6)])
@pytest.mark.parametrize("route", ["single CTAs", "pairs, not persistent"])
def test_host_products_as_separate_steps(kind, S, route):
    hs = lib_ready()
    A, B, _, _ = pair(1100, 1050, 390, 27, "wide")
    C = np.empty((1100, 1050))
    if route == "single CTAs":
        was, restore = hs.pair_kernel(False), hs.pair_kernel
    else:
        was, restore = hs.lib().hsumma_pair_launch(0), hs.lib().hsumma_pair_launch
    try:
        hs.gemm_host(A, B, C, P=8, Q=4, G=16, b=64 if kind == "bf16" else 128, Bouter=256,
                     kind=kind, slices=S)
        assert len(hs.host_row_blocks()) > 1   # block by block
    finally:
        restore(was)
    assert np.array_equal(C, split.split_gemm(A, B, S, kind))
