"""The cost model's backward pass at the edges of its blocks of 16 samples, and
with more samples than its blocks take at once, against the float64 oracle."""
import numpy as np
import pytest

import workloads
from oracle import mlp
from tests.gpu_util import lib_ready, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 15, 16, 17, 257, 5001])
def test_gradient_at_tile_edges(batch):
    torch, hs = torch_cuda(), lib_ready()
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    th = f32(0.3 * workloads.matrix(1, mlp.N_PARAMS, 31, "uniform")[0])
    X, y = f32(workloads.matrix(batch, 10, 32, "uniform")), f32(workloads.matrix(1, batch, 33)[0])
    g = torch.full((mlp.N_PARAMS,), float("nan"), dtype=torch.float32, device="cuda")
    loss = torch.full((1,), float("nan"), dtype=torch.float32, device="cuda")
    hs._check(hs.lib().hsumma_mlp_backward(batch, th.data_ptr(), X.data_ptr(), y.data_ptr(),
                                            g.data_ptr(), loss.data_ptr(), None))
    hs.sync(None)
    L, G = mlp.loss_and_grad(*(t.cpu().numpy().astype(np.float64) for t in (th, X, y)))
    # products of 64 terms over three layers, sums of up to 16 + 20 + 8 terms: about
    # 3 * 64 + 44 roundings of 2^-24 on the largest entries, 1.4e-5
    assert loss.item() == pytest.approx(L, rel=2e-5)
    assert np.max(np.abs(g.cpu().numpy().astype(np.float64) - G)) <= 2e-5 * np.abs(G).max()
