"""The generic path's grouped GEMM at the edges of its tiles: ranks below, at
and above a 16-byte unit and a K chunk (element loads where rows do not start
on 16 bytes), widths that end inside a 64-column tile, buckets of one row, one
tile and a row over it, weights stored tiled, and infinities in the activations.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu


def _forward(src, T, path):
    L = lx.Layer(src)
    L.set_path(path)
    x = synth.tokens(src, T, seed=T)
    y = L.moe_forward(lx.host_to_torch(x, src.dtype).cuda(), src.top_k)
    assert L.info()["device_error"] == 0
    return x, y.float().cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("T", [1, 32, 33, 130])
@pytest.mark.parametrize("H,I,rank", [(8, 8, 1), (72, 136, 7), (128, 64, 8), (264, 200, 33),
                                      (192, 128, 64), (64, 320, 61)])
def test_tile_edges(H, I, rank, T, dtype):
    r = min(rank, H, I)
    src = synth.flat_layer(H, I, [1, 3, 2], [r, max(1, r // 2), r], 3, dtype, seed=rank,
                           factor_std="visible")
    x, y = _forward(src, T, lx.LX_PATH_GENERIC)
    ref = oracle.moe_forward(src, x, src.top_k)
    # fp32 sums throughout; a bf16 layer's result is rounded once (2^-9 of a value)
    bar = 2.0 ** -8 if dtype == "bf16" else 1e-5
    assert np.max(np.abs(y - ref)) <= bar * np.max(np.abs(ref))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_infinite_activations(dtype):
    """A pre-activation of 1e36 squares to an infinite z: the products with it
    are the infinities and NaNs of plain fp32 arithmetic."""
    src = synth.flat_layer(16, 8, [1], [], 1, dtype, seed=3)
    L = lx.Layer(src)
    x = torch.zeros(4, 16)
    x[0, 0], x[1], x[2, 3], x[3] = 3e38, 0.5, -3e38, float("nan")
    x = x.to(L.torch_dtype)
    y = L.moe_forward(x.cuda(), 1).float().cpu()
    g, u, d = [lx.host_to_torch(w, dtype).float() for w in src.node_w[0]]
    xf = x.float()
    h = xf @ g.T
    ref = (torch.nn.functional.silu(h) * (xf @ u.T)) @ d.T
    assert torch.equal(torch.isnan(y), torch.isnan(ref))
    assert torch.equal(torch.isinf(y), torch.isinf(ref))
    assert torch.allclose(y[1], ref[1], rtol=2.0 ** -7, atol=1e-6)
