"""Infinite weights on the generic path.

The bf16 form splits an fp32 activation into three bf16 parts, of which the lower
ones are zero where the value needs fewer bits; their product with an infinite
weight is a NaN that plain fp32 multiply-adds do not have.  The outputs are the
infinities and NaNs of plain fp32 arithmetic, for an infinity in each of the weights
that meet an fp32 activation, in rows of 16-byte units (rank 8) and in others (7).
"""
import numpy as np
import pytest
import torch

import synth
from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu
INF = {"bf16": (0x7F80, 0xFF80), "f32": (np.inf, -np.inf)}


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rank", [7, 8])
@pytest.mark.parametrize("where", ["dominant down", "down V", "down U", "up U"])
def test_infinite_weights(where, rank, dtype):
    src = synth.flat_layer(72, 136, [2], rank, 1, dtype, seed=rank, factor_std="visible")
    anchor = next(n for n in range(src.n_nodes) if src.is_anchor(n))
    member = 1 - anchor
    w = src.node_w[anchor if where == "dominant down" else member]
    target = w[{"dominant down": 2, "down V": 5, "down U": 4, "up U": 2}[where]]
    plus, minus = (np.asarray(v).astype(target.dtype) for v in INF[dtype])
    target[3, 5], target[target.shape[0] - 1, 0] = plus, minus
    L = lx.Layer(src)
    L.set_path(lx.LX_PATH_GENERIC)
    x = lx.host_to_torch(synth.tokens(src, 40, seed=1), dtype)
    y = L.moe_forward(x.cuda(), 1).float().cpu()
    ids = L.route(x.cuda(), 1)[0].cpu()[:, 0]
    f = lambda n: [lx.host_to_torch(a, dtype).float() for a in src.node_w[n]]
    Wg, Wu, Wd = f(anchor)
    Ug, Vg, Uu, Vu, Ud, Vd = f(member)
    xf = x.float()
    low = lambda v, U, V: (v @ V) @ U.T
    is_member = (src.expert_node[ids.numpy()] == member)[:, None]
    pick = lambda a, b: torch.where(torch.from_numpy(is_member), a + b, a)
    act = torch.nn.functional.silu(pick(xf @ Wg.T, low(xf, Ug, Vg))) * pick(xf @ Wu.T, low(xf, Uu, Vu))
    ref = pick(act @ Wd.T, low(act, Ud, Vd))
    assert bool(torch.isinf(ref).any()) or bool(torch.isnan(ref).any())
    assert torch.equal(torch.isnan(y), torch.isnan(ref))
    assert torch.equal(torch.isposinf(y), torch.isposinf(ref))
    assert torch.equal(torch.isneginf(y), torch.isneginf(ref))
    ok = torch.isfinite(ref)
    if bool(ok.any()):  # bf16: the result is rounded once (2^-9); fp32 sums
        bar = (2.0 ** -8 if dtype == "bf16" else 1e-5) * float(ref[ok].abs().max())
        assert float((y[ok] - ref[ok]).abs().max()) <= bar
