"""The screened route's dispatch: both sides of the line by T, E, H and k, and of the
batches whose selection runs four CTAs an SM (rows above 2048), give the full
router's ids and gates bit for bit; and the ids alone never cost more than with the
logits (a small E or long rows at a few hundred tokens did: 56 us against 26).
"""
import pytest
import torch

import synth
from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu


def _layer(E, H):
    return lx.Layer(synth.flat_layer(H, 64, [4] * (E // 4), 64, 8, "bf16", seed=E + H, skew=synth.QWEN_SKEW))


def _tokens(T, H):
    return torch.randn(T, H, generator=torch.Generator().manual_seed(T)).bfloat16().cuda()


@pytest.mark.parametrize("E,H,T,k", [
    (128, 2048, 348, 8), (128, 2048, 349, 8), (64, 7168, 256, 2), (64, 7168, 700, 2), (16, 7168, 1300, 2),
    (16, 7168, 1300, 8), (256, 2560, 256, 8), (128, 2112, 3648, 8), (128, 2560, 3649, 8), (200, 2560, 4864, 4),
    (256, 2560, 4865, 8), (256, 4096, 3700, 8),
])
def test_ids_and_gates_equal_the_full_routers(E, H, T, k):
    L, x = _layer(E, H), _tokens(T, H)
    ids, gates = L.route(x, k)
    ids_f, gates_f, _ = L.route(x, k, want_logits=True)
    assert torch.equal(ids, ids_f)
    assert torch.equal(gates.view(torch.int32), gates_f.view(torch.int32))
    L.free()


def _micros(f):
    a, b = torch.cuda.Event(True), torch.cuda.Event(True)
    best = float("inf")
    for _ in range(5):
        a.record()
        for _ in range(30):
            f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 30 * 1000)
    return best


@pytest.mark.parametrize("E,H,T,k", [(64, 7168, 256, 8), (32, 7168, 512, 8), (16, 7168, 8192, 8),
                                     (128, 2048, 1024, 8), (256, 2560, 4096, 8)])
def test_ids_alone_cost_no_more(E, H, T, k):
    L, x = _layer(E, H), _tokens(T, H)
    out = (torch.empty(T, k, dtype=torch.int32, device="cuda"), torch.empty(T, k, device="cuda"))
    logits = torch.empty(T, E, device="cuda")
    run = lambda lg: lx._check(lx.lib().lx_route(L.handle, lx._ptr(x), T, k, lx._ptr(out[0]), lx._ptr(out[1]),
                                                 lx._ptr(lg) if lg is not None else None, lx._stream(None)))
    assert _micros(lambda: run(None)) <= 1.25 * _micros(lambda: run(logits)) + 3.0
    L.free()
