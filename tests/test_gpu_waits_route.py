"""A wait that runs out in the screened route's tensor-core product is reported
in the layer's device error word, as every other bounded wait of a layer.

The hook makes the product's MMA issuer wait for a condition nothing fulfils; the
wait gives up after about a millisecond, the launch ends normally, and the next
call (hook off) routes as before.
"""
import pytest
import torch

import synth
from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu

SHORT = 2_000_000   # SM clock cycles, about 1 ms


@pytest.mark.parametrize("T", [400, 1500])   # by T E H, and where the tiled router would run
def test_unmet_wait_in_the_route_is_reported(T):
    src = synth.flat_layer(2048, 64, [4] * 32, 64, 8, "bf16", seed=5, factor_std="visible")
    L = lx.Layer(src)
    x = lx.host_to_torch(synth.tokens(src, T, seed=1), "bf16").cuda()
    ids, gates = [t.clone() for t in L.route(x, 8)[:2]]
    torch.cuda.synchronize()
    assert L.info()["device_error"] == 0
    L.set_wait_limit(SHORT)
    L.inject_unmet_wait(lx.LX_WAIT_ROUTER)
    L.route(x, 8)
    torch.cuda.synchronize()
    assert L.info()["device_error"] == lx.LX_ERR_TIMEOUT
    L.inject_unmet_wait(lx.LX_WAIT_NONE)
    L.set_wait_limit(0)
    L.clear_device_error()
    again = L.route(x, 8)
    torch.cuda.synchronize()
    assert L.info()["device_error"] == 0
    assert torch.equal(again[0], ids) and torch.equal(again[1], gates)
    L.free()
