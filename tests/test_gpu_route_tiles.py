"""Screened routing at the edges of its dispatch and tiles: the smallest batches
that take it (T E H at the rule's line), a last CTA of one token, router rows that
end inside a load batch, and E that ends inside a lane's stride.  Ids and gates
equal the full router's bit for bit.  Co-activation counts over chunk edges.
"""
import numpy as np
import pytest
import torch

import synth
from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,E,T", [
    (2048, 128, 305), (2048, 128, 306), (2048, 128, 1217), (2048, 128, 4864), (2048, 100, 4881),
    (2560, 256, 256), (2560, 200, 1223), (3136, 64, 5000), (64, 24, 1300), (4096, 160, 300),
])
def test_screened_equals_full(H, E, T):
    src = synth.flat_layer(H, 64, [4] * (E // 4), 64, 8, "bf16", seed=E, skew=synth.QWEN_SKEW)
    L = lx.Layer(src)
    x = lx.host_to_torch(synth.tokens(src, T, seed=T), "bf16").cuda()
    ids_s, w_s = L.route(x, 8)
    ids_f, w_f, _ = L.route(x, 8, want_logits=True)
    assert torch.equal(ids_s, ids_f)
    assert torch.equal(w_s.view(torch.int32), w_f.view(torch.int32))
    L.free()


@pytest.mark.parametrize("E,T,k", [(1, 1, 1), (31, 33, 4), (128, 2048, 8), (129, 2049, 8), (513, 700, 8),
                                   (1024, 1025, 32)])
def test_coact_chunks(E, T, k):
    """Counts over chunk edges, with invalid and repeated ids, against one-hot products."""
    g = torch.Generator().manual_seed(E + T)
    ids = torch.randint(-2, E + 2, (T, k), generator=g, dtype=torch.int32)
    fire, coact = lx.coact_accumulate(ids.cuda(), E)
    lx.coact_accumulate(ids.cuda(), E, fire, coact)
    hot = torch.zeros(T, E + 1, dtype=torch.float64)
    hot.scatter_(1, torch.where((ids >= 0) & (ids < E), ids, E).long(), 1.0)
    hot = hot[:, :E]
    ref = 2 * (hot.T @ hot)
    assert torch.equal(coact.cpu().double(), ref)
    assert torch.equal(fire.cpu().double(), ref.diagonal())
