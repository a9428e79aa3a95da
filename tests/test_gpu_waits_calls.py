"""A wait that runs out inside a call without a layer shows in its results.

lx_compress_factor and lx_align_cost have no layer whose error word could say so:
when one of their bounded waits gives up, everything they write is NaN.  The hook
makes one wait of the next call run out after about a millisecond; the launches end
normally, and the call after it gives the same bits as the call before.  Jacobi
cases: two CTAs of the cluster busy, all eight with one pair each, uneven runs.
"""
import ctypes

import numpy as np
import pytest
import torch

from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu

SHORT = 2_000_000   # SM clock cycles, about 1 ms


def _randn(shape, seed, dtype):
    g = np.random.default_rng(seed).standard_normal(shape).astype(np.float32)
    return torch.from_numpy(g).cuda().to(dtype)


@pytest.mark.parametrize("l,dtype,site", [
    (3, torch.float32, lx.LX_WAIT_CALL_JACOBI), (16, torch.float32, lx.LX_WAIT_CALL_JACOBI),
    (57, torch.bfloat16, lx.LX_WAIT_CALL_JACOBI), (57, torch.bfloat16, lx.LX_WAIT_CALL_PRODUCT),
])
def test_compression_gives_nan_and_recovers(l, dtype, site):
    Wd, Wm = _randn((256, 192), 1, dtype), _randn((256, 192), 2, dtype)
    om = _randn((192, l), 3, torch.float32)
    run = lambda: [t.clone() for t in lx.compress_factor(Wd, Wm, om, l - 1, 1)]
    before = run()
    assert all(bool(torch.isfinite(t).all()) for t in before)
    lx.inject_unmet_wait_call(site, SHORT)
    bad = run()
    torch.cuda.synchronize()
    assert all(bool(torch.isnan(t).all()) for t in bad)
    assert all(torch.equal(a, b) for a, b in zip(before, run()))


def test_alignment_gives_nan_and_recovers():
    dom, mem = ([_randn(s, q + n, torch.bfloat16) for n, s in enumerate(((96, 256), (96, 256), (256, 96)))]
                for q in (0, 10))
    before = lx.align_cost(dom, mem).clone()
    lx.inject_unmet_wait_call(lx.LX_WAIT_CALL_PRODUCT, SHORT)
    bad = lx.align_cost(dom, mem)
    torch.cuda.synchronize()
    assert bool(torch.isnan(bad).all())
    assert torch.equal(lx.align_cost(dom, mem), before)


def test_short_bound_alone_does_not_fire():
    om = _randn((192, 40), 3, torch.float32)
    Wd, Wm = _randn((256, 192), 1, torch.bfloat16), _randn((256, 192), 2, torch.bfloat16)
    lx.inject_unmet_wait_call(lx.LX_WAIT_NONE, SHORT)
    assert all(bool(torch.isfinite(t).all()) for t in lx.compress_factor(Wd, Wm, om, 32, 1))


def test_unknown_site_is_refused():
    assert lx.lib().lx_inject_unmet_wait_call(lx.LX_WAIT_TC_MMA, ctypes.c_uint64(0)) == lx.LX_ERR_ARG
