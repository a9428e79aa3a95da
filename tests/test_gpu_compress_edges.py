"""The compression kernels at the edges of their tilings: sketch widths l around
the 16-column Cholesky blocks, the Jacobi's values per lane (32, 48, 80, 144 and
192 columns) and the dealing of a column's entries to its lanes (up to 144 columns
and above), fewer pairs than CTAs, and runs of pairs of unequal length.  Same bars
as the parity tests.
"""
import numpy as np
import pytest
import torch

from oracle import compress
from paper_2608_07814_gb300 import lx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,l,r", [
    (1024, 328, 1, 1), (264, 1024, 2, 1), (328, 264, 7, 5), (264, 328, 16, 16), (1024, 328, 17, 9),
    (328, 1024, 64, 60), (264, 328, 65, 65), (264, 1024, 97, 90), (328, 264, 129, 120),
    (1024, 328, 160, 150), (328, 1024, 161, 150), (264, 328, 193, 190), (1024, 512, 255, 240),
])
def test_sketch_widths(rows, cols, l, r):
    rng = np.random.default_rng(l)
    Wd = rng.standard_normal((rows, cols)).astype(np.float32) * np.float32(0.02)
    Wm = rng.standard_normal((rows, cols)).astype(np.float32) * np.float32(0.02)
    om = rng.standard_normal((cols, l)).astype(np.float32)
    R = compress.residual(Wd, Wm)
    Uo, Vo, so = compress.randomized_factors(R, r, om.astype(np.float64), 1)
    U, V, s = [t.cpu().numpy().astype(np.float64) for t in lx.compress_factor(
        torch.from_numpy(Wd).cuda(), torch.from_numpy(Wm).cuda(), torch.from_numpy(om).cuda(), r, 1)]
    Po = Uo @ Vo.T
    assert np.max(np.abs(U @ V.T - Po)) <= 1e-4 * np.max(np.abs(Po))
    assert np.max(np.abs(s - so)) <= 1e-5 * so[0]
    assert np.max(np.abs(U.T @ U - np.diag(s))) <= 1e-4 * s[0]
    assert np.max(np.abs(V.T @ V - np.diag(s))) <= 1e-4 * s[0]
