"""lx_compress_factor follows its stated arithmetic to the bit.

The kernels spread the work over many threads and SMs, but every rounded
operation and the order of every sum are fixed: fp32 products summed by fused
multiply-adds in ascending order, the Gram in four interleaved compensated
chains, a Cholesky factor and its inverse blocked by 16 columns with correctly
rounded roots and divisions, M = L1 L2 and the Rayleigh quotients in float64, and
the one-sided Jacobi in the circle method's order, rotating every pair further
than 1e-6 from orthogonal until a sweep rotates none.  This file restates that
arithmetic in numpy (fp32 weights, whose products with the residual are plain
fp32 sums) and asks for equal bits: a root or a division by a fast
approximation, a shorter iteration, another pair order or a 32-bit sum in
place of a 64-bit one each show.  Sizes: one pair, one CTA's worth and fewer
pairs than CTAs, odd l, uneven runs of pairs, and above 144 columns, where a
column's entries are dealt to the lanes differently.
"""
import numpy as np
import pytest
import torch

from paper_2608_07814_gb300 import lx

F32, F64 = np.float32, np.float64
B = 16  # Cholesky block


def fma(a, b, c):
    """fp32 fused multiply-add: the exact product and a sum rounded to odd in
    float64 (two-sum for its error), then once to fp32."""
    p = np.asarray(a, F32).astype(F64) * np.asarray(b, F32).astype(F64)
    c = np.broadcast_to(np.asarray(c, F32).astype(F64), p.shape)
    s = p + c
    v = s - p
    e = (p - (s - v)) + (c - v)
    bits = np.ascontiguousarray(s).view(np.int64)
    bits = np.where((e != 0) & ((bits & 1) == 0), bits + np.where((e > 0) == (s > 0), 1, -1), bits)
    return bits.view(F64).astype(F32)


def test_fma_rounds_once():
    # (1 + 2^-12)^2 = 1 + 2^-11 + 2^-24: a tie that a tiny addend breaks
    a = F32(1 + 2.0 ** -12)
    for c, up in ((F32(2.0 ** -70), True), (F32(-2.0 ** -70), False)):
        got = fma(np.array([a]), np.array([a]), np.array([c]))[0]
        assert got == F32(1 + 2.0 ** -11 + (2.0 ** -23 if up else 0))


def gemm(A, Bm):
    acc = np.zeros((A.shape[0], Bm.shape[1]), F32)
    for k in range(A.shape[1]):
        acc = fma(A[:, k:k + 1], Bm[k:k + 1, :], acc)
    return acc


def df_add(d, p, e):
    s = d[0] + p
    v = s - d[0]
    err = (d[0] - (s - v)) + (p - v)
    return s, d[1] + (err + e)


def gram(X):
    """hi + lo pairs, added as the Cholesky does; float64 and fp32 values."""
    l = X.shape[1]
    ch = []
    for c in range(4):
        d = (np.zeros((l, l), F32), np.zeros((l, l), F32))
        for m in range(c, X.shape[0], 4):
            x, y = X[m][:, None], X[m][None, :]
            p = x * y
            d = df_add(d, p, fma(x, y, -p))
        ch.append(d)
    s = df_add(df_add(ch[0], *ch[1]), *df_add(ch[2], *ch[3]))
    return s[0].astype(F64) + s[1].astype(F64)


def cholesky(G, shift_rel):
    l = G.shape[0]
    A = G.astype(F32)
    md = G.diagonal().max()
    A[np.arange(l), np.arange(l)] += F32(F64(F32(shift_rel)) * md)
    L, rd = np.zeros((l, l), F32), np.zeros(l, F32)
    for j0 in range(0, l, B):
        j1 = min(j0 + B, l)
        for j in range(j0, j1):
            L[j, j] = np.sqrt(np.maximum(A[j, j], F32(1e-30)))
            rd[j] = F32(1) / L[j, j]
            L[j + 1:, j] = A[j + 1:, j] * rd[j]
            if j + 1 < j1:
                A[j + 1:, j + 1:j1] = fma(-L[j + 1:, j:j + 1], L[j + 1:j1, j][None, :], A[j + 1:, j + 1:j1])
        if j1 < l:
            acc = np.zeros((l - j1, l - j1), F32)
            for m in range(j0, j1):
                acc = fma(L[j1:, m:m + 1], L[j1:, m][None, :], acc)
            A[j1:, j1:] = A[j1:, j1:] - acc
    return L, rd


def inverse_t(L, rd):
    l = L.shape[0]
    X = np.zeros((l, l), F32)
    for j0 in range(0, l, B):  # the diagonal blocks
        j1 = min(j0 + B, l)
        x = np.eye(j1 - j0, dtype=F32)
        for p in range(j1 - j0):
            x[p] *= rd[j0 + p]
            x[p + 1:] = fma(-L[j0 + p + 1:j1, j0 + p:j0 + p + 1], x[p][None, :], x[p + 1:])
        X[j0:j1, j0:j1] = np.tril(x)
    for i0 in range(B, l, B):
        i1 = min(i0 + B, l)
        for j0 in range(0, i0, B):
            S = np.zeros((i1 - i0, B), F32)
            for q in range(j0, i0):
                S = fma(L[i0:i1, q:q + 1], X[q:q + 1, j0:j0 + B], S)
            acc = np.zeros_like(S)
            for p in range(i1 - i0):
                acc = fma(X[i0:i1, i0 + p:i0 + p + 1], S[p:p + 1], acc)
            X[i0:i1, j0:j0 + B] = -acc
    return X.T.copy()


def qr_pass(X, shift_rel):
    L, rd = cholesky(gram(X), shift_rel)
    return gemm(X, inverse_t(L, rd)), L


def jacobi(Mt):
    """W of M W = U S; Mt[j] is column j of M."""
    l = Mt.shape[0]
    lp = l + (l & 1)
    rows = -(-lp // 16) * 16
    M, W = np.zeros((lp, rows), F32), np.zeros((lp, rows), F32)
    M[:l, :l] = Mt
    W[np.arange(lp), np.arange(lp)] = 1
    if lp > 144:
        order = np.arange(rows).reshape(-1, 8)                       # entry 8 v + u of lane u
    else:
        order = np.arange(rows).reshape(-1, 8, 2).transpose(0, 2, 1).reshape(-1, 8)
    for _ in range(30):
        rotated = False
        for r in range(lp - 1):
            g = np.arange(lp // 2)
            p, q = (r + g) % (lp - 1), (r - g) % (lp - 1)
            p[0], q[0] = r, lp - 1
            x, y = M[p], M[q]
            s = np.zeros((3, lp // 2, 8), F32)
            for at in order:
                s = fma(np.stack([x[:, at], y[:, at], x[:, at]]),
                        np.stack([x[:, at], y[:, at], y[:, at]]), s)
            for o in (4, 2, 1):
                s = s + s[:, :, np.arange(8) ^ o]
            a, b, gm = s[:, :, 0]
            with np.errstate(all="ignore"):
                do = (gm != 0) & (np.abs(gm) > F32(1e-6) * np.sqrt(a * b))
                z = (b - a) / (F32(2) * gm)
                t = np.where(z >= 0, F32(1), F32(-1)) / (np.abs(z) + np.sqrt(fma(z, z, F32(1))))
                c = F32(1) / np.sqrt(fma(t, t, F32(1)))
            if not do.any():
                continue
            rotated = True
            p, q = p[do], q[do]
            c, sn = c[do][:, None], (t * c)[do][:, None]
            for A in (M, W):
                x, y = A[p], A[q]
                A[p], A[q] = fma(c, x, -(sn * y)), fma(sn, x, c * y)
        if not rotated:
            break
    return W[:l, :l]


def tree64(v):
    w = np.zeros(256, F64)
    w[:len(v)] = v
    w = w.reshape(8, 32)
    for o in (16, 8, 4, 2, 1):
        w = w + w[:, np.arange(32) ^ o]
    t = 0.0
    for q in range(8):
        t += w[q, 0]
    return t


def factors(Wd, Wm, omega, r, iters):
    R, l = Wm - Wd, omega.shape[1]
    Y = gemm(R, omega)
    for it in range(iters):
        Y, _ = qr_pass(Y, 1e-6)
        Z, _ = qr_pass(gemm(R.T, Y), 1e-6)
        Y = gemm(R, Z)
    Q, _ = qr_pass(qr_pass(Y, 1e-6)[0], 0.0)
    Z, L1 = qr_pass(gemm(R.T, Q), 1e-6)
    Z, L2 = qr_pass(Z, 0.0)
    M = np.zeros((l, l), F64)
    for k in range(l):  # ascending k; the products are exact in float64
        M += L1[:, k].astype(F64)[:, None] * L2[k].astype(F64)[None, :]
    Mt = M.astype(F32).T.copy()
    Wt = jacobi(Mt)
    MWn, Wn, sig = np.zeros((l, l), F32), np.zeros((l, l), F32), np.zeros(l, F64)
    for j in range(l):
        w, v = Wt[j].astype(F64), np.zeros(l, F64)
        for k in range(l):
            v = v + Mt[k].astype(F64) * w[k]
        nw = np.sqrt(tree64(w * w))
        sig[j] = np.sqrt(tree64(v * v)) / nw
        MWn[j], Wn[j] = (v / nw).astype(F32), (w / nw).astype(F32)
    top = np.lexsort((np.arange(l), -sig))[:r]
    rs = np.sqrt(sig[top]).astype(F32)
    keep = (sig[top] > 1e-6 * sig[top[0]])[:, None]
    with np.errstate(all="ignore"):
        Wu, Wv = np.where(keep, MWn[top] / rs[:, None], F32(0)), np.where(keep, Wn[top] * rs[:, None], F32(0))
    U, V = gemm(Q, Wu.T), gemm(Z, Wv.T)
    flip = U[np.argmax(np.abs(U), axis=0), np.arange(r)] < 0
    U[:, flip], V[:, flip] = -U[:, flip], -V[:, flip]
    return U, V, sig[top].astype(F32)


@pytest.mark.gpu
@pytest.mark.parametrize("rows,cols,l,r,iters,kind", [
    (24, 40, 1, 1, 1, "random"), (24, 40, 2, 2, 0, "random"), (40, 24, 9, 7, 1, "random"),
    (64, 56, 24, 20, 2, "random"), (88, 72, 37, 30, 1, "random"), (64, 104, 50, 50, 0, "random"),
    (168, 152, 146, 140, 0, "random"),
    # singular values in near-equal clusters, and graded over five decades
    (64, 72, 40, 32, 1, "clusters"), (72, 64, 33, 33, 0, "clusters"), (64, 72, 40, 32, 1, "graded"),
])
def test_factors_bit_for_bit(rows, cols, l, r, iters, kind):
    rng = np.random.default_rng(rows + l)
    Wd, Wm, om = (rng.standard_normal(s).astype(F32) for s in ((rows, cols), (rows, cols), (cols, l)))
    if kind != "random":
        n = min(rows, cols)
        sv = 10.0 ** (-5 * np.arange(n) / n) if kind == "graded" else \
            0.5 ** (np.arange(n) // 8) * (1 + 1e-5 * rng.random(n))
        Uq, Vq = (np.linalg.qr(rng.standard_normal((m, n)))[0] for m in (rows, cols))
        Wm = Wd + ((Uq * sv) @ Vq.T).astype(F32)
    ref = factors(Wd, Wm, om, r, iters)
    got = lx.compress_factor(*(torch.from_numpy(a).cuda() for a in (Wd, Wm, om)), r, iters)
    for name, a, b in zip("UVs", ref, got):
        assert np.array_equal(a, b.cpu().numpy()), name
