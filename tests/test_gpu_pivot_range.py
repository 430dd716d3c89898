"""Pivots whose reciprocal leaves the normal numbers.  The quotients u / d are ordinary
numbers there and L, D and log det are compared exactly (subnormal pivots: entries
and quotients are short binary fractions, so every step of the elimination is exact;
pivots near the overflow limit: one elimination step, one rounding)."""
import numpy as np
import pytest

from test_gpu_dense_widths import P, stored  # noqa: F401

pytestmark = pytest.mark.gpu


def factor(P, A, kind, wmax):
    import torch
    n = A.shape[0]
    cp, ri, lo, up, _ = stored(A)
    h = P.SelInv(n, cp, ri, unsym=int(kind == "unsym"), max_sn_width=wmax, relax=P.RELAX_NONE)
    dev = lambda v: torch.tensor(v, device="cuda")  # noqa: E731
    if kind == "unsym":
        h.factor_unsym(dev(lo), dev(up))
    else:
        (h.factor_bk if kind == "pivoted" else h.factor)(dev(lo))
    h.sync_status()
    # dense unit lower factors from the panels (supernodes of consecutive columns, full below)
    out = []
    for which in (1, 3) if kind == "unsym" else (1,):
        p = h.panels(which)[0].cpu().numpy()
        M, at = np.zeros((n, n)), 0
        sn = h.symbolic()["sn_start"]
        for f, e in zip(sn[:-1], sn[1:]):
            M[f:, f:e] = p[at:at + (n - f) * (e - f)].reshape(e - f, n - f).T
            at += (n - f) * (e - f)
        out.append(np.tril(M, -1) + np.eye(n))
        if which == 1:
            d = np.diag(M).copy()
    return h, out, d


@pytest.mark.parametrize("wmax", [1, 2, 128])
@pytest.mark.parametrize("kind", ["real", "unsym", "pivoted"])
def test_subnormal_pivots(P, kind, wmax):  # noqa: F811
    L = np.array([[1, 0, 0], [0.5, 1, 0], [-0.25, 0.5, 1]])
    U = np.array([[1, 0, 0], [-0.5, 1, 0], [0.5, 0.25, 1]]) if kind == "unsym" else L
    D = np.ldexp(np.array([4.0, 8.0, 16.0]), -1060)
    A = np.ldexp((L * np.ldexp(D, 1060)) @ U.T, -1060)
    assert (D < np.ldexp(1.0, -1024)).all() and (np.ldexp(A, 1060) == (L * np.ldexp(D, 1060)) @ U.T).all()
    h, lu, d = factor(P, A, kind, wmax)
    assert np.array_equal(d, D)
    assert np.array_equal(lu[0], L) and (kind != "unsym" or np.array_equal(lu[1], U))
    want = np.log(2.0) * (2 + 3 + 4 - 3 * 1060)
    assert abs(h.logdet()[0, 0] - want) <= 1e-13 * abs(want)


@pytest.mark.parametrize("wmax", [1, 128])
@pytest.mark.parametrize("kind", ["real", "unsym", "pivoted"])
def test_pivots_near_the_overflow_limit(P, kind, wmax):  # noqa: F811
    rng = np.random.default_rng(5)
    d0 = 1.7e308
    for _ in range(20):
        c, u = rng.uniform(0.5, 1.0, 2) * 1e300
        A = np.array([[d0, u if kind == "unsym" else c], [c, 1e300]])
        _, lu, d = factor(P, A, kind, wmax)
        assert lu[0][1, 0] == c / d0 and (kind != "unsym" or lu[1][1, 0] == u / d0)
        assert d[0] == d0
