"""Dense matrices whose supernodes have the widths where the blocked kernels of
the diagonal blocks (factorisation, inverse, normalisation) change path: one
fragment, one block, a ragged last block, the widest, with and without rows
below.  Tolerance 1e-10 of max |X|, the bar of every oracle comparison; the
matrices have condition numbers below 1e3, so rounding stays under 1e-12."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
TOL = 1e-10
SIZES = [(1, 128), (8, 128), (9, 8), (31, 128), (32, 128), (33, 32), (64, 128), (65, 128), (96, 33), (127, 128),
         (128, 128), (129, 128), (161, 100), (300, 128)]


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1404_0447_gb300 as P
    return P


def dense(n, cplx, unsym, indefinite=False):
    g = np.random.default_rng(1000 * n + 2 * cplx + unsym)
    a = g.normal(size=(n, n)) + (1j * g.normal(size=(n, n)) if cplx else 0.0)
    if not unsym:
        a = (a + a.T) / 2
    shift = 3.0 * np.sqrt(n) * (np.where(g.random(n) < 0.5, -1.0, 1.0) if indefinite else 1.0)
    return a + np.diag(shift * np.ones(n))


def stored(A):
    n = A.shape[0]
    cols, rows = np.nonzero(np.triu(np.ones((n, n), bool)))
    cp, ri, lo = synth.lower_csc_from_coo(n, rows, cols, A[rows, cols])
    c = np.repeat(np.arange(n), np.diff(cp))
    return cp, ri, lo, A[c, ri], c


@pytest.mark.parametrize("kind", ["real", "complex", "unsym", "unsym_complex", "pivoted", "pivoted_complex"])
@pytest.mark.parametrize("n,wmax", SIZES)
def test_dense_block_widths(P, kind, n, wmax):
    import torch
    cplx, unsym, piv = "complex" in kind, kind.startswith("unsym"), kind.startswith("pivoted")
    A = dense(n, cplx, unsym, indefinite=piv)
    cp, ri, lo, up, c = stored(A)
    h = P.SelInv(n, cp, ri, dtype=P.C128 if cplx else P.F64, max_sn_width=min(wmax, 112 if unsym and cplx else 128),
                 relax=P.RELAX_NONE, unsym=int(unsym))
    dev = lambda v: torch.tensor(v, dtype=h.torch_dtype, device="cuda")  # noqa: E731
    if unsym:
        h.factor_unsym(dev(lo), dev(up))
    elif piv:
        h.factor_bk(dev(lo))
    else:
        h.factor(dev(lo))
    h.selinv(P.LEVEL)
    h.sync_status()
    X = np.linalg.inv(A)
    top = np.abs(X).max()
    assert np.max(np.abs(h.selected()[0].cpu().numpy() - X[ri, c])) / top <= TOL
    if unsym:
        assert np.max(np.abs(h.selected_upper()[0].cpu().numpy() - X[c, ri])) / top <= TOL
