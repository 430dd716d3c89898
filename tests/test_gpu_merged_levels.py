"""Dense matrices whose chain of supernodes crosses the size at which a level's
updates of the ancestors stop running as one launch (9728 tiles of 16 x 8 real,
4864 complex, 1216 pivoted: |C| about 1580, 1110, 550), and small ones on the
merged side with ragged widths; the factorisation, the selected inverse and, on
the pivot-free symmetric factor, the adjoint.  Block inverses at the orders where
their blocks and strips end.  Tolerance 1e-10 of the largest entry: condition
numbers below 10 leave rounding below 1e-12."""
import numpy as np
import pytest

from test_gpu_adjoint import dense_G_from_panels, expected_grad, panel_positions
from test_gpu_dense_widths import P, dense, stored  # noqa: F401
from test_zz_no_alloc import factor_blocks

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("kind,n", [("real", 1800), ("complex", 1300), ("unsym", 1500), ("pivoted", 800)])
def test_chain_crosses_the_merged_limit(P, kind, n):  # noqa: F811
    import torch
    cplx, unsym, piv = kind == "complex", kind == "unsym", kind == "pivoted"
    A = dense(n, cplx, unsym, indefinite=piv)
    cp, ri, lo, up, c = stored(A)
    h = P.SelInv(n, cp, ri, dtype=P.C128 if cplx else P.F64, relax=P.RELAX_NONE, unsym=int(unsym))
    dev = lambda v: torch.tensor(v, dtype=h.torch_dtype, device="cuda")  # noqa: E731
    for _ in range(2):  # launched, then replayed
        h.factor_unsym(dev(lo), dev(up)) if unsym else h.factor_bk(dev(lo)) if piv else h.factor(dev(lo))
        h.selinv(P.LEVEL)
        h.sync_status()
        X = np.linalg.inv(A)
        assert np.abs(h.selected()[0].cpu().numpy() - X[ri, c]).max() <= TOL * np.abs(X).max()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,wmax", [(9, 8), (50, 17), (129, 128), (161, 33), (300, 128), (1800, 128)])
def test_adjoint_merged_updates(P, n, wmax, cplx):  # noqa: F811
    import torch
    A = dense(n, cplx, False)
    cp, ri, lo, _, c = stored(A)
    batch = 1 if n > 1000 else 2
    h = P.SelInv(n, cp, ri, dtype=P.C128 if cplx else P.F64, max_sn_width=wmax, relax=P.RELAX_NONE, batch=batch)
    h.factor(torch.tensor(np.tile(lo, (batch, 1)), dtype=h.torch_dtype, device="cuda"))
    h.selinv(P.LEVEL)
    sym = h.symbolic()
    rows, cols = panel_positions(sym)
    g = np.random.default_rng(n)
    G = g.normal(size=(batch, rows.size)) + (1j * g.normal(size=(batch, rows.size)) if cplx else 0)
    for _ in range(2):  # launched, then replayed
        got = h.adjoint(torch.tensor(G, dtype=h.torch_dtype, device="cuda")).cpu().numpy()
        h.sync_status()
        for b in range(batch):
            want = expected_grad(n, cp, ri, A, dense_G_from_panels(n, sym, G[b], rows, cols), sym["perm"])
            assert np.abs(got[b] - want).max() <= TOL * np.abs(want).max()


@pytest.mark.parametrize("s", [1, 8, 31, 32, 33, 64, 65, 96, 127])
def test_block_inverse_orders(P, s):  # noqa: F811
    mats, Lp, d, _ = factor_blocks(P, s, 3, s)
    M = P.block_inverse_static(Lp, d).cpu().numpy().reshape(3, s, s).transpose(0, 2, 1)
    for b, A in enumerate(mats):
        Ai = np.linalg.inv(A)
        assert np.abs(M[b] - Ai).max() <= TOL * np.abs(Ai).max()
