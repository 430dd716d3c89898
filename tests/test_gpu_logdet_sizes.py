"""log det at the orders where its partial sums change in number (256 per CTA, at most
128 CTAs), batch members included.  Diagonal matrices: the pivots are the entries.
Tolerance: n roundings of 1.1e-16 on sums of |log| <= 1.4 n give 2e-16 n^2 at the very
worst; a tree of 256-term sums stays below 1e-13 n."""
import numpy as np
import pytest

from test_gpu_dense_widths import P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 513, 32767, 32768, 33000])
def test_logdet_of_a_diagonal(P, n, cplx):  # noqa: F811
    import torch
    rng = np.random.default_rng(n)
    d = rng.uniform(0.25, 4.0, (2, n)) * np.where(rng.random((2, n)) < 0.3, -1.0, 1.0)
    if cplx:
        d = d * np.exp(1j * rng.uniform(-1.0, 1.0, (2, n)))
    h = P.SelInv(n, np.arange(n + 1), np.arange(n), dtype=P.C128 if cplx else P.F64, batch=2)
    h.factor(torch.tensor(d, dtype=h.torch_dtype, device="cuda"))
    got = h.logdet()
    want = np.stack([np.log(np.abs(d)).sum(1), np.angle(d).sum(1) if cplx else (d < 0).sum(1)], 1)
    assert np.abs(got - want).max() <= 1e-13 * n
