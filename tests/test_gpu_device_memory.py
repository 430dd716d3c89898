"""Device memory held by a handle."""
import numpy as np
import pytest

import synth
from test_gpu_dense_widths import P, dense, stored  # noqa: F401

pytestmark = pytest.mark.gpu


def test_logdet_partials_are_sized_by_the_order(P):  # noqa: F811
    """A batch of 65,535 matrices of order 5 has one partial sum per member, not 128
    (2 kB each, 134 MB): what a factorisation takes is about the arrays themselves."""
    import torch
    n, batch = 5, 65535
    cp, ri, lo, _, _ = stored(dense(n, False, False))

    def taken(batch):
        h = P.SelInv(n, cp, ri, batch=batch)
        v = torch.tensor(np.tile(lo, (batch, 1)), device="cuda")
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        h.factor(v)
        ld = h.logdet()
        assert np.array_equal(ld, np.tile(ld[:1], (batch, 1)))
        return free - torch.cuda.mem_get_info()[0], h.info["panel_entries"]

    taken(1)  # modules and streams
    used, entries = taken(batch)
    arrays = batch * 8 * (2 * entries + 25 + 5 + 6 + 2)  # L and X, (L_KK)^-1, D, log det and weights
    assert used < arrays + (48 << 20)
