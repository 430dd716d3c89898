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


@pytest.mark.parametrize("what", ["factor", "autotune", "persistent", "pivoted", "adjoint"])
def test_device_bytes_count_every_allocation(P, what):  # noqa: F811
    """device_bytes against what the driver says was taken: an allocation takes whole
    2 MiB blocks at most, and streams, events and graphs take some blocks more."""
    import torch
    p = synth.grid3d(30)
    vals = torch.tensor(p.values, device="cuda")

    def use():
        h = P.SelInv(p.n, p.colptr, p.rowind)
        free = torch.cuda.mem_get_info()[0]
        h.factor_bk(vals) if what == "pivoted" else h.factor(vals)
        if what == "autotune":
            h.autotune()
        h.selinv(P.PERSISTENT if what == "persistent" else P.LEVEL)
        if what == "adjoint":
            h.adjoint(G, out=grad)
        h.sync_status()
        used = free - torch.cuda.mem_get_info()[0]
        return h.info["device_bytes"], used

    h = P.SelInv(p.n, p.colptr, p.rowind)
    G = torch.zeros(h.info["panel_entries"], dtype=torch.float64, device="cuda")
    grad = torch.empty(p.nnz, dtype=torch.float64, device="cuda")
    assert h.info["device_bytes"] == 0
    use()  # modules
    said, used = use()
    assert said <= used <= said + 60 * (2 << 20)


def test_device_bytes_count_the_counters_of_a_batch(P):  # noqa: F811
    """A chain of 40 columns, 65,535 times: the counters of the schedules take some 60
    MB, more than the rounding of all allocations to 2 MiB."""
    import torch
    n, cp, ri, v = synth.laplacian_1d(40)
    batch = 65535
    vals = torch.tensor(v, device="cuda").repeat(batch)

    def use():
        h = P.SelInv(n, cp, ri, batch=batch, max_sn_width=1, relax=P.RELAX_NONE)
        free = torch.cuda.mem_get_info()[0]
        h.factor(vals)
        h.sync_status()
        return h.info["device_bytes"], free - torch.cuda.mem_get_info()[0]

    use()
    said, used = use()
    assert said <= used <= said + (40 << 20)
