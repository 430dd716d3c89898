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
    """device_bytes against what CUDA says was taken: an allocation takes whole
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


@pytest.mark.parametrize("what", ["factor", "pivoted", "persistent", "adjoint", "autotune"])
def test_call_that_ran_out_of_memory_can_be_tried_again(P, what):  # noqa: F811
    """The second of a call's allocations fails (debug switch): ERR_OOM, and the same
    call made again allocates what is missing and gives the right bits."""
    import torch
    p = synth.grid3d(7)
    vals = torch.tensor(p.values, device="cuda")

    def call(h, fail):
        out = []
        steps = {"factor": lambda: h.factor(vals), "pivoted": lambda: h.factor_bk(vals),
                 "persistent": lambda: h.selinv(P.PERSISTENT), "adjoint": lambda: out.append(h.adjoint(X)),
                 "autotune": lambda: h.autotune()}
        if what not in ("factor", "pivoted"):
            h.factor(vals)
            h.selinv(P.LEVEL)
            X = h.panels(0).clone()
        elif what == "pivoted":
            h.factor(vals)
        if fail:
            h.set_debug(16)
            with pytest.raises(P.PselinvError) as e:
                steps[what]()
            assert e.value.code == -5
        if what == "autotune":  # a schedule half replaced: refused until the next factorisation
            if fail:
                with pytest.raises(P.PselinvError) as e:
                    h.selinv(P.LEVEL)
                assert e.value.code == -8
            h.factor(vals)
        else:
            steps[what]()
        h.selinv(P.LEVEL) if what != "persistent" else None
        h.sync_status()
        return [h.panels(0).clone(), h.panels(1).clone()] + out

    new = lambda: P.SelInv(p.n, p.colptr, p.rowind)  # noqa: E731
    tuned = what == "autotune"
    for a, b in zip(call(new(), True), call(new(), False)):
        # autotune: the trial's step-2 slices stay, which sum in another order
        assert torch.allclose(a, b, rtol=0, atol=1e-13 * float(b.abs().max())) if tuned else torch.equal(a, b)
