"""Bounded device waits that run out: what each call reports, the state it leaves
and the recovery of the handle.  The waits are made to run out by the library's
own debug switches; every launch ends by its limit and reports a status."""
import os

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1404_0447_gb300 as P
    return P


def test_persistent_abort_flag_is_read_once_per_cta():
    """Threads of a CTA that each read the flag can see different values and then
    meet different barriers: the flag is read by one thread, before the barrier
    that publishes the task."""
    text = open(os.path.join(ROOT, "paper_1404_0447_gb300", "csrc", "persistent.cu")).read()
    loop = text[text.index("for (;;)"):]
    read = "volatile int*)(status + 2)"
    assert loop.count(read) == 1
    dequeue = loop[:loop.index("__syncthreads()")]
    assert dequeue.index("if (threadIdx.x == 0) {") < dequeue.index(read)


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [1, 6])
def test_persistent_timeouts_with_many_tasks_in_flight(P, batch):
    """Several timeouts in a row on one handle, each while every SM holds tasks; the
    launch after each gives the bits of the first."""
    import torch
    p = synth.grid3d(14)
    h = P.SelInv(p.n, p.colptr, p.rowind, batch=batch, spin_limit_ns=2_000_000)
    h.factor(torch.tensor(np.tile(p.values, batch), device="cuda"))
    h.selinv(P.PERSISTENT)
    h.sync_status()
    good = h.panels(0).clone()
    for _ in range(4):
        h.set_debug(2)
        h.selinv(P.PERSISTENT)
        with pytest.raises(P.PselinvError) as e:
            h.sync_status()
        assert e.value.code == -7
        h.selinv(P.PERSISTENT)
        h.sync_status()
        assert torch.equal(h.panels(0), good)
