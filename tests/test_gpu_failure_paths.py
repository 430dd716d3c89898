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


def merged_handle(P, kind, batch=2):
    """A handle whose small levels hold several groups each, and a function that factors it."""
    import torch
    p = synth.convdiff_problem(dims=(7, 6, 5)) if kind == "unsym" else synth.grid3d(7)
    h = P.SelInv(p.n, p.colptr, p.rowind, dtype=P.C128 if kind == "complex" else P.F64, unsym=int(kind == "unsym"),
                 batch=batch)
    assert np.diff(h.symbolic()["group_ptr"]).max() > 1
    dev = lambda v: torch.tensor(np.tile(v, batch), dtype=h.torch_dtype, device="cuda")  # noqa: E731
    lo = dev(p.values)
    if kind == "unsym":
        up = dev(p.values_up)
        return h, lambda: h.factor_unsym(lo, up)
    return h, lambda: (h.factor_bk if kind == "pivoted" else h.factor)(lo)


def raises(P, code, f, *a):
    with pytest.raises(P.PselinvError) as e:
        f(*a)
    assert e.value.code == code


@pytest.mark.gpu
@pytest.mark.parametrize("report", ["sync_status", "logdet"])
@pytest.mark.parametrize("kind", ["real", "complex", "unsym", "pivoted"])
def test_factorisation_wait_runs_out(P, kind, report):
    """Launched (first call) and replayed: ERR_TIMEOUT, the handle back to "not
    factored", and the next factorisation right."""
    import torch
    h, factor = merged_handle(P, kind)
    good = None
    for _ in range(2):
        h.set_debug(4)
        factor()
        raises(P, -7, getattr(h, report))
        raises(P, -8, h.selinv, P.LEVEL)
        factor()
        h.selinv(P.LEVEL)
        h.sync_status()
        if good is None:
            h2, factor2 = merged_handle(P, kind)
            factor2()
            h2.selinv(P.LEVEL)
            good = h2.panels(0)
        assert torch.equal(h.panels(0), good)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["real", "complex"])
def test_adjoint_wait_runs_out(P, kind):
    import torch
    h, factor = merged_handle(P, kind)
    factor()
    h.selinv(P.LEVEL)
    G = h.panels(0).clone()
    good = h.adjoint(G).clone()
    h.sync_status()
    for _ in range(2):
        h.set_debug(4)
        assert h.adjoint(G).isnan().all()
        raises(P, -7, h.sync_status)
        assert torch.equal(h.adjoint(G), good)  # X and the factor are untouched
        h.sync_status()


@pytest.mark.gpu
def test_adjoint_timeout_outlives_the_next_factorisation(P):
    import torch
    h, factor = merged_handle(P, "real")
    factor()
    h.selinv(P.LEVEL)
    G = h.panels(0).clone()
    good = h.adjoint(G).clone()
    h.set_debug(4)
    h.adjoint(G)
    factor()
    h.selinv(P.LEVEL)
    raises(P, -7, h.sync_status)
    h.sync_status()  # reported once
    assert torch.equal(h.adjoint(G), good)


@pytest.mark.gpu
def test_adjoint_after_an_unreported_timeout_is_right(P):
    import torch
    h, factor = merged_handle(P, "real")
    factor()
    h.selinv(P.LEVEL)
    G = h.panels(0).clone()
    good = h.adjoint(G).clone()
    h.set_debug(4)
    h.adjoint(G)
    assert torch.equal(h.adjoint(G), good)
    raises(P, -7, h.sync_status)


@pytest.mark.gpu
def test_backward_pass_whose_wait_ran_out_is_nan_and_reported(P):
    import torch
    p = synth.grid3d(7)
    h = P.SelInv(p.n, p.colptr, p.rowind)
    v = torch.tensor(p.values, device="cuda")[None].requires_grad_()
    P.selected_inverse(v, h).square().sum().backward()
    good = v.grad.clone()
    v.grad = None
    X = P.selected_inverse(v, h)
    h.set_debug(4)
    X.square().sum().backward()
    assert v.grad.isnan().all()
    raises(P, -7, P.selected_inverse, v, h)
    v.grad = None
    P.selected_inverse(v, h).square().sum().backward()
    assert torch.equal(v.grad, good)


@pytest.mark.gpu
@pytest.mark.parametrize("report", ["sync_status", "logdet"])
def test_timeout_is_reported_before_a_pivot_it_spoilt(P, report):
    """Two leaves of pivot 1 each take 1 off the root's 1: without the update that
    waits, the root's pivot is 0 instead of -1."""
    import torch
    h = P.SelInv(3, np.array([0, 2, 4, 5]), np.array([0, 2, 1, 2, 2]), relax=P.RELAX_NONE)
    assert np.diff(h.symbolic()["group_ptr"]).max() == 2
    vals = torch.ones(5, dtype=torch.float64, device="cuda")
    h.set_debug(4)
    h.factor(vals)
    raises(P, -7, getattr(h, report))
    h.factor(vals)
    assert h.logdet().tolist() == [[0.0, 1.0]]


@pytest.mark.gpu
def test_calls_go_on_without_their_graphs(P):
    """The second call captures its launches: where that fails, it launches them."""
    import torch
    h, factor = merged_handle(P, "real")
    G = None
    ref = []
    for it in range(3):
        h.set_debug(8 if it == 1 else 0)
        factor()
        h.set_debug(8 if it == 1 else 0)
        h.selinv(P.LEVEL)
        G = h.panels(0).clone() if G is None else G
        h.set_debug(8 if it == 1 else 0)
        out = [h.panels(0).clone(), h.panels(1).clone(), h.adjoint(G).clone()]
        h.sync_status()
        ref = ref or out
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["GRAPH", "PERSISTENT"])
def test_schedules_that_are_graphs_report_a_failed_capture(P, mode):
    import torch
    h, factor = merged_handle(P, "real")
    factor()
    h.set_debug(8)
    raises(P, -5, h.selinv, getattr(P, mode))
    h.selinv(getattr(P, mode))
    h.sync_status()
    X = h.panels(0).clone()
    h.selinv(P.LEVEL)
    assert torch.equal(h.panels(0), X)


@pytest.mark.gpu
def test_launches_are_counted_once_after_a_failed_capture(P):
    h, factor = merged_handle(P, "real")
    factor()
    counts = []
    for flag in (0, 8, 0, 0):
        h.set_timing(False)  # resets the counts
        h.set_debug(flag)
        h.selinv(P.LEVEL)
        counts.append(h.get_timing()[1].tolist())
    assert all(c == counts[0] for c in counts)
