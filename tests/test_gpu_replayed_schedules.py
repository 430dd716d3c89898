"""Repeated calls on one handle: the level loops of the factorisation, the
LEVEL sweep and the adjoint are replayed from a graph from the second call on.
New values, the other kind of factor and a rebuilt schedule must give what a
handle used for the first time gives, bit for bit (same kernels, same order)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    import paper_1404_0447_gb300 as P
    return P


def once(P, p, vals, pivoted, **opts):
    h = P.SelInv(p.n, p.colptr, p.rowind, **opts)
    (h.factor_bk if pivoted else h.factor)(vals)
    h.selinv(P.LEVEL)
    return h.panels(0)


@pytest.mark.parametrize("mode", ["LEVEL", "GRAPH", "PERSISTENT"])
def test_values_and_kind_of_factor_change_between_replays(P, mode):
    import torch
    p = synth.grid3d(9)
    g = np.random.default_rng(1)
    h = P.SelInv(p.n, p.colptr, p.rowind, max_sn_width=40)
    for it in range(6):
        v = p.values.copy()
        diag = p.colptr[:-1]
        # indefinite values on the pivoted turns, so that its pivots differ from the identity
        v[diag] += g.uniform(0.0, 1.0, p.n) - (5.0 if it % 3 == 2 else 0.0)
        vals = torch.tensor(v, device="cuda")
        piv = it % 3 == 2
        (h.factor_bk if piv else h.factor)(vals)
        h.selinv(getattr(P, mode))
        assert torch.equal(h.panels(0), once(P, p, vals, piv, max_sn_width=40))


def test_adjoint_replays_and_user_capture(P):
    import torch
    p = synth.grid3d(7)
    h = P.SelInv(p.n, p.colptr, p.rowind)
    vals = torch.tensor(p.values, device="cuda")
    outs = []
    for it in range(4):
        G = torch.randn(h.info["panel_entries"], dtype=torch.float64, device="cuda",
                        generator=torch.Generator("cuda").manual_seed(it % 2))
        h.factor(vals)
        h.selinv(P.LEVEL)
        outs.append(h.adjoint(G, P.G_PANEL))
    assert torch.equal(outs[0], outs[2]) and torch.equal(outs[1], outs[3])
    assert not torch.equal(outs[0], outs[1])
    # inside the caller's own capture the launches themselves are recorded
    ref = h.selected()
    out = torch.zeros_like(ref)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        h.factor(vals)
        h.selinv(P.LEVEL)
        h.selected(out=out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_autotune_drops_the_captured_schedules(P):
    import torch
    p = synth.grid3d(8)
    h = P.SelInv(p.n, p.colptr, p.rowind)
    vals = torch.tensor(p.values, device="cuda")
    for _ in range(3):
        h.factor(vals)
        h.selinv(P.LEVEL)
    x = h.selected()
    h.autotune()
    for _ in range(3):
        h.factor(vals)
        h.selinv(P.LEVEL)
        assert torch.allclose(h.selected(), x, rtol=1e-12, atol=1e-12)
