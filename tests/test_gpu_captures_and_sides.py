"""The adjoint's two streams inside the caller's own capture, and a batch of
non-symmetric matrices (two copies per member in the merged launches) against
handles of their own: equal bits in both."""
import numpy as np
import pytest

import synth
from test_gpu_dense_widths import P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m", [7, 13])
def test_adjoint_in_the_callers_capture(P, m, cplx):  # noqa: F811
    import torch
    p = synth.grid3d(m)
    h = P.SelInv(p.n, p.colptr, p.rowind, dtype=P.C128 if cplx else P.F64)
    c = np.repeat(np.arange(p.n), np.diff(p.colptr))
    values = [torch.tensor(p.values + (p.rowind == c) * (0.5 + k) * (1 + 0.25j if cplx else 1), dtype=h.torch_dtype,
                           device="cuda") for k in range(3)]
    seeds = [torch.randn(h.info["panel_entries"], dtype=h.torch_dtype, device="cuda",
                         generator=torch.Generator("cuda").manual_seed(k)) for k in range(3)]

    def eager(k):
        h.factor(values[k])
        h.selinv(P.LEVEL)
        return h.adjoint(seeds[k], P.G_PANEL).clone()

    want = [eager(k) for k in range(3)]  # launched, captured, replayed
    v, G = values[0].clone(), seeds[0].clone()
    out = torch.empty(1, p.nnz, dtype=h.torch_dtype, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        h.factor(v)
        h.selinv(P.LEVEL)
        h.adjoint(G, P.G_PANEL, out=out)
    for k in (1, 2, 0):
        v.copy_(values[k])
        G.copy_(seeds[k])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want[k])
        assert torch.equal(eager(k), want[k])  # the handle's own graphs beside it
    h.sync_status()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("batch", [3, 40])
def test_unsym_member_bits_do_not_depend_on_the_batch(P, batch, cplx):  # noqa: F811
    import torch
    p = synth.convdiff_problem(dims=(11, 10, 9))
    rng = np.random.default_rng(batch)
    c = np.repeat(np.arange(p.n), np.diff(p.colptr))
    shift = [(p.rowind == c) * rng.uniform(0, 1) * (1 + 1j if cplx else 1) for _ in range(batch)]
    lo, up = (np.stack([v + s for s in shift]) for v in (p.values, p.values_up))

    def run(lo, up):
        h = P.SelInv(p.n, p.colptr, p.rowind, dtype=P.C128 if cplx else P.F64, unsym=1, batch=len(lo))
        dev = lambda v: torch.tensor(v, dtype=h.torch_dtype, device="cuda")  # noqa: E731
        h.factor_unsym(dev(lo), dev(up))
        h.selinv(P.LEVEL)
        h.sync_status()
        return [h.panels(w).clone().view(len(lo), -1) for w in range(4)]

    for a, b in zip(run(lo, up), run(lo[-1:], up[-1:])):
        assert torch.equal(a[-1], b[0])
