"""A batch member's factor, selected inverse and gradient have the bits of a handle
of its own: the rules that choose tiles and merged launches count one member's work.
Batch sizes that would cross those rules' lines if they counted the whole batch."""
import numpy as np
import pytest

import synth
from test_gpu_dense_widths import P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["real", "complex", "pivoted"])
@pytest.mark.parametrize("batch", [3, 40])
def test_member_bits_do_not_depend_on_the_batch(P, kind, batch):  # noqa: F811
    import torch
    p = synth.grid3d(12)
    dt = P.C128 if kind == "complex" else P.F64
    rng = np.random.default_rng(batch)
    c = np.repeat(np.arange(p.n), np.diff(p.colptr))
    vals = np.stack([p.values + (p.rowind == c) * rng.uniform(0, 1) * (1j if kind == "complex" else 1)
                     for _ in range(batch)])

    def run(v):
        h = P.SelInv(p.n, p.colptr, p.rowind, dtype=dt, batch=len(v))
        t = torch.tensor(v, dtype=h.torch_dtype, device="cuda")
        h.factor_bk(t) if kind == "pivoted" else h.factor(t)
        h.selinv(P.LEVEL)
        X = h.panels(0).clone()
        out = [X, h.panels(1).clone()]
        if kind != "pivoted":
            out.append(h.adjoint(X))
        h.sync_status()
        return [o.view(len(v), -1) for o in out]

    whole, last = run(vals), run(vals[-1:])
    for a, b in zip(whole, last):
        assert torch.equal(a[-1], b[0])
