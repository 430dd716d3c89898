"""Batches beyond half the limit of a grid dimension (65,535): two sides per member
must not share one.  Members repeat a few values; each is checked against the same
matrix on a handle of its own, bit for bit."""
import numpy as np
import pytest

import synth
from test_gpu_dense_widths import P, dense, stored  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("batch", [32767, 32768, 65535])
def test_unsym_batch_up_to_the_grid_limit(P, batch, cplx):  # noqa: F811
    import torch
    n, kinds = 5, 3
    mats = [stored(dense(n, cplx, True) + k * np.eye(n)) for k in range(kinds)]
    cp, ri = mats[0][:2]

    def run(members, reps):
        h = P.SelInv(n, cp, ri, dtype=P.C128 if cplx else P.F64, unsym=1, max_sn_width=2, relax=P.RELAX_NONE,
                     batch=len(members))
        assert h.info["nlevels"] == 3  # two levels update others
        dev = lambda q: torch.tensor(np.stack([m[q] for m in members]), dtype=h.torch_dtype, device="cuda")  # noqa: E731
        lo, up = dev(2), dev(3)
        for _ in range(reps):  # launched, then replayed
            h.factor_unsym(lo, up)
            h.selinv(P.LEVEL)
            h.sync_status()
        return h.selected(), h.selected_upper()

    got = run([mats[b % kinds] for b in range(batch)], 2)
    for k in range(kinds):
        for g, w in zip(got, run([mats[k]], 1)):
            assert torch.equal(g[k::kinds], w.expand(g[k::kinds].shape))
