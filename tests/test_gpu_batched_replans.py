"""Batched solves after their plans are destroyed and made anew (often at the
same host addresses, with the same density buffers): the batch is captured
again, for the new plans' workspaces and spectra."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_destroyed_plans_drop_their_batch_graphs():
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2504_19410_gb300 as fsa

    shapes = [(16, 24, 32), (32, 16, 8), (64, 64, 64)]
    rng = np.random.default_rng(9)
    rhos = [torch.from_numpy(rng.standard_normal(n)).cuda() for n in shapes]
    phis = [torch.empty_like(r) for r in rhos]
    keep = []
    for step in range(6):
        scale = 1.0 + 0.25 * step  # another box: another spectrum
        plans = [fsa.Plan(tuple(0.25 * scale * k for k in n), n, "f64", eps=0.5, eps_tol=-1.0) for n in shapes]
        fsa.apply_batched(plans, rhos, phis)
        got = [p.clone() for p in phis]
        for p, r, a in zip(plans, rhos, got):
            assert torch.equal(p.apply(r), a)
        # other device memory in between, so that new workspaces lie elsewhere
        keep.append(torch.empty((1 << 22) * (step + 1), device="cuda"))
        for p in plans:
            p.close()
