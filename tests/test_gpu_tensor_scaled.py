"""Tensor generation through the radial tables whose base is a half or a third of
the smallest step (tests/test_radial_rule.py has these grids' ratios): against
the oracle's tensor.  FP64 tolerance as in the other tensor tests: each of the three transforms
rounds about log2(2n) <= 10 times at 2^-53 relative to the largest entry, the
oracle's FFTs likewise: 64 * 2^-53 of the largest value; FP32 adds one rounding
(2^-24)."""
import numpy as np
import pytest

from oracle import fsa as oracle

pytestmark = pytest.mark.gpu
EPS = 0.5

CASES = [
    ((128, 128, 128), (8.0, 8.0, 12.0)),   # mesh steps 2 : 2 : 3, boxes 3 : 3 : 2, both in halves
    ((192, 192, 96), (12.0, 12.0, 8.0)),   # mesh steps 3 : 3 : 4 in thirds, boxes 2 : 2 : 3 in halves
    ((192, 192, 96), (16.0, 16.0, 12.0)),  # mesh steps 2 : 2 : 3 in halves, boxes 3 : 3 : 4 in thirds
]


@pytest.mark.parametrize("n,L", CASES, ids=lambda v: "x".join(map(str, v)))
def test_spectrum_from_scaled_tables(n, L):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2504_19410_gb300 as fsa
    want = oracle.spectrum_octant(oracle.tensor_T(L, n, EPS), n)
    top = np.abs(want).max()
    for dt in ("f64", "f32"):
        plan = fsa.Plan(L, n, dt, eps=EPS, eps_tol=-1.0)
        got = plan.spectrum().double().cpu().numpy()
        plan.close()
        tol = 64 * 2.0 ** -53 * top + (0 if dt == "f64" else 2.0 ** -24 * np.abs(want))
        assert (np.abs(got - want) <= tol).all(), (dt, np.abs(got - want).max() / top)
