"""Tensor generation: the radial tables and the symmetry-pruned DCT passes
against the oracle's tensor, over every transform length and on both sides of
each rule that picks the tables (common integer ratios of the squared mesh
steps for U^eps, of the squared box lengths for W, a table of at most a quarter
of the octant).  FP64 tolerance: each of the three transforms rounds about
log2(2n) <= 10 times at 2^-53 relative to the largest entry, the oracle's FFTs
likewise: 64 * 2^-53 of the largest value.  FP32 adds one rounding (2^-24)."""
import numpy as np
import pytest

from oracle import fsa as oracle

pytestmark = pytest.mark.gpu
EPS = 0.3

CASES = [
    ((12, 12, 12), (1.5, 1.5, 1.5)),      # cube: both tables (q = 433 of 2197 points)
    ((8, 8, 8), (1.0, 1.0, 1.0)),         # cube too small for a table
    ((24, 48, 96), (1.55, 3.1, 6.2)),     # one mesh step, boxes 1 : 2 : 4
    ((32, 48, 64), (2.0, 3.0, 4.0)),      # boxes 2 : 3 : 4 (squares 4 : 9 : 16 after scaling)
    ((64, 64, 128), (4.0, 4.0, 4.0)),     # one box, mesh steps 2 : 2 : 1
    ((48, 32, 64), (3.0, 4.0, 4.0)),      # mesh steps 1 : 2 : 1
    ((32, 24, 16), (1.3, 1.7, 2.9)),      # no common ratio
    ((16, 6, 4), (2.0, 0.75, 0.5)),       # one mesh step, odd first-stage counts
    ((192, 16, 48), (24.0, 2.0, 6.0)),    # flat box: table above a quarter of the octant
    ((384, 12, 64), (12.0, 0.375, 2.0)), ((8, 512, 16), (0.25, 16.0, 0.5)), ((128, 4, 256), (8.0, 0.25, 16.0)),
    ((96, 192, 64), (6.0, 12.0, 4.0)),
]


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2504_19410_gb300 as fsa
    return fsa


@pytest.mark.parametrize("kernel", ["coulomb3d", "biharmonic3d"])
@pytest.mark.parametrize("n,L", CASES, ids=lambda v: "x".join(map(str, v)))
def test_spectrum_with_and_without_tables(lib, n, L, kernel):
    want = oracle.spectrum_octant(oracle.tensor_T(L, n, EPS, kernel=kernel), n)
    top = np.abs(want).max()
    for dt in ("f64", "f32"):
        plan = lib.Plan(L, n, dt, eps=EPS, eps_tol=-1.0, kernel=kernel)
        first = plan.spectrum().double().cpu().numpy()
        plan.generate()  # again: the tables' memory holds other data by now
        got = plan.spectrum().double().cpu().numpy()
        plan.close()
        assert np.array_equal(first, got)
        tol = 64 * 2.0 ** -53 * top + (0 if dt == "f64" else 2.0 ** -24 * np.abs(want))
        assert (np.abs(got - want) <= tol).all(), (dt, np.abs(got - want).max() / top)
