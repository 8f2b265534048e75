"""Generation 8's kernels for transform lengths 768 and 1024 (n = 384, 512) on
each axis, within the FP32 tolerance of the oracle: grids whose columns do not
fill a tile, grids of many more tiles than CTAs, and densities of one plan
(bit-equal to single solves)."""
import numpy as np
import pytest

from oracle import fsa as oracle

pytestmark = pytest.mark.gpu
TOL = 2e-6
EPS = 0.5
# axis 0 (R2C, C2R), axis 1 (middle), both; ragged columns; many tiles
CASES = [(384, 4, 8), (512, 6, 4), (384, 6, 6), (512, 16, 24), (4, 384, 8), (8, 512, 4), (6, 384, 6), (16, 512, 24),
         (512, 384, 8), (384, 512, 16), (24, 384, 96), (32, 512, 64)]


@pytest.fixture(scope="module")
def lib():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_2504_19410_gb300 as fsa
    from paper_2504_19410_gb300 import capi
    capi.fsa_device_fault(clear=True)
    yield fsa
    capi.fsa_autotune_set(1)
    torch.cuda.synchronize()
    assert capi.fsa_device_fault(clear=True) == 0


def solve(lib, mode, n, rhos):
    import torch
    from paper_2504_19410_gb300 import capi
    capi.fsa_autotune_set(mode)
    plan = lib.Plan(tuple(0.25 * k for k in n), n, "f32", eps=EPS, eps_tol=-1.0)
    t = [torch.from_numpy(r).cuda() for r in rhos]
    if len(t) > 1:
        plan.reserve(len(t))
        out = plan.apply_many(t)
    else:
        out = [plan.apply(t[0])]
    got = [o.cpu().numpy() for o in out]
    plan.close()
    return got


@pytest.mark.parametrize("n", CASES, ids=lambda n: "x".join(map(str, n)))
def test_long_lines(lib, n):
    rng = np.random.default_rng(5)
    rhos = [rng.standard_normal(n).astype(np.float32) for _ in range(3)]
    many = solve(lib, 7, n, rhos)
    for g, r in zip(many, rhos):
        assert np.array_equal(g, solve(lib, 7, n, [r])[0])
    err = oracle.rel_error(many[-1], oracle.solve(tuple(0.25 * k for k in n), n, EPS, rhos[-1].astype(np.float64)))
    assert err <= TOL, err
