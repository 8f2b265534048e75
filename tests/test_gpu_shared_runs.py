"""The shared-spectrum middle pass takes the densities of one plan in runs: every
run length its rule gives (all densities, a divisor, one) is bit-equal to
single solves with the same kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("mode", [5, 7])  # generations 4 and 8
@pytest.mark.parametrize("n,count", [((64, 64, 64), 64), ((64, 64, 64), 12), ((16, 96, 32), 7), ((8, 256, 6), 3),
                                     ((64, 128, 16), 36), ((4, 192, 8), 64)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_runs_equal_single_solves(lib, mode, n, count):
    import torch
    from paper_2504_19410_gb300 import capi
    capi.fsa_autotune_set(mode)
    plan = lib.Plan(tuple(0.25 * k for k in n), n, "f32", eps=0.4, eps_tol=-1.0)
    plan.reserve(count)
    rho = torch.from_numpy(np.random.default_rng(3).standard_normal((count,) + n).astype(np.float32)).cuda()
    got = plan.apply_many(list(rho.unbind(0)))
    one = [plan.apply(r) for r in rho.unbind(0)]
    same = [bool(torch.equal(a, b)) for a, b in zip(got, one)]
    plan.close()
    assert all(same), same
