"""Both shared-spectrum middle passes (the tensor-copy one, and the prefetching
one that widths and lengths without tensor copies take) at run lengths that are
one, a proper divisor, and all of the densities: bit-equal to single solves.
The runs named are those of the rule (shared_run) on 152 SMs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [  # generations, n, count
    (4, (128, 64, 128), 6),   # tensor copies, length 128: run 6 of 6
    (8, (128, 128, 128), 5),  # length 256: run 5 of 5
    (8, (64, 64, 64), 64),    # run 16 of 64
    (8, (64, 192, 64), 9),    # length 384: run 1 of 9
    (4, (256, 32, 128), 6),   # prefetching, length 64: run 6 of 6
    (4, (128, 32, 128), 6),   # run 3 of 6
    (4, (64, 32, 64), 64),    # run 8 of 64
    (8, (64, 64, 12), 32),    # 24 columns, no tensor map: run 2 of 32
    (8, (48, 96, 12), 40),    # run 2 of 40
    (4, (64, 384, 32), 8),    # length 768 without an exact tensor-copy kernel: run 2 of 8
    (4, (16, 512, 32), 16),   # length 1024: run 1 of 16
]


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


@pytest.mark.parametrize("gen,n,count", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_runs_equal_single_solves(lib, gen, n, count):
    import torch
    from paper_2504_19410_gb300 import capi
    capi.fsa_autotune_set({4: 5, 8: 7}[gen])
    plan = lib.Plan(tuple(0.25 * k for k in n), n, "f32", eps=0.4, eps_tol=-1.0)
    plan.reserve(count)
    rho = torch.from_numpy(np.random.default_rng(5).standard_normal((count,) + n).astype(np.float32)).cuda()
    got = plan.apply_many(list(rho.unbind(0)))
    same = [bool(torch.equal(a, plan.apply(r))) for a, r in zip(got, rho.unbind(0))]
    plan.close()
    assert all(same), same
