"""Generating a plan again leaves its stored spectrum readable: solves of the
plan that need neither its workspace nor a native-FP64 spectrum run on another
stream meanwhile and give the same bits.  (Generation's radial tables lie
outside the spectrum; the spectrum itself is overwritten by equal values.)"""
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
    capi.fsa_autotune_set(3)  # FP64 plans compute in double-word arithmetic
    yield fsa
    capi.fsa_autotune_set(1)


@pytest.mark.parametrize("n,L", [((64, 64, 64), (4.0, 4.0, 4.0)), ((32, 64, 48), (2.0, 4.0, 3.0)),
                                 ((32, 24, 16), (1.3, 1.7, 2.9))], ids=lambda v: "x".join(map(str, v)))
@pytest.mark.parametrize("dt", ["f32", "f64"])
def test_solves_during_regeneration(lib, n, L, dt):
    import torch
    from paper_2504_19410_gb300 import capi
    plan = lib.Plan(L, n, dt, eps=0.4, eps_tol=-1.0)
    assert dt == "f32" or plan.info.arithmetic == 2
    rho = torch.from_numpy(np.random.default_rng(4).standard_normal(n)).cuda().to(torch.float32 if dt == "f32" else torch.float64)
    want, spec = plan.apply(rho), plan.spectrum()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(4):
        got = [torch.empty_like(rho) for _ in range(40)]
        torch.cuda.synchronize()
        for i, out in enumerate(got):
            if i % 4 == 0:
                plan.generate(stream=a)
            capi.fsa_apply_noalloc(plan.handle, rho, out, b)
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in got)
    assert torch.equal(plan.spectrum(), spec)
    if dt == "f64":  # the workspace is free too
        got = [torch.empty_like(rho) for _ in range(40)]
        torch.cuda.synchronize()
        for i, out in enumerate(got):
            if i % 4 == 0:
                plan.generate(stream=a)
            plan.apply(rho, out, stream=b)
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in got)
    plan.close()
