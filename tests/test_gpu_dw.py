"""The paired double-word passes (FP64 tier) at the edges of their tiles:
every transform length on every axis, row and column counts that do not fill
a tile, and grids with many times more tiles than the GPU holds CTAs (each CTA
then takes over further tiles).  Tolerance: the FP64 tier's 1e-12 max-norm
relative error against the FP64 oracle on the same seeded input."""
import numpy as np
import pytest

import workloads as W
from oracle import fsa as oracle

pytestmark = pytest.mark.gpu
TOL = 1e-12
EPS = 0.5

# (n, kernel): all lengths 2n = 8 .. 1024 on each axis, ragged tiles, many tiles
CASES = [
    ((4, 6, 8), "coulomb3d"), ((12, 4, 6), "coulomb3d"), ((6, 24, 12), "coulomb3d"), ((16, 48, 24), "coulomb3d"),
    ((96, 4, 48), "coulomb3d"), ((4, 96, 16), "coulomb3d"), ((32, 12, 64), "coulomb3d"), ((64, 192, 4), "coulomb3d"),
    ((192, 6, 96), "coulomb3d"), ((8, 384, 6), "coulomb3d"), ((384, 4, 192), "coulomb3d"), ((6, 512, 8), "coulomb3d"),
    ((512, 6, 384), "coulomb3d"), ((4, 64, 512), "coulomb3d"), ((256, 8, 256), "coulomb3d"), ((128, 256, 32), "coulomb3d"),
    ((128, 128, 128), "coulomb3d"), ((96, 192, 64), "coulomb3d"),
    ((6, 512), "coulomb2d"), ((512, 6), "coulomb2d"), ((384, 192), "coulomb2d"), ((12, 48), "coulomb2d"),
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
    capi.fsa_autotune_set(3)  # FP64 plans: double-word
    yield fsa
    capi.fsa_autotune_set(1)
    torch.cuda.synchronize()
    assert capi.fsa_device_fault(clear=True) == 0


def solve(lib, L, n, kernel, rho, calls=2, **more):
    import torch
    plan = lib.Plan(L, n, "f64", eps=EPS, eps_tol=-1.0, kernel=kernel, **more)
    assert plan.info.arithmetic == 2
    t = torch.from_numpy(rho).cuda()
    outs = [plan.apply(t).cpu().numpy() for _ in range(calls)]
    plan.close()
    for o in outs[1:]:
        assert np.array_equal(o, outs[0])
    return outs[0]


@pytest.mark.parametrize("n,kernel", CASES, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_every_length_and_tile_edge(lib, n, kernel):
    L = tuple(0.25 * k for k in n)
    rho = np.random.default_rng(17).standard_normal(n)
    err = oracle.rel_error(solve(lib, L, n, kernel, rho), oracle.solve(L, n, EPS, rho, kernel=kernel))
    assert err <= TOL, err


@pytest.mark.parametrize("reading", ["grid", "kernel"])
@pytest.mark.parametrize("n", [(96, 48, 128), (24, 192, 8), (12, 16, 384)], ids=lambda n: "x".join(map(str, n)))
def test_ddi_unpadded_lengths(lib, n, reading):
    L = tuple(0.25 * k for k in n)
    dip = W.ddi_dipoles(3)
    rho = np.random.default_rng(18).standard_normal(n)
    got = solve(lib, L, n, "ddi3d", rho, dipoles=dip, ddi_derivative=reading)
    err = oracle.rel_error(got, oracle.ddi3d_solve(L, n, EPS, rho, dip[0], dip[1], reading))
    assert err <= TOL, err
