"""The solves whose speed this repository is measured by.

Each case is work that a user of the package has it do through its public
entry points (``Plan``, ``Plan.apply``, ``Plan.apply_many``, ``Plan.generate``)
on synthetic 8-Gaussian densities:

  apply   one density through one plan that the program keeps
  many    a batch of densities through one plan in one call
  precomp the plan's tensor spectrum (the paper's Precomp phase); the output
          is the spectrum octant that ``Plan.spectrum`` copies out

``exact`` computes the same values in FP64 with plain torch on the doubled
grid: Phi = crop(iDFT((DFT(T1) + W) DFT(pad(rho)))), T1 = prod(h) U^eps on the
doubled grid's offsets, W the transform of U - U^eps.
"""
import math

import torch

import paper_2504_19410_gb300 as fsa

DTYPES = {"f32": torch.float32, "f64": torch.float64}
# dipole orientations of the paper's DDI example
DIP_N = (0.82778, 0.41505, -0.37751)
DIP_M = (0.3118, 0.9378, -0.15214)


def _case(name, op, kernel, dtype, n, L, eps, count=1):
    d = {"name": name} if name else {}
    d.update(op=op, kernel=kernel, dtype=dtype, n0=n[0], n1=n[1], n2=n[2] if len(n) > 2 else 0,
             L0=L[0], L1=L[1], L2=L[2] if len(L) > 2 else 0.0, eps=eps, count=count)
    return d


def listed():
    box = (16.0, 16.0, 16.0)
    return [
        # the smallest 3-D solve in use (the 32^3 isotropic Gaussian on [-8,8]^3): launches and latency
        _case("cube_32_f32", "apply", "coulomb3d", "f32", (32, 32, 32), (8.0, 8.0, 8.0), 1.0),
        # the d = 2 path in the paper's precision
        _case("plane_512_f64", "apply", "coulomb2d", "f64", (512, 512), (16.0, 16.0), 1.0),
        # uneven axes of the 3 * 2^a sizes: every pass has a length of its own
        _case("ragged_96x48x192_f32", "apply", "coulomb3d", "f32", (96, 48, 192), (12.0, 6.0, 24.0), 1.0),
        # an ordinary single-precision solve that fits in cache
        _case("cube_128_f32", "apply", "coulomb3d", "f32", (128, 128, 128), box, 1.0),
        # the dipole-dipole potential of Example 4, grid reading (ten passes), double precision
        _case("ddi_96_f64", "apply", "ddi3d", "f64", (96, 96, 96), (8.0, 8.0, 8.0), 1.0),
        # a time-dependent solver's batch: many small densities through one plan
        _case("many_64x64_f32", "many", "coulomb3d", "f32", (64, 64, 64), box, 1.0, 64),
        # the paper's 192^3 double-precision run (Example 2)
        _case("cube_192_f64", "apply", "coulomb3d", "f64", (192, 192, 192), (12.0, 12.0, 12.0), 1.0),
        # the headline solve, both precisions
        _case("cube_256_f32", "apply", "coulomb3d", "f32", (256, 256, 256), box, 1.0),
        _case("cube_256_f64", "apply", "coulomb3d", "f64", (256, 256, 256), box, 1.0),
        # the pancake: the longest transforms on two axes
        _case("pancake_512x512x128_f32", "apply", "coulomb3d", "f32", (512, 512, 128), (16.0, 16.0, 2.0), 0.4),
        # a new plan's tensor in double precision: what a plan-cache miss pays
        _case("precomp_256_f64", "precomp", "coulomb3d", "f64", (256, 256, 256), box, 1.0),
        # the largest grid the library takes
        _case("cube_512_f32", "apply", "coulomb3d", "f32", (512, 512, 512), box, 1.0),
    ]


SIZES = (16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512)


def draw(rng):
    """Sizes per axis spread evenly over the supported lengths (2^a, 3 2^a), a
    box of the grid's proportions, either precision, every operation."""
    op = rng.choice(("apply", "apply", "apply", "apply", "plane", "ddi", "many", "precomp"))
    dtype = rng.choice(("f32", "f64"))
    h = rng.choice((0.125, 0.25))
    # the largest listed case is 512^3 FP32: a drawn one stays below its cost
    # (double precision costs about six times as much per point)
    most = {"apply": 2 ** 26, "ddi": 2 ** 24, "many": 2 ** 22, "precomp": 2 ** 24, "plane": 2 ** 18}[op]
    if dtype == "f64":
        most //= 4
    while True:
        if rng.random() < 0.3:
            n = (rng.choice(SIZES[1:]),) * 3
        else:
            n = tuple(rng.choice(SIZES) for _ in range(3))
        if op == "plane":
            n = n[:2]
            most = 2 ** 18
        if math.prod(n) <= most and math.prod(n) >= 2 ** 12:
            break
    L = tuple(0.5 * h * k for k in n)
    eps = min(0.5, 2.0 * min(L) / 7.0)
    if op == "plane":
        return _case(None, "apply", "coulomb2d", dtype, n, L, eps)
    if op == "ddi":
        return _case(None, "apply", "ddi3d", dtype, n, L, eps)
    count = rng.randint(2, 64) if op == "many" else 1
    while op == "many" and count > 2 and count * math.prod(n) > 2 ** 24:
        count //= 2
    return _case(None, op, rng.choice(("coulomb3d", "coulomb3d", "biharmonic3d")) if op != "precomp" else "coulomb3d",
                 dtype, n, L, eps, count)


def _shape(case):
    return tuple(case[k] for k in ("n0", "n1", "n2") if case[k])


def _box(case):
    return tuple(case[k] for k in ("L0", "L1", "L2") if case[k])


def _density(case, seed):
    """count densities of 8 Gaussians each (centres in the middle quarter of
    the box, widths 1/32 .. 1/10 of the narrowest half-width's span), FP64."""
    n, L = _shape(case), _box(case)
    g = torch.Generator().manual_seed(int(seed))
    out = torch.zeros((case["count"],) + n, dtype=torch.float64, device="cuda")
    x = [torch.linspace(-Lj, Lj, nj + 1, dtype=torch.float64, device="cuda")[:-1] for Lj, nj in zip(L, n)]
    for k in range(case["count"]):
        for _ in range(8):
            u = torch.rand(5, generator=g, dtype=torch.float64).tolist()
            amp, w = 2.0 * u[0] - 1.0, 1.0 / 16.0 + u[1] * (0.2 - 1.0 / 16.0)
            e = [torch.exp(-0.5 * ((xj / Lj - 0.5 * (u[2 + j] - 0.5)) / w) ** 2) for j, (xj, Lj) in enumerate(zip(x, L))]
            prod = amp * e[0]
            for f in e[1:]:
                prod = prod.unsqueeze(-1) * f
            out[k] += prod
    return out.to(DTYPES[case["dtype"]])


def _plan(case, generate=True):
    more = {"dipoles": (DIP_N, DIP_M), "ddi_derivative": "grid"} if case["kernel"] == "ddi3d" else {}
    return fsa.Plan(_box(case), _shape(case), case["dtype"], eps=case["eps"], eps_tol=-1.0, kernel=case["kernel"],
                    generate=generate, **more)


def prepare(case, seed):
    """A program's own objects: the plan (spectrum and workspace), the
    densities and the buffers for the potentials, on the device."""
    if case["op"] == "precomp":
        # the seed moves the box a little: another plan's tensor
        c = dict(case)
        s = 1.0 + 0.001 * (int(seed) % 97)
        c.update(L0=case["L0"] * s, L1=case["L1"] * s, L2=case["L2"] * s)
        return {"op": "precomp", "plan": _plan(c, generate=False)}
    rho = _density(case, seed)
    plan = _plan(case)
    phi = torch.empty_like(rho)
    if case["op"] == "many":
        plan.reserve(case["count"])
        return {"op": "many", "plan": plan, "rhos": list(rho.unbind(0)), "phis": list(phi.unbind(0)), "phi": phi}
    return {"op": "apply", "plan": plan, "rho": rho[0], "phi": phi[0]}


def run(state):
    plan = state["plan"]
    if state["op"] == "apply":
        return plan.apply(state["rho"], state["phi"])
    if state["op"] == "many":
        plan.apply_many(state["rhos"], state["phis"])
        return state["phi"]
    plan.generate()
    return plan.spectrum()


def work(case):
    """Bytes: densities in, potentials out, the spectrum octant once (precomp:
    the octant out).  Flops: 5 M log2 M per complex transform of length
    M = 2 n (half of it per real one), forward and inverse, the zero half of
    the padded lines skipped, plus the spectrum multiply; the DDI's grid
    derivative adds its own unpadded transforms; precomp counts one real even
    transform per axis and about 60 operations per octant point."""
    n = _shape(case)
    s = 4 if case["dtype"] == "f32" else 8
    vol, octant, count = math.prod(n), math.prod(k + 1 for k in n), case["count"]

    def solve(M, dims):
        k0 = M[0] // 2 + 1
        lg = [5.0 * m * math.log2(m) for m in M]
        lines = [0.5 * math.prod(dims[1:]), k0 * (M[2] if len(M) > 2 else 1)]
        f = 2 * (lines[0] * lg[0] + lines[1] * lg[1])
        if len(M) > 2:
            f += 2 * k0 * dims[1] * lg[2]
        return f + 2.0 * k0 * math.prod(M[1:])

    if case["op"] == "precomp":
        M = [2 * k for k in n]
        e = [k + 1 for k in n]
        f = 60.0 * octant + sum(octant / e[j] * 1.25 * M[j] * math.log2(M[j]) for j in range(len(n)))
        return {"bytes": octant * s, "flops": f}
    f = solve([2 * k for k in n], n)
    if case["kernel"] == "ddi3d":
        f += solve(list(n), n)
    return {"bytes": 2 * count * vol * s + octant * s, "flops": count * f}


def _bih_series(x):
    """(exp(-x)(1 + x + 2x^2) - 1)/x^2 without cancellation near 0."""
    acc = torch.zeros_like(x)
    for j in range(31, 1, -1):
        c = (-1) ** j * (1.0 / math.factorial(j) - 1.0 / math.factorial(j - 1) + 2.0 / math.factorial(j - 2))
        acc = acc * x + c
    big = (torch.exp(-x) * (1.0 + x + 2.0 * x * x) - 1.0) / torch.clamp(x, min=0.5) ** 2
    return torch.where(x < 1.0, acc, big)


def _spectrum(kernel, n, L, eps):
    """DFT(T1) + W on the half spectrum of the doubled grid (real, last axis halved)."""
    d = len(n)
    dev = "cuda"
    r2 = torch.zeros((1,) * d, dtype=torch.float64, device=dev)
    k2 = torch.zeros((1,) * d, dtype=torch.float64, device=dev)
    hv = 1.0
    for j in range(d):
        h = 2.0 * L[j] / n[j]
        hv *= h
        o = torch.arange(2 * n[j], dtype=torch.float64, device=dev)
        o = torch.where(o > n[j], 2 * n[j] - o, o)
        shp = [1] * d
        shp[j] = -1
        r2 = r2 + ((o * h) ** 2).view(shp)
        p = o[: n[j] + 1] if j == d - 1 else o
        k2 = k2 + ((p * (math.pi / (2.0 * L[j]))) ** 2).view(shp)
    r = r2.sqrt_()
    small = r == 0
    rr = torch.where(small, torch.ones_like(r), r)
    t = torch.special.erf(r / eps)
    if kernel == "biharmonic3d":
        t = t * r / (8.0 * math.pi)
    elif kernel == "coulomb2d":
        t = torch.where(small, torch.full_like(r, 1.0 / (math.pi ** 1.5 * eps)), t / (2.0 * math.pi * rr))
    else:
        t = torch.where(small, torch.full_like(r, 1.0 / (2.0 * math.pi ** 1.5 * eps)), t / (4.0 * math.pi * rr))
    del r, rr, r2, small
    s = torch.fft.rfftn(t * hv).real.contiguous()
    del t
    if kernel == "biharmonic3d":
        w = eps ** 4 / 16.0 * _bih_series(0.25 * k2 * eps * eps)
    elif kernel == "coulomb2d":
        k = k2.sqrt()
        w = torch.where(k > 0, torch.special.erf(0.5 * eps * k) / torch.where(k > 0, k, torch.ones_like(k)),
                        torch.full_like(k, eps / math.sqrt(math.pi)))
    else:
        w = torch.where(k2 > 0, -torch.expm1(-0.25 * eps * eps * k2) / torch.where(k2 > 0, k2, torch.ones_like(k2)),
                        torch.full_like(k2, 0.25 * eps * eps))
    return s.add_(w)


def _ddi_source(rho, n, L):
    """d_n d_m rho by the spectral derivative on the n-point grid (multiplier
    -(k.n)(k.m), the Nyquist index at -n/2), real part."""
    nk = torch.zeros((1, 1, 1), dtype=torch.float64, device="cuda")
    mk = torch.zeros((1, 1, 1), dtype=torch.float64, device="cuda")
    for j in range(3):
        q = torch.fft.fftfreq(n[j], d=1.0 / n[j], dtype=torch.float64, device="cuda") * (math.pi / L[j])
        shp = [1] * 3
        shp[j] = -1
        nk, mk = nk + (DIP_N[j] * q).view(shp), mk + (DIP_M[j] * q).view(shp)
    return torch.fft.ifftn(torch.fft.fftn(rho) * (-(nk * mk))).real


def exact(case, seed):
    n, L, eps = _shape(case), _box(case), case["eps"]
    if case["op"] == "precomp":
        s = 1.0 + 0.001 * (int(seed) % 97)
        spec = _spectrum(case["kernel"], n, tuple(v * s for v in L), eps)
        octant = spec[tuple(slice(0, k + 1) for k in n)]
        return octant / math.prod(2 * k for k in n)
    rho = _density(case, seed).double()
    spec = _spectrum("coulomb3d" if case["kernel"] == "ddi3d" else case["kernel"], n, L, eps)
    dims = tuple(range(len(n)))
    M = [2 * k for k in n]
    outs = []
    for k in range(case["count"]):
        src = _ddi_source(rho[k], n, L) if case["kernel"] == "ddi3d" else rho[k]
        f = torch.fft.rfftn(src, s=M, dim=dims).mul_(spec)
        phi = torch.fft.irfftn(f, s=M, dim=dims)[tuple(slice(0, m) for m in n)]
        del f
        if case["kernel"] == "ddi3d":
            phi = -sum(a * b for a, b in zip(DIP_N, DIP_M)) * rho[k] - 3.0 * phi
        outs.append(phi.clone())
    return torch.stack(outs) if case["op"] == "many" else outs[0]
