"""Workloads of the Poisson solver as programs run it, for timing and for comparing outputs.

Every case goes through the public entry points of paper_1211_5244_gb300
(Plan.solve, the autograd function, solve_batched, solve_host_stream) on
synthetic densities: sums of Gaussians with centres in the middle half of the
box, plus noise, neutral where an axis is periodic. ``kind`` says which entry
point, ``n1 n2 n3`` the grid (x fastest), ``bc`` one letter per axis
(p periodic, f free), ``dtype`` the plan's type. Plans are built as a program
builds them: default padding (2n on free axes), default schedule.
"""
import math

import numpy as np
import torch

from paper_1211_5244_gb300 import psolver
from paper_1211_5244_gb300.autograd import hartree

H = 0.3  # grid spacing


def listed():
    def solve(name, n, bc, dtype, energy=True):
        return dict(name=name, kind="solve", n1=n[0], n2=n[1], n3=n[2], bc=bc, dtype=dtype, energy=energy)

    return [
        # a small molecule in vacuum, FP64, solved thousands of times in an SCF loop: latency
        solve("free32_f64", (32, 32, 32), "fff", "f64"),
        # a polymer along x, the ordinary mid-size FP32 grid
        solve("wire128_f32", (128, 128, 128), "pff", "f32"),
        # the same polymer set up along z: the periodic axis is not the first one
        solve("wire_z128_f32", (128, 128, 128), "ffp", "f32"),
        # a slab on the grid its cell happens to give, potential only (forces)
        solve("surface_ragged_f32", (90, 75, 110), "ppf", "f32", False),
        # a cluster on a grid that is no power of two
        solve("free_ragged_f32", (100, 90, 110), "fff", "f32"),
        # a bulk cell in FP64, one axis of odd length
        solve("periodic_f64", (120, 100, 81), "ppp", "f64"),
        # a molecule in vacuum at the paper's precision
        solve("free128_f64", (128, 128, 128), "fff", "f64"),
        # the headline grid, padded to 512^3
        solve("free256_f32", (256, 256, 256), "fff", "f32"),
        # the largest grid, padded to 1024^3
        solve("free512_f32", (512, 512, 512), "fff", "f32"),
        # the differentiable Hartree energy: forward and backward through autograd
        dict(name="hartree192_f32", kind="grad", n1=192, n2=192, n3=192, bc="fff", dtype="f32"),
        # many uneven densities in one call, shapes 24..160 per axis, the four kinds of boundary conditions
        dict(name="batched32_f32", kind="batch", count=32, nmin=24, nmax=160, shapes=401, dtype="f32"),
        # densities that live in pinned host memory, transfers overlapped with the solves
        dict(name="host_stream128_f32", kind="stream", n1=128, n2=128, n3=128, bc="ppp", dtype="f32", count=8),
    ]


ALL_BCS = ("fff", "pff", "fpf", "ffp", "ppf", "pfp", "fpp", "ppp")


def _size(rng, lo, hi):
    """A grid length, spread over the logarithm; half of them made of the factors 2, 3, 5 that FFT users pick."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5:
        while not _smooth(n):
            n += 1
    return min(n, hi)


def _smooth(n):
    for q in (2, 3, 5):
        while n % q == 0:
            n //= q
    return n == 1


def _spectrum(n, bc):
    L = [2 * v if b == "f" else v for v, b in zip(n, bc)]
    return (L[0] // 2 + 1) * L[1] * L[2]


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["grad", "batch", "stream"])
    if kind == "batch":
        nmin = rng.randint(16, 48)
        return dict(kind="batch", count=rng.randint(4, 32), nmin=nmin, nmax=rng.randint(nmin + 8, 160),
                    shapes=rng.randrange(1 << 16), dtype="f32")
    dtype = "f64" if kind == "solve" and rng.random() < 0.35 else "f32"
    most = 8.5e6 if dtype == "f64" else 6e7  # half-spectrum points: no drawn case costs more than 512^3 in FP32
    while True:
        n = [_size(rng, 16, 256) for _ in range(3)]
        bc = rng.choice(ALL_BCS)
        if 16 ** 3 <= _spectrum(n, bc) <= most:
            break
    case = dict(kind=kind, n1=n[0], n2=n[1], n3=n[2], bc=bc, dtype=dtype)
    if kind == "solve":
        case["energy"] = rng.random() < 0.7
    if kind == "stream":
        case["count"] = rng.randint(3, 8)
    return case


def _problems(case):
    """[(n, bc)] of a case: one grid, or the batch's."""
    if case["kind"] != "batch":
        return [((case["n1"], case["n2"], case["n3"]), case["bc"])]
    rng = np.random.default_rng(case["shapes"])
    kinds = ("fff", "pff", "ppf", "ppp")
    out = []
    for _ in range(case["count"]):
        n = tuple(int(v) for v in rng.integers(case["nmin"], case["nmax"] + 1, size=3))
        out.append((n, kinds[int(rng.integers(0, 4))]))
    return out


def _torch_dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _density(n, bc, seed, dtype, ngauss=8):
    """Gaussians plus 1e-3 noise on an (n3, n2, n1) grid, made on the GPU."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n = np.array(n)
    centre = H * (n / 4 + rng.uniform(size=(ngauss, 3)) * n / 2)
    sigma = H * rng.uniform(1.5, 4.0, size=ngauss)
    amp = rng.standard_normal(ngauss)
    g = []
    for j in range(3):
        x = H * np.arange(n[j])
        v = np.exp(-((x[None, :] - centre[:, j:j + 1]) ** 2) / (2 * sigma[:, None] ** 2))
        g.append(torch.from_numpy(v * amp[:, None] if j == 2 else v).to("cuda", dtype))
    rho = torch.rand((int(n[2]), int(n[1]), int(n[0])), generator=gen, device="cuda", dtype=dtype).mul_(2e-3).sub_(1e-3)
    for q in range(ngauss):
        rho += g[2][q][:, None, None] * (g[1][q][:, None] * g[0][q][None, :])
    if "p" in bc:
        rho -= rho.double().mean().to(dtype)
    return rho


def _densities(case, seed):
    dt = _torch_dtype(case)
    if case["kind"] == "stream":
        (n, bc), = _problems(case)
        return [_density(n, bc, seed * 1000 + i, dt) for i in range(case["count"])]
    return [_density(n, bc, seed * 1000 + i, dt) for i, (n, bc) in enumerate(_problems(case))]


def _cotangents(case, seed):
    (n, _), = _problems(case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 7)
    gV = torch.randn((n[2], n[1], n[0]), generator=gen, device="cuda", dtype=torch.float32)
    gE = torch.tensor(1.5, dtype=torch.float64, device="cuda")
    return gV, gE


def prepare(case, seed):
    s = dict(case=case, plans=[psolver.Plan(n, bc, H, case["dtype"]) for n, bc in _problems(case)],
             rho=_densities(case, seed))
    if case["kind"] == "grad":
        s["rho"][0].requires_grad_(True)
        s["gV"], s["gE"] = _cotangents(case, seed)
    if case["kind"] == "stream":
        s["rho"] = [r.cpu().pin_memory() for r in s["rho"]]
        s["V"] = [torch.empty_like(r).pin_memory() for r in s["rho"]]
    return s


def run(state):
    case = state["case"]
    # the energy of an FP32 plan joins the FP32 terms of the program's total
    plan = state["plans"][0]
    if case["kind"] == "solve":
        V, E = plan.solve(state["rho"][0], energy=case["energy"])
        return [V] if E is None else [V, E.to(V.dtype)]
    if case["kind"] == "grad":
        rho = state["rho"][0]
        V, E = hartree(rho, plan)
        grad, = torch.autograd.grad((V, E), rho, (state["gV"], state["gE"]))
        return [V.detach(), E.detach().float(), grad]
    if case["kind"] == "batch":
        Vs, E = psolver.solve_batched(state["plans"], state["rho"])
        return [Vs, E.float()]
    Vs, E = plan.solve_host_stream(state["rho"], state["V"])
    return [Vs, E]


def work(case):
    b = 4 if case["dtype"] == "f32" else 8
    nbytes = flops = 0.0
    for n, bc in _problems(case):
        L = [2 * v if c == "f" else v for v, c in zip(n, bc)]
        # the solve's order: periodic axes first, free axes last; the first takes the real-to-complex transform
        order = [j for j in range(3) if bc[j] == "p"] + [j for j in range(3) if bc[j] == "f"]
        a0, a1, a2 = order
        f = lambda m: 5.0 * m * math.log2(max(m, 2))  # noqa: E731
        c = L[a0] // 2 + 1
        fl = n[a1] * n[a2] * f(L[a0]) / 2 + c * n[a2] * f(L[a1]) + c * L[a1] * f(L[a2])
        octant = (L[0] // 2 + 1) * (L[1] // 2 + 1) * (L[2] // 2 + 1)
        solves = {"grad": 2, "stream": case.get("count", 1)}.get(case["kind"], 1)
        flops += solves * 2 * fl
        nbytes += b * (solves * 2 * n[0] * n[1] * n[2] + octant)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the solve in 64 bits, by plain FFTs


def _cell_mean_wire(k):
    """The average over the H x H cell of the 2D Green's function of Laplacian - k^2."""
    base = (math.log(H) - 1.5 + math.pi / 4 - 0.5 * math.log(2.0)) / (2 * math.pi)
    if k == 0:
        return base
    x, w = np.polynomial.legendre.leggauss(64)
    th, wth = (x + 1) * math.pi / 8, w * math.pi / 8
    s, ws = (x + 1) / 2, w / 2
    R = (H / 2) / np.cos(th)[:, None]
    r = R * s[None, :] ** 4
    k0 = torch.special.modified_bessel_k0(torch.from_numpy(k * r)).numpy()
    f = (k0 + np.log(r)) * r * 4 * R * s[None, :] ** 3
    integral = 8 * float((wth[:, None] * ws[None, :] * f).sum())
    return base - integral / (2 * math.pi * H * H)


def _kernel_fourier(n, bc, L):
    """K^F on the half spectrum (kz, ky, kx <= L1/2), FP64 on the GPU."""
    per = [c == "p" for c in bc]
    k2 = torch.zeros((1, 1, 1), dtype=torch.float64, device="cuda")
    d2 = torch.zeros((1, 1, 1), dtype=torch.float64, device="cuda")
    for j in range(3):
        i = torch.arange(L[j], dtype=torch.float64, device="cuda")
        i = torch.minimum(i, L[j] - i).reshape([-1 if d == 2 - j else 1 for d in range(3)])
        if per[j]:
            k2 = k2 + (2 * math.pi * i / (n[j] * H)) ** 2
        else:
            d2 = d2 + (H * i) ** 2
    nper = sum(per)
    if nper == 3:
        G = torch.where(k2 > 0, -1.0 / k2, torch.zeros_like(k2))
    elif nper == 2:
        k, z = k2.sqrt(), d2.sqrt()
        G = H * torch.where(k > 0, -torch.exp(-k * z) / (2 * k.clamp_min(1e-300)), z / 2)
    elif nper == 1:
        k, r = k2.sqrt(), d2.sqrt()
        one = torch.ones_like(r)
        rs = torch.where(r > 0, r, one)
        G = torch.where(k > 0, -torch.special.modified_bessel_k0(torch.where(k > 0, k, torch.ones_like(k)) * rs),
                        torch.log(rs)) / (2 * math.pi)
        mean = torch.tensor([_cell_mean_wire(float(v)) for v in k.reshape(-1)], dtype=torch.float64, device="cuda")
        G = H * H * torch.where(r > 0, G, mean.reshape(k.shape))
    else:
        r = d2.sqrt()
        c3 = 3 * math.log(2 + math.sqrt(3.0)) - math.pi / 2
        G = torch.where(r > 0, -H ** 3 / (4 * math.pi * torch.where(r > 0, r, torch.ones_like(r))),
                        torch.full_like(r, -H * H * c3 / (4 * math.pi)))
    free = [2 - j for j in range(3) if not per[j]]
    if free:
        G = torch.fft.fftn(G, dim=free).real
    return G[..., : L[0] // 2 + 1]


def _convolve(KF, rho, n, L):
    spec = torch.fft.rfftn(rho, s=(L[2], L[1], L[0])).mul_(KF)
    V = torch.fft.irfftn(spec, s=(L[2], L[1], L[0]))
    return V[: n[2], : n[1], : n[0]].contiguous()


def exact(case, seed):
    rhos = _densities(case, seed)
    problems = _problems(case)
    if case["kind"] == "stream":
        problems = problems * case["count"]
    Vs, Es, KF, last = [], [], None, None
    for (n, bc), r in zip(problems, rhos):
        L = [2 * v if c == "f" else v for v, c in zip(n, bc)]
        if last != (n, bc):
            KF, last = _kernel_fourier(n, bc, L), (n, bc)
        r = r.double()
        V = _convolve(KF, r, n, L)
        Vs.append(V)
        Es.append(0.5 * H ** 3 * (r * V).sum())
    if case["kind"] == "solve":
        return [Vs[0], Es[0]] if case["energy"] else [Vs[0]]
    if case["kind"] == "grad":
        gV, gE = _cotangents(case, seed)
        (n, bc), = problems
        L = [2 * v if c == "f" else v for v, c in zip(n, bc)]
        return [Vs[0], Es[0], _convolve(KF, gV.double(), n, L) + H ** 3 * gE * Vs[0]]
    return [Vs, torch.stack(Es) if case["kind"] == "batch" else Es]
