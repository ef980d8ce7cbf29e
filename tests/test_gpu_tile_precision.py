"""Precision of the passes on the tile kernels against their wider forms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# the fused pass (last axis of the order) in two steps (L = 100), two odd steps
# (81), three steps (343), ending in a prime radix (38), in Bluestein form (37, 82);
# along y (pfp: order x, z, y)
@pytest.mark.parametrize("n,bc", [((64, 30, 50), "pff"), ((64, 20, 81), "ppp"), ((64, 10, 343), "ppp"),
                                  ((64, 30, 38), "ppp"), ((64, 20, 37), "ppp"), ((64, 12, 41), "ppf"),
                                  ((64, 50, 30), "pfp")])
def test_energy_sum_over_the_lanes(gpu_lib, n, bc):
    """FP32 plans add the energy across threads in 64 bits.

    Two densities whose spectra share no kx: one constant along x (kx = 0 alone),
    one b (delta(x) - delta(x - n1/2)) (the odd kx), b = 2^-8. Their x
    transforms are exact, the later passes treat each kx on its own, and a thread of
    the fused pass holds lines of one kx. So every thread's FP32 value is the same in the solve of
    the sum as in the two solves apart, and in 64 bits the energies add up to
    within (adders in all) x 2^-53: 1e-12 is above that for the 2^11 threads
    and CTAs of the longest chain. Adding lanes of both kinds in 32 bits rounds each
    warp's sum to 2^-24."""
    import torch
    from paper_1211_5244_gb300 import psolver
    rng = np.random.default_rng(17)
    n1, n2, n3 = n
    g = rng.choice([-2.0, -1.0, -0.5, 0.5, 1.0, 2.0], size=(n3, n2, 1)).astype(np.float32)
    fa = np.ones((1, 1, n1), np.float32)
    fb = np.zeros((1, 1, n1), np.float32)
    fb[..., 0], fb[..., n1 // 2] = 2.0 ** -8, -(2.0 ** -8)
    plan = psolver.Plan(n, bc, 0.3, "f32")
    assert tuple(plan.info().order)[0] == 0
    Ea, Eb, Eab = (plan.solve(torch.from_numpy(np.ascontiguousarray(g * f)).cuda())[1].item()
                   for f in (fa, fb, fa + fb))
    assert Ea != 0.0 and Eb != 0.0
    assert abs(Eab - Ea - Eb) <= 1e-12 * (abs(Ea) + abs(Eb)), (Ea, Eb, Eab - Ea - Eb)


def _round_trip(n, bc, dtype, **plan_args):
    """rms error of a solve with K^F = 1, relative to its result.

    The kernel delta(r) makes V = rho, so the rounding of the transforms shows alone
    (with a Poisson kernel a few long waves carry it), on white noise (every mode alike)."""
    import torch
    from paper_1211_5244_gb300 import psolver
    plan = psolver.Plan(n, bc, 0.3, dtype, **plan_args)
    L = list(plan.info().L)
    delta = np.zeros((L[2] // 2 + 1, L[1] // 2 + 1, L[0] // 2 + 1))
    delta[0, 0, 0] = 1.0
    plan.set_kernel_real(delta)
    k = plan.kernel_octant()
    k0 = float(k[0, 0, 0])
    assert float((k.double() - k0).abs().max()) <= 1e-6 * k0
    rng = np.random.default_rng(sum(n))
    rho = rng.standard_normal(n[::-1]).astype(np.float32 if dtype == "f32" else np.float64)
    V = plan.solve(torch.from_numpy(rho).cuda())[0].cpu().numpy()
    wide = np.longdouble
    ref = rho.astype(wide) * (wide(k0) * wide(L[0]) * wide(L[1]) * wide(L[2]))
    return float(np.sqrt(((V.astype(wide) - ref) ** 2).sum() / (ref ** 2).sum()))


# every axis of one length: powers of two, odd prime powers, composite radices,
# prime radices, the Bluestein form. FP32 powers of two run the tile kernels in
# orders that do not start with x
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,bc", [(16, "fff"), (32, "ffp"), (64, "fpf"), (64, "fpp"), (49, "ppp"), (81, "ppp"),
                                  (50, "fff"), (45, "ppf"), (60, "ppp"), (36, "ffp"), (55, "ppp"), (34, "fff"),
                                  (62, "ppp"), (37, "ppp")])
def test_rounding_of_the_tile_kernels(gpu_lib, n, bc, dtype):
    """The tile kernels round no more than the Stockham stages (schedule radix = 1).

    The rms over n^3 >= 4096 errors of random inputs has a sampling error below
    1/sqrt(2 x 4096) = 1.1%; 2% covers both sides."""
    tile = _round_trip((n, n, n), bc, dtype)
    stockham = _round_trip((n, n, n), bc, dtype, schedule=dict(radix=1))
    assert tile <= 1.02 * stockham, (tile, stockham)


@pytest.mark.parametrize("ykind", [0, 2])  # the persistent and the plain kernels
@pytest.mark.parametrize("n,bc", [((32, 16, 512), "ppf"), ((32, 16, 1024), "ppp"), ((32, 512, 16), "pfp"),
                                  ((32, 1024, 16), "ppp")])
def test_rounding_of_the_1024_point_kernels(gpu_lib, n, bc, ykind):
    """The register z and y kernels of length 1024 against the Stockham stages, in an
    order that does not start with x. 2^17 or more values: a sampling error below 0.2% on
    each side; 2% leaves the register kernels of the short axes their own rounding."""
    order = (1, 0, 2) if n[2] > n[1] else (2, 0, 1)
    fast = _round_trip(n, bc, "f32", schedule=dict(ykind=ykind))
    stockham = _round_trip(n, bc, "f32", order=order, schedule=dict(radix=1))
    assert fast <= 1.02 * stockham, (fast, stockham)
