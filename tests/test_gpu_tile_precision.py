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
