"""FP32 plans in the order x, z, y whose fused pass has a register kernel and whose
second pass has none, on the Stockham kernels (schedule radix = 1): the strided
kernels then run every pass on tiles of their own width. L = 1024, 128, 256, 384 and
512 along y: the register kernel's tile is wider than the strided one, narrower (the
energy takes more CTAs' partials), and the same."""
import numpy as np
import pytest

from oracle import poisson as op
from paper_1211_5244_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5  # FP32, of the parity tests


@pytest.mark.parametrize("how", ["plan", "axis", "autotune"])
@pytest.mark.parametrize("n,bc", [((32, 512, 16), "pfp"), ((24, 1024, 10), "ppp"), ((24, 64, 20), "pfp"),
                                  ((70, 128, 9), "ppp"), ((24, 128, 18), "pfp"), ((24, 192, 10), "pfp"),
                                  ((40, 256, 12), "pfp")])
def test_strided_kernels_beside_register_lengths(gpu_lib, n, bc, how):
    import torch
    from paper_1211_5244_gb300 import psolver
    kw = {"plan": dict(schedule=dict(radix=1)), "axis": dict(axis_schedule={1: dict(radix=1)}),
          "autotune": dict(autotune=True)}[how]
    plan = psolver.Plan(n, bc, 0.3, "f32", order=(0, 2, 1), **kw)
    rho = synth.random_density(n, seed=sum(n), subtract_mean=True).astype(np.float32)
    V, E = plan.solve(torch.from_numpy(rho).cuda())
    Vo, Eo = op.solve(rho.astype(np.float64), bc, 0.3)
    V = V.double().cpu().numpy()
    assert np.linalg.norm(V - Vo) <= TOL * np.linalg.norm(Vo)
    assert np.abs(V - Vo).max() <= TOL * np.abs(Vo).max()
    assert abs(E.item() - Eo) <= TOL * abs(Eo)
