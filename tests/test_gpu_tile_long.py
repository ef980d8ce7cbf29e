"""The longest lines against the FP64 oracle: three register steps (1920, 2048, 3072) and
smooth lengths that need a fourth radix and stay on the Stockham kernels (625, 1250, 2000;
tests/test_tile_radix.py has the rule). Tolerances of the other parity tests."""
import numpy as np
import pytest

from oracle import poisson as op
from paper_1211_5244_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5}


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("N", [625, 1250, 1920, 2000, 2048, 3072])
def test_long_lines(gpu_lib, N, axis, dtype):
    import torch
    from paper_1211_5244_gb300 import psolver
    n = [6, 5, 9]
    free = N % 2 == 0
    n[axis] = N // 2 if free else N
    bc = "".join("f" if free and j == axis else "p" for j in range(3))
    npd = np.float32 if dtype == "f32" else np.float64
    rho = synth.random_density(n, seed=N + axis, subtract_mean=True).astype(npd)
    V, E = psolver.Plan(n, bc, 0.3, dtype).solve(torch.from_numpy(rho).cuda())
    Vo, Eo = op.solve(rho.astype(np.float64), bc, 0.3)
    d = V.double().cpu().numpy() - Vo
    assert np.linalg.norm(d) <= TOL[dtype] * np.linalg.norm(Vo)
    assert np.abs(d).max() <= TOL[dtype] * np.abs(Vo).max()
    assert abs(E.item() - Eo) <= TOL[dtype] * abs(Eo)
