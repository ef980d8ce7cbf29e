"""The vector-Jacobian product with both cotangents, rhobar = K vbar + h^3 gE V,
against the FP64 oracle: the last pass adds the energy term where its kernel does
(register x kernels, tile kernels), a pass of its own does elsewhere. V is an
array of its own here, not K rho, so that a wrong element of it shows."""
import numpy as np
import pytest

from oracle import poisson as op
from paper_1211_5244_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5}  # of the parity tests
H = 0.3

CASES = [
    # FP32 register x kernels: periodic and free, even rows; odd rows shorter than L1 / 2
    ((64, 9, 10), "pff", None, {}),
    ((32, 10, 9), "fff", None, {}),
    ((45, 10, 9), "fff", (96, 20, 18), {}),
    ((33, 7, 10), "fff", (128, 14, 20), {}),
    # tile kernels, packed rows (even L1): odd and even n1
    ((35, 10, 9), "fff", None, {}),
    ((30, 9, 10), "fff", None, {}),
    ((90, 7, 5), "ppf", None, {}),
    # tile kernels, pairs of rows (odd L1): an even and an odd number of rows
    ((33, 6, 5), "ppp", None, {}),
    ((33, 5, 7), "ppp", None, {}),
    # pairs of columns along y and z: odd and even n1
    ((21, 22, 14), "fpf", None, {}),
    ((22, 26, 13), "fpp", None, {}),
    ((21, 14, 22), "ffp", None, {}),
    ((18, 14, 25), "ffp", None, {}),
    # Bluestein form: pairs of rows, packed rows, columns
    ((37, 6, 5), "pff", None, {}),
    ((74, 5, 6), "pff", None, {}),
    ((15, 37, 6), "fpf", None, {}),
    # the term as a pass of its own: Stockham last pass, chunked x and y passes
    ((5, 12, 9), "fff", None, {}),
    ((30, 9, 10), "fff", None, dict(radix=1)),
    ((64, 128, 12), "fff", None, dict(chunks=3)),
]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,bc,L,schedule", CASES)
def test_vjp_of_both_outputs(gpu_lib, n, bc, L, schedule, dtype, offset):
    """offset: vbar, V and rhobar one element off the alignment of a pair of reals."""
    import torch
    from paper_1211_5244_gb300 import psolver
    plan = psolver.Plan(n, bc, H, dtype, L=L, schedule=schedule or None)
    npd = np.float32 if dtype == "f32" else np.float64
    vbar = synth.random_density(n, seed=sum(n), subtract_mean="p" in bc).astype(npd)
    V = synth.random_density(n, seed=sum(n) + 1).astype(npd)
    gE = -37.5  # h^3 gE is about 1: both terms count

    def place(a):
        t = torch.full((a.size + 8,), float("nan"), dtype=plan.torch_dtype, device="cuda")
        v = t[4 + offset:4 + offset + a.size].view(plan.shape)
        v.copy_(torch.from_numpy(a))
        return t, v

    _, tv = place(vbar)
    _, tV = place(V)
    whole, out = place(np.zeros_like(V))
    plan.solve_vjp(vbar=tv, V=tV, gE=torch.tensor(gE, dtype=torch.float64, device="cuda"), out=out)
    ref = op.solve(vbar.astype(np.float64), bc, H)[0] + H ** 3 * gE * V.astype(np.float64)
    d = out.double().cpu().numpy() - ref
    assert np.linalg.norm(d) <= TOL[dtype] * np.linalg.norm(ref)
    assert np.abs(d).max() <= TOL[dtype] * np.abs(ref).max()
    # nothing outside rhobar is written
    w = whole.cpu().numpy()
    assert np.isnan(w[:4 + offset]).all() and np.isnan(w[4 + offset + V.size:]).all()
