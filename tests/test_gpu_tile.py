"""The tile kernels (register DFT steps for lengths with factors up to 13) against
the FP64 oracle: every radix in every step, two and three steps, odd lengths,
padded and periodic lines, line counts that end inside a tile, along each axis and
with each processing order. Tolerances of the other parity tests."""
import numpy as np
import pytest

from oracle import poisson as op
from paper_1211_5244_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5}

# 4 = 2 x 2 is the shortest; 26, 33, 91, 169 use 11 and 13; 343 and 2197 three odd
# steps; 2000 and 4096 the longest tables; the others mix the composite radices;
# the second row ends in a prime radix from 17 to 31, behind one step, two or none; the
# third runs in Bluestein form
LENGTHS = [4, 6, 9, 15, 22, 26, 33, 63, 70, 90, 91, 126, 150, 169, 208, 220, 231, 343, 420, 1000, 2000, 2197, 4096,
           17, 19, 31, 34, 46, 62, 93, 116, 221, 247, 406, 1085, 1472,
           37, 74, 106, 127, 289, 323, 487, 578, 1022, 1031]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("N", LENGTHS)
def test_tile_lengths(gpu_lib, N, axis, dtype):
    import torch
    from paper_1211_5244_gb300 import psolver
    free = N % 2 == 0 and N > 200  # a padded axis of length N, else a periodic one
    n = [5, 7, 3]
    n[axis] = N // 2 if free else N
    bc = "".join("f" if free and j == axis else "p" for j in range(3))
    rho = synth.random_density(n, seed=N + axis, subtract_mean=True)
    npd = np.float32 if dtype == "f32" else np.float64
    if N == 4096 and axis == 0 and dtype == "f64":
        # complex FP64 lines of 4096 along x: the plan refuses them, since its
        # Stockham form would need more shared memory than a CTA has
        with pytest.raises(psolver.PsError):
            psolver.Plan(n, bc, 0.3, dtype)
        return
    for order in ([None, (1, 2, 0)] if N < 200 else [None]):
        plan = psolver.Plan(n, bc, 0.3, dtype, order=order)
        r = torch.from_numpy(np.ascontiguousarray(rho.astype(npd))).cuda()
        V, E = plan.solve(r)
        Vo, Eo = op.solve(rho.astype(npd).astype(np.float64), bc, 0.3)
        V = V.double().cpu().numpy()
        l2 = np.linalg.norm(V - Vo) / np.linalg.norm(Vo)
        mx = np.abs(V - Vo).max() / np.abs(Vo).max()
        assert max(l2, mx, abs(float(E) - Eo) / abs(Eo)) <= TOL[dtype], (order, l2, mx, float(E), Eo)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,bc", [((30, 9, 10), "pff"), ((31, 10, 9), "fpf"), ((18, 25, 14), "fpp")])
def test_tile_unaligned_rows(gpu_lib, n, bc, dtype):
    """rho and V one element off the alignment of a pair of reals."""
    import torch
    from paper_1211_5244_gb300 import psolver
    rho = synth.random_density(n, seed=3, subtract_mean=True)
    plan = psolver.Plan(n, bc, 0.3, dtype)
    t = torch.zeros(2 * rho.size + 4, dtype=plan.torch_dtype, device="cuda")
    r = t[1:1 + rho.size].view(plan.shape)
    off = rho.size + 2 + (rho.size + 1) % 2  # odd
    V = t[off:off + rho.size].view(plan.shape)
    r.copy_(torch.from_numpy(rho))
    plan.solve(r, V=V)
    Vo, _ = op.solve(r.double().cpu().numpy(), bc, 0.3)
    d = V.double().cpu().numpy() - Vo
    assert np.linalg.norm(d) <= TOL[dtype] * np.linalg.norm(Vo)
