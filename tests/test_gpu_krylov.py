"""The Gram-Schmidt kernels of the Newton-Krylov solver at the sizes where
their passes over eight vectors, their partial sums and their vector loads have
edges: the linear residual that GMRES reports after m steps is the true one of
the step it returns, ||R - (D - J) dU|| / ||R|| with the oracle's exact J."""
import numpy as np
import pytest

import coronal_inputs as ci
import oracle
from _util import oracle_grid, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
VR = 1935.07 / ci.V_REF


@pytest.mark.parametrize("m", [1, 3, 7, 8, 9, 16, 25])
@pytest.mark.parametrize("basis", [0, 1])
@pytest.mark.parametrize("precond", [0, 1])
def test_reported_linear_residual_is_the_true_one(m, basis, precond):
    import paper_2209_04481_gb300 as pg
    shape = (5, 7, 16) if m % 2 else (12, 8, 24)
    U, Br = problem(shape, dipole_only=True)
    g = pg.Grid(*shape, precision="fp64", p_b=ci.parker_sound_speed2(), inner_bc="low_e_wp", vr_star=VR)
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    U64 = torch.from_numpy(U.copy()).cuda()
    dU = torch.zeros_like(U64)
    cfl = 2.0
    st = g.newton_krylov_step(U64, cfl, dU=dU, krylov_dim=m, lin_rtol=1e-12, basis_fp32=basis, precond=precond)
    assert st["krylov_iters"] == m and st["residual_evals"] == 1 + 2 * m
    og = oracle_grid(shape, inner_bc="low_e_wp", vr_star=VR)
    x = dU.cpu().numpy()
    R = oracle.residual(og, U, Br)["R"]
    _, Jx = oracle.residual_jvp(og, U, Br, x, np.zeros_like(Br))
    r = R - x / (cfl * oracle.local_dt(og, U))[None] + Jx
    rel = np.linalg.norm(r) / np.linalg.norm(R)
    # finite-difference products: 1e-5 of the step (the bar of the one-step
    # tests) in each of m directions; an FP32 basis adds its rounding, below that
    assert abs(rel - st["lin_rel"]) <= 1e-5 * np.sqrt(m) + 1e-3 * st["lin_rel"]
    g.close()
