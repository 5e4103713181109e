"""The Newton-Krylov workspace and its finite-difference step at the ends of
their ranges: the first step of a grid on a stream of its own, directions
beyond the range of FP32, and the memory a central difference takes."""
import numpy as np
import pytest

import coronal_inputs as ci
import oracle
from _util import oracle_grid, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
VR = 1935.07 / ci.V_REF


def make(shape, precision="fp64"):
    import paper_2209_04481_gb300 as pg
    U, Br = problem(shape, dipole_only=True)
    g = pg.Grid(*shape, precision=precision, p_b=ci.parker_sound_speed2(), inner_bc="low_e_wp", vr_star=VR)
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    torch.cuda.synchronize()
    return g, U, Br


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_first_step_on_a_side_stream(precision):
    """The workspace is set up by the first step, on that step's stream."""
    out = []
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        g, U, _ = make((8, 8, 16), precision)
        U64 = torch.from_numpy(U.copy()).cuda()
        torch.cuda.synchronize()
        st = g.newton_krylov_step(U64, 4.0, stream=stream, krylov_dim=10)
        stream.synchronize()
        out.append((U64, st))
        g.close()
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("cfl", [1e42, 1e60, 1e-60])
@pytest.mark.parametrize("m", [2, 5])
def test_directions_beyond_fp32(cfl, m):
    """z = dtau . v with entries far outside FP32 (precond 0, FP64 basis): the
    linear residual reported is the true one of the step returned."""
    shape = (5, 7, 16)
    g, U, Br = make(shape)
    U64 = torch.from_numpy(U.copy()).cuda()
    dU = torch.zeros_like(U64)
    st = g.newton_krylov_step(U64, cfl, dU=dU, krylov_dim=m, lin_rtol=1e-12, basis_fp32=0, precond=0)
    og = oracle_grid(shape, inner_bc="low_e_wp", vr_star=VR)
    x = dU.cpu().numpy()
    R = oracle.residual(og, U, Br)["R"]
    _, Jx = oracle.residual_jvp(og, U, Br, x, np.zeros_like(Br))
    r = R - x / (cfl * oracle.local_dt(og, U))[None] + Jx
    rel = np.linalg.norm(r) / np.linalg.norm(R)
    # the bar of the steps at ordinary directions: 1e-5 per finite-difference product
    assert abs(rel - st["lin_rel"]) <= 1e-5 * np.sqrt(m) + 1e-3 * st["lin_rel"], (rel, st)
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_central_difference_takes_no_memory_of_its_own(precision):
    """9.4 (4.7) MB of a second perturbed state on 64 x 32 x 64 would show."""
    used = {}
    for central in (0, 1):
        g, U, _ = make((64, 32, 64), precision)
        U64 = torch.from_numpy(U.copy()).cuda()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        g.newton_krylov_step(U64, 1.0, krylov_dim=2, fd_central=central)
        torch.cuda.synchronize()
        used[central] = before - torch.cuda.mem_get_info()[0]
        g.close()
    assert used[0] > 0 and used[1] <= used[0]
