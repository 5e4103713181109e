"""The FP64 VJP without room for its scratch: the tiled passes (two launches
where the others take three), the same gradient, and the three passes again
once there is room."""
import numpy as np
import pytest

import coronal_inputs as ci
import oracle
from _util import oracle_grid, problem
from test_gpu_adjoint import objectives, steady

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LIMIT = "CRN_VJP_SCRATCH_LIMIT"


def test_vjp_without_room_for_the_scratch(monkeypatch):
    import paper_2209_04481_gb300 as pg
    shape = (12, 9, 24)
    U, Br = problem(shape, perturb=3)
    g = pg.Grid(*shape, precision="fp64", p_b=ci.parker_sound_speed2())
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    Ud = torch.from_numpy(U).cuda()
    Rb = np.random.default_rng(1).standard_normal(U.shape)
    need = 1000 * 12 * 9 * 24
    monkeypatch.setenv(LIMIT, str(need))
    Ub, Bb = g.residual_vjp(Ud, torch.from_numpy(Rb).cuda(), want_br=True)
    assert g.last_launch_count == 2
    rng = np.random.default_rng(2)
    v, dB = rng.standard_normal(U.shape) * np.abs(U), rng.standard_normal(Br.shape)
    _, Jv = oracle.residual_jvp(oracle_grid(shape), U, Br, v, dB)

    def check(Ub, Bb):
        a, b = Ub.cpu().numpy() * v, Bb.cpu().numpy() * dB
        assert abs(np.sum(a) + np.sum(b) - np.sum(Rb * Jv)) <= 1e-11 * (np.sum(np.abs(a)) + np.sum(np.abs(b)))

    check(Ub, Bb)
    monkeypatch.setenv(LIMIT, str(2 * need))       # a shortage that has passed
    Ub, Bb = g.residual_vjp(Ud, torch.from_numpy(Rb).cuda(), want_br=True)
    assert g.last_launch_count == 3
    check(Ub, Bb)
    monkeypatch.setenv(LIMIT, "0")                 # the scratch it holds stays in use
    g.residual_vjp(Ud, torch.from_numpy(Rb).cuda())
    assert g.last_launch_count == 3
    g.sync_status()
    g.close()


@pytest.mark.parametrize("fgmres", [30, 0])
def test_adjoint_without_room_for_the_scratch(monkeypatch, fgmres):
    monkeypatch.setenv(LIMIT, "0")
    shape = (6, 6, 16)
    g, U64, Br, og = steady(shape, "low_e_wp", "fp64")
    gbar = objectives(shape, None)["rho"]
    gb = torch.from_numpy(gbar).cuda()
    sens, _, st = g.adjoint_solve(U64, gb, krylov_dim=30, lin_rtol=1e-10, precond=1, adjoint_cfl=100.0,
                                  adjoint_outer=400, adjoint_fgmres=fgmres)
    assert st["lin_rel"] <= 1e-10
    g.residual_vjp(U64, gb)
    assert g.last_launch_count == 2                # still without it
    g.sync_status()
    s = sens.cpu().numpy()
    dB = np.random.default_rng(5).standard_normal(Br.shape)
    ref = oracle.steady_sensitivity(og, U64.cpu().numpy(), Br, gbar, dB, rtol=1e-11)
    assert abs(float(np.sum(s * dB)) - ref) <= 1e-6 * np.sum(np.abs(s * dB))
    g.close()
