"""The Newton-Krylov workspace and its finite-difference step at the ends of
their ranges: the first step of a grid on a stream of its own."""
import pytest

import coronal_inputs as ci
from _util import problem

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
