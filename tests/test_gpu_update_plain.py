"""Pseudo-time steps without the res(a) monitor run a kernel of their own: the
same states bit for bit as the monitored steps (one FMA per entry in both), at
sizes around its blocks, for a state on a 16-byte boundary and off it, alone and
in an ensemble."""
import numpy as np
import pytest

import coronal_inputs as ci
from _util import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
VR = 1935.07 / ci.V_REF


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", [(2, 2, 8), (7, 9, 24), (33, 16, 32)])
def test_plain_steps_equal_monitored_steps(shape, precision):
    import paper_2209_04481_gb300 as pg
    U, Br = problem(shape, dipole_only=True)
    g = pg.Grid(*shape, precision=precision, p_b=ci.parker_sound_speed2(), inner_bc="low_e_wp", vr_star=VR)
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    log = torch.zeros(27, dtype=torch.float64, device="cuda")
    a = g.pseudo_time_step(torch.from_numpy(U.copy()).cuda(), 3, 0.3, res_log10=log)
    buf = torch.empty(U.size + 1, dtype=torch.float64, device="cuda")
    for off in (0, 1):
        b = buf[off:off + U.size].view(U.shape)
        b.copy_(torch.from_numpy(U))
        g.pseudo_time_step(b, 3, 0.3)
        assert torch.equal(a, b), off
    ens = pg.Ensemble([g])
    c = torch.from_numpy(U.copy()).cuda()
    ens.pseudo_time_step([c], 3, 0.3)
    assert torch.equal(a, c)
    g.sync_status()
    assert torch.isfinite(log).all()
    ens.close()
    g.close()
