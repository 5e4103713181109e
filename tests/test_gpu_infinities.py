"""Zeros and infinities in the FP64 reciprocal and square root of
mhd_device.cuh, and what they decide in the residual: a state whose signal speed
overflows has the step bound 0 (not the one of the slowest admissible speed),
and the cell is reported."""
import numpy as np
import pytest

import coronal_inputs as ci
import oracle
from _util import oracle_grid, problem
from test_gpu_fp64_ops import lib, ops  # noqa: F401  (fixtures)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_reciprocal_and_root_at_zero_and_infinity(ops):  # noqa: F811
    rcp, root = ops(np.array([0.0, -0.0, np.inf, -np.inf, np.nan]))
    assert rcp[0] == np.inf and rcp[1] == -np.inf
    assert rcp[2] == 0.0 and rcp[3] == 0.0 and np.signbit(rcp[3])
    assert np.isnan(rcp[4])
    assert root[2] == np.inf and np.isnan(root[3]) and np.isnan(root[4])


@pytest.mark.parametrize("kernel", ["tiled", "cellwise"])
@pytest.mark.parametrize("limiter", ["none", "minmod", "vanalbada"])
def test_step_bound_of_an_overflowing_speed(limiter, kernel):
    """Energy 1e160 in one cell: c_f^2 overflows, lambda is infinite there and the
    step bound 0 (van Albada's slopes overflow first: NaN states, as the oracle's)."""
    import paper_2209_04481_gb300 as pg
    shape = (6, 8, 16)
    U, Br = problem(shape, perturb=3)
    U = U.copy()
    U[7, 3, 4, 5] = 1e160
    g = pg.Grid(*shape, precision="fp64", limiter=limiter, kernel=kernel, p_b=ci.parker_sound_speed2())
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    Ud = torch.from_numpy(U).cuda()
    with np.errstate(all="ignore"):
        ref = oracle.residual(oracle_grid(shape, limiter=limiter), U, Br)["dtmin"]
    assert (ref == 0.0) == (limiter != "vanalbada")
    for norms in (torch.zeros(9, dtype=torch.float64, device="cuda"), None):
        dtmin = torch.ones(1, dtype=torch.float64, device="cuda")
        R = g.residual(Ud, norms=norms, dtmin=dtmin)
        assert abs(float(dtmin) - ref) <= 1e-12 * ref
        assert not torch.isfinite(R[:, 3, 4, 5]).all()
        with pytest.raises(pg.CoronaError, match="non-physical"):
            g.sync_status()
    g.close()
