"""The tiled residual where its tiling has edges: shells smaller than a tile,
rows and columns that leave a remainder in both precisions' tiles (8 x 32 in
FP32, 8 x 16 in FP64), one-plane and ragged radial chunks, and chunks that
start one and two planes above the inner boundary; the norms and the step
bound over one and over many CTAs.  Against the oracle at the bounds of the
parity tests."""
import numpy as np
import pytest

import coronal_inputs as ci
import oracle
from _util import check_fp32, oracle_grid, problem, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 8), (3, 9, 24), (4, 7, 40), (5, 17, 32), (7, 8, 16), (33, 16, 48)]


@pytest.mark.parametrize("kchunk", [None, 1, 2, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_tile_and_chunk_edges(shape, precision, kchunk, monkeypatch):
    import paper_2209_04481_gb300 as pg
    if kchunk is not None:
        monkeypatch.setenv("CRN_KCHUNK", str(kchunk))
    limiter = "vanalbada" if shape[0] % 2 else "minmod"
    U, Br = problem(shape, perturb=5)
    g = pg.Grid(*shape, precision=precision, limiter=limiter, p_b=ci.parker_sound_speed2())
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    Ud = torch.from_numpy(U).to("cuda", g.dtype)
    norms = torch.zeros(9, dtype=torch.float64, device="cuda")
    dtmin = torch.zeros(1, dtype=torch.float64, device="cuda")
    R = g.residual(Ud, norms=norms, dtmin=dtmin)
    g.sync_status()
    og = oracle_grid(shape, limiter=limiter)
    ref = oracle.residual(og, U, Br, want_scale=True)
    Rn, nn, dn = R.double().cpu().numpy(), norms.cpu().numpy(), float(dtmin)
    if precision == "fp64":
        assert np.all(rel_err(Rn, ref["R"], ref["scale"]) <= 1e-12)
        np.testing.assert_allclose(nn, ref["norms"], rtol=1e-12)
        assert abs(dn - ref["dtmin"]) <= 1e-12 * ref["dtmin"]
    else:
        check_fp32(Rn, ref, og, U, nn, dn)
    # bitwise repeatable, norms included
    R2 = g.residual(Ud, norms=(n2 := torch.zeros_like(norms)))
    assert torch.equal(R, R2) and torch.equal(norms, n2)
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_flags_of_the_tiled_kernel(precision):
    """The lowest flagged cell: a negative density, a negative pressure and a
    non-finite entry, each alone in its shell."""
    import paper_2209_04481_gb300 as pg
    shape = (6, 9, 24)
    U, Br = problem(shape)
    cells = [(4, 8, 23), (0, 0, 0), (2, 5, 17)]
    for cell, (var, val) in zip(cells, ((0, -1.0), (7, -1.0), (4, np.inf))):
        V = U.copy()
        V[(var,) + cell] = val
        g = pg.Grid(*shape, precision=precision, p_b=ci.parker_sound_speed2())
        g.set_inner_boundary(torch.from_numpy(Br).cuda())
        g.residual(torch.from_numpy(V).to("cuda", g.dtype))
        with pytest.raises(pg.CoronaError, match="non-physical"):
            g.sync_status()
        # a bad cell spoils the residuals of cells whose stencil holds it, so
        # the lowest flagged cell is at most two planes below
        k = g.last_bad_cell // (shape[1] * shape[2])
        assert cell[0] - 2 <= k <= cell[0]
        g.close()
