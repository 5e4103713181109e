"""R when neither the norms nor the step bound is asked for (the kernel without
the reductions), and the members of an ensemble that fills the GPU (radial
chunks of its own).  R does not depend on either: bitwise the same numbers."""
import pytest

import coronal_inputs as ci
from _util import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def make(shape, precision, limiter, seed=0):
    import paper_2209_04481_gb300 as pg
    U, Br = problem(shape, seed=seed, perturb=3 + seed)
    g = pg.Grid(*shape, precision=precision, limiter=limiter, p_b=ci.parker_sound_speed2())
    g.set_inner_boundary(torch.from_numpy(Br).cuda())
    return g, torch.from_numpy(U).to("cuda", g.dtype)


def scratch():
    return (torch.zeros(9, dtype=torch.float64, device="cuda"),
            torch.zeros(1, dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("limiter", ["none", "minmod", "vanalbada"])
@pytest.mark.parametrize("shape", [(2, 2, 8), (5, 17, 40), (33, 16, 48)])
def test_residual_alone(shape, limiter, precision):
    g, U = make(shape, precision, limiter)
    norms, dtmin = scratch()
    both = g.residual(U, norms=norms, dtmin=dtmin)
    alone = g.residual(U)
    n1, d1 = scratch()
    assert torch.equal(both, alone)
    assert torch.equal(both, g.residual(U, norms=n1)) and torch.equal(norms, n1)
    assert torch.equal(both, g.residual(U, dtmin=d1)) and torch.equal(dtmin, d1)
    assert float(norms.min()) > 0 and float(dtmin) > 0
    g.sync_status()
    # a bad cell is still reported
    U[0, 1, 1, 3] = -1
    import paper_2209_04481_gb300 as pg
    g.residual(U)
    with pytest.raises(pg.CoronaError, match="non-physical"):
        g.sync_status()
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("limiter", ["none", "vanalbada"])
def test_ensemble_that_fills_the_gpu(precision, limiter):
    """Work for more than four planes a resident CTA: balanced chunks, the last
    one of a member shorter than the rest; a tall, a flat and a small shell."""
    import paper_2209_04481_gb300 as pg
    shapes = [(64, 32, 96), (47, 40, 80), (96, 30, 64), (9, 48, 128), (3, 4, 8)]
    gs, Us = zip(*(make(s, precision, limiter, seed=m) for m, s in enumerate(shapes)))
    ens = pg.Ensemble(list(gs))
    n = len(gs)
    norms = torch.zeros((n, 9), dtype=torch.float64, device="cuda")
    dtmin = torch.zeros(n, dtype=torch.float64, device="cuda")
    Rs = [R.clone() for R in ens.residual(list(Us), norms=norms, dtmin=dtmin)]
    alone = [R.clone() for R in ens.residual(list(Us))]
    d1 = torch.zeros_like(dtmin)
    for a, b in zip(alone, ens.residual(list(Us), dtmin=d1)):
        assert torch.equal(a, b)
    assert torch.equal(dtmin, d1)
    for m, g in enumerate(gs):
        nm, dm = scratch()
        R = g.residual(Us[m], norms=nm, dtmin=dm)
        g.sync_status()
        assert torch.equal(Rs[m], alone[m]) and torch.equal(R, Rs[m]), m
        # one sum of squares in two orders: FP32 partial sums of a column
        # (at most nr planes) round at 2^-24 each, FP64 at 2^-53
        tol = shapes[m][0] * (2.0 ** -24 if precision == "fp32" else 2.0 ** -53) + 2.0 ** -40
        assert torch.allclose(norms[m], nm, rtol=tol, atol=0), m
        assert torch.equal(dtmin[m:m + 1], dm), m
    ens.close()
