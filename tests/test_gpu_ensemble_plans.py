"""The ensemble's chunks, tiles and tuner where the defaults and the launches'
limits meet: one-plane chunks of FP64 members, more members than the longest
chunk can balance, a chunk set without a tile, and a tuner that leaves the
default where the default is faster."""
import pytest

import coronal_inputs as ci
from _util import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def make(shapes, precision):
    import paper_2209_04481_gb300 as pg
    gs, Us, cache = [], [], {}
    for shape in shapes:
        if shape not in cache:
            U, Br = problem(shape, perturb=3)
            cache[shape] = torch.from_numpy(U), torch.from_numpy(Br).cuda()
        U, Br = cache[shape]
        g = pg.Grid(*shape, precision=precision, p_b=ci.parker_sound_speed2())
        g.set_inner_boundary(Br)
        gs.append(g)
        Us.append(U.to("cuda", g.dtype))
    return gs, Us, pg.Ensemble(gs)


def close(gs, ens):
    gs[0].sync_status()
    ens.close()
    for g in gs:
        g.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kchunk", [1, 2])
def test_shortest_chunks(precision, kchunk):
    gs, Us, ens = make([(80, 64, 128), (5, 8, 16)], precision)
    norms = torch.zeros((2, 9), dtype=torch.float64, device="cuda")
    ens.kchunk = kchunk
    Rs = ens.residual(Us, norms=norms)
    for g, U, R in zip(gs, Us, Rs):
        assert torch.equal(R, g.residual(U))
    ref = torch.stack([torch.linalg.vector_norm(R.double().reshape(9, -1), dim=1) for R in Rs])
    # FP32 sums of at most 2 squares a thread and a 5-level tree; FP64 elsewhere
    torch.testing.assert_close(norms, ref, rtol=1e-6 if precision == "fp32" else 1e-12, atol=0)
    close(gs, ens)


@pytest.mark.parametrize("precision,n", [("fp32", 100), ("fp64", 50)])
def test_more_members_than_chunks_can_balance(precision, n):
    """Many flat shells: more (tile, plane) pairs than eight items per CTA of the
    tallest member's full height.  Every member is taken whole."""
    shapes = [(8, 64, 128) if m % 3 else (5, 64, 128) for m in range(n)]
    gs, Us, ens = make(shapes, precision)
    assert [ens.member_config(m)[1] for m in range(n)] == [s[0] for s in shapes]
    Rs = ens.residual(Us)
    for m in (0, 1, n - 1):
        assert torch.equal(Rs[m], gs[m].residual(Us[m])), m
    close(gs, ens)


@pytest.mark.parametrize("precision,own", [("fp64", (8, 16)), ("fp32", (8, 32))])
def test_chunk_without_a_tile_keeps_the_own_tile(precision, own):
    gs, Us, ens = make([(12, 8, 32), (9, 24, 64)], precision)
    assert ens.member_config(0)[0] == own
    ens.set_member_config(0, kchunk=3)
    assert ens.member_config(0) == (own, 3)
    ens.set_member_config(0, tile=(16, 16), kchunk=5)
    assert ens.member_config(0) == ((16, 16), 5)
    ens.set_member_config(0)
    assert ens.member_config(0)[0] == own
    close(gs, ens)


def _time(ens, Us, Rs):
    for _ in range(3):
        ens.residual(Us, Rs)
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            ens.residual(Us, Rs)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_tuned_is_never_slower_than_the_default(precision):
    """Shells that fill the GPU.  3 % for the runs of one configuration."""
    gs, Us, ens = make([(64, 32, 96), (47, 40, 80), (96, 30, 64), (60, 48, 128)], precision)
    Rs = [torch.empty_like(U) for U in Us]
    default = _time(ens, Us, Rs)
    ref = [R.clone() for R in Rs]
    k = ens.autotune(Us, Rs)
    assert ens.kchunk == k
    tuned = _time(ens, Us, Rs)
    assert tuned <= 1.03 * default, (tuned, default, [ens.member_config(m) for m in range(4)])
    tol = 1e-13 if precision == "fp64" else 1e-6
    for a, b in zip(ref, Rs):
        assert torch.all((a - b).abs() <= tol * a.abs().amax(dim=(1, 2, 3), keepdim=True))
    close(gs, ens)
