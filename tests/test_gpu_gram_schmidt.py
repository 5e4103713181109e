"""The Gram-Schmidt kernels of the Newton-Krylov solver against sums in 64 bits:
long FP32 chains, more rows of partials than one trip of the last block adds,
the second pass, and short vectors."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
U32 = 2.0 ** -24   # rounding of one FP32 operation


@pytest.fixture(scope="module")
def gs(tmp_path_factory):
    from paper_2209_04481_gb300 import build
    out = str(tmp_path_factory.mktemp("gs") / "gs.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-shared", "-o", out,
                    os.path.join(HERE, "gram_schmidt_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    nsm = torch.cuda.get_device_properties(0).multi_processor_count

    def run(V, w):
        """(h, |w|^2 before, |w|^2 after, repeated, w / |w|) of w against the rows of V."""
        f = lib.run32 if V.dtype == torch.float32 else lib.run64
        f.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int] + [ctypes.c_void_p] * 5 + [ctypes.c_int]
        cnt, n = V.shape
        x = w.clone()
        d = dict(dtype=torch.float64, device="cuda")
        part, coef, out = torch.zeros((cnt + 1) * nsm, **d), torch.zeros(cnt + 1, **d), torch.zeros(cnt + 4, **d)
        counter = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert f(V.data_ptr(), n, cnt, x.data_ptr(), part.data_ptr(), coef.data_ptr(), counter.data_ptr(),
                 out.data_ptr(), nsm) == 0
        o = out.cpu()
        assert int(counter) == 0
        return o[:cnt], float(o[cnt]), float(o[cnt + 1]), bool(o[cnt + 3]), x
    return run


@pytest.mark.parametrize("shape", [(128, 64, 128), (96, 48, 96), (33, 17, 40)])
def test_long_chains(gs, shape):
    """Equal positive products, whose FP32 sums round the same way term after
    term: an uncompensated chain of L terms loses up to L / 2 roundings.  The
    sums may lose one rounding a term (that of the product)."""
    n = 9 * shape[0] * shape[1] * shape[2]
    w = torch.full((n,), 1.0 + 2.0 ** -18 - 2.0 ** -23, dtype=torch.float32, device="cuda")
    wd = float(w[0])
    for v in (1.0, 1.0 + 2.0 ** -20 - 2.0 ** -23, 0.7):
        V = torch.full((1, n), v, dtype=torch.float32, device="cuda")
        h, ww, after, redo, _ = gs(V, w)
        assert not redo                       # V is far from unit length: w grows
        vd = float(V[0, 0])
        assert abs(float(h[0]) / (n * vd * wd) - 1.0) <= 1.25 * U32
        assert abs(ww / (n * wd * wd) - 1.0) <= 1.25 * U32
        # an entry of w after the pass: its coefficient and its FMA rounded once each
        y = wd - float(h[0]) * vd
        assert abs(after / (n * y * y) - 1.0) <= (2 * 2 + 1.25) * U32


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("cnt", [1, 8, 9, 127, 128, 150, 500])
@pytest.mark.parametrize("n", [72, 9 * 5 * 7 * 16])
def test_columns_of_many_vectors(gs, cnt, n, dtype):
    """Random rows (not orthonormal: cnt may exceed n), small against w, so that one pass is enough."""
    gen = torch.Generator(device="cuda").manual_seed(cnt)
    V = torch.randn((cnt, n), dtype=torch.float64, device="cuda", generator=gen).to(dtype) / (4.0 * n * cnt) ** 0.5
    w = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen).to(dtype)
    h, ww, after, redo, x = gs(V, w)
    assert not redo
    u = U32 if dtype == torch.float32 else 2.0 ** -53
    Vd, wd = V.double(), w.double()
    mag = (Vd.abs() @ wd.abs()).cpu()
    # one rounding a term, and the FP64 sums' (n terms at most)
    assert torch.all((h - (Vd @ wd).cpu()).abs() <= (1.25 * u + n * 2.0 ** -53) * mag)
    assert abs(ww / float(wd @ wd) - 1.0) <= 1.25 * u + n * 2.0 ** -53
    y = wd - h.cuda() @ Vd
    # cnt FMAs with coefficients of one rounding
    err = (cnt + 2) * u * (wd.abs() + h.abs().cuda() @ Vd.abs())
    assert torch.all((x.double() * after ** 0.5 - y).abs() <= err + 2 * u * y.abs())


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("cnt", [3, 24])
def test_second_pass(gs, cnt, dtype):
    """w almost in the span of an orthonormal V: the pass is repeated, and w leaves orthogonal to working precision."""
    n = 9 * 12 * 8 * 24
    gen = torch.Generator(device="cuda").manual_seed(cnt)
    Q, _ = torch.linalg.qr(torch.randn((n, cnt + 1), dtype=torch.float64, device="cuda", generator=gen))
    V = Q.T[:cnt].contiguous().to(dtype)
    c = torch.randn(cnt, dtype=torch.float64, device="cuda", generator=gen)
    w = (c @ Q.T[:cnt] + 1e-2 * Q.T[cnt]).to(dtype)
    h, _, after, redo, x = gs(V, w)
    assert redo
    u = U32 if dtype == torch.float32 else 2.0 ** -53
    ref = (V.double() @ w.double()).cpu()
    # cnt FMAs and a coefficient a pass, V orthonormal to 2 u: relative to |w| and
    # the coefficients in the first pass, to what is left in the second
    first = (cnt + 8) * u * (float(ref.abs().sum()) + float(w.double().norm()))
    assert torch.all((V.double() @ x.double()).abs() <= (cnt + 8) * u)
    assert torch.all((h - ref).abs() <= first)
    assert abs(after ** 0.5 - 1e-2) <= first
