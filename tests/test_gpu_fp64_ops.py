"""The FP64 building blocks of mhd_device.cuh: reciprocal and square root within
one unit in the last place of the correctly rounded result over the exponents a
state can hold, with their edge values; and the face's lambda, which forms only
the signal speeds an FP32 bound leaves open, bit for bit that of both speeds."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2209_04481_gb300 import build
    out = str(tmp_path_factory.mktemp("ops") / "fp64_ops.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-shared", "-o", out,
                    os.path.join(HERE, "fp64_ops_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    lib.run_ops.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    lib.run_quotients.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    lib.run_lambdas.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_double] + [ctypes.c_void_p] * 2 + [ctypes.c_int]
    return lib


@pytest.fixture(scope="module")
def ops(lib):
    def run(x):
        xd = torch.from_numpy(x).cuda()
        a, b = torch.empty_like(xd), torch.empty_like(xd)
        torch.cuda.synchronize()
        assert lib.run_ops(xd.data_ptr(), a.data_ptr(), b.data_ptr(), x.size) == 0
        return a.cpu().numpy(), b.cpu().numpy()
    return run


def test_within_one_ulp(ops):
    rng = np.random.default_rng(1)
    m = rng.uniform(1.0, 2.0, 400000)
    x = np.concatenate([m * 2.0 ** rng.integers(-300, 300, m.size), 1.0 + np.arange(2000) * 2.0 ** -52,
                        2.0 - np.arange(1, 2000) * 2.0 ** -52])
    rcp, root = ops(x)
    assert np.all(np.abs(rcp - 1.0 / x) <= np.spacing(1.0 / x))
    assert np.all(np.abs(root - np.sqrt(x)) <= np.spacing(np.sqrt(x)))
    rcp, _ = ops(-x)
    assert np.all(np.abs(rcp + 1.0 / x) <= np.spacing(1.0 / x))


def test_root_of_a_rounded_square_is_its_base(ops):
    m = np.random.default_rng(2).uniform(1.0, 2.0, 300000) * 2.0 ** np.random.default_rng(3).integers(-100, 100, 300000)
    _, root = ops(m * m)
    assert np.array_equal(root, m)


def test_edge_values(ops):
    _, root = ops(np.array([0.0, -0.0, 5e-324, -1.0, np.nan]))
    assert root[0] == 0.0 and root[1] == 0.0 and root[2] == 0.0
    assert np.isnan(root[3]) and np.isnan(root[4])


def _quotient(lib, a, b):
    x, y = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    q = torch.empty_like(x)
    torch.cuda.synchronize()
    assert lib.run_quotients(x.data_ptr(), y.data_ptr(), q.data_ptr(), a.size) == 0
    return q.cpu().numpy()


def test_quotient_within_one_ulp(lib):
    rng = np.random.default_rng(4)
    n = 2000000
    near1 = 1.0 + rng.integers(0, 2000, n // 4) * 2.0 ** -52
    near2 = 2.0 - rng.integers(1, 2000, n // 4) * 2.0 ** -52
    a = np.concatenate([rng.uniform(1, 2, n // 2), near1, near2]) * 2.0 ** rng.integers(-200, 200, n)
    a *= np.where(rng.random(n) < 0.5, -1.0, 1.0)
    b = rng.permutation(np.concatenate([rng.uniform(1, 2, n // 2), near1, near2])) * 2.0 ** rng.integers(-200, 200, n)
    q = _quotient(lib, a, b)
    assert np.all(np.abs(q - a / b) <= np.spacing(np.abs(a / b)))
    # 0.51 units of the exact quotient (the values near 1 and 2 give many next to
    # a rounding boundary, where the correctly rounded one is the neighbour)
    for i in range(0, n, 101):
        e = abs(Fraction(q[i]) - Fraction(a[i]) / Fraction(b[i])) / Fraction(np.spacing(abs(q[i])))
        assert e <= Fraction(51, 100), (a[i], b[i], q[i], float(e))
    assert np.array_equal(_quotient(lib, b, b), np.ones(n))


def test_quotient_edge_values(lib):
    a = np.array([0.0, -0.0, 5e-324, 1e-300, np.inf, -np.inf, np.nan, 1.0, 3.0])
    b = np.array([2.0, 2.0, 1.0, 1e300, 2.0, 2.0, 2.0, np.inf, np.nan])
    q = _quotient(lib, a, b)
    assert np.all(q[:4] == 0.0) and np.signbit(q[1])
    assert np.isnan(q[4:9]).all()


def _faces(kind, n, rng):
    """Two primitive states per face; (9, n) each."""
    if kind == "range":  # every magnitude a unit system could give
        m = 10.0 ** rng.uniform(-30, 10, (9, n))
    else:
        m = 10.0 ** np.array([rng.uniform(-5, 0.5, n)] + [rng.uniform(-4, 0.5, n)] * 3 + [rng.uniform(-4, 0.5, n)] * 3
                             + [rng.uniform(-7, -0.5, n), rng.uniform(-6, -2, n)])
    wl = m * np.where(rng.random((9, n)) < 0.5, -1.0, 1.0)
    wl[0], wl[7] = np.abs(wl[0]), np.abs(wl[7])
    rel = {"close": 1e-6, "wind": 1e-2, "range": 1.0, "bad": 0.3}[kind]
    wr = wl * (1.0 + rel * rng.standard_normal((9, n)))
    if kind == "close":
        wr[:, ::3] = wl[:, ::3]              # equal sides
    if kind == "bad":                        # negative, zero, infinite and NaN entries
        for w in (wl, wr):
            for v, x in ((0, -1.0), (7, -1.0), (0, 0.0), (7, 0.0), (0, np.nan), (7, np.inf), (5, np.nan), (2, np.inf)):
                hit = rng.random(n) < 0.05
                w[v, hit] = x if not np.isfinite(x) else x * w[v, hit]
    return wl, wr


@pytest.mark.parametrize("kind", ["wind", "close", "range", "bad"])
@pytest.mark.parametrize("ch", [1.0, 0.0, 0.05, 30.0])
def test_lambda_is_that_of_both_speeds(lib, kind, ch):
    n = 60000
    rng = np.random.default_rng(11)
    wl, wr = _faces(kind, n, rng)
    nrm = rng.standard_normal((3, n))
    nrm /= np.linalg.norm(nrm, axis=0)
    nrm[:, ::7] = np.array([1.0, 0.0, 0.0])[:, None]
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (wl, wr, nrm)]
    lam, ref = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.run_lambdas(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), ch, lam.data_ptr(), ref.data_ptr(), n) == 0
    a, b = lam.cpu().numpy(), ref.cpu().numpy()
    bad = ~((a == b) | (np.isnan(a) & np.isnan(b)))
    assert not bad.any(), (int(bad.sum()), a[bad][:4], b[bad][:4], wl[:, bad][:, :2], wr[:, bad][:, :2])
