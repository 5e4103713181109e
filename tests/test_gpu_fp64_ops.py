"""The FP64 reciprocal and square root of mhd_device.cuh: within one unit in
the last place of the correctly rounded result over the exponents a state can
hold, and their edge values."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    from paper_2209_04481_gb300 import build
    out = str(tmp_path_factory.mktemp("ops") / "fp64_ops.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-shared", "-o", out,
                    os.path.join(HERE, "fp64_ops_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    lib.run_ops.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]

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
