"""The FP32 momentum flux rounds the product that costs less: on the radial faces
of a perturbed wind its mean error against 64 bits lies below that of the sum
with the pressure's product rounded instead of the mass flux's."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import coronal_inputs as ci

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2209_04481_gb300 import build
    out = str(tmp_path_factory.mktemp("flux") / "flux.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, *build.EXTRA["residual_fp32.cu"], "-shared", "-o", out,
                    os.path.join(HERE, "fp32_flux_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    lib.run_fluxes.argtypes = [ctypes.c_void_p] * 5 + [ctypes.c_int]
    return lib


def momentum_flux(wl, wr, n):
    """Rusanov momentum flux of the primitive states, gamma 1.05, c_h = 1, in float64."""
    def side(w):
        rho, v, b, p = w[0], w[1:4], w[4:7], w[7]
        un, bn, b2 = (v * n).sum(0), (b * n).sum(0), (b * b).sum(0)
        a2, s = 1.05 * p / rho, (1.05 * p + b2) / rho
        cf = np.sqrt(0.5 * (s + np.sqrt(np.maximum(s * s - 4 * a2 * bn * bn / rho, 0.0))))
        return rho * un * v + (p + 0.5 * b2) * n - bn * b, rho * v, np.abs(un) + cf
    FL, ML, sl = side(wl)
    FR, MR, sr = side(wr)
    lam = np.maximum(np.maximum(sl, sr), 1.0)
    return 0.5 * (FL + FR) - 0.5 * lam * (MR - ML)


def test_momentum_flux_rounds_the_mass_flux(lib):
    shape = (96, 48, 96)
    W = ci.background(*shape)[1]["W"]
    rng = np.random.default_rng(6)
    W = (W * (1.0 + 0.01 * rng.standard_normal(W.shape))).astype(np.float32)
    _, tc, pc = ci.cell_centres(*shape)
    t, p = np.meshgrid(tc, pc, indexing="ij")
    e = np.stack([np.sin(t) * np.cos(p), np.sin(t) * np.sin(p), np.cos(t)]).astype(np.float32)
    n = np.ascontiguousarray(np.broadcast_to(e[:, None], (3, shape[0] - 1) + shape[1:]).reshape(3, -1))
    wl, wr = (np.ascontiguousarray(W[:, s].reshape(9, -1)) for s in (slice(0, -1), slice(1, None)))
    ref = momentum_flux(wl.astype(np.float64), wr.astype(np.float64), n.astype(np.float64))
    d = [torch.from_numpy(x).cuda() for x in (wl, wr, n)]
    f, other = torch.empty_like(d[2]), torch.empty_like(d[2])
    torch.cuda.synchronize()
    assert lib.run_fluxes(*[x.data_ptr() for x in d], f.data_ptr(), other.data_ptr(), n.shape[1]) == 0
    rel = [np.abs(x.double().cpu().numpy() - ref) / np.abs(ref).max(axis=0) for x in (f, other)]
    assert rel[0].mean() < rel[1].mean(), (rel[0].mean(), rel[1].mean())
    assert rel[0].max() <= 100 * 2.0 ** -24   # nine products and sums a side, the step's difference
