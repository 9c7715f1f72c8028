"""Legendre <-> Fourier products in tiles of 128 x 64 at their edges: a last row tile of
one row, a last column tile of one column, odd lmax (the parities differ in size), against
the FP64 plan, which takes the small tiles; forward through the FP32 pipes, and transposed."""

import numpy as np
import pytest

from helpers import per_l_error
from oracle import hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,B", [(128, 256, 19), (128, 255, 19), (128, 129, 38), (128, 128, 65),
                                          (256, 511, 7), (256, 512, 9)])
def test_large_tiles(nside, lmax, B):
    import paper_1904_10514_gb300 as hp
    rng = np.random.default_rng(lmax + B)
    n = hp2sph.n_alm(lmax)
    x = rng.standard_normal((B, 12 * nside * nside)).astype(np.float32)
    a = (rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n))).astype(np.complex64)
    out = {}
    for prec in ("fp32", "fp64"):
        rd, cd = (torch.float64, torch.complex128) if prec == "fp64" else (torch.float32, torch.complex64)
        plan = hp.Plan(nside, lmax, B, prec, sweeps=True, simt=True)
        out[prec] = (plan.analyze(torch.as_tensor(x, dtype=rd, device="cuda")).cpu().numpy().astype(np.complex128),
                     plan.synthesize(torch.as_tensor(a, dtype=cd, device="cuda")).cpu().numpy().astype(np.float64))
        plan.close()
    for b in range(B):
        e = per_l_error(out["fp32"][0][b], out["fp64"][0][b], lmax)
        assert e.max() < 1e-5, (b, e)     # the parity gate
        d = np.linalg.norm(out["fp32"][1][b] - out["fp64"][1][b]) / np.linalg.norm(out["fp64"][1][b])
        assert d < 2e-5, (b, d)           # the adjoint's
