"""Spreading and grid FFT at the edges of their work split: the last tile of 32 orders
with 1, 2 or 3 orders in it, an unpaired last order, every pass structure of the grid
length M = 8 nside, FP32 (differenced from M = 4096 on) and FP64."""

import numpy as np
import pytest

import skies
from helpers import per_l_error, per_l_norms
from oracle import hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 1e-5}   # the parity gates of the FP64 and FP32 plans


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nside,lmax", [(2, 3), (4, 7), (8, 15), (16, 32), (32, 33), (64, 34), (128, 64), (256, 5),
                                        (512, 6), (512, 7)])
def test_order_tails(nside, lmax, prec):
    import paper_1904_10514_gb300 as hp
    # a band of 2 nside, or at most 64: the degrees above lmax only add to what the analysis must reject
    band = min(2 * nside, 64)
    maps, _ = skies.small_powerlaw_maps(nside, 2, seed=900 + nside, alpha=1.5, noise=1e-3, lmax=band)
    dt = torch.float64 if prec == "fp64" else torch.float32
    x = torch.as_tensor(maps, dtype=dt, device="cuda")
    got = hp.Plan(nside, lmax, 2, prec).analyze(x).cpu().numpy().astype(np.complex128)
    f = x.cpu().numpy().astype(np.float64)
    ref = hp2sph.analyze(f, nside, lmax)
    for b in range(2):
        e = per_l_error(got[b], ref[b], lmax)
        # degrees without power in the sky: against the norm of all that is compared
        e[:2] = per_l_norms(got[b] - ref[b], lmax)[:2] / np.linalg.norm(per_l_norms(ref[b], lmax))
        assert e.max() < TOL[prec], (b, e)
