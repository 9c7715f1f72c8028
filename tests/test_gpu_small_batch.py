"""The operators applied to small batches and to FP64 batches (matrix-vector form of
the analysis): sizes at the edges of its row tiles, k chunks and map groups."""

import numpy as np
import pytest

import skies
from helpers import per_l_error, per_l_norms
from oracle import hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 1e-5}   # the parity gates of the FP64 and FP32 plans


@pytest.mark.parametrize("prec,batches", [("fp32", (1, 2, 3, 4, 5, 8)), ("fp64", (1, 2, 3, 4, 5, 7, 9))])
@pytest.mark.parametrize("nside,lmax", [(2, 4), (4, 0), (16, 31), (64, 127), (128, 256), (128, 129)])
def test_every_batch_gives_the_same_coefficients(nside, lmax, prec, batches):
    """nside 2: fewer k than one 16-byte load per lane needs; 16, 64: one partly
    filled chunk of k; 128: whole chunks and the odd last term; chains of 1 .. 129
    rows against tiles of 64.  Map by map the coefficients are those of the
    one-map plan to the last bit, and those meet the oracle (the degrees below 2,
    where the sky has no power, against the norm of its whole band, also when lmax
    cuts that band off)."""
    import paper_1904_10514_gb300 as hp
    B = max(batches)
    maps, _ = skies.small_powerlaw_maps(nside, B, seed=500 + nside, alpha=2.0, noise=1e-3, lmax=2 * nside)
    dt = torch.float64 if prec == "fp64" else torch.float32
    x = torch.as_tensor(maps, dtype=dt, device="cuda")
    got = {b: hp.Plan(nside, lmax, b, prec).analyze(x[:b].contiguous()) for b in batches}
    one = hp.Plan(nside, lmax, 1, prec)
    f = x.cpu().numpy().astype(np.float64)
    ref = hp2sph.analyze(f, nside, lmax)
    band = [np.linalg.norm(per_l_norms(v, 2 * nside)) for v in hp2sph.analyze(f, nside, 2 * nside)]
    for k in range(B):
        alone = one.analyze(x[k:k + 1].contiguous())
        a = alone[0].cpu().numpy().astype(np.complex128)
        e = per_l_error(a, ref[k], lmax)
        e[:2] = per_l_norms(a - ref[k], lmax)[:2] / band[k]
        assert e.max() < TOL[prec]
        for b in batches:
            if k < b:
                assert torch.equal(got[b][k], alone[0]), (b, k)
