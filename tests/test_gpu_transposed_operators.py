"""Transposed per-order operators against the same transforms through the transposed
sweeps and the Legendre-to-Fourier table: one map, the last batch of the small-batch
kernels and the first of the tensor-core ones, a column tile with one map in it and
several tiles, row tails (odd and even lmax, lmax below the grid's order)."""

import numpy as np
import pytest

from oracle import hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# two evaluations that each stay within the adjoint's gate of the exact result
TOL = {"fp64": 2e-12, "fp32": 2e-5}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("B", [1, 7, 8, 9, 16, 33, 65])
@pytest.mark.parametrize("nside,lmax", [(2, 4), (8, 13), (16, 0), (32, 57), (64, 128)])
def test_operators_match_sweeps(nside, lmax, B, prec):
    import paper_1904_10514_gb300 as hp
    cd = torch.complex128 if prec == "fp64" else torch.complex64
    rng = np.random.default_rng(nside + lmax + B)
    n = hp2sph.n_alm(lmax)
    a = torch.as_tensor(rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n)), dtype=cd, device="cuda")
    out = {}
    for sweeps in (False, True):
        plan = hp.Plan(nside, lmax, B, prec, sweeps=sweeps, synthesis=True)
        r = [plan.synthesize(a), plan.analyze_vjp(a), plan.sh_synthesis(a)]
        x = r[2].clone()
        if sweeps:
            x = out[False][2]
        r.append(plan.sh_synthesis_adjoint(x))
        out[sweeps] = [v.clone() for v in r]
        torch.cuda.synchronize()
        plan.close()
    for name, u, v in zip(("synthesize", "analyze_vjp", "sh_synthesis", "sh_synthesis_adjoint"), out[False], out[True]):
        u, v = u.reshape(B, -1), v.reshape(B, -1)
        d = torch.linalg.vector_norm(u - v, dim=1) / torch.linalg.vector_norm(v, dim=1)
        assert float(d.max()) <= TOL[prec], (name, d)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nside,lmax,B", [(128, 0, 1), (128, 61, 3), (256, 31, 8), (256, 33, 5)])
def test_last_k(nside, lmax, B, prec):
    """Nside + 1 modes: one past the tiles of 128 (FP32) or 64 (FP64)."""
    test_operators_match_sweeps(nside, lmax, B, prec)


@pytest.mark.parametrize("B", [8, 9, 33])
@pytest.mark.parametrize("nside,lmax", [(16, 21), (64, 128)])
def test_equal_weight_analysis(nside, lmax, B):
    """hpx_healpix_analysis through the transposed synthesis tiles."""
    import paper_1904_10514_gb300 as hp
    x = torch.as_tensor(np.random.default_rng(B).standard_normal((B, 12 * nside * nside)), dtype=torch.float32,
                        device="cuda")
    out = []
    for sweeps in (False, True):
        plan = hp.Plan(nside, lmax, B, "fp32", sweeps=sweeps, synthesis=True)
        out.append(plan.healpix_analysis(x, niter=1).clone())
        torch.cuda.synchronize()
        plan.close()
    d = torch.linalg.vector_norm(out[0] - out[1], dim=1) / torch.linalg.vector_norm(out[1], dim=1)
    assert float(d.max()) <= TOL["fp32"], d
