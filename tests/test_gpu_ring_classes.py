"""Ring transforms at the edges of their launch classes: the shortest and the longest
ring of every kind (plain, Bluestein, quarter-length Bluestein), several classes in one
map, and the work list of an uneven batch with classes of both of its launches."""

import numpy as np
import pytest

import skies
from helpers import per_l_error, per_l_norms
from oracle import hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 1e-5}   # the parity gates of the FP64 and FP32 plans


def _check(got, ref, lmax, tol):
    e = per_l_error(got, ref, lmax)
    # degrees without power in the sky: against the norm of all that is compared
    e[:2] = per_l_norms(got - ref, lmax)[:2] / np.linalg.norm(per_l_norms(ref, lmax))
    assert e.max() < tol, e


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nside,lmax", [(2, 4), (32, 9), (128, 8), (512, 9), (1024, 6)])
def test_ring_kinds(nside, lmax, prec):
    """Both ring forms, on a sky with power up to 4 lmax, so that the rings carry
    orders that the output drops."""
    import paper_1904_10514_gb300 as hp
    maps, _ = skies.small_powerlaw_maps(nside, 2, seed=70 + nside, alpha=1.5, noise=1e-3, lmax=min(2 * nside, 4 * lmax))
    x = torch.as_tensor(maps, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    ref = hp2sph.analyze(x.cpu().numpy().astype(np.float64), nside, lmax)
    plan = hp.Plan(nside, lmax, 2, prec)
    t = list(plan.tuning)
    for form in (0, 1):
        t[4] = form
        plan.tuning = tuple(t)
        got = plan.analyze(x).cpu().numpy().astype(np.complex128)
        for b in range(2):
            _check(got[b], ref[b], lmax, TOL[prec])
    plan.close()


def test_ring_forms_agree_at_nside2048():
    """Rings of up to 8192 points and Bluestein convolutions of 16384: per degree
    within half the gate of each other (both are FP32 evaluations of the same DFTs)."""
    import paper_1904_10514_gb300 as hp
    maps, _ = skies.small_powerlaw_maps(2048, 1, seed=77, alpha=1.5, noise=1e-3, lmax=32)
    x = torch.as_tensor(maps, dtype=torch.float32, device="cuda")
    plan = hp.Plan(2048, 24, 1, "fp32")
    t = list(plan.tuning)
    res = []
    for form in (0, 1):
        t[4] = form
        plan.tuning = tuple(t)
        res.append(plan.analyze(x).cpu().numpy().astype(np.complex128)[0])
    plan.close()
    _check(res[1], res[0], 24, 0.5 * TOL["fp32"])


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_uneven_work_list(prec):
    import paper_1904_10514_gb300 as hp
    nsides, lmaxs = [512, 16, 256, 512], [5, 9, 6, 3]
    maps = [skies.small_powerlaw_maps(ns, 1, seed=80 + k, alpha=1.5, noise=1e-3, lmax=32)[0][0]
            for k, ns in enumerate(nsides)]
    plan = hp.Plan(nsides=nsides, lmaxs=lmaxs, precision=prec)
    x = torch.as_tensor(np.concatenate(maps), dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    got = plan.analyze(x).cpu().numpy().astype(np.complex128)
    f = x.cpu().numpy().astype(np.float64)
    ia = ip = 0
    for ns, L in zip(nsides, lmaxs):
        na, npix = hp2sph.n_alm(L), 12 * ns * ns
        _check(got[ia:ia + na], hp2sph.analyze(f[None, ip:ip + npix], ns, L)[0], L, TOL[prec])
        ia, ip = ia + na, ip + npix
    plan.close()
