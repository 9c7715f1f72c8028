"""The backward ring and grid stages at the edges of their launch classes: every pass
structure of the inverse grid FFT, plain, Bluestein and quarter-length rings in both
directions' forms, one order, an unpaired last order, and a row tail of the interpolation."""

import numpy as np
import pytest

from oracle import dense, hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DOT = {"fp64": 1e-12, "fp32": 2e-5}   # the gates of the dot and synthesis tests
SYN = {"fp64": 1e-11, "fp32": 1e-5}
SIZES = [(2, 3), (4, 8), (16, 0), (32, 31), (64, 6), (128, 5), (256, 6), (512, 7)]


def _alm(L, B, seed):
    rng = np.random.default_rng(seed)
    n = hp2sph.n_alm(L)
    return rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nside,lmax", SIZES + [(1024, 5), (2048, 4)])
def test_transpose_of_analysis(nside, lmax, prec):
    """<A f, a> = <f, A^T a> in both ring forms, for every map of the batch."""
    import paper_1904_10514_gb300 as hp
    if nside == 2048 and prec == "fp64":
        pytest.skip("FP32 only")
    B = 3 if nside <= 512 else 1
    rng = np.random.default_rng(nside + lmax)
    plan = hp.Plan(nside, lmax, B, prec)
    rd, cd = (torch.float64, torch.complex128) if prec == "fp64" else (torch.float32, torch.complex64)
    f = torch.as_tensor(rng.standard_normal((B, plan.npix)), dtype=rd, device="cuda")
    a = torch.as_tensor(_alm(lmax, B, nside), dtype=cd, device="cuda")
    fn, an = f.cpu().numpy().astype(np.float64), a.cpu().numpy().astype(np.complex128)
    t = list(plan.tuning)
    for form in (0, 1):
        t[4] = form
        plan.tuning = tuple(t)
        Af = plan.analyze(f).cpu().numpy().astype(np.complex128)
        Ata = plan.synthesize(a).cpu().numpy().astype(np.float64)
        for b in range(B):
            lhs, rhs = dense.alm_dot(Af[b], an[b], lmax), float(np.dot(fn[b], Ata[b]))
            assert abs(lhs - rhs) <= DOT[prec] * np.linalg.norm(fn[b]) * np.linalg.norm(Ata[b]), (form, b, lhs, rhs)
    plan.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nside,lmax", SIZES + [(1024, 5)])
def test_synthesis(nside, lmax, prec):
    import paper_1904_10514_gb300 as hp
    B = 2 if nside <= 512 else 1
    a = _alm(lmax, B, 7 * nside).astype(np.complex128 if prec == "fp64" else np.complex64)
    plan = hp.Plan(nside, lmax, B, prec, synthesis=True)
    ref = hp2sph.synthesize(a.astype(np.complex128), nside, lmax)
    t = list(plan.tuning)
    for form in (0, 1):
        t[4] = form
        plan.tuning = tuple(t)
        f = plan.sh_synthesis(torch.as_tensor(a, device="cuda")).cpu().numpy()
        assert np.max(np.abs(f - ref)) <= SYN[prec] * np.max(np.abs(ref)), form
    plan.close()
