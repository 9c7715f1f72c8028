"""The synthesis at Nside 2048 against scipy's Y_l^m on rings of every transform class, ring by
ring, so that an error in one class is not lost in the norm of the whole sphere."""

import numpy as np
import pytest

from oracle import geometry, hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sample(nside):
    """Ring indices: ends and middles of the transform classes, both hemispheres, the equator."""
    polar = [1, 2, 25, 100, 127, 128, 129, 200, 256, 257, 400, 512, 513, 700, 1023, 1025, 1600, 2047]
    north = [k - 1 for k in polar if k < nside] + [nside - 1, nside, 2 * nside - 2]
    return [r if k % 2 else 4 * nside - 2 - r for k, r in enumerate(north)] + [2 * nside - 1]


def _coefficients(L, seed):
    rng = np.random.default_rng(seed)
    n = hp2sph.n_alm(L)
    a = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    a[:L + 1].imag = 0
    return a.astype(np.complex64)


def test_synthesis_at_nside2048():
    from scipy.special import sph_harm_y

    import paper_1904_10514_gb300 as hp
    nside, L = 2048, 4
    plan = hp.Plan(nside, L, 1, "fp32", synthesis=True)
    a = _coefficients(L, 3)
    f = plan.sh_synthesis(torch.as_tensor(a, device="cuda")[None])[0].cpu().numpy().astype(np.float64)
    plan.close()
    table = geometry.ring_table(nside)
    for r in _sample(nside):
        q = table[r]
        phi = q["phi0"] + 2 * np.pi * np.arange(q["nphi"]) / q["nphi"]
        ref = np.zeros(q["nphi"])
        for m in range(L + 1):
            for l in range(m, L + 1):
                y = a[hp2sph.alm_index(l, m, L)] * sph_harm_y(l, m, q["theta"], phi)
                ref += (1 if m == 0 else 2) * y.real
        got = f[q["start"]:q["start"] + q["nphi"]]
        assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(a)) * (L + 1), (r, q["nphi"])
