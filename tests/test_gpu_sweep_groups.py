"""Real-lane sweeps with several orders per warp against the complex-lane form, which
applies the same rotations to the same values: batches that leave 1 to 32 orders per
warp, part of a warp idle, and more maps than lanes; odd and even lmax."""

import numpy as np
import pytest

from oracle import dense, hp2sph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 8, 9, 16, 17, 33])
@pytest.mark.parametrize("nside,lmax", [(2, 1), (16, 32), (32, 57), (64, 128)])
def test_forms_identical_and_adjoint(nside, lmax, B):
    import paper_1904_10514_gb300 as hp
    rng = np.random.default_rng(B + lmax)
    plan = hp.Plan(nside, lmax, B, "fp32", sweeps=True)
    x = torch.as_tensor(rng.standard_normal((B, plan.npix)), dtype=torch.float32, device="cuda")
    n = hp2sph.n_alm(lmax)
    a_np = rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n))
    a = torch.as_tensor(a_np, dtype=torch.complex64, device="cuda")
    t = list(plan.tuning)
    fwd, adj = [], []
    for form in (0, 1, 2):
        t[2] = form
        plan.tuning = tuple(t)
        fwd.append(plan.analyze(x).clone())
        adj.append(plan.synthesize(a).cpu().numpy().astype(np.float64))
    assert torch.equal(fwd[0], fwd[1]) and torch.equal(fwd[0], fwd[2])
    xn, Af = x.cpu().numpy().astype(np.float64), fwd[2].cpu().numpy().astype(np.complex128)
    for b in range(B):
        lhs = dense.alm_dot(Af[b], a[b].cpu().numpy().astype(np.complex128), lmax)
        for v in adj:
            rhs = float(np.dot(xn[b], v[b]))
            assert abs(lhs - rhs) <= 2e-5 * np.linalg.norm(xn[b]) * np.linalg.norm(v[b]), (b, lhs, rhs)
    plan.close()
