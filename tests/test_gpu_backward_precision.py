"""Rounding of the FP32 synthesis against the FP64 plan: no larger than with radix-2 passes
and directly tabulated twiddles, whose relative errors on these inputs are the figures in
the list, but for 6%."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rounding(nside, lmax, B, parity=None):
    import paper_1904_10514_gb300 as hp
    rng = np.random.default_rng(nside + B)
    n = (lmax + 1) * (lmax + 2) // 2
    a = rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n))
    if parity is not None:   # the orders of one parity alone
        a = a * (np.repeat(np.arange(lmax + 1), lmax + 1 - np.arange(lmax + 1)) % 2 == parity)
    a = torch.as_tensor(a, device="cuda").to(torch.complex64)
    f = {}
    for prec in ("fp32", "fp64"):
        plan = hp.Plan(nside, lmax, B, prec, synthesis=True)
        f[prec] = plan.sh_synthesis(a.to(plan.cdtype)).double().clone()
        torch.cuda.synchronize()
        plan.close()
    return float(torch.linalg.vector_norm(f["fp32"] - f["fp64"]) / torch.linalg.vector_norm(f["fp64"]))


@pytest.mark.parametrize("nside,lmax,B,radix2", [(64, 128, 16, 2.290e-7), (256, 512, 9, 2.446e-7),
                                                 (512, 700, 9, 2.801e-7), (128, 256, 4, 2.545e-7)])
def test_synthesis_rounding(nside, lmax, B, radix2):
    assert _rounding(nside, lmax, B) <= 1.06 * radix2


@pytest.mark.parametrize("nside,lmax,B,even,odd", [(64, 128, 16, 2.254e-7, 2.292e-7), (128, 256, 16, 2.332e-7, 2.367e-7),
                                                   (256, 512, 9, 2.413e-7, 2.451e-7)])
def test_orders_of_one_parity(nside, lmax, B, even, odd):
    """An even and an odd order share an FFT: neither parity takes on the other's rounding."""
    assert _rounding(nside, lmax, B, 0) <= 1.06 * even
    assert _rounding(nside, lmax, B, 1) <= 1.06 * odd
