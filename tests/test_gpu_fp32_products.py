"""FP32 plans of more than 8 maps take FP16 pairs (22 bits) of their operators in the
analysis and the synthesis only: the transposed synthesis and the adjoint keep FP32
products, and give the bits of a plan that never leaves the FP32 pipes there."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,B", [(8, 16, 9), (64, 128, 16), (128, 255, 33)])
def test_transposed_synthesis(nside, lmax, B):
    import paper_1904_10514_gb300 as hp
    x = torch.as_tensor(np.random.default_rng(nside).standard_normal((B, 12 * nside * nside)), dtype=torch.float32,
                        device="cuda")
    out = []
    for simt in (False, True):
        plan = hp.Plan(nside, lmax, B, "fp32", simt=simt, jacobi=True)
        out.append((plan.sh_synthesis_adjoint(x).clone(), plan.healpix_analysis(x, niter=0).clone()))
        torch.cuda.synchronize()
        plan.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("nside,lmax,B", [(8, 16, 9), (64, 128, 16), (128, 255, 33)])
def test_adjoint(nside, lmax, B):
    import paper_1904_10514_gb300 as hp
    rng = np.random.default_rng(nside + 1)
    n = (lmax + 1) * (lmax + 2) // 2
    a = torch.as_tensor(rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n)), device="cuda").to(torch.complex64)
    out = []
    for sweeps in (False, True):
        plan = hp.Plan(nside, lmax, B, "fp32", sweeps=sweeps)
        out.append((plan.synthesize(a).clone(), plan.analyze_vjp(a).clone()))
        torch.cuda.synchronize()
        plan.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
