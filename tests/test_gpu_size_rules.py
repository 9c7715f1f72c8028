"""Both sides of the rules that choose a form by the size of the work: the same maps in a
batch of one and in batches that take the other form."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# two FP32 evaluations with relative errors up to 5e-7 each; FP64 as the adjoint's gate
TOL = {"fp32": 1e-6, "fp64": 2e-12}


def _coefficients(L, B, prec):
    rng = np.random.default_rng(L + B)
    n = (L + 1) * (L + 2) // 2
    a = rng.standard_normal((B, n)) + 1j * rng.standard_normal((B, n))
    return torch.as_tensor(a, device="cuda").to(torch.complex64 if prec == "fp32" else torch.complex128)


@pytest.mark.parametrize("nside,lmax,B", [(256, 512, 8), (256, 511, 4), (512, 1024, 4), (512, 900, 8)])
def test_orders_per_warp(nside, lmax, B):
    """Sweeps of 2 and 4 orders per warp (one in the small plans of the other tests): the analysis has
    the bits of the complex-lane form, the transposed sweeps agree with those of another batch."""
    import paper_1904_10514_gb300 as hp
    x = torch.as_tensor(np.random.default_rng(B).standard_normal((B, 12 * nside * nside)), dtype=torch.float32,
                        device="cuda")
    a = _coefficients(lmax, 32, "fp32")
    plan = hp.Plan(nside, lmax, B, "fp32", sweeps=True, synthesis=True)
    t = list(plan.tuning)
    fwd = []
    for form in (0, 2):
        t[2] = form
        plan.tuning = tuple(t)
        fwd.append(plan.analyze(x).clone())
    assert torch.equal(*fwd)
    many, adj = plan.sh_synthesis(a[:B]).clone(), plan.synthesize(a[:B]).clone()
    torch.cuda.synchronize()
    plan.close()
    plan = hp.Plan(nside, lmax, 32, "fp32", sweeps=True, synthesis=True)   # one order per warp
    for u, v in ((many, plan.sh_synthesis(a)), (adj, plan.synthesize(a))):
        d = torch.linalg.vector_norm(u - v[:B]) / torch.linalg.vector_norm(u)
        assert float(d) <= TOL["fp32"]
    torch.cuda.synchronize()
    plan.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nside,lmax,B", [(4, 7, 1300), (8, 16, 310), (16, 32, 80), (32, 64, 20), (64, 33, 19),
                                          (64, 128, 5)])
def test_backward_grid(nside, lmax, B, prec):
    """One block per column for small grids in few columns, grid FFT and interpolation else."""
    import paper_1904_10514_gb300 as hp
    a = _coefficients(lmax, B, prec)
    out = []
    for b in (B, 1):
        plan = hp.Plan(nside, lmax, b, prec, sweeps=True, synthesis=True)
        out.append((plan.sh_synthesis(a[:b]).clone(), plan.synthesize(a[:b]).clone()))
        torch.cuda.synchronize()
        plan.close()
    for many, one in zip(*out):
        d = torch.linalg.vector_norm(many[0] - one[0]) / torch.linalg.vector_norm(one[0])
        assert float(d) <= TOL[prec]


@pytest.mark.parametrize("prec,nside,lmax,B", [("fp32", 4, 8, 2), ("fp32", 16, 32, 70), ("fp32", 64, 33, 17),
                                               ("fp64", 4, 8, 2), ("fp64", 16, 9, 33), ("fp64", 64, 33, 9)])
def test_short_rings(prec, nside, lmax, B):
    """One warp per ring pair in large batches of short rings (and at Nside 4), four in the plan
    of one map: the same bits."""
    import paper_1904_10514_gb300 as hp
    x = torch.as_tensor(np.random.default_rng(nside).standard_normal((B, 12 * nside * nside)), device="cuda")
    x = x.to(torch.float32 if prec == "fp32" else torch.float64)
    # (FP32 sweeps and FP64 operators sum in one order for every batch)
    out = []
    for b in (B, 1):
        plan = hp.Plan(nside, lmax, b, prec, sweeps=prec == "fp32", simt=True)
        out.append(plan.analyze(x[:b].contiguous()).clone())
        torch.cuda.synchronize()
        plan.close()
    assert torch.equal(out[0][0], out[1][0])


@pytest.mark.parametrize("nside,lmax,B", [(64, 128, 5), (128, 255, 8), (256, 300, 7), (64, 127, 8)])
def test_synthesis_operators_of_5_to_8_maps(nside, lmax, B):
    """Stored in groups of rows from lmax 128 on, by rows below: both directions against FP64."""
    import paper_1904_10514_gb300 as hp
    a = _coefficients(lmax, B, "fp64")
    out = {}
    for prec in ("fp32", "fp64"):
        plan = hp.Plan(nside, lmax, B, prec, synthesis=True)
        f = plan.sh_synthesis(a.to(plan.cdtype)).clone()
        x = f if prec == "fp32" else out["fp32"][0].double()
        out[prec] = (f, plan.sh_synthesis_adjoint(x).clone())
        torch.cuda.synchronize()
        plan.close()
    for u, v in zip(out["fp32"], out["fp64"]):
        assert float(torch.linalg.vector_norm(u - v) / torch.linalg.vector_norm(v)) <= 5e-7
