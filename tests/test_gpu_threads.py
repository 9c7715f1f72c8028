"""Host threads with plans of different sizes launch the same kernels at the same time: no
launch is refused, and the results are those of the same calls made alone."""

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,B,small", [(256, 1, (2, 4, 2)), (512, 8, (16, 2, 4))])
def test_threads_with_plans_of_several_sizes(nside, B, small):
    import paper_1904_10514_gb300 as hp
    L = hp.lib()
    jobs = []
    for ns, b in [(nside, B)] + [(s, 1) for s in small]:
        plan = hp.Plan(ns, min(2 * ns, 32), b, "fp32")
        x = torch.as_tensor(np.random.default_rng(ns).standard_normal((b, plan.npix)), dtype=torch.float32,
                            device="cuda")
        ref = plan.analyze(x).clone()
        back = plan.synthesize(ref).clone()
        stream = torch.cuda.Stream()
        hp.hpx_set_stream(plan.handle, stream.cuda_stream)
        jobs.append((plan, x, ref, back, torch.empty_like(ref), torch.empty_like(back), stream))
    torch.cuda.synchronize()
    start, done, errors = threading.Barrier(len(jobs)), threading.Event(), []

    def work(k):
        plan, x, ref, back, out, m, _ = jobs[k]
        h, px, pr, po, pm = plan.handle, x.data_ptr(), ref.data_ptr(), out.data_ptr(), m.data_ptr()
        start.wait()
        n = 0
        while n < 6000 if k == 0 else not done.is_set():
            rc = L.hpx_analyze(h, px, po) or L.hpx_synthesize(h, pr, pm)
            n += 1
            if n % 200 == 0:   # keeps the queue of launches short
                rc = rc or L.hpx_sync(h)
            if rc != hp.HPX_OK:
                errors.append((k, n, rc))
                break
        if k == 0:
            done.set()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for plan, x, ref, back, out, m, _ in jobs:
        if not errors and not (torch.equal(out, ref) and torch.equal(m, back)):
            errors.append("results differ")
        plan.close()
    assert not errors, errors
