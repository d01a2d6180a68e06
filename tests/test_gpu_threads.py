"""Products of different plans from several threads at once: the kernels' launch settings depend on the plan's
sizes, and no thread's setting may break another's launch.  Every product equals the one that its plan
gave alone, up to the order of the floating-point sums (5e-6 of the 2-norm: FP32 sums of a few thousand terms)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


def _run(plans, rounds):
    """plans: (plan, u).  One thread each, `rounds` products on a stream of its own."""
    alone = [p.apply(u).cpu().numpy() for p, u in plans]
    torch.cuda.synchronize()
    got, errors = [None] * len(plans), []
    gate = threading.Barrier(len(plans))

    def work(i):
        try:
            p, u = plans[i]
            s = torch.cuda.Stream()
            out = torch.empty_like(torch.as_tensor(alone[i], device="cuda"))
            gate.wait()
            with torch.cuda.stream(s):
                for _ in range(rounds):
                    p.apply(u, out=out, stream=s)
            s.synchronize()
            got[i] = out.cpu().numpy()
        except Exception as e:  # the launch that was refused
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(plans))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(len(plans)):
        assert O.rel_l2(got[i], alone[i]) < 5e-6


@pytest.mark.parametrize("shapes", [((6, ffm.LAG_TC_TRANSLATION), (7, ffm.LAG_TC_TRANSLATION), (8, ffm.LAG_TC_TRANSLATION)),
                                    ((2, ffm.LAG_TC_TARGET), (3, ffm.LAG_TC_TARGET), (2, ffm.LAG_TC_TARGET))])
def test_lagrange_transfers_of_different_sizes(shapes):
    plans = []
    for i, (r1, variant) in enumerate(shapes):
        n = 2000 + 300 * i
        X, Y = (torch.as_tensor(W.cube_volume(n, s), device="cuda") for s in (2 * i + 1, 2 * i + 2))
        u = torch.as_tensor(np.random.default_rng(i).standard_normal(n).astype(np.float32), device="cuda")
        plans.append((ffm.Plan(X, Y, ffm.LAPLACE, 0.0, 1e-3, r1_override=r1, n_leaf=16, lagrange_transfer=variant), u))
    _run(plans, 400)
    for p, _ in plans:
        assert p.info()["device_errors"] == 0
        p.close()


def test_nufft_levels_of_different_sizes():
    plans = []
    for i, (n, eps) in enumerate(((8000, 1e-3), (12000, 1e-4), (16000, 1e-3))):
        prob = W.helmholtz_sphere(n, seed=i + 1)
        t = lambda a: torch.as_tensor(a, device="cuda")
        plans.append((ffm.Plan(t(prob.X), t(prob.Y), ffm.HELMHOLTZ, prob.k, eps, weights=t(prob.w),
                               pw_transform=ffm.PW_NUFFT, precision=ffm.PREC_F32), t(prob.u)))
    assert any(p.info()["nufft"][l] for p, _ in plans for l in range(22))
    _run(plans, 200)
    for p, _ in plans:
        assert p.info()["device_errors"] == 0
        p.close()
