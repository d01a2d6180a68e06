"""The double-float plane-wave levels against the same plan in FP64: what their sums lose.

The error is that of the double-float phases, factors and sums (2^-44 .. 2^-47 relative) times the quadrature's
cancellation (8e4 at eps 1e-4, 8e7 at 1e-6 on the finest level).  The bounds are the measured errors of sums that are
normalised after every term (5.2e-12 and 4.8e-9) plus an eighth: a cheaper form of the sums may not cost
digits.  Sums normalised every eight terms give 7.2e-12 and 7.0e-9."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs,eps,bound", [(1, 1e-4, 5.85e-12), (8, 1e-4, 6.25e-12), (16, 1e-6, 5.4e-9), (3, 1e-6, 5.4e-9)])
def test_sums_keep_the_accuracy_of_terms_normalised_one_by_one(nrhs, eps, bound):
    P = W.helmholtz_cube_multirhs(30000, nrhs=max(nrhs, 2), eps=eps)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    u = P.u.T.astype(np.complex128)[:nrhs]
    out = []
    for prec in (ffm.PREC_F32X2, ffm.PREC_F64):
        with ffm.Plan(t(P.X), t(P.Y), ffm.HELMHOLTZ, P.k, eps, weights=t(P.w), precision=prec,
                      pw_transform=ffm.PW_DIRECT) as p:
            out.append(p.apply(t(u)).cpu().numpy())
            info = p.info()
        assert 2 in info["mode"]
    assert np.linalg.norm(out[0] - out[1]) / np.linalg.norm(out[1]) < bound
