"""Complex Lagrange levels lose nothing against FP32 multiply-adds that a user could see: error against the oracle's
FFM with the tensor-core transfer and with the CUDA-core one.

Bound on the difference along the result (a tensor-core accumulation truncates, so its error has one sign): a
fill of four chunks is eight truncating steps, which lose at most 3 ulps (3 2^-24 = 1.8e-7).  Fills of half
the K extent and more lost 2.3e-7 to 5e-7.  Bounds on the error itself: what FP32 multiply-adds gave before the
transfer moved to tensor cores."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


def _errors(X, Y, u, k, eps, w, ref):
    t = lambda a: torch.as_tensor(a, device="cuda")
    out = []
    for variant in (ffm.LAG_DEFAULT, ffm.LAG_CUDA_CORES):
        with ffm.Plan(t(X), t(Y), ffm.HELMHOLTZ, k, eps, weights=t(w), precision=ffm.PREC_F64,
                      lagrange_transfer=variant) as p:
            d = p.apply(t(u)).cpu().numpy().astype(np.complex128) - ref
            assert 1 in p.info()["mode"] and p.info()["device_errors"] == 0
        out.append((np.linalg.norm(d) / np.linalg.norm(ref), (np.vdot(ref, d) / np.vdot(ref, ref)).real))
    return out


@pytest.mark.parametrize("k,eps,before", [(1e-3, 1e-4, 5.4e-7), (1e-3, 1e-3, 2.7e-7)])
def test_constant_density(k, eps, before):
    n = 20000
    X, Y, w = W.cube_volume(n, 1), W.cube_volume(n - 7, 2), np.full(n - 7, 1.0 / n)
    u = np.ones(n - 7, np.complex64)
    ref = O.ffm(X, Y, u.astype(np.complex128), O.HELMHOLTZ, k, eps, w=w)[:, 0]
    (tc, along), (cc, along_cc) = _errors(X, Y, u, k, eps, w, ref)
    assert abs(along - along_cc) < 1.8e-7
    assert tc < before and cc < before


def test_surface_with_plane_wave_levels():
    n, k = 20000, 12.0
    X, w = W.cube_surface(n, 31), np.full(n, 6.0 / n)
    u = np.exp(1j * k * X @ np.array([0.0, 0.6, 0.8])).astype(np.complex64)
    ref = O.ffm(X, X, u.astype(np.complex128), O.HELMHOLTZ, k, 1e-4, w=w)[:, 0]
    for err, _ in _errors(X, X, u, k, 1e-4, w, ref):
        assert err < 3.1e-7
