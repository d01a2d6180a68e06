"""Densities near the ends of the FP32 range: a product that is finite term by term stays finite, whatever the
powers of two that scale the tensor-core operands.  Reference: the CUDA-core transfer; tolerance as in
test_gpu_pair_transfer.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,variant,scale,size", [
    (ffm.LAPLACE, ffm.LAG_TC_TRANSLATION, 1.0, 1e35), (ffm.LAPLACE, ffm.LAG_TC_TARGET, 1.0, 1e35),
    (ffm.HELMHOLTZ, ffm.LAG_TC_TRANSLATION, 1.0, 1e35), (ffm.LAPLACE_DL, ffm.LAG_TC_TRANSLATION, 10.0, 1e35),
    (ffm.LAPLACE_GRAD, ffm.LAG_TC_TRANSLATION, 1e3, 2e36), (ffm.LAPLACE, ffm.LAG_TC_TRANSLATION, 1.0, 1e-24),
    (ffm.LAPLACE, ffm.LAG_TC_TARGET, 1.0, 1e-24), (ffm.LAPLACE_GRAD, ffm.LAG_TC_TRANSLATION, 1e-10, 1e-24)])
def test_large_and_small_densities(kernel, variant, scale, size):
    n = 3000
    X, Y = scale * W.cube_volume(n, 1), scale * W.cube_volume(n - 7, 2)
    rng = np.random.default_rng(4)
    helm = kernel == ffm.HELMHOLTZ
    u = rng.standard_normal(n - 7) + (1j * rng.standard_normal(n - 7) if helm else 0.0)
    t = lambda a: torch.as_tensor(a, device="cuda")
    u = t((size * u).astype(np.complex64 if helm else np.float32))
    normals = t(Y / scale) if kernel == ffm.LAPLACE_DL else None
    out = []
    for v in (variant, ffm.LAG_CUDA_CORES):
        with ffm.Plan(t(X), t(Y), kernel, 1.0 if helm else 0.0, 1e-3, r1_override=4, n_leaf=16, kappa_switch=1e9,
                      normals=normals, lagrange_transfer=v) as p:
            out.append(p.apply(u).cpu().numpy().astype(np.complex128))
            info = p.info()
        assert all(info["tune_tc"][l] == v - 1 for l in range(info["l_stop"] + 1) if info["n_adm"][l] > 0)
    assert np.isfinite(out[1]).all() and out[1].any()
    assert O.rel_l2(out[0] / size, out[1] / size) < 3e-6
