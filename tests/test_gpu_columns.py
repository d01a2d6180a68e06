"""The right-hand sides of one product are independent in the tensor-core transfers: their magnitudes may
differ by any factor, and a non-finite density stays in its own column.

Reference: the CUDA-core transfer of the same plan constants, column by column.  Tolerance as in
test_gpu_pair_transfer.py: the same products up to the split's error and FP32 sums in another order, 3e-6 of
a column's 2-norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu
TOL = 3e-6


def _products(u, variant, r1, n, **kw):
    X, Y = W.cube_volume(n, 1), W.cube_volume(n - 7, 2)
    t = lambda a: torch.as_tensor(a, device="cuda")
    out = []
    for v in (variant, ffm.LAG_CUDA_CORES):
        with ffm.Plan(t(X), t(Y), ffm.LAPLACE, 0.0, 1e-3, r1_override=r1, n_leaf=16, lagrange_transfer=v, **kw) as p:
            out.append(p.apply(t(u)).cpu().numpy().astype(np.float64))
            info = p.info()
        lag = [l for l in range(info["l_stop"] + 1) if info["n_adm"][l] > 0]
        assert lag and all(info["tune_tc"][l] == v - 1 for l in lag) and info["device_errors"] == 0
    return out


def _densities(n, nrhs):
    return np.random.default_rng(nrhs).standard_normal((nrhs, n - 7)).astype(np.float32)


@pytest.mark.parametrize("variant", [ffm.LAG_TC_TARGET, ffm.LAG_TC_TRANSLATION])
@pytest.mark.parametrize("r1", [2, 4])
@pytest.mark.parametrize("scales", [(1.0, 1e-10), (1e10, 1.0, 1e-10), (1.0, 0.0, 1e-30, 1e8, 1e-8)])
def test_columns_of_different_magnitude(scales, r1, variant):
    n = 3000
    u = _densities(n, len(scales)) * np.asarray(scales, np.float32)[:, None]
    a, b = _products(u, variant, r1, n)
    for m, s in enumerate(scales):
        if s == 0.0:
            assert not a[m].any()
        else:
            assert O.rel_l2(a[m], b[m]) < TOL, (m, s)


@pytest.mark.parametrize("variant", [ffm.LAG_TC_TARGET, ffm.LAG_TC_TRANSLATION])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_a_non_finite_density_stays_in_its_column(bad, variant):
    n = 3000
    u = _densities(n, 4)
    u[0] *= 1e-6
    u[3] *= 1e6
    u[1, 17] = bad
    a, b = _products(u, variant, 4, n)
    assert not np.isfinite(a[1]).any()
    for m in (0, 2, 3):
        assert O.rel_l2(a[m], b[m]) < TOL, m


def test_densities_over_ten_orders_of_magnitude_in_one_column():
    """A target-stationary level has one scale per column; what it loses of a small source is far below the
    large sources' own potential at every target (error 2^-38 of the largest u~ per term)."""
    n = 3000
    rng = np.random.default_rng(5)
    u = _densities(n, 1) * (10.0 ** rng.uniform(-5, 5, (1, n - 7))).astype(np.float32)
    a, b = _products(u, ffm.LAG_TC_TARGET, 4, n)
    assert np.max(np.abs(a - b) / np.abs(b).max()) < TOL and O.rel_l2(a, b) < TOL
