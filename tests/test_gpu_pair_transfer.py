"""The f16 hi / lo tensor-core transfers (by translation, and target-stationary) against the CUDA-core transfer of the same
plan constants, at the edges of its tiles: operator rows that pad (r1 = 2, 3, 5, 7), fill one, two and
four row blocks, K chunks with remainders, tiles of one pair, rows of several right-hand sides that
cross tiles, complex operators, stacked and component operators.

Tolerance: both sum the same FP32 products up to the split's error (2^-22 of an operand value, twice,
plus 2^-24) and FP32 accumulation in another order (K up to 1536: about sqrt(K) 2^-24 = 2.3e-6 of a
term's size at worst), so the products agree to 3e-6 in the 2-norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu
TOL = 3e-6


def _pair(kernel, r1, nrhs, n=3000, scale=1.0, spread=False, variant=ffm.LAG_TC_TRANSLATION):
    rng = np.random.default_rng(r1 + 10 * nrhs)
    X, Y = scale * W.cube_volume(n, 1), scale * W.cube_volume(n - 7, 2)
    k = 1.0 / scale if kernel == ffm.HELMHOLTZ else 0.0
    u = rng.standard_normal((nrhs, n - 7))
    if spread:  # densities over ten orders of magnitude, zeros among them
        u *= 10.0 ** rng.uniform(-5, 5, u.shape)
        u[:, ::11] = 0.0
    u = u + 1j * rng.standard_normal(u.shape) if kernel == ffm.HELMHOLTZ else u
    u = torch.as_tensor(u.astype(np.complex64 if kernel == ffm.HELMHOLTZ else np.float32), device="cuda")
    t = lambda a: torch.as_tensor(a, device="cuda")
    out = []
    for variant in (variant, ffm.LAG_CUDA_CORES):
        with ffm.Plan(t(X), t(Y), kernel, k, 1e-3, r1_override=r1, n_leaf=16, kappa_switch=1e9,
                      normals=t(Y) if kernel == ffm.LAPLACE_DL else None, lagrange_transfer=variant) as p:
            v = p.apply(u)
            torch.cuda.synchronize()
            info = p.info()
        lag = [l for l in range(info["l_stop"] + 1) if info["n_adm"][l] > 0]
        assert lag and all(info["tune_tc"][l] == variant - 1 for l in lag)
        out.append(v.cpu().numpy().astype(np.complex128))
    return out


@pytest.mark.parametrize("r1", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kernel", [ffm.LAPLACE, ffm.HELMHOLTZ, ffm.LAPLACE_DL, ffm.LAPLACE_GRAD])
def test_matches_the_cuda_core_transfer(kernel, r1):
    a, b = _pair(kernel, r1, 1)
    assert O.rel_l2(a, b) < TOL


@pytest.mark.parametrize("nrhs", [2, 3, 37, 130])
@pytest.mark.parametrize("kernel", [ffm.LAPLACE, ffm.HELMHOLTZ])
def test_several_right_hand_sides(kernel, nrhs):
    a, b = _pair(kernel, 4, nrhs, n=1200)
    assert O.rel_l2(a, b) < TOL


@pytest.mark.parametrize("nrhs,n", [(1, 3000), (3, 1200), (1, 12000)])
@pytest.mark.parametrize("r1", [2, 3, 4])
def test_target_stationary(r1, nrhs, n):
    a, b = _pair(ffm.LAPLACE, r1, nrhs, n=n, variant=ffm.LAG_TC_TARGET)
    assert O.rel_l2(a, b) < TOL


def test_the_rule_takes_a_level_of_many_pairs_to_the_target_stationary_transfer():
    n = 700_000
    X, Y = (torch.as_tensor(W.cube_volume(n, s), device="cuda") for s in (1, 2))
    u = torch.as_tensor(np.random.default_rng(3).standard_normal(n).astype(np.float32), device="cuda")
    out = []
    for variant in (ffm.LAG_DEFAULT, ffm.LAG_TC_TRANSLATION):
        with ffm.Plan(X, Y, ffm.LAPLACE, 0.0, 1e-3, lagrange_transfer=variant) as p:
            out.append(p.apply(u).double())
            info = p.info()
        assert info["device_errors"] == 0
        many = [l for l in range(22) if info["n_adm"][l] >= 4000 * info["n_trans"][l] * -(-info["n_tgt_boxes"][l] // 19456) > 0]
        assert many
        for l in range(22):
            if info["n_adm"][l]:
                assert info["tune_tc"][l] == (2 if variant == ffm.LAG_DEFAULT and l in many else 1)
    assert float((out[0] - out[1]).norm() / out[1].norm()) < TOL


@pytest.mark.parametrize("scale", [1e-12, 1e12])
def test_scales_of_points_and_densities(scale):
    a, b = _pair(ffm.LAPLACE, 4, 1, scale=scale, spread=True)
    assert O.rel_l2(a, b) < TOL


def test_non_finite_densities_stay_visible():
    X = torch.as_tensor(W.cube_volume(2000, 1), device="cuda")
    u = torch.ones(2000, device="cuda")
    u[3] = float("inf")
    with ffm.Plan(X, X, ffm.LAPLACE, 0.0, 1e-3, n_leaf=16, lagrange_transfer=ffm.LAG_TC_TRANSLATION) as p:
        v = p.apply(u)
    assert not torch.isfinite(v).any()


def test_wait_give_up_of_a_complex_level():
    X = torch.as_tensor(W.cube_volume(3000, 1), device="cuda")
    u = torch.ones(3000, dtype=torch.complex64, device="cuda")
    with ffm.Plan(X, X, ffm.HELMHOLTZ, 1.0, 1e-3, n_leaf=16, wait_tries=-1) as p:
        p.apply(u)
        with pytest.raises(ffm.FFMError) as e:
            p.info()
        assert e.value.status == 4
    with ffm.Plan(X, X, ffm.HELMHOLTZ, 1.0, 1e-3, n_leaf=16) as p:
        p.apply(u)
        assert p.info()["device_errors"] == 0


@pytest.mark.parametrize("shift", [0.0, 0.3, 1.7])
def test_pair_lists_of_a_target_stationary_level_come_back_on_request(shift):
    """Such a level keeps no pair lists: the export makes them from the near lists, the autotuner (which
    times the transfers by translation) makes and keeps them; both equal the other plan's."""
    X = torch.as_tensor(W.gaussian_mixture(20000, 1), device="cuda")
    Y = torch.as_tensor(W.gaussian_mixture(15000, 2) + shift, device="cuda")
    u = torch.ones(15000, device="cuda")
    with ffm.Plan(X, Y, ffm.LAPLACE, 0.0, 1e-3, lagrange_transfer=ffm.LAG_TC_TARGET) as p, \
            ffm.Plan(X, Y, ffm.LAPLACE, 0.0, 1e-3, lagrange_transfer=ffm.LAG_TC_TRANSLATION) as q:
        info = q.info()
        levels = [l for l in range(info["l_stop"] + 1) if info["n_adm"][l]]
        assert levels and p.info()["n_adm"] == info["n_adm"]
        assert any(p.info()["tune_tc"][l] == 2 for l in levels)
        for l in levels:
            np.testing.assert_array_equal(p.pairs(l, "adm"), q.pairs(l, "adm"))
        a, b = p.apply(u).double(), q.apply(u).double()
        assert float((a - b).norm() / b.norm()) < TOL
        p.autotune()
        for l in levels:
            np.testing.assert_array_equal(p.pairs(l, "adm"), q.pairs(l, "adm"))
        assert float((p.apply(u).double() - b).norm() / b.norm()) < TOL
        assert p.info()["device_errors"] == 0
