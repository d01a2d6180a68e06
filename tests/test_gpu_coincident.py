"""Pairs of coincident points contribute nothing, also where the two sets have different root cubes (their leaf-relative
coordinates then differ by rounding), and pairs that are merely close keep their contribution.

One leaf: only the near field, FP64 direct sums; tolerance as in test_gpu_near_sizes.py (5e-6 in the 2-norm; the double
layer and the gradient sum terms of both signs, 2e-5).  Many leaves: the plan's accuracy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu
KERNELS = [ffm.LAPLACE, ffm.HELMHOLTZ, ffm.LAPLACE_DL, ffm.LAPLACE_GRAD]


def _sets(n, shift, dtype):
    """Y in a cube at `shift`; X: every third point of Y, and points of a larger cube (so the root cubes differ)."""
    Y = (W.cube_volume(n, 2) + shift).astype(dtype)
    X = np.concatenate([Y[::3], (1.3 * W.cube_volume(n // 2, 1) + shift - 0.1).astype(dtype)])
    return np.ascontiguousarray(X), Y


def _reference(kernel, X, Y, k, u):
    X, Y = X.astype(np.float64), Y.astype(np.float64)
    if kernel == ffm.LAPLACE_DL:
        v = np.stack([np.asarray(O.direct_dl(X, Y, Y, c)).reshape(len(X)) for c in u.astype(np.float64)])
    elif kernel == ffm.LAPLACE_GRAD:
        v = np.stack([np.asarray(O.direct_grad(X, Y, c)).reshape(len(X), 3).T for c in u.astype(np.float64)])
    else:
        kind = O.HELMHOLTZ if kernel == ffm.HELMHOLTZ else O.LAPLACE
        v = np.stack([O.direct(X, Y, c.astype(np.complex128 if k else np.float64), kind, k)[:, 0] for c in u])
    return v if kernel == ffm.HELMHOLTZ else v.real


def _product(kernel, X, Y, k, u, **kw):
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    with ffm.Plan(t(X), t(Y), kernel, k, 1e-3, normals=t(Y) if kernel == ffm.LAPLACE_DL else None, **kw) as p:
        info = p.info()
        v = p.apply(t(u if len(u) > 1 else u[0])).cpu().numpy()
    assert info["oX"] != info["oY"]
    return info, v.reshape((len(u),) + v.shape[v.ndim - (2 if kernel == ffm.LAPLACE_GRAD else 1):])


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("dtype,shift", [(np.float64, 0.0), (np.float64, 37.3), (np.float32, 0.7)])
@pytest.mark.parametrize("kernel", KERNELS)
def test_one_leaf(kernel, dtype, shift, nrhs):
    X, Y = _sets(300, shift, dtype)
    k = 2.0 if kernel == ffm.HELMHOLTZ else 0.0
    u = np.random.default_rng(3).uniform(0.5, 1.0, (nrhs, len(Y))).astype(np.complex64 if k else np.float32)
    info, v = _product(kernel, X, Y, k, u, n_leaf=1 << 20)
    assert info["l_stop"] == 0
    ref = _reference(kernel, X, Y, k, u)
    assert O.rel_l2(v, ref) < (5e-6 if kernel in (ffm.LAPLACE, ffm.HELMHOLTZ) else 2e-5)


@pytest.mark.parametrize("kernel", [ffm.LAPLACE, ffm.HELMHOLTZ])
def test_many_leaves(kernel):
    X, Y = _sets(6000, 0.25, np.float64)
    k = 2.0 if kernel == ffm.HELMHOLTZ else 0.0
    u = np.random.default_rng(4).uniform(0.5, 1.0, (1, len(Y))).astype(np.complex64 if k else np.float32)
    info, v = _product(kernel, X, Y, k, u, n_leaf=8)
    assert info["l_stop"] >= 3
    assert O.rel_l2(v, _reference(kernel, X, Y, k, u)) < 1e-3


@pytest.mark.parametrize("gap", [1e-6, 1e-9, 1e-12])
def test_close_pairs_keep_their_contribution(gap):
    """Points `gap` apart, along the axis on which the two root cubes agree least: 1e-12 of a unit cube is about ten
    times the radius, and the error of its distance (about the radius) is allowed for."""
    X, Y = _sets(300, 0.0, np.float64)
    X[:100] = Y[::3] + np.array([gap, 0.0, 0.0])
    u = np.random.default_rng(5).uniform(0.5, 1.0, (1, len(Y))).astype(np.float32)
    info, v = _product(ffm.LAPLACE, X, Y, 0.0, u, n_leaf=1 << 20)
    a = max(abs(x - y) for x, y in zip(info["oX"], info["oY"]))
    tau = 4.0 * (2.0 ** -52 * 3.0 * info["d0"] + 2.0 ** -46 * (a + info["d0"]))
    assert tau < 0.2 * gap
    assert O.rel_l2(v, _reference(ffm.LAPLACE, X, Y, 0.0, u)) < 5e-6 + tau / gap
