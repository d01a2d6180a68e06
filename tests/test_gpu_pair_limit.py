"""A level with more admissible pairs than a list with 32-bit offsets holds: the target-stationary transfer, which
needs no list, takes it; everything that would need one is refused with a status.

One point per cell of two grids of 256^3 cells that are shifted by half a cell: at level 8 a target keeps the
children of up to 4^3 near parents, of which up to 4^3 stay near."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1909_05600_gb300 import ffm

pytestmark = pytest.mark.gpu
N = 256
UNSUPPORTED = 5


def _grids():
    g = torch.arange(N, dtype=torch.float64, device="cuda") / (N - 1)
    X = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3).contiguous()
    return X, X + 0.5 / N * (1.0 + 2.0 ** -20)


def _counts(sigma8):
    """Near and admissible pairs of level 8 by the definition, per axis (|sigma 2^l + k| < 2 is near)."""
    near = lambda l, k: abs(sigma8 * 2.0 ** (l - 8) + k) < 2.0
    x = np.arange(N)
    k8, k7 = x[:, None] - x[None, :], (x[:, None] >> 1) - (x[None, :] >> 1)
    cand = near(7, k7)
    both = cand & near(8, k8)
    c, n = cand.sum(1).astype(object), both.sum(1).astype(object)
    tot = lambda a: int(a.sum()) ** 3
    return tot(n), tot(c) - tot(n)


def test_more_pairs_than_a_list_holds():
    X, Y = _grids()
    u = torch.rand(N ** 3, dtype=torch.float32, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) + 0.5
    for variant in (ffm.LAG_CUDA_CORES, ffm.LAG_TC_TRANSLATION):
        with pytest.raises(ffm.FFMError) as e:
            ffm.Plan(X, Y, ffm.LAPLACE, 0.0, 1e-2, n_leaf=4, lagrange_transfer=variant)
        assert e.value.status == UNSUPPORTED
    with pytest.raises(ffm.FFMError) as e:
        ffm.Plan(X, Y, ffm.LAPLACE_GRAD, 0.0, 1e-1, n_leaf=4)
    assert e.value.status == UNSUPPORTED
    with ffm.Plan(X, Y, ffm.LAPLACE, 0.0, 1e-3, n_leaf=4) as p:
        info = p.info()
        assert info["l_stop"] == 8 and info["tune_tc"][8] == 2
        sigma8 = (info["oX"][0] - info["oY"][0]) / info["d0"] * 256
        near, adm = _counts(sigma8)
        assert adm > 2 ** 32 and info["n_adm"][8] == adm and info["n_near"][8] == near
        v = p.apply(u)
        assert p.info()["device_errors"] == 0
        with pytest.raises(ffm.FFMError) as e:
            p.pairs(8, "adm")
        assert e.value.status == UNSUPPORTED
    t = torch.randint(0, N ** 3, (32,), generator=torch.Generator().manual_seed(2)).cuda()
    ref = torch.stack([(u.double() / (4.0 * np.pi * (X[i] - Y).norm(dim=1))).sum() for i in t])
    assert float((v[t].double() - ref).norm() / ref.norm()) < 1e-3
