"""An accuracy that needs more than eight Chebyshev nodes per axis is refused with a status wherever a level
would use them, whichever transfer is asked for, and before anything is sized by the node count; a plan
without such a level takes any accuracy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu
UNSUPPORTED = 5


@pytest.mark.parametrize("variant", [ffm.LAG_DEFAULT, ffm.LAG_CUDA_CORES, ffm.LAG_TC_TRANSLATION, ffm.LAG_TC_TARGET])
@pytest.mark.parametrize("kernel,eps", [(ffm.LAPLACE, 2.3e-7), (ffm.LAPLACE, 1e-9), (ffm.HELMHOLTZ, 1e-8),
                                        (ffm.LAPLACE_DL, 3e-6), (ffm.LAPLACE_DL, 1e-9), (ffm.LAPLACE_GRAD, 1e-8)])
def test_too_many_nodes(kernel, eps, variant):
    X = torch.as_tensor(W.cube_volume(2000, 1), device="cuda")
    kw = dict(lagrange_transfer=variant, normals=X if kernel == ffm.LAPLACE_DL else None, kappa_switch=1e9)
    with pytest.raises(ffm.FFMError) as e:
        ffm.Plan(X, X, kernel, 1.0 if kernel == ffm.HELMHOLTZ else 0.0, eps, n_leaf=16, **kw)
    assert e.value.status == UNSUPPORTED
    with ffm.Plan(X, X, kernel, 1.0 if kernel == ffm.HELMHOLTZ else 0.0, eps, n_leaf=1 << 20, **kw) as p:
        assert not any(p.info()["n_adm"])
