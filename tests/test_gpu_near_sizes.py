"""The Laplace near field alone (one leaf, no far field) at the edges of its thread groups, target
chunks and source batches, against the FP64 direct sum.

Tolerance: a term is off by at most a few FP32 roundings (2e-7), and a target's sum of up to 4100 positive
terms runs in FP32 partial sums of at most 4100 terms (about sqrt(4100) 2^-24 = 3.8e-6 at worst): 5e-6 in
the 2-norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [1, 3, 1023, 1024, 1025, 4100])
@pytest.mark.parametrize("nx", [1, 4, 5, 33, 64, 65, 127, 128, 129, 300])
def test_one_leaf(nx, ny):
    X, Y = W.cube_volume(nx, 1), W.cube_volume(ny, 2)
    u = np.random.default_rng(3).uniform(0.5, 1.0, ny).astype(np.float32)
    t = lambda a: torch.as_tensor(a, device="cuda")
    with ffm.Plan(t(X), t(Y), ffm.LAPLACE, 0.0, 1e-3, n_leaf=1 << 20) as p:
        info = p.info()
        v = p.apply(t(u)).cpu().numpy().astype(np.float64)
    assert info["l_stop"] == 0 and info["p2p_pairs"] == nx * ny
    ref = O.direct(X, Y, u.astype(np.float64), O.LAPLACE)[:, 0].real
    assert O.rel_l2(v, ref) < 5e-6
