"""The Lagrange basis, the operators and the matrices between the levels belong to the same (rounded) nodes: a constant
density, for which every error of the basis has one sign, keeps the oracle's far field.

The product's error along the exact result: the basis constants' own rounding leaves at most 2.8e-8 per axis (r1 = 8)
on six axes, 1.7e-7; the FP32 sums of equal terms add about as much as half a rounding, 1e-7.  Constants of the exact
nodes beside rounded ones gave 6.0e-7 at r1 = 4 and 5.0e-7 at 6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r1,n", [(3, 20000), (4, 20000), (5, 20000), (6, 20000), (8, 8000)])
def test_a_constant_density_keeps_its_far_field(r1, n):
    X, Y, w = W.cube_volume(n, 1), W.cube_volume(n - 7, 2), np.full(n - 7, 1.0 / n)
    u = np.ones(n - 7, np.float32)
    t = lambda a: torch.as_tensor(a, device="cuda")
    ref = O.ffm(X, Y, u.astype(np.float64), O.LAPLACE, 0.0, 1e-3, w=w, r1_override=r1)[:, 0].real
    with ffm.Plan(t(X), t(Y), ffm.LAPLACE, 0.0, 1e-3, weights=t(w), r1_override=r1,
                  lagrange_transfer=ffm.LAG_CUDA_CORES) as p:
        v = p.apply(t(u)).cpu().numpy().astype(np.float64)
    assert abs(np.vdot(ref, v - ref) / np.vdot(ref, ref)) < 2.7e-7
