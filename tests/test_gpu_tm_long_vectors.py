"""TM solves whose Gram-Schmidt sweeps run in fixed point (vectors beyond two rows per thread of a
full launch): a TM vector's second plane is zero and stays exactly zero through products, sweeps
and deflation, in the solution and in every basis vector.  Sizes on both sides of the boundaries
of the projections' rows per thread and of one chunk per block, plain, FP32-inner and deflated.
The reported residual and the one recomputed from the solution agree to the product's rounding."""
import numpy as np
import pytest
import torch

from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,inner,r", [(300, 270, die.DIE_FP64, 0), (290, 281, die.DIE_FP32_INNER, 0),
                                           (401, 389, die.DIE_FP64, 0), (523, 522, die.DIE_FP64, 0),
                                           (300, 280, die.DIE_FP32_INNER, 2)])
def test_second_plane_stays_zero(n1, n2, inner, r):
    rng = np.random.default_rng(n1)
    eps = np.full((n2, n1), 1.0 + 0j)
    eps[n2 // 4:3 * n2 // 4, n1 // 4:3 * n1 // 4] = 1.5 + 0.2j * rng.random((3 * n2 // 4 - n2 // 4, 3 * n1 // 4 - n1 // 4))
    op = die.Operator(eps, 1.0 / 60.0, pol=die.DIE_TM)
    b = op.plane_wave(0.4)
    D = die.Deflation(op, r, regularized=True, inner=inner) if r else None
    m = 11
    x, rep = op.solve(b, restart=m, tol=0.0, max_iters=2 * m, inner=inner, regularized=bool(r), deflation=D)
    assert bool((x[1] == 0).all())
    V = op.basis(0, m - 1)
    assert bool((V[:, 1] == 0).all()) and bool((V[:, 0] != 0).any())
    res = float(torch.linalg.norm(op.apply(x) - b) / torch.linalg.norm(b))
    assert abs(res - rep["rel_res_orig"]) <= 1e-10 and res < 0.1
