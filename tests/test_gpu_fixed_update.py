"""Gram-Schmidt updates in fixed point (vectors beyond two rows per thread of a full launch):
orthogonality and the reported residual on both sides of the size where they start, basis
counts around the groups of eight, and right-hand sides near the ends of the FP64 range.  An
always re-orthogonalised basis is orthonormal to a few roundings; the residual estimate of the
cycle and the recomputed one agree to the rounding of the product (1e-10 with room)."""
import numpy as np
import pytest
import torch

from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(270, 285), (288, 271), (512, 301)])
@pytest.mark.parametrize("m", [1, 2, 9, 17, 33])
def test_basis_and_residual(n1, n2, m):
    rng = np.random.default_rng(n1 + m)
    op = die.Operator(W.random_field(rng, n1, n2, lo=1.0, hi=4.0), 1.0 / 60.0)
    b = torch.from_numpy(W.random_vector(rng, n1, n2)).cuda()
    x, rep = op.solve(b, restart=m, tol=0.0, max_iters=m, reorth_eta=1.0, history=m)
    r = torch.linalg.norm(op.apply(x) - b) / torch.linalg.norm(b)
    assert abs(float(r) - rep["rel_res_solved"]) <= 1e-10
    assert abs(rep["history"][-1] - rep["rel_res_solved"]) <= 1e-10
    if m > 2:
        V = op.basis(1, m - 1).reshape(m - 1, -1)
        G = (V.conj() @ V.T).cpu().numpy()
        assert np.abs(G - np.eye(m - 1)).max() < 1e-13


@pytest.mark.parametrize("s", [1e-140, 1e140])
def test_range(s):
    rng = np.random.default_rng(3)
    op = die.Operator(W.random_field(rng, 300, 290, lo=1.0, hi=4.0), 1.0 / 60.0)
    b = torch.from_numpy(W.random_vector(rng, 300, 290)).cuda()
    x, rep = op.solve(b, restart=12, tol=0.0, max_iters=12)
    # the solve is homogeneous in b, as long as the square of its norm is in range
    y, rs = op.solve(b * s, restart=12, tol=0.0, max_iters=12)
    assert abs(rs["rel_res_solved"] - rep["rel_res_solved"]) <= 1e-10
    assert float(torch.linalg.norm(y / s - x) / torch.linalg.norm(x)) <= 1e-9
