"""Fixed-point projections at every number of rows per thread (three to seven), with one, two and more
chunks per block and groups of rows of the grid, and the folded deflated updates beyond one chunk: an
always re-orthogonalised basis is orthonormal to a few roundings, and the residual estimate of the
cycle and the recomputed one agree to the rounding of the product (1e-10 with room)."""
import numpy as np
import pytest
import torch

from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,m", [(250, 240, 72), (279, 279, 9), (300, 291, 18), (342, 342, 10), (397, 396, 9),
                                     (430, 429, 10), (461, 460, 17), (501, 499, 9), (523, 521, 10), (560, 559, 9),
                                     (601, 600, 10), (702, 700, 9), (1024, 901, 10)])
def test_basis_and_residual(n1, n2, m):
    rng = np.random.default_rng(n1 + m)
    op = die.Operator(W.random_field(rng, n1, n2, lo=1.0, hi=4.0), 1.0 / 60.0)
    b = torch.from_numpy(W.random_vector(rng, n1, n2)).cuda()
    x, rep = op.solve(b, restart=m, tol=0.0, max_iters=m, reorth_eta=1.0, history=m)
    r = torch.linalg.norm(op.apply(x) - b) / torch.linalg.norm(b)
    assert abs(float(r) - rep["rel_res_solved"]) <= 1e-10
    assert abs(rep["history"][-1] - rep["rel_res_solved"]) <= 1e-10
    V = op.basis(1, m - 1).reshape(m - 1, -1)
    G = (V.conj() @ V.T).cpu().numpy()
    assert np.abs(G - np.eye(m - 1)).max() < 1e-13


@pytest.mark.parametrize("n1,n2,r", [(430, 429, 2), (640, 560, 9)])
def test_folded_deflation(n1, n2, r):
    """Deflated FP32-inner cycles (the projections onto the deflation basis inside the update): the
    cycle's estimate follows the products in complex64, 1e-5 of the start."""
    p = W.config1(max(n1, n2))
    eps = np.ascontiguousarray(p.eps_r[:n2, :n1])
    op = die.Operator(eps, p.h)
    D = die.Deflation(op, r, regularized=True, inner=die.DIE_FP32_INNER)
    b = op.plane_wave(0.3)
    m = 10
    x, rep = op.solve(b, restart=m, tol=0.0, max_iters=m, regularized=True, inner=die.DIE_FP32_INNER, deflation=D,
                      reorth_eta=1.0, history=m)
    res = torch.linalg.norm(op.apply(x) - b) / torch.linalg.norm(b)
    assert abs(float(res) - rep["rel_res_orig"]) <= 1e-10
    assert abs(rep["history"][-1] - rep["rel_res_solved"]) <= 1e-5
    V = op.basis(1, m - 1).reshape(m - 1, -1)
    G = (V.conj() @ V.T).cpu().numpy()
    assert np.abs(G - np.eye(m - 1)).max() < 1e-13
