"""Gram-Schmidt on vectors shorter than a full reduction launch (small blocks, groups of basis
vectors side by side in the grid) and just beyond it: an always re-orthogonalised basis is
orthonormal to a few roundings (1e-13 for 40 vectors), and the reported residual is the true
one."""
import numpy as np
import pytest
import torch

from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(2, 2), (5, 3), (17, 16), (61, 61), (110, 90), (139, 140), (200, 195)])
def test_short_vector_gram_schmidt(n1, n2):
    """One long cycle on vectors that take small blocks and side-by-side groups: the basis is
    orthonormal and the solve's residual is the true one."""
    rng = np.random.default_rng(n1)
    op = die.Operator(W.random_field(rng, n1, n2, lo=1.0, hi=3.0), 1.0 / 60.0)
    b = torch.from_numpy(W.random_vector(rng, n1, n2)).cuda()
    m = min(40, 2 * n1 * n2 - 1)
    x, rep = op.solve(b, restart=m, tol=0.0, max_iters=m, reorth_eta=1.0)
    r = torch.linalg.norm(op.apply(x) - b) / torch.linalg.norm(b)
    assert abs(float(r) - rep["rel_res_solved"]) <= 1e-10
    k = rep["iters"]
    if rep["rel_res_solved"] > 1e-8 and k > 2:      # no breakdown: v_1 .. v_{k-1} are kept
        V = op.basis(1, k - 1).reshape(k - 1, -1)
        G = (V.conj() @ V.T).cpu().numpy()
        assert np.abs(G - np.eye(k - 1)).max() < 1e-13
