"""FP64 products at scales that a transform's common exponent has to follow: vectors of subnormal
numbers, and TM planes of very different size (the TM operator acts on each plane by itself)."""
import numpy as np
import pytest
import torch

from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(12, 9), (31, 20), (64, 64), (100, 70)])
@pytest.mark.parametrize("k", [1010, 1030, 1050])
def test_subnormal_vectors(n1, n2, k):
    """A x of x = 2^-k x0: every stored intermediate is rounded to multiples of 2^-1074, half a unit
    in each of the four passes' values, which the passes before the last carry on with a factor
    below 16 (a few |chi| times the kernel's norm): 64 units of 2^(k - 1074) of x0."""
    rng = np.random.default_rng(k + n1)
    op = die.Operator(W.random_field(rng, n1, n2, lo=1.0, hi=4.0), 1.0 / 60.0)
    x = torch.from_numpy(W.random_vector(rng, n1, n2)).cuda()
    lo, hi = float(2.0 ** -(k // 2)), float(2.0 ** -(k - k // 2))
    xs = x * lo * hi                                   # rounded to what FP64 holds
    x = xs / hi / lo                                   # exactly those values, scaled back
    for reg in (False, True):
        y = op.apply_regularized(xs) if reg else op.apply(xs)
        ref = op.apply_regularized(x) if reg else op.apply(x)
        err = float((y / hi / lo - ref).abs().max())
        assert err <= 64 * 2.0 ** (k - 1074) + 1e-13 * float(ref.abs().max()), (reg, err)


@pytest.mark.parametrize("n1,n2", [(24, 17), (64, 64), (130, 100), (520, 36)])
@pytest.mark.parametrize("k", [-60, 40, 200])
def test_tm_planes_of_different_size(n1, n2, k):
    rng = np.random.default_rng(n1 + 3)
    op = die.Operator(W.random_field(rng, n1, n2, lo=1.0, hi=4.0), 1.0 / 60.0, pol=die.DIE_TM)
    x = torch.from_numpy(W.random_vector(rng, n1, n2)).cuda()
    xs = torch.stack([x[0], x[1] * 2.0 ** k])
    for reg in (False, True):
        f = op.apply_regularized if reg else op.apply
        y = f(xs)
        for p in (0, 1):
            alone = torch.zeros_like(xs)
            alone[0] = xs[p]
            ref = f(alone)[0]
            assert float(torch.linalg.norm(y[p] - ref) / torch.linalg.norm(ref)) < 1e-14, (p, reg)
