"""Complex64 products with both planes of a column in one thread (column transforms of length 512) and
the tall row tiles of large batches (row transforms of length 256): against the FFT oracle, in the
relative 2-norm at the complex64 tolerance of the other product tests (2e-5), batches equal to single
products bit for bit, a zero TM plane zero, and a value that is not finite everywhere."""
import math

import numpy as np
import pytest
import torch

from oracle import fftmv
from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu
H = 1.0 / 60.0


@pytest.mark.parametrize("n1,n2,nb", [(256, 256, 3), (129, 200, 2), (20, 255, 5), (600, 193, 2), (128, 203, 13),
                                      (128, 128, 32)])
@pytest.mark.parametrize("reg", [False, True])
def test_batch(n1, n2, nb, reg):
    rng = np.random.default_rng(n1 * 7 + n2)
    eps = W.random_field(rng, n1, n2, lo=1.0, hi=4.0)
    op, ref = die.Operator(eps, H, prec=die.DIE_FP32_INNER), fftmv.FFTOperator(eps, H)
    X = torch.from_numpy(np.stack([W.random_vector(rng, n1, n2) for _ in range(nb)])).to(torch.complex64).cuda()
    Y = op.apply_batch(X, regularized=reg)
    f = op.apply_regularized if reg else op.apply
    for k in range(nb):
        assert torch.equal(Y[k], f(X[k].contiguous()))
    x = X[nb - 1].cpu().numpy().astype(np.complex128)
    y = ref.apply_regularized(x) if reg else ref.apply(x)
    assert np.linalg.norm(Y[nb - 1].cpu().numpy() - y) / np.linalg.norm(y) < 2e-5


def test_planes_and_not_finite():
    rng = np.random.default_rng(2)
    n1, n2 = 40, 256
    op = die.Operator(W.random_field(rng, n1, n2, lo=1.0, hi=4.0), H, prec=die.DIE_FP32_INNER, pol=die.DIE_TM)
    x = torch.from_numpy(W.random_vector(rng, n1, n2)).to(torch.complex64).cuda()
    x[1] = 0
    y = op.apply_regularized(x)
    assert bool((y[1] == 0).all()) and bool((y[0] != 0).any())
    x[0, 7, 5] = math.nan
    assert not bool(torch.isfinite(torch.view_as_real(op.apply(x))).any())
