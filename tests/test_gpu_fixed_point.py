"""FP64 products on the fixed-point transforms, against the FFT oracle: every transform
length (2^a and 3 * 2^a), grids that fill half a transform and ragged ones, the three-plane
system, batches, and values at the ends of the FP64 range.

Tolerance: the products' rounding (some 2^-53 per pass, 1e-14 with room) plus the error of
CUDA's Bessel functions in the Green table, documented as 5e-12 absolute beyond |x| = 8; the
oracle takes its table from scipy."""
import math

import numpy as np
import pytest
import torch

from oracle import fftmv, te_mag
from paper_1104_4263_gb300 import die, workloads as W

pytestmark = pytest.mark.gpu
H = 1.0 / 60.0


def _tol(n1, n2):
    return 1e-14 if 2 * math.pi * H * math.hypot(n1, n2) < 8 else 2e-11


def _err(y, ref):
    return np.linalg.norm(y - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("n1,n2", [(2, 2), (8, 8), (9, 12), (16, 13), (17, 24), (32, 31), (33, 48), (64, 57), (65, 128),
                                   (97, 192), (129, 256), (200, 384), (257, 512), (768, 391), (1024, 36), (40, 1536),
                                   (2048, 20)])
@pytest.mark.parametrize("reg", [False, True])
def test_product_every_length(n1, n2, reg):
    rng = np.random.default_rng(n1 * 4099 + n2)
    eps = W.random_field(rng, n1, n2)
    x = W.random_vector(rng, n1, n2)
    ref = fftmv.FFTOperator(eps, H)
    op = die.Operator(eps, H)
    xt = torch.from_numpy(x).cuda()
    y = (op.apply_regularized(xt) if reg else op.apply(xt)).cpu().numpy()
    assert _err(y, ref.apply_regularized(x) if reg else ref.apply(x)) < _tol(n1, n2)


@pytest.mark.parametrize("n1,n2", [(7, 12), (12, 20)])
def test_three_planes(n1, n2):
    rng = np.random.default_rng(n1)
    eps, mu = W.random_field(rng, n1, n2), 1.0 + 0.5 * W.random_field(rng, n1, n2)
    A, AR = te_mag.dense_A(eps, mu, H), te_mag.dense_AR(eps, mu, H)
    op = die.Operator(eps, H, pol=die.DIE_TE_MAG, mu_r=mu)
    x = rng.standard_normal((3, n2, n1)) + 1j * rng.standard_normal((3, n2, n1))
    y = op.apply_regularized(torch.from_numpy(x).cuda()).cpu().numpy()
    assert _err(y.reshape(-1), AR @ (A @ x.reshape(-1))) < 1e-14


@pytest.mark.parametrize("scale", [1e-300, 1e-250, 1e-30, 1e30, 1e250, 1e290])
def test_range(scale):
    """Magnitudes near the ends of the FP64 range: the products are homogeneous."""
    rng = np.random.default_rng(5)
    n1, n2 = 30, 23
    eps = W.random_field(rng, n1, n2)
    x = W.random_vector(rng, n1, n2)
    op = die.Operator(eps, H)
    y = op.apply(torch.from_numpy(x * scale).cuda()).cpu().numpy()
    ref = fftmv.FFTOperator(eps, H).apply(x * scale / scale)
    assert _err(y / scale, ref) < 1e-14


def test_rows_of_very_different_size_zero_and_not_finite():
    rng = np.random.default_rng(6)
    n1, n2 = 40, 35
    eps = W.random_field(rng, n1, n2)
    ref, op = fftmv.FFTOperator(eps, H), die.Operator(eps, H)
    x = W.random_vector(rng, n1, n2)
    x[0] *= 10.0 ** rng.uniform(-12, 0, size=(n2, 1))
    x[1, 3:9] = 0.0
    xt = torch.from_numpy(x).cuda()
    assert _err(op.apply(xt).cpu().numpy(), ref.apply(x)) < 1e-14
    assert not op.apply(torch.zeros_like(xt)).any()
    for bad in (math.nan, math.inf):
        xt[1, 20, 7] = bad
        y = op.apply(xt)
        assert not bool(torch.isfinite(torch.view_as_real(y)).any())


def test_batch_equals_single_and_in_place():
    rng = np.random.default_rng(7)
    n1, n2 = 45, 61
    op = die.Operator(W.random_field(rng, n1, n2), H)
    x = torch.from_numpy(np.stack([W.random_vector(rng, n1, n2) * 10.0 ** k for k in (0, -9, 7)])).cuda()
    for reg in (False, True):
        one = torch.stack([(op.apply_regularized(v) if reg else op.apply(v)) for v in x])
        assert torch.equal(op.apply_batch(x, regularized=reg), one)
        y = x.clone()
        assert torch.equal(op.apply_batch(y, y, regularized=reg), one)
