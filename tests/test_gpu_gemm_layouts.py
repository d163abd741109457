"""The tensor-core GEMM over operand layouts and tile edges: k or the row index of unit
stride, neither, rows that are not 16-byte aligned, batches against one shared operand (run
as one tall matrix), and the row counts on both sides of the tile variants.

The operands are rounded to BF16 on the way in, so the reference is the FP64 product of the
rounded operands; what remains is FP32 accumulation, at most K roundings of 2^-23 relative to
the sum of magnitudes."""
import pytest
import torch

from paper_1104_4263_gb300 import die

pytestmark = pytest.mark.gpu


def _operand(rows, K, layout, batch, g):
    """(batch, rows, K) float32 with the strides of a layout."""
    if layout == "k":
        x = torch.randn((batch, rows, K + (-K) % 4), generator=g, device="cuda")[:, :, :K]
    elif layout == "r":
        x = torch.randn((batch, K, rows + (-rows) % 4), generator=g, device="cuda")[:, :, :rows].transpose(1, 2)
    elif layout == "odd":         # unit stride, rows one float off the 16-byte boundaries
        x = torch.randn((batch, rows, K + 1 + K % 2), generator=g, device="cuda")[:, :, 1:K + 1]
    else:
        x = torch.randn((batch, rows, 2 * K), generator=g, device="cuda")[:, :, ::2]
    return x


def _check(C, A, B, alpha=1.0, beta=0.0, C0=None):
    a, b = A.bfloat16().double(), B.bfloat16().double()
    ref = alpha * (a @ b.transpose(-1, -2))
    mag = abs(alpha) * (a.abs() @ b.abs().transpose(-1, -2))
    if beta:
        ref, mag = ref + beta * C0.double(), mag + abs(beta) * C0.double().abs()
    K = A.shape[-1]
    assert bool(((C.double() - ref).abs() <= (K + 4) * 2.0 ** -23 * mag + 1e-30).all())


@pytest.mark.parametrize("la", ["k", "r", "odd", "strided"])
@pytest.mark.parametrize("lb", ["k", "r", "odd", "strided"])
def test_layouts(la, lb):
    g = torch.Generator(device="cuda").manual_seed(1)
    for M, N, K, batch in ((1, 1, 1, 1), (32, 32, 64, 3), (33, 31, 65, 2), (129, 64, 100, 2), (32, 33, 300, 2),
                           (7, 128, 17, 5), (300, 130, 33, 1)):
        A, B = _operand(M, K, la, batch, g), _operand(N, K, lb, batch, g)
        C0 = torch.randn((batch, M, N), generator=g, device="cuda")
        C = C0.clone()
        die.gemm_bf16(A, B, C, alpha=0.5, beta=-2.0)
        _check(C, A, B, 0.5, -2.0, C0)


@pytest.mark.parametrize("M", [1, 16, 48, 128, 200])
def test_batch_against_one_operand(M):
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn((37, M, 72), generator=g, device="cuda")
    B = torch.randn((1, 40, 72), generator=g, device="cuda").expand(37, 40, 72)
    for C in (torch.empty((37, M, 40), device="cuda"), torch.empty((37, 40, M), device="cuda").transpose(1, 2)):
        die.gemm_bf16(A, B, C)
        _check(C, A, B)


def test_long_k_and_many_tiles():
    g = torch.Generator(device="cuda").manual_seed(9)
    for M, N, K, batch in ((32, 32, 5000, 4), (4, 128, 3001, 3), (128, 32, 2049, 2), (5000, 96, 40, 3)):
        A, B = _operand(M, K, "k", batch, g), _operand(N, K, "k", batch, g)
        _check(die.gemm_bf16(A, B), A, B)
