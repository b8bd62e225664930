"""k_gemm_x3, the split product of the frame merge and the optimizer step, on
its own: both tile widths at odd and even multiples of 128 columns (an odd one
leaves the second half of a 256-wide tile out of range), contractions of one
stage, of fewer stages than the ring holds and of many, the second product of
the same launch, and the epilogue that adds to a base.

Operands hi + lo with hi multiples of 1/8 up to 1 and lo multiples of 2^-17
below 2^-14: the hi hi products sum exactly in binary32, and so do the two
cross products, so the result is their sum rounded once to binary32."""
import numpy as np
import pytest
import torch

import paper_2607_19331_gb300 as iso

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _operand(rows, kc, seed):
    g = torch.Generator().manual_seed(seed)
    hi = torch.randint(-8, 9, (rows, kc), generator=g).float() / 8
    lo = torch.randint(-7, 8, (rows, kc), generator=g).float() * 2.0 ** -17
    return hi.double().numpy(), lo.double().numpy(), torch.cat([hi, lo], 1).contiguous().to(DEV)


def _product(a, b):
    hh = a[0] @ b[0].T
    cross = a[0] @ b[1].T + a[1] @ b[0].T
    return (hh.astype(np.float32) + cross.astype(np.float32)).astype(np.float32)


SHAPES = [(128, 128, 32), (256, 384, 64), (384, 128, 96), (128, 256, 160), (256, 640, 1056), (128, 1152, 32)]


@pytest.mark.parametrize("M,N,Kc", SHAPES)
@pytest.mark.parametrize("width", [128, 256, 0])
def test_products(M, N, Kc, width):
    a, b = _operand(M, Kc, 1), _operand(N, Kc, 2)
    C = torch.full((M, N), float("nan"), device=DEV)
    iso.gemm_x3(a[2], b[2], C, width=width)
    torch.cuda.synchronize()
    assert np.array_equal(C.cpu().numpy(), _product(a, b))


@pytest.mark.parametrize("M,N,Kc", SHAPES[:4])
@pytest.mark.parametrize("width", [128, 256])
def test_two_products_in_one_launch(M, N, Kc, width):
    a, b, a2, b2 = (_operand(r, Kc, 3 + i) for i, r in enumerate((M, N, M, N)))
    C, C2 = (torch.full((M, N), float("nan"), device=DEV) for _ in range(2))
    iso.gemm_x3(a[2], b[2], C, a2[2], b2[2], C2, width=width)
    torch.cuda.synchronize()
    assert np.array_equal(C.cpu().numpy(), _product(a, b))
    assert np.array_equal(C2.cpu().numpy(), _product(a2, b2))


# outputs that end inside a tile, inside the 256-wide tile's second half and at its edges
@pytest.mark.parametrize("m,n", [(1, 1), (128, 128), (129, 257), (200, 383), (256, 384), (255, 300)])
@pytest.mark.parametrize("width", [128, 256])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_product_added_to_a_base(m, n, width, dtype):
    M, N, Kc = (m + 127) // 128 * 128, (n + 127) // 128 * 128, 64
    a, b = _operand(M, Kc, 7), _operand(N, Kc, 8)
    W0 = torch.randn(m, n, generator=torch.Generator().manual_seed(9)).to(dtype).to(DEV)
    out = torch.full_like(W0, float("nan"))
    iso.gemm_x3(a[2], b[2], W0=W0, out=out, width=width)
    torch.cuda.synchronize()
    want = (W0.float().cpu() + torch.from_numpy(_product(a, b)[:m, :n])).to(dtype)
    assert torch.equal(out.cpu(), want)
