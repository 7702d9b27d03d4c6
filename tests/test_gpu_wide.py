"""Transform passes in wide radices (float, double): every radix, one to five stages, both sides of
the field sizes where the radix class changes, ragged blocks, against a library transform in 64 bits.

Bound: a transform of N points errs by at most about eps log2 N per stage chain in relative 2-norm
(Higham, Accuracy and Stability of Numerical Algorithms, ch. 24, with small constants); 4 eps log2 N
is asked."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd

pytestmark = pytest.mark.gpu

SIZES = [(4,), (6,), (250,), (486,), (750,), (972,), (1024,),            # 1D: one line
         (4, 4), (8, 6), (18, 10), (60, 54), (90, 30), (144, 90),        # small fields, radices 2..5
         (540, 810), (512, 500), (1000, 270),                           # about 2^17 points
         (10, 12, 4), (64, 6, 1000), (324, 50, 6), (30, 240, 18),
         (180, 150, 96), (128, 162, 200), (320, 256, 60)]               # about 2^20 and 2^21


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", SIZES)
def test_wide_transforms(n, precision):
    eps, rdt, cdt = ((2.0 ** -53, torch.float64, torch.complex128) if precision == "fp64" else
                     (2.0 ** -24, torch.float32, torch.complex64))
    gen = torch.Generator(device="cuda").manual_seed(31)
    x = torch.randn(tuple(reversed(n)), generator=gen, dtype=torch.float64, device="cuda").to(rdt)
    G = vd.Grid(n, (2 * math.pi,) * len(n))
    bound = 4.0 * eps * math.log2(math.prod(n))
    ref = torch.fft.rfftn(x.double())
    got = G.fft_r2c(x, precision=precision)
    assert (torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)).item() < bound
    h = ref.to(cdt).contiguous()
    back = torch.fft.irfftn(h.to(torch.complex128), s=tuple(reversed(n)))
    got = G.fft_c2r(h, precision=precision)
    assert (torch.linalg.vector_norm(got - back) / torch.linalg.vector_norm(back)).item() < bound
