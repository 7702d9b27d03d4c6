"""Narrowing of the refinement's right-hand side to float: coefficients far below the largest one keep
their float value, subnormal ones included.

On four points f = c cos x + e sin x has the spectrum (2 c, -2 e) exactly, and so has every quantity of a
constant-density solve (-f to float accuracy): the small part never meets the large one.  Bound: a float of
exponent x has spacing max(2^(x - 23), 2^-149); the narrowing, two operator applies of about ten
roundings each and the CG update stay below 64 spacings of the normalised part, e / (sqrt(2) c)."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", [-20, -60, -73, -75, -100, -126, -130, -138])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 40 * 1.3, 2.0 ** -200 * 1.7])
@pytest.mark.parametrize("solver", ["cg", "rmr", "gmres"])
def test_small_coefficients(solver, scale, small):
    e = 1.3 * 2.0 ** small
    f = torch.tensor([1.0, e, -1.0, -e], dtype=torch.float64, device="cuda") * scale
    G = vd.Grid((4,), (2 * math.pi,))
    G.set_density(torch.ones(4, dtype=torch.float64, device="cuda"))
    x, info = G.solve("pressure", solver, f, tol=1e-5, max_it=5, precision="mixed")
    assert info["status"] == "converged"
    got = (x / scale).tolist()
    spacing = max(2.0 ** (small - 23), 2.0 ** -149)
    assert abs(got[1] + e) <= 64 * spacing and abs(got[3] - e) <= 64 * spacing
    assert abs(got[0] + 1.0) <= 64 * 2.0 ** -24 and abs(got[2] - 1.0) <= 64 * 2.0 ** -24
