"""Arithmetic on the bits of doubles (density quotients, narrowing of the refinement's right-hand side,
Parseval weights): a density or right-hand side scaled by a power of two scales the results by exactly
that power, also at scales far outside the range of floats; quotients stay within 2 ulp."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd
from paper_2403_06654_gb300 import inputs

pytestmark = pytest.mark.gpu

N, L = (30, 18, 20), (2 * math.pi, 3.0, 4.0)


def fields():
    rho = torch.from_numpy(inputs.slab_density(N, L, 7.0, 1, 1.0, 1.5, 0.6)).cuda()
    f = torch.from_numpy(inputs.smooth_random_field(N, L, 51, kmax=4)).cuda()
    return rho, f


@pytest.mark.parametrize("k", [-900, -300, -130, -1, 1, 126, 300, 900])
def test_density_scale(k):
    rho, f = fields()
    G = vd.Grid(N, L)
    G.set_density(rho)
    ref = G.apply("pressure", f)
    G.set_density(rho * 2.0 ** k)
    got = G.apply("pressure", f)
    # (2^-k may itself leave the doubles: scale in two steps)
    assert torch.equal(got * 2.0 ** (k // 2) * 2.0 ** (k - k // 2), ref)


@pytest.mark.parametrize("c", [1.0, 3.0, 0.1, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1e-200, 7e150])
def test_density_quotient(c):
    """A constant density divides every coefficient by the same c: each stored quotient is within 2 ulp
    of its value, so the applies agree to that and the transforms' rounding (64 eps in 2-norm)."""
    _, f = fields()
    G = vd.Grid(N, L)
    G.set_density(torch.ones_like(f))
    ref = G.apply("pressure", f)
    G.set_density(torch.full_like(f, c))
    got = G.apply("pressure", f) * c
    assert (torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)).item() < 64 * 2.0 ** -53


@pytest.mark.parametrize("solver", ["cg", "gmres", "rmr"])
@pytest.mark.parametrize("k", [-60, 1, 60])
def test_rhs_scale(k, solver):
    # (precision "mixed": the float-pair transforms of "mixed_dd" hold their fields in floats, whose
    # low parts underflow for fields near 2^-60)
    precision = "mixed"
    rho, f = fields()
    G = vd.Grid(N, L)
    G.set_density(rho)
    ref, i0 = G.solve("pressure", solver, f, tol=1e-9, max_it=300, precision=precision)
    got, i1 = G.solve("pressure", solver, f * 2.0 ** k, tol=1e-9, max_it=300, precision=precision)
    assert i0["status"] == i1["status"] == "converged" and i0["iters"] == i1["iters"]
    assert torch.equal(got * 2.0 ** -k, ref)


def test_rhs_scale_beyond_floats():
    rho, f = fields()
    G = vd.Grid(N, L)
    G.set_density(rho)
    ref, i0 = G.solve("pressure", "cg", f, tol=1e-9, max_it=300, precision="mixed")
    for k in (-400, 400):
        got, i1 = G.solve("pressure", "cg", f * 2.0 ** k, tol=1e-9, max_it=300, precision="mixed")
        assert i0["iters"] == i1["iters"] and torch.equal(got * 2.0 ** -k, ref)
