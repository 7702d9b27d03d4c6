"""The stored coefficients 1/(N rho) against the division of the same doubles, element by element: random
significands at scale one and over the whole range of exponents, neighbours of powers of two, quotients
and densities that leave the normal doubles.

Bound: the quotient is formed from a float-pair reciprocal (relative error 2^-47) and corrected by its own
residual, so before its last rounding it errs by 2^-94, 2^-41 of the spacing of doubles: it is the
correctly rounded quotient unless that lies this close to a rounding boundary, one in 2^40 of random
values.  Equality is asked of these 2^21."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd

pytestmark = pytest.mark.gpu


def _densities(kind, count, gen):
    m = 1.0 + torch.randint(0, 2 ** 52, (count,), generator=gen, device="cuda").double() * 2.0 ** -52
    if kind == "unit":
        return m
    if kind == "edges":   # 1 +- k ulp, k small
        k = torch.randint(-64, 65, (count,), generator=gen, device="cuda")
        one = torch.full((count,), 1.0, dtype=torch.float64, device="cuda").view(torch.int64)
        return (one + k).view(torch.float64)
    low, high = (-1074, 1023) if kind == "range" else (1000, 1023)
    e = torch.randint(low, high + 1, (count,), generator=gen, device="cuda")
    half = torch.div(e, 2, rounding_mode="floor")
    return m * torch.exp2(half.double()) * torch.exp2((e - half).double())


@pytest.mark.parametrize("kind", ["unit", "edges", "range", "largest"])
@pytest.mark.parametrize("n", [(128, 128, 128), (250, 90, 96)])
def test_quotients(n, kind):
    gen = torch.Generator(device="cuda").manual_seed(97)
    count = math.prod(n)
    rho = _densities(kind, count, gen)
    rho = torch.where(torch.isfinite(rho) & (rho > 0), rho, torch.ones_like(rho))
    G = vd.Grid(n, (2 * math.pi,) * 3)
    G.set_density(rho.reshape(tuple(reversed(n))))
    at = -(-8 * count // 256) * 256   # the copy of rho first, then 1/(N rho)
    got = G._dens[at:at + 8 * count].view(torch.float64)
    # (the scalar division on the host is IEEE; the device's division too)
    ref = torch.full_like(rho, 1.0 / count) / rho
    assert torch.equal(got, ref)
