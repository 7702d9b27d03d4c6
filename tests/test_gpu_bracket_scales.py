"""The float velocity bracket at density scales inside and far outside the range of floats: one Richardson
step of the inner float operator against the oracle's step.  With inv_sc fixed the density-gradient
terms do not change with the scale of the density, so they have to survive any of them.

Bound: as for the step at scale one, the float transforms err by about eps log2 N <= 16 eps each, three
deep, and the step length is a quotient of two such products: 1e-5 (about 170 eps)."""

import math

import numpy as np
import pytest
import torch

import paper_2403_06654_gb300 as vd
from paper_2403_06654_gb300 import inputs
from oracle import operators as op
from oracle import solvers as sv
from oracle import spectral as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [-62, -50, 60, 84, 110, 130, 400])
@pytest.mark.parametrize("n", [(300,), (18, 20), (12, 10, 6)])
def test_one_float_step_at_density_scale(n, k):
    L = tuple([2 * math.pi, 3.0, 5.0][:len(n)])
    g = sp.Grid(n, L)
    rho = (2.0 + 0.1 * inputs.smooth_random_field(n, L, 41, kmax=2)) * 2.0 ** k
    b = np.stack([inputs.smooth_random_field(n, L, 42 + c, kmax=2) for c in range(len(n))])
    a, isc = 0.3, 0.7
    A, M = op.velocity_system(rho, g, a, isc)
    ref = sv.solve("rmr", A, M, b, tol=0.0, maxit=1)
    G = vd.Grid(n, L)
    G.set_density(torch.from_numpy(rho).cuda(), "velocity")
    x, info = G.solve("velocity", "rmr", torch.from_numpy(b).cuda(), a=a, inv_sc=isc, tol=0.0, max_it=1,
                      precision="mixed")
    assert info["iters"] == 1
    assert np.linalg.norm(x.cpu().numpy() - ref.x) / np.linalg.norm(ref.x) < 1e-5
