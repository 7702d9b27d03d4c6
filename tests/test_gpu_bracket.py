"""The float velocity bracket (density data split into float pairs): one Richardson step of the inner
float operator in 1D, 2D and 3D, on sizes that leave a ragged last block, against the oracle's step.

Bound: the float transforms err by about eps log2 N <= 16 eps each, three deep, and the step length
is a quotient of two such products: 1e-5 (about 170 eps) covers it; a wrong pairing of a second
derivative or a dropped term moves the step by percents at a = 0.3."""

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


@pytest.mark.parametrize("n", [(10,), (300,), (18, 20), (50, 36), (12, 10, 6), (20, 18, 30)])
def test_one_float_step_of_the_velocity_operator(n):
    L = tuple([2 * math.pi, 3.0, 5.0][:len(n)])
    g = sp.Grid(n, L)
    rho = 2.0 + 0.1 * inputs.smooth_random_field(n, L, 41, kmax=2)
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
