"""Single-launch 1D solves over the lengths their transforms treat differently: radix 2 only, with 3
and 5, one element per thread and several, the shortest and the longest.  Iterates after two
iterations agree with the oracle's within the parity bound (1e-10)."""

import math

import numpy as np
import pytest
import torch

import paper_2403_06654_gb300 as vd
from oracle import operators as op
from oracle import solvers as sv
from oracle import spectral as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 6, 8, 10, 18, 30, 64, 90, 256, 250, 486, 512, 750, 972, 1000, 1024])
@pytest.mark.parametrize("solver", ["cg", "gmres", "rmr"])
def test_two_iterations(solver, n):
    L = (3.0,)
    g = sp.Grid((n,), L)
    x = L[0] * np.arange(n) / n
    rho = 2.0 + np.cos(2 * math.pi * x / L[0])
    f = np.cos(2 * math.pi * x / L[0] + 0.3) + (0.2 * np.sin(4 * math.pi * x / L[0]) if n > 6 else 0.0)
    A, M = op.pressure_system(rho, g)
    ref = sv.solve(solver, A, M, sp.project_range(f, g), tol=1e-9, maxit=2, restart=20)
    G = vd.Grid((n,), L)
    G.set_density(torch.from_numpy(rho).cuda())
    got, info = G.solve("pressure", solver, torch.from_numpy(f).cuda(), tol=1e-9, max_it=2, restart=20)
    assert info["iters"] == ref.iters
    assert np.linalg.norm(got.cpu().numpy() - ref.x) / np.linalg.norm(ref.x) < 1e-10
