"""GMRES orthogonalisation kernels at the edges of their vector counts (2, 4, 8, 16 and 32 basis
vectors per kernel, and the separate dots and updates beyond 32): the iterate after k steps of one
cycle against the oracle's, within the parity bound of equal iterates (1e-10)."""

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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 40])
def test_gmres_iterates_at_vector_counts(k):
    n, L = (40, 36), (2 * math.pi, 2 * math.pi)
    g = sp.Grid(n, L)
    # a density ratio of 200 keeps the residual far above rounding for 40 steps
    rho = inputs.slab_density(n, L, 200.0, 1, 2.0, math.pi, 3 * L[1] / n[1])
    f = sp.project_range(inputs.random_field(g.shape, 21), g)
    A, M = op.pressure_system(rho, g)
    ref = sv.solve("gmres", A, M, f, tol=0.0, maxit=k, restart=64)
    G = vd.Grid(n, L)
    G.set_density(torch.from_numpy(rho).cuda())
    x, info = G.solve("pressure", "gmres", torch.from_numpy(f).cuda(), tol=0.0, max_it=k, restart=64)
    assert info["iters"] == k and info["status"] == "max_iter"
    assert np.linalg.norm(x.cpu().numpy() - ref.x) / np.linalg.norm(ref.x) < 1e-10
