"""Recorded GMRES cycles run in groups of steps: restarts that end inside, at and past group boundaries,
cycles that converge at once and budgets that end a cycle early give the host-driven solve's iterations
and, within the recorded solves' bound (1e-13), its solution."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd
from paper_2403_06654_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed_dd"])
@pytest.mark.parametrize("restart,max_it", [(1, 40), (3, 200), (4, 200), (5, 200), (17, 200), (40, 200), (64, 6)])
def test_recorded_gmres_groups(restart, max_it, precision):
    n, L = (24, 20), (2 * math.pi, 2 * math.pi)
    rho = torch.from_numpy(inputs.slab_density(n, L, 9.0, 0, 2.0, math.pi, 3 * L[0] / n[0])).cuda()
    bv = torch.stack([torch.from_numpy(inputs.smooth_random_field(n, L, 61 + c, kmax=4)).cuda() for c in range(2)])
    bp = torch.from_numpy(inputs.smooth_random_field(n, L, 63, kmax=4)).cuda()
    item = {"n": n, "L": L, "rho": rho, "a": 5e-2, "inv_sc": 1.0, "b_vel": bv, "x_vel": torch.zeros_like(bv),
            "b_pres": bp, "x_pres": torch.zeros_like(bp)}
    B = vd.Batch([item], vel_solver="gmres", pres_solver="gmres", tol=1e-9, max_it=max_it, restart=restart,
                 precision=precision)
    B.run()
    iv, ip = B.info(0)
    G = vd.Grid(n, L)
    G.set_density(rho, "velocity")
    kw = {"tol": 1e-9, "max_it": max_it, "restart": restart, "precision": precision}
    xv, jv = G.solve("velocity", "gmres", bv, a=5e-2, inv_sc=1.0, **kw)
    xp, jp = G.solve("pressure", "gmres", bp, **kw)
    for got, ref, i, j in ((item["x_vel"], xv, iv, jv), (item["x_pres"], xp, ip, jp)):
        assert i["iters"] == j["iters"] and i["status"] == j["status"]
        assert (torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)).item() < 1e-13
