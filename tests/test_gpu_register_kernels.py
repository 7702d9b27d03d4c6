"""The float register kernels (four-step transforms held in registers) forced through the launch table on small
grids, where the built-in choice is the general kernel: x passes of 128, 256 and 512 points in their
three forms, y and z passes of 128 and 256, each with its TMA-staged variant where there is one.

Transforms are compared with a library transform in 64 bits; bound 4 eps log2 N, as for the general kernels.
The fused x pass and the operator programs of y and z passes run inside mixed-precision solves at a
density ratio below and above the one from which the coefficient is a float pair: refinement in double
converges only if the inner float operator is the operator to float accuracy.  At half the accuracy a
sweep gains less than half of its digits, so twice the general kernels' iterations bound a sound one."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd
from paper_2403_06654_gb300 import inputs

pytestmark = pytest.mark.gpu

REGISTER, STAGED = 0, 128
X_GRIDS = [(128, 20, 10), (256, 18, 6), (512, 10, 4), (128, 30), (512, 6)]
YZ_GRIDS = [(20, 128, 6), (18, 256, 4), (20, 6, 128), (24, 10, 256), (30, 256), (18, 128, 128)]


def _keys(n):
    """(kind, length, axis, direction or form) of the passes of n that have a register kernel"""
    keys = []
    if n[0] in (128, 256, 512):
        keys += [(1, n[0] // 2, 0, mode) for mode in (0, 1, 2)]
    for axis in range(1, len(n)):
        if n[axis] in (128, 256):
            keys += [(0, n[axis], axis, d) for d in (-1, 1)]
    return keys


@pytest.fixture
def force():
    done = []

    def set_all(n, choice):
        for kind, length, axis, d in _keys(n):
            c = REGISTER if kind == 1 and d != 0 else choice   # (the fused form alone has a staged variant)
            vd.vd_autotune_set(kind, 1, length, axis, d, c)
            done.append((kind, 1, length, axis, d))

    yield set_all
    for key in done:
        vd.vd_autotune_set(*key, -1)


@pytest.mark.parametrize("choice", [REGISTER, STAGED])
@pytest.mark.parametrize("n", X_GRIDS + YZ_GRIDS)
def test_transforms(n, choice, force):
    gen = torch.Generator(device="cuda").manual_seed(33)
    x = torch.randn(tuple(reversed(n)), generator=gen, dtype=torch.float32, device="cuda")
    G = vd.Grid(n, (2 * math.pi,) * len(n))
    force(n, choice)
    ref = torch.fft.rfftn(x.double())
    bound = 4.0 * 2.0 ** -24 * math.log2(math.prod(n))
    got = G.fft_r2c(x, precision="mixed")
    assert (torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)).item() < bound
    h = ref.to(torch.complex64).contiguous()
    back = torch.fft.irfftn(h.to(torch.complex128), s=tuple(reversed(n)))
    got = G.fft_c2r(h, precision="mixed")
    assert (torch.linalg.vector_norm(got - back) / torch.linalg.vector_norm(back)).item() < bound


@pytest.mark.parametrize("ratio", [3.0, 300.0])
@pytest.mark.parametrize("choice", [REGISTER, STAGED])
@pytest.mark.parametrize("n", X_GRIDS + YZ_GRIDS)
def test_solves(n, choice, ratio, force):
    L = tuple([2 * math.pi, 3.0, 4.0][:len(n)])
    ax = len(n) - 1
    rho = torch.from_numpy(inputs.slab_density(n, L, ratio, ax, 0.4 * L[ax], 0.5 * L[ax], 3 * L[ax] / n[ax])).cuda()
    f = torch.from_numpy(inputs.smooth_random_field(n, L, 35, kmax=3)).cuda()
    G = vd.Grid(n, L)
    G.set_density(rho, "velocity")
    runs = [("pressure", "cg", f, {})]
    if ratio <= 10.0:   # (the velocity coefficient is no float pair, and GMRES(30) stalls at high ratios in double too)
        runs.append(("velocity", "gmres", torch.stack([f] * len(n)), {"a": 0.05, "inv_sc": 1.0}))
    kw = {"tol": 1e-10, "precision": "mixed"}
    general = [G.solve(op, solver, b, max_it=2000, **kw, **p) for op, solver, b, p in runs]
    assert all(i["status"] == "converged" for _, i in general)
    force(n, choice)
    for (op, solver, b, p), (_, ref) in zip(runs, general):
        x, info = G.solve(op, solver, b, max_it=2 * ref["iters"], **kw, **p)
        assert info["status"] == "converged" and info["relres_true"] <= 1.05e-10
