"""Launch-table entries are kept by length; the shared memory of a shape also depends on the field's size.
Every number of lines per block that an entry may ask for gives a transform on a small field too, with the
built-in shape's bits (a shape only distributes whole lines), whether it fits there (it is used) or
not (the built-in shape is)."""

import math

import pytest
import torch

import paper_2403_06654_gb300 as vd

pytestmark = pytest.mark.gpu

TYPES = {"fp64": (0, torch.float64), "mixed": (1, torch.float32), "mixed_dd": (2, torch.float64)}


@pytest.mark.parametrize("precision", sorted(TYPES))
@pytest.mark.parametrize("n", [108, 128, 160, 240, 256, 432, 512, 750, 1000])
def test_any_lines_per_block(n, precision):
    code, rdt = TYPES[precision]
    grids = [(0, (8, n, 6), n, 1, (-1, 1)), (0, (8, 6, n), n, 2, (-1, 1))]
    if 2 * n <= 1024:
        grids.append((1, (2 * n, 6, 4), n, 0, (1, 2)))
    for kind, shape, length, axis, dirs in grids:
        gen = torch.Generator(device="cuda").manual_seed(71)
        x = torch.randn(tuple(reversed(shape)), generator=gen, dtype=torch.float64, device="cuda").to(rdt)
        G = vd.Grid(shape, (2 * math.pi,) * 3)
        ref = G.fft_r2c(x, precision=precision)
        back = G.fft_c2r(ref, precision=precision)
        try:
            for lines in (1, 2, 4, 8, 16, 32, 64):
                for d in dirs:
                    vd.vd_autotune_set(kind, code, length, axis, d, lines)
                got = G.fft_r2c(x, precision=precision)
                assert torch.equal(got, ref), (shape, lines)
                assert torch.equal(G.fft_c2r(got, precision=precision), back), (shape, lines)
        finally:
            for d in dirs:
                vd.vd_autotune_set(kind, code, length, axis, d, -1)
