"""What the tuner finds on one field holds for fields of about its size: a small field with axes of the same
lengths keeps its built-in shapes.  Shown by the bits: on the large float field the register four-step
kernels win or are the built-in choice, on the small one the general kernel, which rounds differently."""

import math
import os
import subprocess
import sys

import pytest
import torch

import paper_2403_06654_gb300 as vd

pytestmark = pytest.mark.gpu

BIG, SMALL = (256, 256, 160), (256, 256)


def _transforms(n, precision):
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(tuple(reversed(n)), generator=gen, dtype=torch.float64, device="cuda")
    x = x.float() if precision == "mixed" else x
    G = vd.Grid(n, (2 * math.pi,) * len(n))
    xh = G.fft_r2c(x, precision=precision)
    return xh, G.fft_c2r(xh, precision=precision)


def _erase():
    for e in vd.vd_autotune_table():
        vd.vd_autotune_set(*e[:5], -1)


def test_tuning_a_large_field_leaves_small_ones():
    _erase()
    small, big = _transforms(SMALL, "mixed"), _transforms(BIG, "mixed")
    # the register kernel where the tuner's choice for the large field would reach the small one
    for d in (-1, 1):
        vd.vd_autotune_set(0, 1, 256, 1, d, 0)
    forced = _transforms(SMALL, "mixed")
    assert not torch.equal(forced[0], small[0])   # (the two kernels can be told apart)
    _erase()
    try:
        vd.vd_autotune(vd.Grid(BIG, (2 * math.pi,) * 3), ("mixed",))
        assert vd.vd_autotune_table()
        again = _transforms(SMALL, "mixed")
        assert torch.equal(again[0], small[0]) and torch.equal(again[1], small[1])
        tuned = _transforms(BIG, "mixed")
        err = torch.linalg.vector_norm(tuned[1] - big[1]) / torch.linalg.vector_norm(big[1])
        assert err.item() < 8 * 2.0 ** -24 * math.log2(math.prod(BIG))   # two transforms' rounding each
        # an entry set by hand holds for every size, also after tuning
        for d in (-1, 1):
            vd.vd_autotune_set(0, 1, 256, 1, d, 0)
        assert torch.equal(_transforms(SMALL, "mixed")[0], forced[0])
    finally:
        _erase()
    assert vd.vd_autotune_table() == []


def test_tuned_table_survives_its_file(tmp_path, monkeypatch):
    """A later process reads the tuner's file into the same entries."""
    _erase()
    f = tmp_path / "tune.txt"
    monkeypatch.setenv("VD_TUNE_FILE", str(f))
    try:
        vd.vd_autotune(vd.Grid((24, 20, 18), (2 * math.pi,) * 3), ("fp64", "mixed_dd"))
        table = sorted(vd.vd_autotune_table())
    finally:
        _erase()
    code = "import paper_2403_06654_gb300 as vd; print(sorted(vd.vd_autotune_table()))"
    env = dict(os.environ, PYTHONPATH=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    out = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, check=True).stdout
    assert table and out.strip() == str(table)
    # scope and built-in flag follow the six numbers of an entry
    assert all(len(line.split()) == 8 for line in f.read_text().splitlines())
