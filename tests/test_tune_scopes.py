"""Table files: entries with a field-size scope beside entries for every size; setting or erasing an entry
by hand replaces the scoped ones of its key.  Host computations, no GPU."""

import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import paper_2403_06654_gb300 as vd
print(sorted(vd.vd_autotune_table()))
vd.vd_autotune_set(0, 1, 256, 2, -1, 4)
print(sorted(vd.vd_autotune_table()))
vd.vd_autotune_set(0, 1, 256, 2, -1, -1)
print(sorted(vd.vd_autotune_table()))
"""


def test_scoped_entries(tmp_path):
    f = tmp_path / "tune.txt"
    # every size; radix class 2 and 2^15 lines; the same with the built-in shape; a line of neither form
    f.write_text("0 1 256 2 -1 0\n0 1 256 2 -1 16 80 0\n0 1 256 2 -1 128 81 1\n0 1 256 2 1 8 80\n1 0 80 0 2 16\n")
    env = dict(os.environ, VD_TUNE_FILE=str(f), PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", CODE], env=env, capture_output=True, text=True, check=True).stdout
    key, other = (0, 1, 256, 2, -1), (1, 0, 80, 0, 2, 16)
    assert out.splitlines() == [str(sorted([key + (0,), key + (16,), key + (128,), other])),
                                str(sorted([key + (4,), other])), str([other])]
