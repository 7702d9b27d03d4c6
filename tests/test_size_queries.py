"""Size queries are made per request (server) and per item (batch) on the host: they form no launch plans.
Host computations, no GPU."""

import ctypes
import math
import time

import paper_2403_06654_gb300 as vd


def test_batch_bytes_makes_no_plans():
    """The plans of the wide passes took 60 to 114 us per axis of 480 to 1024 points; the query itself
    takes about a microsecond.  The least of many calls is compared, so a busy host cannot fail it."""
    item = (vd.vd_batch_item * 1)()
    item[0].ndim = 3
    item[0].n = (ctypes.c_int * 3)(960, 1000, 1024)
    item[0].L = (ctypes.c_double * 3)(*([2 * math.pi] * 3))
    item[0].b_pres = item[0].x_pres = item[0].rho = 1   # (only tested against null)
    params = vd.vd_batch_params(vd.SOLVERS["gmres"], vd.SOLVERS["cg"], 1e-10, 100, 30, vd.PRECISIONS["mixed"])
    query = vd.lib().vd_batch_bytes
    assert query(item, 1, ctypes.byref(params)) > 0
    least = math.inf
    for _ in range(50):
        t = time.perf_counter()
        query(item, 1, ctypes.byref(params))
        least = min(least, time.perf_counter() - t)
    assert least < 50e-6, least
