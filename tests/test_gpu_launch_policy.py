"""The launch policy belongs to a solve, not to the handle.  Needs a GB300."""
import threading
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1605_01522_gb300 import inputs, mfs

pytestmark = pytest.mark.gpu


def _best(handle, b, n=60):
    best = 1e9
    for _ in range(n):
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        t = time.perf_counter()
        handle.solve(b, x, tol=1e-8)
        best = min(best, time.perf_counter() - t)
    return best


def test_first_solve_beside_another_does_not_fix_the_launches():
    """Solves take programmatic launches only while they run alone in the
    process.  A handle whose iteration graphs were captured beside another
    solve replayed ordinary launches ever after: 1.26 times the time of this
    small system (1.93 against 1.53 ms), bound 1.12 for the best of 60 solves."""
    s = inputs.thermo_elastic_2d(ne=32)
    kw = dict(precond="bgs_amg", max_levels=3, coarse_max=0)
    b = torch.from_numpy(s.rhs).cuda()
    big = inputs.coupled_box_3d(ne=20, nfields=3)
    bb = torch.from_numpy(big.rhs).cuda()
    with mfs.Solver(s, **kw) as alone, mfs.Solver(s, **kw) as beside, \
            mfs.Solver(big, precond="amg_bgs", max_iters=3000, max_levels=4, coarse_max=500) as other:
        xa, ia, _ = alone.solve(b, tol=1e-8)
        t = threading.Thread(target=lambda: other.solve(bb, torch.zeros_like(bb), tol=1e-30, check=False))
        t.start()
        time.sleep(0.1)
        xb, ib, _ = beside.solve(b, tol=1e-8)
        assert t.is_alive()  # the other solve ran meanwhile
        t.join()
        assert ia["iters"] == ib["iters"] and torch.equal(xa, xb)
        ta, tb = _best(alone, b), _best(beside, b)
        ta, tb = min(ta, _best(alone, b)), min(tb, _best(beside, b))
        assert max(ta, tb) <= 1.12 * min(ta, tb), (ta, tb)
        assert torch.equal(xa, beside.solve(b, tol=1e-8)[0])
