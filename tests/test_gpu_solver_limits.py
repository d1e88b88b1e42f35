"""The slab solve at the ends of its iteration cap: the largest value solves, zero and negative values
stop at the first check with a report of it.  The end state against the oracle's direct solve, bar 1e-9 (the
solver stops at 1e-12 of the reference residual)."""
import numpy as np
import pytest

from oracle import stdg
from paper_1307_5310_gb300 import meshgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_it", [2**31 - 1, 2**31 - 2, 0, -1, -2, -(2**31)])
def test_iteration_cap(max_it):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_5310_gb300 import stm

    m = meshgen.box_mesh(2, 2, 1, p=2, q=1)
    meshgen.random_materials(m, 91, 92)
    u0 = np.random.Generator(np.random.PCG64(93)).uniform(-1, 1, 4 * 6 * 27)
    for precision in (stm.STM_FP64, stm.STM_MIXED):
        s = stm.Slab(m, precision=precision, tol=1e-12, max_it=max_it)
        s.set_state(u0)
        rc, rep = s.slab_solve(0.1)
        if max_it > 0:
            o = stdg.Oracle(m)
            ref = o.end_state(o.slab_solve(u0, 0.0, 0.1))
            u, _ = s.get_state()
            assert rc == stm.STM_OK and np.linalg.norm(u - ref) < 1e-9 * np.linalg.norm(ref), rep
        else:
            assert rc == stm.STM_ENOTCONV and rep["iterations"] == 0 and rep["restarts"] == 0
            assert 1e-12 < rep["rel_residual"] < 1e3
        s.close()
