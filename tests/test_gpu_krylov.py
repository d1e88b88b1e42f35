"""The GMRES reductions and their device-side control at their edges: restart lengths up to the
largest (15 basis vectors and a norm in one reduction), with and without the second Gram-Schmidt
pass, unknown counts below one block, at a whole number of vectors and with a scalar tail.

The slab's end state against the oracle's direct solve: GMRES stops at 1e-12 of the reference
residual; the bar 1e-9 is the solver's stated accuracy.
"""
import numpy as np
import pytest

from oracle import stdg
from paper_1307_5310_gb300 import meshgen

pytestmark = pytest.mark.gpu

# unknowns: 192 (one block), 162 (p = 2: not a multiple of 4 or 8), 1,296
MESHES = [(2, 2, 1, 1, 1), (1, 1, 1, 2, 1), (2, 2, 1, 2, 2)]


@pytest.fixture(scope="module")
def stm():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_5310_gb300 import stm as s

    return s


@pytest.mark.parametrize("nx,ny,nz,p,q", MESHES)
def test_restart_lengths(stm, nx, ny, nz, p, q):
    m = meshgen.box_mesh(nx, ny, nz, hi=(1.0, 0.9, 0.7), p=p, q=q)
    meshgen.random_materials(m, 91, 92)
    o = stdg.Oracle(m)
    u0 = np.random.Generator(np.random.PCG64(93)).uniform(-1, 1, nx * ny * nz * 6 * (p + 1) ** 3)
    dt = 0.1
    uo = o.end_state(o.slab_solve(u0, 0.0, dt))
    for restart in (3, 9, 15):
        for reorth in (True, False):
            for precision in (stm.STM_FP64, stm.STM_MIXED):
                s = stm.Slab(m, precision=precision, tol=1e-12, restart=restart, reorth=reorth, max_it=3000)
                s.set_state(u0)
                rc, rep = s.slab_solve(dt)
                assert rc == stm.STM_OK, rep
                u, _ = s.get_state()
                assert np.linalg.norm(u - uo) < 1e-9 * np.linalg.norm(uo), (restart, reorth, precision)
                s.close()
    # the iteration cap ends the solve with the warning and keeps the iterate
    s = stm.Slab(m, tol=1e-12, restart=15, max_it=1)
    s.set_state(u0)
    rc, rep = s.slab_solve(dt)
    assert rc == stm.STM_ENOTCONV and rep["iterations"] == 1
