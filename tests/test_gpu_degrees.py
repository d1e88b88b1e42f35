"""Residual and GMRES operator over every compiled degree (p = 0..7, q = 1..6), both precisions,
against the plain torch FP64 evaluation of perf/cases.py (quadrature tables and dense 1-D
contractions; itself equal to the oracle to 2e-15).

Bars, as in the other parity tests: FP64 1e-12 relative L2.  FP32 2e-6: inputs rounded to float
(6e-8 relative) and sums of at most a few dozen terms of either sign.
"""
import numpy as np
import pytest

from paper_1307_5310_gb300 import meshgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_5310_gb300 import stm
    from perf import cases

    return stm, cases


def _check(mods, m, dt):
    import torch

    stm, cases = mods
    x = cases._Exact(m, dt)
    s = stm.Slab(m)
    g = torch.Generator(device="cuda").manual_seed(5)
    # the 32-bit vectors start 4 bytes past a 16-byte boundary: entry points take any aligned float
    U = torch.empty(s.n_trial + 1, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)[1:]
    V = torch.empty(s.n_test + 1, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)[1:]
    for prec, dtype, bar in ((stm.STM_FP64, torch.float64, 1e-12), (stm.STM_FP32, torch.float32, 2e-6)):
        u = torch.empty(s.n_trial + 1, dtype=dtype, device="cuda")[1:].copy_(U)
        v = torch.empty(s.n_test + 1, dtype=dtype, device="cuda")[1:].copy_(V)
        out = torch.empty(s.n_test + 1, dtype=dtype, device="cuda")[1:]
        s.residual_apply(u, out, 0.0, dt, prec=prec)
        ref = x.residual(x.gather(U, True))
        assert float((out.double() - ref).norm() / ref.norm()) < bar, ("residual", prec)
        s.operator_apply(v, out, dt, prec=prec)
        ref = x.operator(x.precondition(V))
        assert float((out.double() - ref).norm() / ref.norm()) < bar, ("operator", prec)
        s.operator_apply(v, out, dt, pre=False, prec=prec)
        ref = x.operator(V)
        assert float((out.double() - ref).norm() / ref.norm()) < bar, ("operator without P", prec)


@pytest.mark.parametrize("p", range(8))
@pytest.mark.parametrize("geom", ["brick", "affine", "curved"])
def test_every_degree(mods, geom, p):
    for q in range(1, 7):
        kw = {"affine": [[1.0, 0.3, 0.1], [0.0, 0.9, -0.2], [0.15, 0.0, 1.1]]} if geom == "affine" else {}
        m = meshgen.box_mesh(3, 2, 2, hi=(1.0, 0.8, 1.2), p=p, q=q, order="morton" if q % 2 else "lex",
                             perturb=0.1 if geom == "curved" else 0.0, **kw)
        meshgen.random_materials(m, 71 + q, 72)
        _check(mods, m, 0.04)


@pytest.mark.parametrize("n,p,q", [((16, 16, 15), 1, 1), ((16, 16, 16), 1, 1), ((16, 16, 16), 0, 3),
                                   ((32, 32, 31), 2, 1), ((32, 32, 32), 2, 1), ((32, 33, 32), 2, 4)])
def test_low_degree_mesh_sizes(mods, n, p, q):
    """Either side of the sizes where low-degree FP32 meshes change from one kernel to two."""
    m = meshgen.box_mesh(*n, hi=(1.0, 0.8, 1.2), p=p, q=q)
    meshgen.random_materials(m, 81, 82)
    _check(mods, m, 0.01)


def test_first_apply_under_capture(mods):
    """A low-degree FP32 mesh whose first apply is captured (no scratch may be allocated then) runs the
    single pass; later applies run the two kernels.  Both against the FP64 evaluation, bar 2e-6."""
    import torch

    stm, cases = mods
    m = meshgen.box_mesh(16, p=1, q=1)
    meshgen.random_materials(m, 83, 84)
    dt = 0.01
    x = cases._Exact(m, dt)
    side = torch.cuda.Stream()
    s = stm.Slab(m, stream=side.cuda_stream)
    U = torch.empty(s.n_trial, dtype=torch.float64, device="cuda").uniform_(-1, 1)
    u, out = U.float(), torch.zeros(s.n_test, dtype=torch.float32, device="cuda")
    ref = x.residual(x.gather(U, True))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        s.residual_apply(u, out, 0.0, dt, prec=stm.STM_FP32)
    g.replay()
    torch.cuda.synchronize()
    assert float((out.double() - ref).norm() / ref.norm()) < 2e-6
    out.zero_()
    torch.cuda.synchronize()
    s.residual_apply(u, out, 0.0, dt, prec=stm.STM_FP32)
    torch.cuda.synchronize()
    assert float((out.double() - ref).norm() / ref.norm()) < 2e-6
    g.replay()
    torch.cuda.synchronize()
    assert float((out.double() - ref).norm() / ref.norm()) < 2e-6


@pytest.mark.parametrize("qmax", [2, 6])
def test_uneven_degrees_and_partitions(mods, qmax):
    m = meshgen.corner_octree_mesh(3, [0.7, 0.3])
    meshgen.random_hp(m, 73, p_range=(0, 7), q_range=(1, qmax))
    _check(mods, m, 0.02)
    m = meshgen.box_mesh(4, 3, 3, p=2, q=1)
    m["p"] = np.random.Generator(np.random.PCG64(74)).integers(0, 6, 36).astype(np.uint8)
    m["q"] = np.random.Generator(np.random.PCG64(75)).integers(1, qmax + 1, 36).astype(np.uint8)
    meshgen.random_nk(m, 76, choices=(1, 2, 4, 8))
    meshgen.random_materials(m, 77, 78)
    _check(mods, m, 0.03)
