"""The curved mass kernel at the edges of its launch shapes: one element and few (several CTAs per
element, two threads per coefficient plane in FP64), meshes of several element groups per CTA, and a last
group that is not full.  Residual and operator of trilinear meshes against the plain torch FP64
evaluation of perf/cases.py.

Bars, as in the other parity tests: FP64 1e-12 relative L2, FP32 2e-6 (inputs rounded to float, short
sums of either sign).
"""
import pytest

from paper_1307_5310_gb300 import meshgen

pytestmark = pytest.mark.gpu

# small: fewer elements than SMs.  full: at least two element groups per CTA of one wave (152 SMs, up to
# 32 CTAs of up to 8 elements each at p = 1, one or two CTAs at p = 7), with an odd element count
SMALL = [(1, 1, 1), (5, 3, 3)]
FULL = {0: (45, 43, 41), 1: (45, 43, 41), 2: (31, 29, 33), 3: (23, 21, 25), 4: (19, 17, 15), 5: (13, 11, 15),
        6: (11, 9, 11), 7: (9, 11, 9)}


@pytest.fixture(scope="module")
def mods():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_5310_gb300 import stm
    from perf import cases

    return stm, cases


def _check(mods, n, p, q):
    import torch

    stm, cases = mods
    m = meshgen.box_mesh(*n, hi=(1.0, 0.8, 1.2), p=p, q=q, perturb=0.1)
    meshgen.random_materials(m, 71 + q, 72)
    x = cases._Exact(m, 0.02)
    s = stm.Slab(m)
    g = torch.Generator(device="cuda").manual_seed(5)
    U = torch.empty(s.n_trial, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)
    V = torch.empty(s.n_test, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)
    refs = x.residual(x.gather(U, True)), x.operator(V)
    for prec, dtype, bar in ((stm.STM_FP64, torch.float64, 1e-12), (stm.STM_FP32, torch.float32, 2e-6)):
        out = torch.empty(s.n_test, dtype=dtype, device="cuda")
        s.residual_apply(U.to(dtype), out, 0.0, 0.02, prec=prec)
        assert float((out.double() - refs[0]).norm() / refs[0].norm()) < bar, ("residual", prec)
        s.operator_apply(V.to(dtype), out, 0.02, pre=False, prec=prec)
        assert float((out.double() - refs[1]).norm() / refs[1].norm()) < bar, ("operator", prec)
    s.close()


@pytest.mark.parametrize("p", range(8))
def test_small_meshes(mods, p):
    for q in range(1, 7):
        for n in SMALL:
            _check(mods, n, p, q)


@pytest.mark.parametrize("q", [1, 2, 3])
@pytest.mark.parametrize("p", range(8))
def test_several_groups(mods, p, q):
    _check(mods, FULL[p], p, q)
