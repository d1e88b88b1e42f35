"""Low-degree FP32 meshes large enough for the two-kernel passes, in the forms other than plain bricks:
constant 3x3 metric, curved elements, the dissipative term; and a mixed solve whose captured cycles run
them.  FP32 residual and operator against FP64 of the same context (which other tests compare with the
oracle), bar 2e-6: inputs rounded to float and short sums.  Solves: mixed to 1e-11 against FP64 to 1e-12,
bar 1e-8 on the end state.
"""
import pytest

from paper_1307_5310_gb300 import meshgen

pytestmark = pytest.mark.gpu

FORMS = {"affine": dict(affine=[[1.0, 0.3, 0.1], [0.0, 0.9, -0.2], [0.15, 0.0, 1.1]]),
         "curved": dict(perturb=0.1), "dissipative": {}}


@pytest.fixture(scope="module")
def stm():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_5310_gb300 import stm as s

    return s


def _vec(n, seed):
    import torch

    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.empty(n, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)


@pytest.mark.parametrize("n,p,q", [(16, 0, 2), (16, 1, 1), (17, 1, 6), (32, 2, 1), (33, 2, 4)])
@pytest.mark.parametrize("form", sorted(FORMS))
def test_two_kernel_forms(stm, form, n, p, q):
    import torch

    m = meshgen.box_mesh(n, n, n, hi=(1.0, 0.8, 1.2), p=p, q=q, order="morton", **FORMS[form])
    meshgen.random_materials(m, 81, 82)
    s = stm.Slab(m, c_diss=0.7 if form == "dissipative" else 0.0)
    dt = 0.01
    U, V = _vec(s.n_trial, 5), _vec(s.n_test, 6)
    ref, out = torch.empty(s.n_test, dtype=torch.float64, device="cuda"), torch.empty(s.n_test, device="cuda")

    def err():
        return float((out.double() - ref).norm() / ref.norm())

    s.residual_apply(U, ref, 0.0, dt)
    s.residual_apply(U.float(), out, 0.0, dt, prec=stm.STM_FP32)
    assert err() < 2e-6
    for pre in (True, False):
        s.operator_apply(V, ref, dt, pre=pre)
        s.operator_apply(V.float(), out, dt, pre=pre, prec=stm.STM_FP32)
        assert err() < 2e-6, pre
    s.close()


@pytest.mark.parametrize("form", ["brick", "affine", "curved", "dissipative"])
def test_mixed_solve(stm, form):
    import torch

    m = meshgen.box_mesh(16, 16, 16, p=1, q=1, **FORMS.get(form, {}))
    meshgen.random_materials(m, 83, 84)
    ends = []
    for precision, tol in ((stm.STM_FP64, 1e-12), (stm.STM_MIXED, 1e-11)):
        s = stm.Slab(m, precision=precision, tol=tol, max_it=2000, c_diss=0.7 if form == "dissipative" else 0.0)
        s.set_state(_vec(s.n_state, 7))
        for _ in range(2):
            rc, rep = s.slab_solve(0.01)
            assert rc == stm.STM_OK, rep
        ends.append(torch.from_numpy(s.get_state()[0]))
        s.close()
    assert float((ends[1] - ends[0]).norm() / ends[0].norm()) < 1e-8
