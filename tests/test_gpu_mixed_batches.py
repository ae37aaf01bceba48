"""rlt2_iterate_many on contexts whose z moves take different forms (folded in
integers, kz != 1, unequal phi_z, the F variant): the contexts of a batch need
only share dual_mode, warm and two_phase, and each ends exactly where rlt2_iterate
alone takes it."""
import numpy as np
import pytest

from paper_1710_03732_gb300 import instances as I

pytestmark = pytest.mark.gpu

FORMS = [{}, dict(kz=0.75), dict(phi_z=(0.1, 0.2, 0.3, 0.15, 0.25)), dict(variant=1), dict(ky=0.25)]


@pytest.mark.parametrize("order", ["folded first", "folded last"])
@pytest.mark.parametrize("mode,two_phase", [(1, 0), (1, 1), (2, 0), (0, 1)])
def test_each_context_moves_as_alone(mode, two_phase, order):
    from paper_1710_03732_gb300 import rlt2 as R
    inst = I.random_instance(9, 71, with_b=True, asymmetric=True)
    forms = FORMS if order == "folded first" else FORMS[::-1]

    def make():
        return [R.Context(inst.F, inst.D, inst.B,
                          prm=R.params(dual_mode=mode, two_phase=two_phase, warm=1, feas_tol=0.0, **kw)) for kw in forms]

    many, single = make(), make()
    assert (R.rlt2_iterate_many(many, 8) == 8).all()
    for a, b in zip(many, single):
        assert b.iterate(8)[1] == 8
        assert a.bound()[:3] == b.bound()[:3]
        for x, y in zip(a.export_state(), b.export_state()):
            assert np.array_equal(x, y)
        da, db = a.duals(), b.duals()
        for k in ("xi", "psi", "gamma", "alpha"):
            assert np.array_equal(da[k], db[k]), k
    for c in many + single:
        c.close()
