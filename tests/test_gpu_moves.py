"""The class moves (FP64 z move, second-phase move) at the sizes where the lanes'
(p, q, r) groups have remainders, and the second phase's exponent shortcut at the
ends of its tolerance, against the oracle bit for bit (raw duals)."""
import numpy as np
import pytest

import oracle as O
from paper_1710_03732_gb300 import instances as I

pytestmark = pytest.mark.gpu
PHI = (0.1, 0.2, 0.3, 0.15, 0.25)


@pytest.mark.parametrize("n", [3, 4, 5, 6, 10, 11, 13])
@pytest.mark.parametrize("form", ["folded", "uniform", "partners"])
def test_fp64_move_remainders(n, form):
    from paper_1710_03732_gb300 import rlt2 as R
    inst = I.random_instance(n, 60 + n, with_b=True, asymmetric=True)
    kw = {"folded": {}, "uniform": dict(kz=0.75), "partners": dict(kz=0.75, phi_z=PHI)}[form]
    iters = 3
    with R.Context(inst.F, inst.D, inst.B, prm=R.params(dual_mode=0, feas_tol=0.0, **kw)) as ctx:
        lbs, done = ctx.iterate(iters)
        D, C = ctx.export_state()
    _, ref, _ = O.run(inst.F, inst.D, inst.B, iters=iters, dual_mode=0, prm=O.params_array(**kw))
    assert done == iters and np.array_equal(lbs, np.array(ref))
    # the context's last ascent step is pending: its costs are the oracle's one step before
    st, _, _ = O.run(inst.F, inst.D, inst.B, iters=iters - 1, dual_mode=0, prm=O.params_array(**kw))
    assert np.array_equal(D, st.Dhat) and np.array_equal(C, st.Chat)


@pytest.mark.parametrize("tol", [0.0, 5e-324, 1e-300, 1e-12, 1e-9, 1e-3, 0.25, 1.0, 1e6, 1e300])
@pytest.mark.parametrize("n", [5, 9, 12])
def test_second_phase_tolerances(n, tol):
    from paper_1710_03732_gb300 import rlt2 as R
    inst = I.random_instance(n, 80 + n, with_b=True)
    st, _, _ = O.run(inst.F, inst.D, inst.B, iters=4, dual_mode=0)
    D0 = st.Dhat.copy()
    D0[::7] += 1e-9 * np.abs(D0[::7])  # slacks near the usual tolerance
    D0[3::11] = 0.0
    with R.Context(inst.F, inst.D, inst.B, prm=R.params(dual_mode=0, feas_tol=0.0, two_phase=1, phase2_tol=tol)) as ctx:
        ctx.import_state(D0, st.Chat)
        ctx.iterate(1)
        D, _ = ctx.export_state()
    _, xi, psi, _, _ = O.stage_z(n, D0, dual_mode=0)
    assert np.array_equal(D, O.phase2_z(n, D0, xi, psi, tol=tol))
