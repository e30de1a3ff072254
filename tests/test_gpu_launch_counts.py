"""hkbe_get_timing counts every kernel of a phase: a sweep in two launches around
a ring kernel counts three, and a mixed component computed by the retarded
sweep's launch none of its own."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


# instances; launches per iteration of the retarded sweep and the mixed component, and of the lesser sweep
@pytest.mark.parametrize("n,before,after", [(1, (1, 0, 1), (3, 0, 3)), (153, (1, 1, 1), (1, 1, 3))])
def test_split_sweep_counts(n, before, after):
    nt = 270
    w = wk.bethe_workload(nt=nt, h=0.02, k=5, beta=5.0, n_inst=n, quench=(0.0, 1.0, 1.0))
    st = pk.Stepper(nt, 0.02, 5, 5.0, n_inst=n, tol=1e-12, max_iter=60, svd_tol=1e-8, leaf=64, r_max=64)
    mid, mp = pk.model_params_for(w)
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mp)
    st.bootstrap()
    for upto, per in ((190, before), (265, after)):
        st.step(upto - pk.hkbe_current_step(st.h))
        pk.hkbe_reset_counters(st.h)
        st.step(3)
        t = st.timing()
        it = t["ctrl"][1]   # one per iteration
        assert it >= 3
        assert tuple(t[p][1] for p in ("ret", "mixed", "les")) == tuple(it * x for x in per)
