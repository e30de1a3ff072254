"""Handles of one orbital count and storage form, but of different length (and
so of different shared-memory needs), stepped by two host threads at once: each
gives what it gives alone."""
import threading

import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [False, True])
def test_two_threads(mixed):
    w = wk.nambu_workload(nt=2048, h=0.02, k=5, beta=5.0, v=1.0, eps0=0.2, U=0.5, A0=0.3, rho_mode=1)
    mid, mp = pk.model_params_for(w)

    def stepper(nt):
        st = pk.Stepper(nt, 0.02, 5, 5.0, nao=2, rho_mode=1, tol=1e-7 if mixed else 1e-12, max_iter=60,
                        precision=pk.PREC_MIXED if mixed else pk.PREC_FP64, svd_tol=1e-8, leaf=64, r_max=64)
        st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"][:, :nt + 1], mid, mp)
        pk.hkbe_set_drive(st.h, w["drive_A"][:, :nt + 1], w["drive_U"][:, :nt + 1])
        st.bootstrap()
        return st

    def steps(st, out):
        try:
            for _ in range(245):
                st.step(1)
            out.append(st.row(0, 250) + (st.tv(0, 250),))
        except pk.HKBEError as e:
            out.append(e)

    sts = [stepper(256), stepper(2048)]
    alone, both = [[], []], [[], []]
    for st, o in zip(sts, alone):
        steps(st, o)
        pk.hkbe_rewind(st.h)
    th = [threading.Thread(target=steps, args=a) for a in zip(sts, both)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for a, b in zip(alone, both):
        assert not isinstance(a[0], Exception) and not isinstance(b[0], Exception), (a[0], b[0])
        assert all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))
