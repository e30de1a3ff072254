"""hkbe_snapshot_restore brings back the model that the snapshot was taken
with, whatever hkbe_set_model set since: the steps after it repeat bit for
bit."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,params", [(pk.MODEL_NAMBU, [[1.0, 0.5, 1.7]]), (pk.MODEL_NAMBU, [[1.0]]),
                                          (pk.MODEL_BETHE, [[1.0]]), (pk.MODEL_NONE, None)])
@pytest.mark.parametrize("mixed", [False, True])
def test_model_between_save_and_restore(model, params, mixed):
    nt, n = 60, 2
    w = wk.nambu_workload(nt=nt, h=0.02, k=5, beta=5.0, n_inst=n, v=1.0, eps0=0.2, A0=0.3, g=0.5, w0=0.6)
    st = pk.Stepper(nt, 0.02, 5, 5.0, nao=2, n_inst=n, tol=1e-7 if mixed else 1e-12, max_iter=60,
                    precision=pk.PREC_MIXED if mixed else pk.PREC_FP64, svd_tol=1e-8 if mixed else 0.0, leaf=32, r_max=64)
    mid, mp = pk.model_params_for(w)
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mp)
    pk.hkbe_set_drive(st.h, w["drive_A"], w["drive_U"])
    st.bootstrap()
    st.step(20)
    pk.hkbe_snapshot_save(st.h)
    it = st.step(nt - 26)[0]
    first = [st.row(i, nt - 1) + (st.tv(i, nt - 1),) for i in range(n)]
    pk.hkbe_snapshot_restore(st.h)
    pk.hkbe_set_model(st.h, model, None if params is None else np.repeat(params, n, axis=0))
    st.step(3)
    pk.hkbe_snapshot_restore(st.h)
    assert np.array_equal(it, st.step(nt - 26)[0])
    for i in range(n):
        assert all(np.array_equal(x, y) for x, y in zip(first[i], st.row(i, nt - 1) + (st.tv(i, nt - 1),)))
