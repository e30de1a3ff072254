"""A step whose values overflow is reported (HKBE_ERR_NAN) and not taken as
converged: every measure of an iteration's change keeps a NaN.  The overflow
comes from finite inputs: an interaction that jumps to a value whose square
leaves the range of the storage form."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compressed,mixed,rho_mode,n", [(False, False, 0, 1), (False, False, 1, 9), (True, False, 1, 1),
                                                         (True, True, 0, 2), (True, True, 1, 9)])
def test_overflowing_step(compressed, mixed, rho_mode, n):
    nt, jump = 110, 100
    w = wk.nambu_workload(nt=nt, h=0.02, k=5, beta=5.0, n_inst=n, v=1.0, eps0=0.2, U=1.0, rho_mode=rho_mode)
    w["drive_U"][:] = w["drive_U"][0]   # (U = 1 everywhere: the complex64 bootstrap of U = 3 stays above 1e-7)
    w["drive_U"][:, jump + 1:] = 1e40 if mixed else 1e200
    form = dict(svd_tol=1e-8, leaf=32, r_max=64) if compressed else {}
    st = pk.Stepper(nt, 0.02, 5, 5.0, nao=2, n_inst=n, rho_mode=rho_mode, tol=1e-7 if mixed else 1e-12, max_iter=60,
                    precision=pk.PREC_MIXED if mixed else pk.PREC_FP64, **form)
    mid, mp = pk.model_params_for(w)
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mp)
    pk.hkbe_set_drive(st.h, w["drive_A"], w["drive_U"])
    st.bootstrap()
    st.step(jump - 1 - 5)
    with pytest.raises(pk.HKBEError) as e:
        st.step(3)
    assert e.value.code == pk.HKBE_ERR_NAN
    assert pk.hkbe_current_step(st.h) == jump - 1
    assert all(np.isfinite(x).all() for x in st.row(n - 1, jump - 1) + st.row(0, 40))
