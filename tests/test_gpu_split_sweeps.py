"""Sweeps in two launches around a ring kernel (from 192 compressed rows; the
retarded one only where its CTAs leave SMs idle) and in one: a batch beyond that
line against one instance below it, and both against the dense form, which has
neither.  Leaves of 32 and 64, the first row of a split and the last."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


def _run(w, n, mixed, leaf):
    wl = w["wl"]
    form = dict(svd_tol=1e-8 if mixed else 1e-12, leaf=leaf, r_max=128 if wl.nao > 2 else 64) if leaf else {}
    st = pk.Stepper(wl.nt, wl.h, wl.k, wl.beta, nao=wl.nao, n_inst=n, rho_mode=wl.rho_mode, tol=1e-7 if mixed else 1e-13,
                    max_iter=80, precision=pk.PREC_MIXED if mixed else pk.PREC_FP64, **form)
    mid, mp = pk.model_params_for(w)
    rep = lambda a: np.repeat(np.asarray(a)[:1], n, axis=0)
    st.set_inputs(w["tau"], w["omega"], rep(w["gm"]), rep(w["eps"]), mid, rep(mp))
    st.run()
    return st


@pytest.mark.parametrize("no,nt,leaf,batch,mixed", [(1, 262, 32, 153, True), (1, 300, 64, 153, False), (2, 268, 32, 77, True),
                                                    (3, 240, 32, 51, False), (4, 236, 32, 39, True)])
def test_split_sweeps(no, nt, leaf, batch, mixed):
    if no == 1:
        w = wk.bethe_workload(nt=nt, h=0.02, beta=5.0, quench=(0.0, 1.0, 2.0))
    else:
        rng = np.random.default_rng(10 + no)
        A = rng.uniform(-0.5, 0.5, size=(no, no)) + 1j * rng.uniform(-0.5, 0.5, size=(no, no))
        V, e0 = rng.uniform(-0.5, 0.5, size=(no, 2)) + 0j, 0.5 * (A + A.conj().T)
        tau, om = wk.dlr_grid(100.0, 1e-10, 5.0)
        wl = wk.Workload(name="bath", model="bath", nt=nt, h=0.02, k=5, beta=5.0, nao=no, rho_mode=no % 2)
        w = {"wl": wl, "tau": tau, "omega": om, "eps": np.broadcast_to(e0, (1, nt + 1, no, no)).astype(complex),
             "gm": wk.bath_gm(tau, 5.0, e0, V, wk.C5_BATH_LEVELS)[None],
             "model_params": np.concatenate([[2.0], wk.C5_BATH_LEVELS, V.view(np.float64).ravel()])[None]}
    one, many, dense = _run(w, 1, mixed, leaf), _run(w, batch, mixed, leaf), _run(w, 1, False, 0)
    # the compressed FP64 form's rounding floor; the complex64 form's bar plus ten times its SVD tolerance
    bound = 1e-6 + 1e-7 if mixed else 1e-9
    for T in (nt - 1, nt - 34, 230, 200):
        ref = dense.row(0, T) + (dense.tv(0, T),)
        for st, i in ((one, 0), (many, 0), (many, batch - 1)):
            for x, y in zip(st.row(i, T) + (st.tv(i, T),), ref):
                assert np.abs(x - y).max() < bound, (T, i)
