"""Compressed FP64 runs against dense FP64 runs of the same inputs: block sides
longer than one chunk of the source projections, and ranks, levels and orbitals
for which the sweeps leave the projections in global memory (N_o >= 3, r_max
128).  The two forms share no history kernel, so each checks the other."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


def _run(w, svd_tol, leaf, r_max):
    wl = w["wl"]
    st = pk.Stepper(wl.nt, wl.h, wl.k, wl.beta, nao=wl.nao, rho_mode=wl.rho_mode, tol=1e-13, max_iter=80,
                    svd_tol=svd_tol, leaf=leaf, r_max=r_max)
    mid, mp = pk.model_params_for(w)
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mp)
    st.run()
    return st


@pytest.mark.parametrize("no,nt,leaf,r_max", [(1, 620, 32, 64), (2, 600, 64, 64), (3, 170, 32, 128), (4, 200, 32, 128)])
def test_rows_agree(no, nt, leaf, r_max):
    if no == 1:
        w = wk.bethe_workload(nt=nt, h=0.02, beta=5.0, quench=(0.0, 1.0, 2.0))
    else:
        rng = np.random.default_rng(no)
        A = rng.uniform(-0.5, 0.5, size=(no, no)) + 1j * rng.uniform(-0.5, 0.5, size=(no, no))
        V, e0 = rng.uniform(-0.5, 0.5, size=(no, 2)) + 0j, 0.5 * (A + A.conj().T)
        tau, om = wk.dlr_grid(100.0, 1e-10, 5.0)
        wl = wk.Workload(name="bath", model="bath", nt=nt, h=0.02, k=5, beta=5.0, nao=no, rho_mode=no % 2)
        w = {"wl": wl, "tau": tau, "omega": om, "eps": np.broadcast_to(e0, (1, nt + 1, no, no)).astype(complex),
             "gm": wk.bath_gm(tau, 5.0, e0, V, wk.C5_BATH_LEVELS)[None],
             "model_params": np.concatenate([[2.0], wk.C5_BATH_LEVELS, V.view(np.float64).ravel()])[None]}
    a, b = _run(w, 1e-12, leaf, r_max), _run(w, 0.0, 64, 64)
    # SVD tolerance 1e-12: the compressed form's own FP64 rounding floor (1e-9 absolute) is the bound
    for T in (nt - 1, nt - 40, nt // 2, 70):
        for x, y in zip(a.row(0, T) + (a.tv(0, T),), b.row(0, T) + (b.tv(0, T),)):
            assert np.abs(x - y).max() < 1e-9, T
