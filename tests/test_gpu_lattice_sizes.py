"""Grid sizes of the lattice self-energies: the transforms of 8 and 16 points,
and the direct sums of every other L (odd ones and the reflection-reduced k-set
among them), against the lockstep oracle in real time and the host solver on the
imaginary axis.  T + 1 and the node count are no multiples of the times and
nodes per CTA."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk
from oracle.lattice import LatticeOracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,ys,mixed", [(2, 0, 0), (3, 0, 0), (6, 1, 0), (8, 0, 0), (8, 1, 1), (9, 0, 0)])
def test_real_time(L, ys, mixed):
    w = wk.lattice_workload(L=L, nt=15, h=0.05, k=2, beta=4.0, U=1.5, A0=0.4, tc=0.3, width=0.2, dlr_eps=1e-8)
    wl = w["wl"]
    o = LatticeOracle(L, wl.nt, wl.h, wl.k, wl.beta, w["eps"], w["gm"], w["tau"], w["omega"], w["drive_U"][0],
                      tol=1e-14)
    o.run()
    keep = range(L * L)
    if ys:
        w = wk.lattice_workload(L=L, nt=15, h=0.05, k=2, beta=4.0, U=1.5, A0=0.4, tc=0.3, width=0.2, dlr_eps=1e-8,
                                ysymm=True)
        keep = [mx * L + my for mx in range(L) for my in range(L // 2 + 1)]
    st = pk.Stepper(wl.nt, wl.h, wl.k, wl.beta, n_inst=len(keep), tol=1e-7 if mixed else 1e-13, max_iter=80,
                    precision=pk.PREC_MIXED if mixed else pk.PREC_FP64)
    mid, mp = pk.model_params_for(w)
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mp)
    pk.hkbe_set_drive(st.h, w["drive_A"], w["drive_U"])
    st.run()
    bar = 1e-6 if mixed else 1e-10       # the suite's bars, relative to the largest element
    for i, q in enumerate(keep):
        GR, GL, GTV = st.dense(i)
        t = np.tril_indices(wl.nt)
        oq = o.orcs[q]
        ref = max(np.abs(oq.GR[t]).max(), np.abs(oq.GLs[t]).max(), np.abs(oq.GTV).max())
        assert max(np.abs(GR[t] - oq.GR[t]).max(), np.abs(GL[t] - oq.GLs[t]).max(), np.abs(GTV - oq.GTV).max()) < bar * ref


@pytest.mark.parametrize("L,ys", [(2, 0), (5, 0), (8, 1), (12, 0), (15, 0)])
def test_equilibrium(L, ys):
    tau, om = wk.dlr_grid(60.0, 1e-8, 4.0)
    kx, ky = np.meshgrid(2 * np.pi * np.arange(L) / L, 2 * np.pi * np.arange(L // 2 + 1 if ys else L) / L, indexing="ij")
    e = -2 * (np.cos(kx) + np.cos(ky)).ravel()
    n, mp = len(e), np.array([[float(L), float(ys)]] * len(e))
    st = pk.Stepper(16, 0.02, 5, 4.0, n_inst=n, tol=1e-13)
    st.set_inputs(tau, om, None, np.broadcast_to(e[:, None, None, None], (n, 17, 1, 1)).astype(complex),
                  pk.MODEL_LATTICE2B, mp)
    G, _, _ = pk.hkbe_solve_matsubara(st.h, n, len(tau), 1, U_eq=1.5, mix=0.5, tol=1e-12, max_iter=500)
    Gh, _, _, _ = pk.hkbe_matsubara_solve(tau, om, 4.0, pk.MODEL_LATTICE2B, e[:, None, None].astype(complex), mp,
                                          U_eq=1.5, mix=0.5, tol=1e-12, max_iter=500)
    assert np.abs(G - Gh).max() < 1e-11   # both converge the same iteration to 1e-12 with a factor 1/2 per step
