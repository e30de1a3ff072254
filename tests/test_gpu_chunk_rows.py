"""Chunk inverses of the sweeps grow by a row per time step: parity with the
oracle where a chunk starts, ends or is one point long, where the retarded head
covers every point (T <= 2k), and from snapshots taken in the middle of a chunk
(the growing rows are rebuilt then: the steps repeat bit for bit)."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk
from oracle.kbe import from_workload

pytestmark = pytest.mark.gpu

# FP64 forms: 1e-10 of the largest element (the suite's bar); complex64 form: 1e-6 plus ten times the SVD tolerance
CASES = [  # N_o, k, N_t, step of the snapshot, density-matrix scheme, leaf (0: dense), complex64
    (1, 5, 75, 40, 0, 0, False), (1, 1, 36, 34, 0, 0, False), (1, 5, 12, 8, 0, 0, False), (1, 4, 98, 64, 0, 32, False),
    (2, 5, 44, 20, 1, 0, False), (2, 3, 70, 38, 0, 0, False), (2, 5, 107, 75, 1, 32, True), (1, 5, 140, 69, 0, 64, True),
    (3, 5, 45, 33, 0, 0, False), (4, 5, 42, 11, 1, 0, False), (4, 2, 76, 37, 0, 32, True),
]


def _workload(no, k, nt, rho):
    if no == 1:
        w = wk.bethe_workload(nt=nt, h=0.05, k=k, beta=5.0, quench=(0.0, 0.7, 0.05 * (nt // 3)), rho_mode=rho)
        return w, {}
    rng = np.random.default_rng(no)
    A = rng.uniform(-0.5, 0.5, size=(no, no)) + 1j * rng.uniform(-0.5, 0.5, size=(no, no))
    V = rng.uniform(-0.5, 0.5, size=(no, 2)) + 0j
    e0, eb = 0.5 * (A + A.conj().T), wk.C5_BATH_LEVELS
    tau, om = wk.dlr_grid(100.0, 1e-10, 5.0)
    wl = wk.Workload(name="bath", model="bath", nt=nt, h=0.05, k=k, beta=5.0, nao=no, rho_mode=rho)
    mp = np.concatenate([[2.0], eb, V.view(np.float64).ravel()])
    w = {"wl": wl, "tau": tau, "omega": om, "eps": np.broadcast_to(e0, (1, nt + 1, no, no)).astype(complex),
         "gm": wk.bath_gm(tau, 5.0, e0, V, eb)[None], "model_params": mp[None]}
    return w, {"model_params": {"V": V, "eb": eb}}


@pytest.mark.parametrize("no,k,nt,snap,rho,leaf,mixed", CASES)
def test_growing_chunks(no, k, nt, snap, rho, leaf, mixed):
    w, kw = _workload(no, k, nt, rho)
    svd = 1e-8 if mixed else 1e-12
    st = pk.Stepper(nt, 0.05, k, 5.0, nao=no, rho_mode=rho, tol=1e-7 if mixed else 1e-13, max_iter=80,
                    precision=pk.PREC_MIXED if mixed else pk.PREC_FP64, svd_tol=svd if leaf else 0.0, leaf=leaf or 64,
                    r_max=64)
    mid, mp = pk.model_params_for(w)
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mp)
    st.bootstrap()
    st.step(snap - k)
    pk.hkbe_snapshot_save(st.h)
    st.step(nt - 1 - snap)
    first = st.dense()
    pk.hkbe_snapshot_restore(st.h)
    st.step(nt - 1 - snap)
    assert all(np.array_equal(a, b) for a, b in zip(first, st.dense()))
    o = from_workload(w, 0, tol=1e-14, **kw).run()
    i = np.tril_indices(nt)
    ref = max(np.abs(o.GR[i]).max(), np.abs(o.GLs[i]).max())
    err = max(np.abs(first[0][i] - o.GR[i]).max(), np.abs(first[1][i] - o.GLs[i]).max(), np.abs(first[2] - o.GTV).max())
    assert err <= ((1e-6 if mixed else 1e-10) * ref + (10 * svd if leaf else 0.0))
