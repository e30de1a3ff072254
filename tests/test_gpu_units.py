"""Other units of energy and time.  Energies times 2^m, times by 2^-m: G^R, G^<
and G^tv are the same numbers, Sigma is 2^2m times as large, and a power of two
commutes with every rounding, so an FP64 run gives the same bits as long as
nothing leaves the range of FP64 (pivots and reciprocals included).  With
compressed history (an absolute tolerance) the compressed run is compared with the
dense run of the same units, at Sigma about 2^72: its squares are beyond FP32."""
import numpy as np
import pytest

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

pytestmark = pytest.mark.gpu


def _run(no, nt, m, rho_mode=0, mixed=False, **form):
    s = 2.0 ** m
    rng = np.random.default_rng(no)
    V, e0, eb = rng.uniform(-0.5, 0.5, size=(no, 2)) + 0j, np.diag(rng.uniform(-0.5, 0.5, size=no)), wk.C5_BATH_LEVELS
    tau, om = wk.dlr_grid(100.0, 1e-10, 5.0)
    gm = wk.bath_gm(tau, 5.0, e0, V, eb)[None]
    st = pk.Stepper(nt, 0.05 / s, 5, 5.0 / s, nao=no, rho_mode=rho_mode, tol=1e-7 if mixed else 1e-13, max_iter=80,
                    precision=pk.PREC_MIXED if mixed else pk.PREC_FP64, **form)
    mp = np.concatenate([[2.0], eb * s, (V * s).view(np.float64).ravel()])[None]
    st.set_inputs(tau / s, om * s, gm, np.broadcast_to(e0 * s, (1, nt + 1, no, no)).astype(complex), pk.MODEL_BATH, mp)
    st.run()
    return st


@pytest.mark.parametrize("no,rho_mode,m", [(1, 0, 70), (2, 1, 70), (3, 1, 70), (4, 0, 70), (2, 1, -90)])
def test_dense_bits(no, rho_mode, m):
    a, b = _run(no, 75, 0, rho_mode).dense(), _run(no, 75, m, rho_mode).dense()
    assert all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("no,nt,mixed", [(1, 160, False), (2, 150, False), (1, 160, True), (2, 150, True)])
def test_compressed(no, nt, mixed):
    # blocks of 64 columns at most, so no rank exceeds r_max; bounds: the compressed FP64 form's rounding
    # floor; the complex64 form's bar plus ten times its SVD tolerance
    a = _run(no, nt, 36, mixed=mixed, svd_tol=1e-8 if mixed else 1e-12, leaf=32, r_max=64)
    b = _run(no, nt, 36)
    bound = 1e-6 + 1e-7 if mixed else 1e-9
    for T in (nt - 1, nt - 40, 90, 70):
        for x, y in zip(a.row(0, T) + (a.tv(0, T),), b.row(0, T) + (b.tv(0, T),)):
            assert np.abs(x - y).max() < bound, T


def test_large_occupations_complex64():
    # G^M and with it G^<, G^tv times 2^100 (the equations are linear in them): the change from one iterate to
    # the next has squares beyond FP32; bound: the complex64 form's bar, relative to the largest element
    nt, no, V = 75, 2, np.array([[0.3, -0.4], [0.2, 0.5]]) + 0j
    e0, eb = np.diag([0.2, -0.3]), wk.C5_BATH_LEVELS
    tau, om = wk.dlr_grid(100.0, 1e-10, 5.0)
    gm = wk.bath_gm(tau, 5.0, e0, V, eb)[None] * 2.0 ** 100
    mp = np.concatenate([[2.0], eb, V.view(np.float64).ravel()])[None]
    out = []
    for prec in (pk.PREC_FP64, pk.PREC_MIXED):
        st = pk.Stepper(nt, 0.05, 5, 5.0, nao=no, tol=1e-7, max_iter=80, precision=prec)
        st.set_inputs(tau, om, gm, np.broadcast_to(e0, (1, nt + 1, no, no)).astype(complex), pk.MODEL_BATH, mp)
        st.run()
        out.append(st.dense())
    for x, y in zip(*out):
        assert np.abs(x - y).max() < 1e-6 * np.abs(x).max()
