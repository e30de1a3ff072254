"""Performance cases of the Kadanoff-Baym stepper: what its users run, over the range of sizes they run it at.

A user's program builds a ``Stepper`` (grid, G^M, eps(t), model, drive), bootstraps it and advances it, either all
the way ("run": every pass starts again from the bootstrapped state) or from a checkpoint taken part of the way
("window": every pass restores the in-memory snapshot and takes the next steps, one leaf compression among every
64).  A pass ends by reading what was computed: the last retarded row, lesser column and mixed row of every instance,
an older row (reconstructed from the compressed history), and the density matrices of all its steps.  "solve" cases are the equilibrium problem that precedes a propagation.

The inputs are those of ``kbe_workloads`` (the configurations that the benchmark and the tests use), with the level,
quench, drive and interaction strengths drawn from the seed.

``exact`` is a dense 64-bit propagation of the same discrete scheme in numpy and torch, with every step's integral
equations written as one (block) triangular system.
"""
import math
from fractions import Fraction

import numpy as np
import torch

import kbe_workloads as wk
import paper_2604_05319_gb300 as pk

K = 5                     # integration order of every configuration
MIXED_TOL, FP64_TOL = 1e-7, 1e-12   # self-consistency tolerance of the two storage forms, as in the benchmark


def _case(name, model, form, n_inst, nt, **kw):
    c = dict(name=name, kind="run", model=model, form=form, n_inst=n_inst, nt=nt, nao=1, start=K, compressed=False,
             per_step=False, uneven=False)
    c.update(kw)
    return c


def listed():
    return [
        # a first try of a model: one impurity, a few dozen steps; launches and latencies are all there is
        _case("bethe fp64 1x64", "bethe", "fp64", 1, 64),
        # the plain uncompressed configuration at full length, three on-site levels at once
        _case("bethe fp64 3x256", "bethe", "fp64", 3, 256),
        # a small multi-orbital impurity with fixed bath, odd length, FP64, density matrix integrated separately
        _case("bath3 fp64 2x151", "bath", "fp64", 2, 151, nao=3),
        # the level quench with compressed history in FP64: single system, tight tolerance
        _case("bethe hodlr fp64 1x384", "bethe", "fp64", 1, 384, kind="window", start=319, compressed=True),
        # the same in complex64 storage, a parameter scan that fills the device
        _case("bethe hodlr mixed 304x384", "bethe", "mixed", 304, 384, kind="window", start=319, compressed=True),
        # one driven Nambu impurity far into its propagation: the longest history, one instance
        _case("nambu hodlr mixed 1x1089", "nambu", "mixed", 1, 1089, kind="window", nao=2, start=1024, compressed=True),
        # an amplitude scan of the driven Nambu impurity, complex64 storage: the configuration of the headline number
        _case("nambu hodlr mixed 128x600", "nambu", "mixed", 128, 600, kind="window", nao=2, start=535, compressed=True),
        # its FP64 partner, eps(t) supplied and the density matrix read at every step
        _case("nambu hodlr fp64 16x300", "nambu", "fp64", 16, 300, kind="window", nao=2, start=267, compressed=True,
              per_step=True),
        # the 16 x 16 Hubbard lattice in second Born: 256 k-points coupled through Sigma, observables every step
        _case("lattice16 hodlr mixed 256x360", "lattice", "mixed", 256, 360, kind="window", start=295, compressed=True,
              per_step=True),
        # four-orbital impurities of uneven length in one batch
        _case("bath4 hodlr mixed 16x290", "bath", "mixed", 16, 290, kind="window", nao=4, start=225, compressed=True,
              uneven=True),
        # interacting equilibrium of the lattice (second Born on the imaginary axis), before any propagation
        _case("lattice16 equilibrium 256", "lattice", "fp64", 256, 16, kind="solve"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "bethe", "bethe", "nambu", "nambu", "lattice", "bath", "solve"])
    form = rng.choice(["fp64", "mixed"])
    if kind == "dense":
        nao = rng.choice([1, 1, 2, 3])
        c = _case("", "bethe" if nao == 1 else "bath", "fp64", _log(rng, 1, 6), _log(rng, 40, 260 if nao == 1 else 150),
                  nao=nao)
    elif kind == "solve":
        c = _case("", rng.choice(["lattice", "nambu"]), "fp64", 0, 16, kind="solve")
        c["nao"] = 2 if c["model"] == "nambu" else 1
        c["n_inst"] = _log(rng, 1, 128) if c["nao"] == 2 else rng.choice([4, 6, 8, 10, 12, 14, 16]) ** 2
    else:
        nt = _log(rng, 150, 520)
        steps = rng.randint(32, 64)
        c = _case("", kind, form, 1, nt, kind="window", start=nt - 1 - steps, compressed=True,
                  per_step=rng.random() < 0.3)
        if kind == "bethe":
            c["n_inst"] = _log(rng, 1, 300 if form == "mixed" else 32)
        elif kind == "nambu":
            c["nao"] = 2
            c["n_inst"] = _log(rng, 1, 100 if form == "mixed" else 12)
        elif kind == "bath":
            c["nao"] = rng.choice([2, 3, 4])
            c["n_inst"] = _log(rng, 1, 16)
            c["uneven"] = c["n_inst"] > 1 and rng.random() < 0.5
        else:
            c["n_inst"] = rng.choice([6, 8, 10, 12, 16]) ** 2
            c["form"] = "mixed"
    c.pop("name")
    return c


# ---- inputs ------------------------------------------------------------------------------------------------------

def _inputs(case, seed):
    """The workload of a case: grid, G^M, eps(t), model parameters, drive; its strengths drawn from the seed."""
    rng = np.random.default_rng(seed)
    n, nt, nao = case["n_inst"], case["nt"], case["nao"]
    if case["model"] == "bethe":
        if not case["compressed"]:
            w = wk.c1_workload(seed=seed, nt=nt, n_inst=n)
        else:
            h = 0.02
            w = wk.bethe_workload(nt=nt, h=h, n_inst=n, svd_tol=1e-8, quench=(0.0, 1.0, min(5.0, nt // 3 * h)))
            w["eps"][:, 1:, 0, 0] *= rng.uniform(0.5, 1.5, size=n)[:, None]
    elif case["model"] == "nambu":
        w = wk.c4_batch_workload(n, seed, nt=nt)
        w["drive_A"] = w["drive_A"] * rng.uniform(0.8, 1.2)
    elif case["model"] == "lattice":
        w = wk.lattice_workload(L=math.isqrt(n), nt=nt, U=rng.uniform(1.5, 2.0), A0=rng.uniform(0.1, 0.5),
                                svd_tol=1e-6, leaf=64)
    else:
        draws = []
        while len(draws) < n:
            draws += [d for d in wk.c5_draws(64, int(rng.integers(1 << 30)), nt, nt) if d["nao"] == nao]
        draws = draws[:n]
        if case["uneven"]:
            for d in draws[1:]:
                d["nt"] = int(rng.integers(case["start"] // 2 + 1, nt + 1))
        w = wk.c5_group_workload(nao, draws) if nao > 2 else _bath2(draws, nt)
        w["wl"].rho_mode = 1
    return w


def _bath2(draws, nt, h=0.02, beta=5.0):
    """Two-orbital level matrices on two bath levels (the group workload has them for three and four orbitals)."""
    tau, om = wk.dlr_grid(100.0, 1e-10, beta)
    t = np.concatenate([[0.0], np.arange(nt) * h])
    eb = wk.C5_BATH_LEVELS
    eps = np.array([d["eps0"] + (d["A0"] * np.sin(d["Omega"] * t) * (np.arange(nt + 1) > 0))[:, None, None] * np.eye(2)
                    for d in draws])
    V = [np.asarray(d["V"], complex) for d in draws]
    mp = np.array([np.concatenate([[2.0], eb, np.stack([v.real, v.imag], -1).ravel()]) for v in V])
    gm = np.array([wk.bath_gm(tau, beta, d["eps0"], v, eb) for d, v in zip(draws, V)])
    wl = wk.Workload(name="bath2", model="bath", nt=nt, h=h, k=K, beta=beta, nao=2, n_inst=len(draws), svd_tol=1e-7)
    return {"wl": wl, "tau": tau, "omega": om, "eps": eps, "gm": gm, "model_params": mp,
            "nt_per_inst": np.array([d["nt"] for d in draws], np.int32)}


def prepare(case, seed):
    w = _inputs(case, seed)
    wl = w["wl"]
    mixed = case["form"] == "mixed"
    st = pk.Stepper(case["nt"], wl.h, K, wl.beta, nao=case["nao"], n_inst=case["n_inst"], rho_mode=wl.rho_mode,
                    max_iter=80, tol=MIXED_TOL if mixed else FP64_TOL,
                    precision=pk.PREC_MIXED if mixed else pk.PREC_FP64,
                    svd_tol=wl.svd_tol if case["compressed"] else 0.0, leaf=64, r_max=64,
                    nt_per_inst=w["nt_per_inst"] if case["uneven"] else None)
    mid, mpar = pk.model_params_for(w)
    state = dict(case=case, st=st, w=w, U_eq=np.random.default_rng(seed).uniform(1.0, 1.5))
    if case["kind"] == "solve":
        st.set_inputs(w["tau"], w["omega"], None, w["eps"], mid, mpar)
        return state
    st.set_inputs(w["tau"], w["omega"], w["gm"], w["eps"], mid, mpar)
    if "drive_A" in w:
        pk.hkbe_set_drive(st.h, w["drive_A"], w["drive_U"])
    st.bootstrap()
    if case["kind"] == "window":
        st.step(case["start"] - K)
        pk.hkbe_snapshot_save(st.h)
    state["rho"] = np.zeros((case["nt"], case["n_inst"], case["nao"], case["nao"]), np.complex128)
    return state


def _early(case):
    """An older row that is read as well: in compressed storage one that the window's steps compress."""
    return case["start"] // 2 if case["uneven"] else case["start"] - 32 if case["kind"] == "window" else case["nt"] // 2


# ---- one pass ----------------------------------------------------------------------------------------------------

def run(state):
    case, st, w = state["case"], state["st"], state["w"]
    if case["kind"] == "solve":
        gm, _, _ = pk.hkbe_solve_matsubara(st.h, case["n_inst"], st.r, case["nao"], U_eq=state["U_eq"], mix=0.5,
                                           tol=1e-12, max_iter=2000)
        return {"gm": gm}
    T0, T1 = case["start"], case["nt"] - 1
    if case["kind"] == "window":
        pk.hkbe_snapshot_restore(st.h)
    else:
        pk.hkbe_rewind(st.h)
    rho = state["rho"][T0 + 1:T1 + 1]
    obs = None
    if case["per_step"]:   # a driver that computes eps(t) as it goes and records the observables
        obs = np.zeros((T1 - T0, 3))
        for i, T in enumerate(range(T0 + 1, T1 + 1)):
            pk.hkbe_set_hamiltonian_at(st.h, T, w["eps"][:, T + 1])
            st.step(1)
            pk.hkbe_get_density_at(st.h, T, rho[i])
            if case["model"] == "lattice":
                obs[i] = pk.hkbe_get_lattice_observables(st.h, T)
    else:
        st.step(T1 - T0)
        for i, T in enumerate(range(T0 + 1, T1 + 1)):
            pk.hkbe_get_density_at(st.h, T, rho[i])
    # The mixed form holds its rows in complex64: they are handed on in that type.
    dt, ft = (np.complex64, np.float32) if case["form"] == "mixed" else (np.complex128, np.float64)
    last = [int(x) - 1 for x in w["nt_per_inst"]] if case["uneven"] else [T1] * case["n_inst"]
    n, no, Te = case["n_inst"], case["nao"], _early(case)
    gr = np.zeros((n, T1 + 1, no, no), dt)
    gl = np.zeros((n, T1 + 1, no, no), dt)
    tv = np.zeros((n, st.r, no, no), dt)
    gr0 = np.zeros((n, Te + 1, no, no), dt)
    gl0 = np.zeros((n, Te + 1, no, no), dt)
    for i, T in enumerate(last):
        gr[i, :T + 1], gl[i, :T + 1] = st.row(i, T)
        tv[i] = st.tv(i, T)
        gr0[i], gl0[i] = st.row(i, Te)
    out = {"gr": gr, "gl": gl, "tv": tv, "rho": rho.astype(dt), "gr_early": gr0, "gl_early": gl0}
    if obs is not None and case["model"] == "lattice":
        out["obs"] = obs.astype(ft)
    return out


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def work(case):
    """Per corrector iteration (two of them per step at least): the Sigma^R history once for the two sweeps, the
    Sigma^< history once for the lesser source, the mixed rows once; 8 flops per complex multiply-add.  Compressed
    history: leaf triangles, the k + 1 newest rows and factors of rank sqrt(block size) / 2."""
    n, no, nt = case["n_inst"], case["nao"], case["nt"]
    r = 40
    if case["kind"] == "solve":
        return {"bytes": 2 * 16.0 * n * r * no * no, "flops": 20.0 * n * r * r * no ** 3 * 8}
    esz = 8 if case["form"] == "mixed" else 16
    elements = mixed = 0.0
    for T in range(case["start"] + 1, nt):
        if case["compressed"]:
            e = 64 * T / 2 + (K + 1) * T
            size = 64
            while size < T:
                e += 2 * T * math.sqrt(size) / 2
                size *= 2
            elements += min(e, T * T / 2)
        else:
            elements += T * T / 2
        mixed += T * r
    iters = 2
    return {"bytes": iters * n * no * no * (2 * elements * esz + 2 * mixed * 16.0),
            "flops": iters * n * no ** 3 * 8.0 * (4 * elements + 2 * mixed)}


# ---- 64-bit reference --------------------------------------------------------------------------------------------

def _lagrange(nodes, j):
    """Coefficients (rising powers) of the Lagrange polynomial of node j, exact."""
    c = [Fraction(1)]
    for x in nodes:
        if x != nodes[j]:
            d = Fraction(1, nodes[j] - x)
            c = [((c[p - 1] if p else 0) - x * (c[p] if p < len(c) else 0)) * d for p in range(len(c) + 1)]
    return c


def _area(c, a, b):
    return sum(x * (Fraction(b) ** (p + 1) - Fraction(a) ** (p + 1)) / (p + 1) for p, x in enumerate(c))


def _weight_matrices(N):
    """Bd[s, l] (derivative at s) and Wt[s, l] (integral from 0 to s) on unit spacing, rows s = 0..N-1."""
    base = [_lagrange(list(range(K + 1)), l) for l in range(K + 1)]
    D = [[float(sum(p * c[p] * Fraction(m) ** (p - 1) for p in range(1, K + 1))) for c in base] for m in range(K + 1)]
    I0 = [[float(_area(c, 0, m)) for c in base] for m in range(K + 1)]
    am = [_area(_lagrange(list(range(K + 2)), K + 1 - j), K, K + 1) for j in range(K + 2)]
    omega = [float(sum(am[:i + 1])) for i in range(K + 1)]
    M = max(N, 2 * K + 2)
    Bd, Wt = np.zeros((M, M)), np.zeros((M, M))
    for s in range(M):
        if s <= K:
            Bd[s, :K + 1], Wt[s, :K + 1] = D[s], I0[s]
            continue
        Bd[s, s - K:s + 1] = [-D[0][s - l] for l in range(s - K, s + 1)]
        if s < 2 * K + 1:
            Wt[s, :K + 1] += I0[s - K]
            Wt[s, s - K:s + 1] += I0[K]
        else:
            Wt[s, :s + 1] = 1.0
            Wt[s, :K + 1] = omega
            Wt[s, s - K:s + 1] = omega[::-1]
    return Bd[:N, :N], Wt[:N, :N]


class _Imaginary:
    """Cardinal functions l_a of the imaginary-time grid and their integrals."""

    def __init__(self, tau, om, beta):
        self.tau, self.om, self.beta = tau, om, beta
        self.K = self._kernel(tau)

    def _kernel(self, t):
        t, w = np.asarray(t)[:, None], self.om[None]
        return np.exp(-t * np.maximum(w, 0) + (self.beta - t) * np.minimum(w, 0)) / (1 + np.exp(-self.beta * abs(w)))

    def at(self, t):
        return np.linalg.solve(self.K.T, self._kernel(t).T).T

    @staticmethod
    def _nodes(a, b):
        """Gauss-Legendre panels that halve toward both ends."""
        x, w = np.polynomial.legendre.leggauss(20)
        e = np.concatenate([[0.0], 0.5 * 0.5 ** np.arange(16, -1, -1)])
        e = a + (b - a) * np.concatenate([e, 1 - e[-2::-1]])
        m, d = (e[1:] + e[:-1]) / 2, (e[1:] - e[:-1]) / 2
        return (m[:, None] + d[:, None] * x).ravel(), (d[:, None] * w).ravel()

    def product(self):
        x, w = self._nodes(0.0, self.beta)
        f = self.at(x)
        return (f * w[:, None]).T @ f

    def convolution(self, gm):
        """[a, i] = int l_a(t) G^M(t - tau_i) dt, G^M antiperiodic."""
        out = np.zeros((len(self.tau),) * 2 + gm.shape[1:], complex)
        for i, ti in enumerate(self.tau):
            for a, b, sign, shift in ((0.0, ti, -1.0, self.beta), (ti, self.beta, 1.0, 0.0)):
                x, w = self._nodes(a, b)
                out[:, i] += np.einsum("pa,pxy->axy", self.at(x) * (sign * w[:, None]),
                                       np.einsum("pc,cxy->pxy", self.at(x - ti + shift), gm))
        return out


def _dag(a):
    return np.conj(np.swapaxes(a, -1, -2))


def _solve(A, B, no):
    """A X = B for A block triangular but for its first k block rows (no: block size)."""
    c = K * no
    X = np.empty((A.shape[0], B.shape[1]), complex)
    X[:c] = np.linalg.solve(A[:c, :c], B[:c])
    if A.shape[0] > c:
        R, L = torch.from_numpy(B[c:] - A[c:, :c] @ X[:c]), torch.from_numpy(np.ascontiguousarray(A[c:, c:]))
        X[c:] = (torch.linalg.solve_triangular(L, R, upper=False) if no == 1 else torch.linalg.solve(L, R)).numpy()
    return X


class _Dense:
    """One instance: rows G^R(T, t), G^<(t, T), G^tv(T, tau); Sigma over the whole square as [t, x, l, y]."""

    def __init__(self, w, i, nt, v, bath, rho_diag):
        wl = w["wl"]
        self.h, self.no, self.nt, self.v, self.bath, self.diag = wl.h, wl.nao, nt, v, bath, rho_diag
        self.eps, self.gm = w["eps"][i], w["gm"][i]
        self.im = im = _Imaginary(w["tau"], w["omega"], wl.beta)
        self.r = r = len(w["tau"])
        self.Bd, self.Wt = _weight_matrices(nt)
        self.rev, self.e0, self.Q, self.conv = im.at(wl.beta - w["tau"]), im.at([0.0])[0], im.product(), im.convolution(self.gm)
        no = self.no
        self.SR, self.SL = np.zeros((nt, no, nt, no), complex), np.zeros((nt, no, nt, no), complex)
        self.STV, self.GTV = np.zeros((nt, r, no, no), complex), np.zeros((nt, r, no, no), complex)
        self.GR, self.GL = np.zeros((nt, nt, no, no), complex), np.zeros((nt, nt, no, no), complex)
        self.one = np.eye(no)

    def sigma(self, T):
        if self.bath is None:
            sr, sl, tv = (self.v ** 2 * x for x in (self.GR[T, :T + 1], self.GL[T, :T + 1], self.GTV[T]))
        else:
            eb, V = self.bath
            n = 0.5 * (1 - np.tanh(0.5 * self.im.beta * eb))
            ph = np.exp(1j * np.outer(np.arange(T + 1) - T, eb) * self.h)       # e^{-i eb (T - t)}
            sr = np.einsum("xb,tb,yb->txy", V, -1j * ph, V.conj())
            sl = np.einsum("xb,tb,yb->txy", V, 1j * n * ph.conj(), V.conj())
            tv = np.einsum("xb,tb,yb->txy", V, 1j * n * np.exp(np.outer(self.im.tau, eb) - 1j * eb * T * self.h), V.conj())
        for t in range(T + 1):
            self.SR[t, :, T, :] = -_dag(sr[t])
            self.SL[T, :, t, :] = -_dag(sl[t])
        self.SR[T, :, :T + 1, :] = sr.transpose(1, 0, 2)
        self.SL[:T + 1, :, T, :] = sl
        self.STV[T] = tv

    def _matrix(self, S, eps, rows, cols):
        """(i/h) Bd - eps - h Wt S on the given points, [s, x, l, y]."""
        A = -self.h * self.Wt[rows, cols][:, None, :, None] * S
        for x in range(self.no):
            A[:, x, :, x] += (1j / self.h) * self.Bd[rows, cols]
        s = np.arange(rows.start, rows.stop)
        if cols.stop >= rows.stop:
            A[s - rows.start, :, s - cols.start, :] -= eps
        return A

    def retarded(self, T):
        n, no = T + 1, self.no
        S = self.SR[T::-1, :, T::-1, :].transpose(2, 3, 0, 1)      # [s, j, l, m] = SR(T - l, T - s)[m, j]
        A = self._matrix(S[1:], np.swapaxes(self.eps[T:0:-1], 1, 2), slice(1, n), slice(0, n))
        B = 1j * A[:, :, 0, :].reshape(T * no, no)                # y_0 = -i
        Y = _solve(A[:, :, 1:].reshape(T * no, T * no), B, no).reshape(T, no, no)
        self.GR[T, T] = -1j * self.one
        self.GR[T, :T] = np.swapaxes(Y, 1, 2)[::-1]

    def mixed(self, T):
        w = self.h * self.Wt[T, :T]
        rhs = np.einsum("axy,aiyz->ixz", self.STV[T], self.conv)
        rhs += np.einsum("xly,liyz->ixz", self.SR[T, :, :T] * w[:, None], self.GTV[:T])
        rhs -= (1j / self.h) * np.einsum("l,lixy->ixy", self.Bd[T, :T], self.GTV[:T])
        M = (1j * self.Bd[T, T] / self.h) * self.one - self.eps[T + 1] - self.h * self.Wt[T, T] * self.SR[T, :, T]
        self.GTV[T] = np.linalg.solve(M, rhs)

    def source(self, T, GA, n):
        """q(t), t = 0..n-1; GA[l] = G^A(l, T)."""
        gvt = _dag(np.einsum("bc,cxy->bxy", self.rev, self.GTV[T]))
        v = np.einsum("ab,bxy->axy", self.Q, gvt)
        q = self.h * np.tensordot(self.SL[:n, :, :n], self.Wt[T, :n, None, None] * GA, ((2, 3), (0, 1)))
        return q - 1j * np.einsum("taxy,ayz->txz", self.STV[:n], v)

    def lesser(self, T, n, GA):
        """Column x(t), t = 0..n-1, all of them by the equation in t."""
        no = self.no
        q = self.source(T, GA, n)
        A = self._matrix(self.SR[1:n, :, :n], self.eps[2:n + 1], slice(1, n), slice(0, n))
        x = np.empty((n, no, no), complex)
        x[0] = -_dag(np.einsum("c,cxy->xy", self.e0, self.GTV[T]))
        B = q[1:].reshape(-1, no) - A[:, :, 0].reshape(-1, no) @ x[0]
        x[1:] = _solve(A[:, :, 1:].reshape((n - 1) * no, (n - 1) * no), B, no).reshape(n - 1, no, no)
        return x, q

    def density(self, T, x, q):
        """G^<(T, T) from the equation of motion of the density matrix."""
        no, h = self.no, self.h
        A = self.eps[T + 1] + h * self.Wt[T, T] * self.SR[T, :, T]
        r0 = q[T] + h * np.einsum("l,xly,lyz->xz", self.Wt[T, :T], self.SR[T, :, :T], x[:T])
        rhs = -(r0 + _dag(r0)) + (1j / h) * sum(self.Bd[T, l] * self.GL[l, l] for l in range(T - K, T))
        L = (self.Bd[T, T] / h) * np.eye(no * no) + 1j * (np.kron(A, self.one) - np.kron(self.one, A.conj()))
        return 1j * np.linalg.solve(L, rhs.ravel()).reshape(no, no)

    def step(self, T):
        for it in range(60):
            old = self.GR[T, :T + 1].copy(), self.GL[T, :T + 1].copy(), self.GTV[T].copy()
            if it == 0:
                for l, c in enumerate([(-1) ** l * math.comb(K + 1, l + 1) for l in range(K + 1)]):
                    self.GR[T, K + 1:T + 1] += c * self.GR[T - 1 - l, K - l:T - l]
                    self.GL[T, K + 1:T + 1] += c * self.GL[T - 1 - l, K - l:T - l]
                    self.GTV[T] += c * self.GTV[T - 1 - l]
                self.GR[T, :K + 1], self.GL[T, :K + 1] = self.GR[T - 1, :K + 1], self.GL[T - 1, :K + 1]
            self.sigma(T)
            self.retarded(T)
            self.mixed(T)
            x, q = self.lesser(T, T + 1, _dag(self.GR[T, :T + 1]))
            if self.diag:
                x[T] = self.density(T, x, q)
            self.GL[T, :T + 1] = x
            d = max(abs(a - b).max() for a, b in zip(old, (self.GR[T, :T + 1], self.GL[T, :T + 1], self.GTV[T])))
            if d < 1e-13 or (self.bath is not None and it):
                return

    def start(self):
        """Rows 0..k: mixed rows together, retarded columns in the first argument, lesser columns."""
        k, no, h, one = K, self.no, self.h, self.one
        g0 = -1j * np.einsum("bc,cxy->bxy", self.rev, self.gm)
        for t in range(k + 1):      # guess (a fixed bath needs none): free evolution of the scalar level
            ph = np.exp(-1j * self.eps[0, 0, 0] * h * np.arange(-t, 1))[::-1]
            self.GR[t, :t + 1] = -1j * ph.conj()[:, None, None] * one
            self.GL[t, :t + 1] = 0.5j * ph[:, None, None] * one
            self.GTV[t] = np.exp(-1j * self.eps[0, 0, 0] * h * t) * g0
        for it in range(200):
            old = self.GR[:k + 1].copy(), self.GL[:k + 1].copy(), self.GTV[:k + 1].copy()
            for t in range(k + 1):
                self.sigma(t)
            E = self._matrix(self.SR[1:k + 1, :, :k + 1], self.eps[2:k + 2], slice(1, k + 1), slice(0, k + 1))
            Em, E0 = E[:, :, 1:].reshape(k * no, k * no), E[:, :, 0].reshape(k * no, no)
            C = np.einsum("taxy,aiyz->txiz", self.STV[1:k + 1], self.conv).reshape(k * no, -1)
            X = np.linalg.solve(Em, C - E0 @ g0.transpose(1, 0, 2).reshape(no, -1))
            self.GTV[0], self.GTV[1:k + 1] = g0, X.reshape(k, no, self.r, no).transpose(0, 2, 1, 3)
            self.GR[k, k] = -1j * one
            for c in range(k):      # column c: the integral runs from c to m
                self.GR[c, c] = -1j * one
                W = self.Wt[:k + 1, :k + 1] - self.Wt[c, :k + 1]
                A = -h * W[:, None, :, None] * self.SR[:k + 1, :, :k + 1]
                for x in range(no):
                    A[:, x, :, x] += (1j / h) * self.Bd[:k + 1, :k + 1]
                for m in range(k + 1):
                    A[m, :, m, :] -= self.eps[m + 1]
                known = np.array([-_dag(self.GR[c, l]) if l < c else self.GR[l, c] for l in range(c + 1)]).reshape(-1, no)
                rhs = -A[c + 1:, :, :c + 1].reshape((k - c) * no, -1) @ known
                Y = np.linalg.solve(A[c + 1:, :, c + 1:].reshape((k - c) * no, -1), rhs)
                self.GR[c + 1:k + 1, c] = Y.reshape(k - c, no, no)
            for m in range(k + 1):
                GA = np.array([_dag(self.GR[m, l]) if l <= m else -self.GR[l, m] for l in range(k + 1)])
                x, _ = self.lesser(m, k + 1, GA)
                self.GL[m, :m + 1] = x[:m + 1]
            d = max(abs(a - b).max() for a, b in zip(old, (self.GR[:k + 1], self.GL[:k + 1], self.GTV[:k + 1])))
            if d < 1e-14 or (self.bath is not None and it >= 2):
                break
        for t in range(k + 1):
            self.sigma(t)


def exact(case, seed):
    n, nt, no = case["n_inst"], case["nt"], case["nao"]
    if case["kind"] == "solve" or case["model"] not in ("bethe", "bath"):
        return None               # hundreds of coupled instances, or two-orbital histories of a thousand steps
    cost = n * nt ** 3 * (2e-7 if no == 1 else 3.5e-8 * no ** 3)
    if cost > 12:                 # seconds, about
        return None
    w = _inputs(case, seed)
    diag = w["wl"].rho_mode == 1
    last = w["nt_per_inst"] - 1 if case["uneven"] else np.full(n, nt - 1)
    T0 = case["start"]
    out = {"gr": np.zeros((n, nt, no, no), complex), "gl": np.zeros((n, nt, no, no), complex), "tv": [],
           "rho": np.zeros((nt - 1 - T0, n, no, no), complex), "gr_early": [], "gl_early": []}
    for i in range(n):
        p = w["model_params"][i]
        bath = None
        if case["model"] == "bath":
            nb = int(p[0])
            bath = p[1:1 + nb], p[1 + nb:].view(complex).reshape(no, nb)
        d = _Dense(w, i, int(last[i]) + 1, p[0], bath, diag)
        d.start()
        for T in range(K + 1, last[i] + 1):
            d.step(T)
        out["gr"][i, :last[i] + 1], out["gl"][i, :last[i] + 1] = d.GR[last[i]], d.GL[last[i]]
        out["tv"].append(d.GTV[last[i]])
        out["gr_early"].append(d.GR[_early(case), :_early(case) + 1])
        out["gl_early"].append(d.GL[_early(case), :_early(case) + 1])
        for j, T in enumerate(range(T0 + 1, last[i] + 1)):
            out["rho"][j, i] = -1j * d.GL[T, T]
    return {k: np.array(v) for k, v in out.items()}
