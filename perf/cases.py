"""The work that a program using this library has it do, as sized cases.

Every case goes through the binding's public calls.  A pass of most cases resumes
checkpointed states (``State.import_``), advances them (``State.step`` or
``Group.step``) and reads the observables back, as a preempted or monitored solve, a
sweep and a served request do.  One case reads many results from a state without
advancing it, and one admits a new solve: operators, start state, first steps.

The states are made here from the seed alone, in numpy: a purification of a few
weighted vectors, each a superposition of coherent states of every mode (for the
transmon, of its low levels with a displaced resonator), cut into right-canonical
sites at the solve's own relative weight and laid out as ``State.export`` does.
Systems, mode sizes, cutoffs and caps are those of this package's configurations
(`inputs`) and of their check sizes; the cat's time step is the smaller of 1e-3 and
1.6 / N^2, inside the stability bound of the explicit scheme.

A state's sites are fixed only up to a unitary on every bond, so what comes back is
what a program reads: the observables of every state.  The FP64 and the double-float (mixed) form are both in use; the three-pass TF32 form
is not listed, as its products carry no more than 21 bits and its results move by
more than the other forms' errors with any change of an operand's last bits.
"""
from __future__ import annotations

import functools
import struct

import numpy as np
import torch

from paper_2605_27515_gb300 import inputs
from paper_2605_27515_gb300 import qlb as Q
from paper_2605_27515_gb300 import systems

PRECISION = {"f64": Q.PREC_F64, "mixed": Q.PREC_MIXED}


def _case(name, work, system, R, precision, steps, chi=64, chi_mu=16, tol=1e-12, rank=6, terms=3, members=1):
    """R: the configuration's mode sizes log2 N, comma-separated; rank: weighted
    vectors of the start's purification; terms: product terms of each."""
    c = dict(work=work, system=system, R=R, precision=precision, steps=steps, chi=chi, chi_mu=chi_mu, tol=tol,
             rank=rank, terms=terms, members=members)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest solve (the size of the smoke run), one step at a time with its
        # observables read after each: launches and host latency
        _case("cat N=8 monitored", "steps", "cat", "3", "f64", 1, chi_mu=8, rank=2, terms=1),
        # the small cat of the configurations at its own caps, both forms
        _case("cat N=32", "steps", "cat", "5", "f64", 2, chi_mu=8, rank=4),
        _case("cat N=32 mixed", "steps", "cat", "5", "mixed", 4, chi_mu=8, rank=4),
        # the large cat at its check size and at its full size
        _case("cat N=128 mixed", "steps", "cat", "7", "mixed", 2),
        _case("cat N=512 mixed", "steps", "cat", "9", "mixed", 2),
        _case("cat N=512", "steps", "cat", "9", "f64", 1),
        # memory and buffer of the gate experiment (two modes, loose cutoff)
        _case("z_gate N=64x16", "steps", "z_gate", "6,4", "f64", 2, tol=1e-8),
        # driven transmon and resonator at full size: 17 sites, two branches, wide bonds
        _case("transmon 128x1024", "steps", "transmon", "7,10", "f64", 1, chi=128, rank=4, terms=2),
        # two coupled cats with buffers (four modes, five branches) at their check size
        _case("cat_pair 4x8x8x4", "steps", "cat_pair", "3,2,3,2", "mixed", 1, rank=4, terms=2),
        # a bucket of served requests: one group, capped bonds
        _case("served bucket of 12", "group", "cat", "7", "mixed", 2, chi=32, chi_mu=8, rank=4, members=12),
        # everything a program reads from one state: expectation values, fidelity,
        # purity, trace
        _case("read a 17-site state", "read", "transmon", "7,10", "f64", 0, chi=128, rank=8, terms=4),
        # a new solve as the serving admission makes it
        _case("admit cat N=64", "admit", "cat", "6", "mixed", 2, chi=48, chi_mu=8),
    ]


def draw(rng):
    work = rng.choice(["steps", "steps", "steps", "steps", "steps", "group", "read", "admit"])
    if work == "group":
        return _case(None, work, "cat", str(rng.randint(5, 7)), "mixed", rng.randint(1, 2), chi=rng.choice([24, 32]),
                     chi_mu=8, rank=rng.randint(2, 4), terms=rng.randint(2, 3), members=rng.randint(2, 12))
    if work == "admit":
        return _case(None, work, "cat", str(rng.randint(4, 6)), rng.choice(["f64", "mixed"]), rng.randint(1, 2),
                     chi=rng.choice([32, 48, 64]), chi_mu=rng.randint(4, 8))
    system = rng.choice(["cat", "cat", "z_gate", "transmon", "cat_pair"]) if work == "steps" else rng.choice(
        ["cat", "transmon"])
    if system == "cat":
        R = rng.randint(3, 9)
        precision = rng.choice(["f64", "mixed"])
        return _case(None, work, "cat", str(R), precision, 0 if work == "read" else rng.randint(1, 1 if R > 7 else 3),
                     chi=rng.randint(20, 64), chi_mu=rng.randint(6, 16), rank=rng.randint(2, 6),
                     terms=rng.randint(1, 3))
    if system == "z_gate":
        return _case(None, work, "z_gate", "%d,%d" % (rng.randint(4, 7), rng.randint(2, 4)), "f64", 1,
                     chi=rng.randint(32, 64), tol=1e-8, rank=rng.randint(2, 6), terms=rng.randint(2, 3))
    if system == "transmon":
        return _case(None, work, "transmon", "%d,%d" % (rng.randint(5, 7), rng.randint(6, 10)), "f64",
                     0 if work == "read" else 1, chi=rng.choice([96, 128]), rank=rng.randint(2, 4),
                     terms=rng.randint(1, 2))
    return _case(None, work, "cat_pair", rng.choice(["3,2,3,2", "3,2,2,2", "3,3,3,2"]), "mixed", 1,
                 chi=rng.randint(40, 64), rank=rng.randint(2, 4), terms=rng.randint(1, 2))


# ---------------------------------------------------------------- systems


def _config(case):
    """This package's parameter set of the case's system at the case's mode sizes."""
    cfg = inputs.config("cat_r9" if case["system"] == "cat" else case["system"])
    cfg["R"] = [int(r) for r in case["R"].split(",")]
    if case["system"] == "cat":
        N = 2 ** cfg["R"][0]
        cfg["alpha2"] = min(32.0, N / 8.0)
        cfg["dt"] = min(1e-3, 1.6 / N ** 2)
    elif case["system"] == "transmon":
        cfg["dt"] = 2e-6 * max(1.0, 1024 / 2 ** cfg["R"][1])
    return cfg


def _modes(case, cfg):
    """log2 of the mode sizes in the system's own mode order."""
    R = cfg["R"]
    return [R[1], R[0], R[2], R[3]] if case["system"] == "cat_pair" else R


def _drive(cfg):
    """The resonator drive on the plateau of its ramp."""
    return cfg["eps_over_kappa"] * cfg["kappa"]


def _context(case):
    return Q.Ctx(device=0, precision=PRECISION[case["precision"]], tol=case["tol"], chi_max=case["chi"],
                 chi_mu_max=case["chi_mu"])


@functools.lru_cache(maxsize=1)
def _system(key):
    """Context, system and operators, which a program makes once for all its states."""
    case = dict(key)
    ctx, cfg = _context(case), _config(case)
    if case["system"] == "transmon":
        b = systems.build_transmon(ctx, cfg, nsteps=1)
        b.sys.set_hamiltonian(b.ops["H0"], b.ops["H1"], np.full(1 << 20, _drive(cfg)))
    else:
        b = systems.build(ctx, cfg)
    return ctx, b, cfg


# ---------------------------------------------------------------- inputs


def _coherent(N, beta):
    n = np.arange(N)
    logs = np.concatenate([[0.0], np.cumsum(np.log(np.arange(1, N)))])
    r = abs(beta)
    return np.exp(n * np.log(max(r, 1e-300)) - 0.5 * logs - 0.5 * r * r + 1j * n * np.angle(beta))


def _disc(rng, radius):
    return radius * np.sqrt(rng.uniform()) * np.exp(2j * np.pi * rng.uniform())


def _transmon_levels(N, cfg):
    n = np.arange(N) - N // 2
    ej = cfg["ej_over_ec"] * cfg["ec"]
    H = np.diag(4 * cfg["ec"] * n.astype(float) ** 2) - 0.5 * ej * (np.eye(N, k=1) + np.eye(N, k=-1))
    v = np.linalg.eigh(H)[1][:, :4]
    return v * np.sign(v[N // 2] + v[N // 2 + 1])


def _product(case, cfg, rng):
    """One product term of a purification vector: a vector of every mode."""
    N = [2 ** r for r in _modes(case, cfg)]
    if case["system"] == "cat":
        return [_coherent(N[0], _disc(rng, np.sqrt(cfg["alpha2"])))]
    if case["system"] == "z_gate":
        return [_coherent(N[0], _disc(rng, np.sqrt(N[0] / 4.0))), _coherent(N[1], _disc(rng, 0.4))]
    if case["system"] == "transmon":
        c = rng.normal(size=4) * np.array([1.0, 0.3, 0.1, 0.03])
        return [_transmon_levels(N[0], cfg) @ c, _coherent(N[1], _disc(rng, np.sqrt(N[1] / 8.0)))]
    return [_coherent(N[0], _disc(rng, 0.3)), _coherent(N[1], _disc(rng, np.sqrt(N[1] / 5.0))),
            _coherent(N[2], _disc(rng, np.sqrt(N[2] / 5.0))), _coherent(N[3], _disc(rng, 0.3))]


def _kron(vectors):
    return functools.reduce(np.kron, vectors)


def _purification(case, cfg, rng):
    """(mu, 2^L): the rows sqrt(p_k) psi_k of a mixed state, weights falling as 10^-1.2 k."""
    rows = []
    for k in range(case["rank"]):
        psi = sum((rng.normal() + 1j * rng.normal()) * _kron(_product(case, cfg, rng)) for _ in range(case["terms"]))
        rows.append(psi / np.linalg.norm(psi) * 10.0 ** (-0.6 * k))
    P = np.array(rows)
    return P / np.linalg.norm(P)


def _sites(P, L, tol, chi, chi_mu):
    """Right-canonical sites [left][s][right]; the first carries the purification index."""
    out = []
    T, r = P, 1
    for _ in range(L - 1):
        T = T.reshape(-1, 2 * r)
        w, V = np.linalg.eigh(T.conj().T @ T)
        w, V = np.maximum(w[::-1], 0.0), V[:, ::-1]
        tail = np.cumsum(w[::-1])[::-1]
        k = max(1, min(chi, int(np.sum(tail > tol * tail[0]))))
        out.append(np.ascontiguousarray(V[:, :k].conj().T).reshape(k, 2, r))
        T, r = T @ V[:, :k], k
    A = T.reshape(-1, 2 * r)
    Y = np.linalg.eigh(A @ A.conj().T)[1][:, ::-1][:, :chi_mu]
    A = Y.conj().T @ A
    out.append((A / np.linalg.norm(A)).reshape(-1, 2, r))
    return out[::-1]


def _start(case, seed, member=0):
    cfg = _config(case)
    rng = np.random.default_rng([int(seed), member])
    return _sites(_purification(case, cfg, rng), sum(cfg["R"]), case["tol"], case["chi"], case["chi_mu"])


def _checkpoint(cores):
    """The sites in the layout of ``State.export``."""
    d = [c.shape[0] for c in cores] + [1]
    return struct.pack("<Qii", 0x31424C51, len(cores), 0) + np.array(d, np.int32).tobytes() + b"".join(
        np.ascontiguousarray(c, dtype=np.complex128).tobytes() for c in cores)


def _admission(case, seed):
    """Parameters and start vectors of a new solve."""
    cfg = _config(case)
    rng = np.random.default_rng([int(seed), 1])
    cfg["alpha2"] *= rng.uniform(0.5, 1.0)
    cfg["k1"] = float(10 ** rng.uniform(-4.0, -2.0))
    return cfg, [_coherent(2 ** r, _disc(rng, np.sqrt(cfg["alpha2"]))) for r in cfg["R"]]


# ---------------------------------------------------------------- the cases


class _Held:
    """What a program holds between passes."""

    def __init__(self, case, seed):
        self.case = case
        self.group, self.states, self.blobs = None, [], []
        if case["work"] == "admit":
            self.ctx = _context(case)
            self.cfg, self.start = _admission(case, seed)
            return
        key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "steps", "members", "rank", "terms", "work")))
        self.ctx, self.b, self.cfg = _system(key)
        for m in range(case["members"]):
            self.blobs.append(_checkpoint(_start(case, seed, m)))
            self.states.append(self.b.sys.state(self.b.init))
            self.states[m].import_(self.blobs[m])
        if case["work"] == "group":
            self.group = Q.Group(self.ctx, self.states)
        if case["work"] == "read":
            self.target = _target(case, seed)
            for st in self.states:
                self.ops = list(self.b.observables.values()) + [self.b.ops["H0"] if "H0" in self.b.ops else self.b.ops["H"]]
        else:
            self.ops = list(self.b.observables.values())
            self._advance()

    def _advance(self):
        for st, blob in zip(self.states, self.blobs):
            st.import_(blob)
        if self.group:
            self.group.step(self.cfg["dt"], self.case["steps"])
        else:
            self.states[0].step(self.cfg["dt"], self.case["steps"])

    def __del__(self):
        if self.group:
            self.group.close()
        for st in self.states:
            st.close()


def _target(case, seed):
    """Product target of the fidelity: the first product term of the state's leading vector."""
    cfg = _config(case)
    rng = np.random.default_rng([int(seed), 0])
    rng.normal(), rng.normal()
    return _product(case, cfg, rng)


def prepare(case, seed):
    return _Held(case, seed)


def run(s):
    work = s.case["work"]
    if work == "admit":
        b = systems.build(s.ctx, s.cfg)
        st = b.sys.state(s.start)
        st.step(s.cfg["dt"], s.case["steps"])
        out = np.array([st.expectation(o).real for o in b.observables.values()])
        st.close()
        for o in list(b.ops.values()) + list(b.observables.values()):
            o.close()
        b.sys.close()
        return {"observables": out}
    if work == "read":
        st = s.states[0]
        return {"observables": np.array([st.expectation(o).real for o in s.ops]), "purity": st.purity(),
                "trace": st.trace(), "fidelity": st.fidelity(s.target)}
    s._advance()
    return {"observables": np.array([[st.expectation(o).real for o in s.ops] for st in s.states])}


def work(case):
    """One read of the sites and operators and one write of the sites per step; the
    products that apply an operator of bond 8 (the rank of a) per branch and term, and
    one Gram matrix and one triangular factorisation of every bond."""
    if case["work"] == "admit":
        case = dict(case, rank=1, terms=1)
    cores = _start(dict(case, members=1), 0)
    d = np.array([c.shape[0] for c in cores] + [1], dtype=float)
    branches = {"cat": 3, "z_gate": 2, "transmon": 2, "cat_pair": 5}[case["system"]]
    D = 8.0
    entries = float(np.sum(2 * d[:-1] * d[1:]))
    mpo = 4 * D * D * (len(d) - 1)
    passes = max(1, case["steps"]) * case["members"]
    contract = float(np.sum(8 * (2 * d[:-1] * d[1:] * D * d[:-1] + 4 * d[:-1] * d[1:] * D * D)))
    truncate = float(np.sum(8 * ((2 * d[1:]) ** 2 * d[:-1] + (2 * d[1:]) ** 3 / 3)))
    if case["work"] == "read":
        n = 4
        return {"bytes": 16 * (entries + n * mpo), "flops": n * contract}
    return {"bytes": passes * 16 * (2 * entries + mpo), "flops": passes * (contract * (1 + (branches - 1) / 8) + truncate)}


# ---------------------------------------------------------------- exact values


class _Dense:
    """The case's operators applied to columns of length 2^L, in complex128."""

    def __init__(self, case, cfg):
        self.dims = N = [2 ** r for r in _modes(case, cfg)]
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"

        def dev(x):
            return torch.as_tensor(np.asarray(x, dtype=np.complex128)).to(self.dev)

        a = [dev(np.diag(np.sqrt(np.arange(1.0, n)), 1)) for n in N]
        ad = [x.conj().T.contiguous() for x in a]
        num = [dev(np.diag(np.arange(float(n)))) for n in N]
        par = [dev(np.diag((-1.0) ** np.arange(n))) for n in N]
        if case["system"] == "cat":
            k2 = np.sqrt(cfg["k2"])
            self.H = [(cfg["eps_z"], {0: a[0] + ad[0]})]
            self.Ls = [[(k2, {0: a[0] @ a[0]}), (-k2 * cfg["alpha2"], {})], [(np.sqrt(cfg["k1"]), {0: a[0]})]]
            self.obs = [[(1.0, {0: num[0]})], [(1.0, {0: par[0]})]]
        elif case["system"] == "z_gate":
            eps_d, eps_z = -cfg["g2"] * N[0] / 3.0, 0.4 * cfg["g2"] ** 2 / cfg["kb"]
            self.H = [(cfg["g2"], {0: ad[0] @ ad[0], 1: a[1]}), (cfg["g2"], {0: a[0] @ a[0], 1: ad[1]}),
                      (eps_d, {1: a[1] + ad[1]}), (eps_z, {0: a[0] + ad[0]})]
            self.Ls = [[(np.sqrt(cfg["kb"]), {1: a[1]})]]
            self.obs = [[(1.0, {0: par[0]})], [(1.0, {0: num[0]})], [(1.0, {1: num[1]})]]
        elif case["system"] == "transmon":
            ec, ej, g = cfg["ec"], cfg["ej_over_ec"] * cfg["ec"], cfg["g_over_ec"] * cfg["ec"]
            charge = np.arange(N[0]) - float(N[0] // 2)
            cos_phi = 0.5 * (np.eye(N[0], k=1) + np.eye(N[0], k=-1))
            x = a[1] + ad[1]
            H0 = [(1.0, {0: dev(np.diag(4 * ec * charge ** 2) - ej * cos_phi)}), (cfg["wr"], {1: num[1]}),
                  (g, {0: dev(np.diag(charge)), 1: x})]
            self.H = H0 + [(_drive(cfg), {1: x})]
            self.Ls = [[(np.sqrt(cfg["kappa"]), {1: a[1]})]]
            self.obs = [[(1.0, {1: num[1]})], [(1.0, {0: dev(np.diag(charge ** 2))})]]
        else:  # buffer, storage, storage, buffer
            g2, eb, J = cfg["g2"], -cfg["g2"] * cfg["alpha2"], cfg["J"]
            self.H = [(J, {1: ad[1], 2: a[2]}), (J, {2: ad[2], 1: a[1]})]
            for m, b in ((1, 0), (2, 3)):
                self.H += [(g2, {m: a[m] @ a[m], b: ad[b]}), (g2, {m: ad[m] @ ad[m], b: a[b]}), (eb, {b: a[b] + ad[b]})]
            rates = [(0, cfg["kb"]), (3, cfg["kb"]), (1, cfg["k1"]), (2, cfg["k1"])]
            self.Ls = [[(np.sqrt(k), {m: a[m]})] for m, k in rates]
            self.obs = [[(1.0, {1: num[1]})], [(1.0, {2: num[2]})], [(1.0, {1: par[1]})]]
        if case["work"] == "read":
            self.obs = self.obs + [H0 if case["system"] == "transmon" else self.H]

    def apply(self, terms, X, dagger=False):
        out = torch.zeros_like(X)
        for c, factors in terms:
            Z = X.reshape(*self.dims, -1)
            for m, A in factors.items():
                Z = torch.movedim(torch.tensordot(A.conj().T if dagger else A, Z, dims=([1], [m])), 0, m)
            out = out + c * Z.reshape(X.shape)
        return out

    def step(self, X, h):
        """One first-order Kraus step on the columns X of a purification, renormalised."""
        U = X - 1j * h * self.apply(self.H, X)
        parts = []
        for L in self.Ls:
            LX = self.apply(L, X)
            U = U - 0.5 * h * self.apply(L, LX, dagger=True)
            parts.append(np.sqrt(h) * LX)
        X = torch.cat([U] + parts, dim=1)
        return X / torch.linalg.norm(X)

    def observables(self, X):
        return np.array([float(torch.sum(X.conj() * self.apply(o, X)).real) for o in self.obs])


def _columns(cores):
    """The purification that the sites hold, as columns of length 2^L."""
    mu = cores[0].shape[0]
    T = cores[0].reshape(2 * mu, -1)
    for c in cores[1:]:
        T = (T @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    return np.ascontiguousarray(T.reshape(mu, -1).T)


def exact(case, seed):
    if case["work"] == "admit":
        cfg, start = _admission(case, seed)
        v = _kron(start)
        columns = [(v / np.linalg.norm(v)).reshape(-1, 1)]
    else:
        cfg = _config(case)
        columns = [_columns(_start(case, seed, m)) for m in range(case["members"])]
    ops = _Dense(case, cfg)
    columns = [torch.from_numpy(c).to(ops.dev) for c in columns]
    if case["work"] == "read":
        X = columns[0]
        G = X.conj().T @ X
        v = _kron(_target(case, seed))
        v = torch.from_numpy(v / np.linalg.norm(v)).to(ops.dev)
        tr = float(torch.trace(G).real)
        return {"observables": ops.observables(X), "purity": float(torch.sum(G.abs() ** 2)) / tr ** 2, "trace": tr,
                "fidelity": float(torch.sum((v.conj() @ X).abs() ** 2))}
    rows = []
    for X in columns:
        for _ in range(case["steps"]):
            X = ops.step(X, cfg["dt"])
        rows.append(ops.observables(X))
    return {"observables": rows[0] if case["work"] == "admit" else np.array(rows)}
