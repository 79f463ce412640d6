"""What a program asks of this package, as cases whose time can be taken.

Every case goes through the public entry points of ``paper_1109_1205_gb300``
on synthetic model Hamiltonians: the Hubbard ring (one hopping amplitude), the
chain and the star of a single-impurity Anderson model (the star: one real
amplitude per bond) and a fully connected random cluster with complex hopping.
All data are FP64 / complex FP64.  Sizes follow the workloads of this
repository: L = 6 to 16 sites, d = 300 to 9.2e7 states per vector, M = 20 or
40 Krylov vectors per step.

``exact`` computes the same results with torch in FP64 from the model alone:
spin strings in numeric order, Jordan-Wigner signs, Lanczos with full
orthogonalisation for the ground state and Taylor sub-steps for e^{-iHt}.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1109_1205_gb300 as kg


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: H applied to a vector of a 10-site star (an
        # iterative solver of the caller's own around it)
        {"name": "hpsi_star10", "kind": "hpsi", "model": "star", "L": 10, "n_up": 5, "n_dn": 5},
        # H applied to one column of the 12-site ring's Keldysh calculation
        {"name": "hpsi_ring12", "kind": "hpsi", "model": "ring", "L": 12, "n_up": 5, "n_dn": 6},
        # the largest vectors: one column of the 16-site chain (1.5 GB each)
        {"name": "hpsi_chain16", "kind": "hpsi", "model": "chain", "L": 16, "n_up": 6, "n_dn": 7},
        # time evolution of a state on a small cluster with complex hopping
        {"name": "propagate_random8", "kind": "propagate", "model": "random", "L": 8, "n_up": 4, "n_dn": 4,
         "M": 20, "dt": 0.05, "n_steps": 10},
        # time evolution of one state of the half-filled 12-site ring
        {"name": "propagate_ring12", "kind": "propagate", "model": "ring", "L": 12, "n_up": 6, "n_dn": 6,
         "M": 20, "dt": 0.05, "n_steps": 5},
        # G(t) of a small impurity model, 401 times (the 6-site star, M = 40)
        {"name": "green_star6", "kind": "green", "model": "star", "L": 6, "n_up": 3, "n_dn": 3, "M": 40, "dt": 0.05,
         "n_steps": 400, "n_orb": 1},
        # one impurity solve of an embedding loop, from the parameters on:
        # tables, ground state and G(t) of the 10-site star
        {"name": "solve_star10", "kind": "solve", "model": "star", "L": 10, "n_up": 5, "n_dn": 5, "M": 20, "dt": 0.05,
         "n_steps": 100, "n_orb": 1},
        # G(t,t') after a local quench on a short chain, both spins
        {"name": "keldysh_chain8", "kind": "keldysh", "model": "chain", "L": 8, "n_up": 4, "n_dn": 4, "M": 20,
         "dt": 0.1, "n_t": 10, "n_orb": 2},
        # rows and Gram matrix of the 12-site ring's quench, all 12 orbitals
        {"name": "keldysh_ring12", "kind": "staged", "model": "ring", "L": 12, "n_up": 6, "n_dn": 6, "M": 20,
         "dt": 0.05, "n_t": 4, "n_orb": 12},
        # many impurity models of uneven size solved together
        {"name": "batched_star", "kind": "batched", "model": "star", "n_inst": 48, "L_min": 6, "L_max": 10, "M": 20,
         "dt": 0.05, "n_steps": 60},
        # a training step: G(t) of a 10-site star and the gradient of a loss
        # of it with respect to every parameter
        {"name": "gradient_star10", "kind": "gradient", "model": "star", "L": 10, "n_up": 5, "n_dn": 5, "M": 20,
         "dt": 0.05, "n_steps": 40},
        # spectra from two long series (dt = 0.01 to t = 1000)
        {"name": "fourier_100k", "kind": "fourier", "n_series": 2, "n_t": 100001, "n_omega": 4001, "dt": 0.01,
         "eta": 0.01},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _filling(rng, L, off=1):
    return max(1, min(L - 1, L // 2 + rng.randint(-off, off)))


def draw(rng):
    kind = rng.choice(["hpsi", "hpsi", "propagate", "propagate", "green", "solve", "keldysh", "staged", "batched",
                       "gradient", "fourier"])
    model = rng.choice(["ring", "chain", "star", "random"])
    dt = rng.choice([0.02, 0.05, 0.1])
    if kind == "hpsi":
        L = rng.randint(6, 15)
        if model == "random":
            L = min(L, 12)
        return {"kind": kind, "model": model, "L": L, "n_up": _filling(rng, L), "n_dn": _filling(rng, L)}
    if kind == "propagate":
        L = rng.randint(5, 12 if model in ("ring", "chain") else 11)
        return {"kind": kind, "model": model, "L": L, "n_up": _filling(rng, L), "n_dn": _filling(rng, L),
                "M": rng.randint(12, 40) if L < 11 else rng.randint(12, 24), "dt": rng.choice([-1, 1]) * min(dt, 0.05),
                "n_steps": rng.randint(1, 12) if L < 11 else rng.randint(1, 4)}
    if kind in ("green", "solve"):
        L = rng.randint(5, 10) if kind == "green" else rng.randint(6, 10)
        if model == "ring":
            L -= L % 2  # half filling of an odd ring is degenerate
        return {"kind": kind, "model": model, "L": L, "n_up": L // 2, "n_dn": L // 2, "M": rng.randint(16, 40),
                "dt": min(dt, 0.05), "n_steps": _log_int(rng, 10, 400 if L < 9 else 60), "n_orb": rng.randint(1, 3)}
    if kind == "keldysh":
        L = rng.randint(5, 9)
        return {"kind": kind, "model": rng.choice(["chain", "star"]), "L": L, "n_up": L // 2, "n_dn": L // 2,
                "M": rng.randint(16, 24), "dt": dt, "n_t": rng.randint(2, 12), "n_orb": rng.randint(1, 4)}
    if kind == "staged":
        L = rng.choice([8, 10, 12])
        return {"kind": kind, "model": "ring", "L": L, "n_up": L // 2, "n_dn": L // 2, "M": rng.randint(16, 22),
                "dt": min(dt, 0.05), "n_t": rng.randint(2, 3) if L == 12 else rng.randint(3, 6),
                "n_orb": rng.randint(2, min(L, 9))}
    if kind == "batched":
        lo = rng.randint(5, 7)
        return {"kind": kind, "model": "star", "n_inst": _log_int(rng, 4, 48), "L_min": lo,
                "L_max": lo + rng.randint(1, 10 - lo), "M": 20, "dt": min(dt, 0.05), "n_steps": _log_int(rng, 10, 60)}
    if kind == "gradient":
        L = rng.randint(6, 9)
        return {"kind": kind, "model": "star", "L": L, "n_up": L // 2, "n_dn": L // 2, "M": 20, "dt": min(dt, 0.05),
                "n_steps": _log_int(rng, 10, 60)}
    return {"kind": kind, "n_series": rng.randint(1, 4), "n_t": _log_int(rng, 300, 50000),
            "n_omega": _log_int(rng, 50, 4001), "dt": rng.choice([0.01, 0.02, 0.05]), "eta": rng.choice([0.01, 0.05, 0.1])}


# ------------------------------------------------------------------ models
def _model(name, L, seed, field=0.0, scale_U=1.0, n_up=0, n_dn=0):
    """h (L x L), eps (2 x L), U (L): the model `name` with seeded parameters."""
    r = np.random.default_rng(seed)
    h = np.zeros((L, L), dtype=np.complex128)
    eps = np.zeros((2, L))
    U = np.zeros(L)
    u0 = float(r.uniform(4.0, 8.0)) * scale_U
    if name == "ring":  # T = 1, periodic
        for i in range(L):
            h[i, (i + 1) % L] = h[(i + 1) % L, i] = -1.0
        U[:] = u0
    elif name == "chain":  # impurity at site 0 of an open chain, T = 1
        for i in range(L - 1):
            h[i, i + 1] = h[i + 1, i] = -1.0
        U[0] = u0
        eps[:, 0] = -u0 / 2
    elif name == "star":  # impurity 0 coupled to each bath site
        h[0, 1:] = h[1:, 0] = r.uniform(0.2, 1.0, L - 1)
        eps[:, 1:] = r.uniform(-3.0, 3.0, L - 1)
        U[0] = u0
        eps[:, 0] = -u0 / 2
    else:  # fully connected, complex Hermitian
        a = r.uniform(-1, 1, (L, L)) + 1j * r.uniform(-1, 1, (L, L))
        h = 0.5 * (a + a.conj().T)
        np.fill_diagonal(h, 0.0)
        eps = r.uniform(-1, 1, (2, L))
        U = r.uniform(0, 4, L)
    eps[0, 0] -= field
    eps[1, 0] += field
    return {"L": L, "n_up": n_up, "n_dn": n_dn, "h": h, "eps": eps, "U": U}


def _case_model(case, seed, **kw):
    return _model(case["model"], case["L"], seed, n_up=case["n_up"], n_dn=case["n_dn"], **kw)


def _pair(case, seed):
    """Initial and final Hamiltonian of a quench: U halved on the ring, the
    local field h = 2 switched off on the chain and the star."""
    if case["model"] == "ring":
        return _case_model(case, seed, scale_U=2.0), _case_model(case, seed)
    return _case_model(case, seed, field=2.0), _case_model(case, seed)


def _instances(case, seed):
    r = np.random.default_rng(seed)
    out = []
    for i in range(case["n_inst"]):
        L = int(r.integers(case["L_min"], case["L_max"] + 1))
        nu, nd = int(r.integers(1, L)), int(r.integers(1, L))
        out.append(_model("star", L, [seed, i], n_up=nu, n_dn=nd))
    return out


def _orbitals(case):
    n, L = case["n_orb"], case["L"]
    if case["kind"] == "staged":
        return [(i % L, 0) for i in range(n)]
    return [(a // 2, a % 2) for a in range(n)]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _vector(d, seed):
    g = torch.Generator(device=_device()).manual_seed(int(seed))
    v = torch.randn(d, dtype=torch.complex128, device=_device(), generator=g)
    return v / torch.linalg.vector_norm(v)


def _series(case, seed):
    """G(t)-like series: eight poles with normalised weights each."""
    r = np.random.default_rng(seed)
    t = np.arange(case["n_t"]) * case["dt"]
    out = np.zeros((case["n_series"], case["n_t"]), dtype=np.complex128)
    for s in range(case["n_series"]):
        E, w = r.uniform(-8, 8, 8), r.uniform(0, 1, 8)
        for e, x in zip(E, w / w.sum()):
            out[s] += -1j * x * np.exp(-1j * e * t)
    return out, np.linspace(-10, 10, case["n_omega"])


def _cotangents(case, seed):
    r = np.random.default_rng([seed, 3])
    n = case["n_steps"] + 1
    return [torch.from_numpy(r.standard_normal((n, 1, 1)) + 1j * r.standard_normal((n, 1, 1))).to(_device())
            for _ in range(2)]


# ----------------------------------------------------------------- the runs
def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "hpsi":
        s = kg.Sector(_case_model(case, seed))
        st.update(sector=s, x=_vector(s.dim, seed), y=torch.empty(s.dim, dtype=torch.complex128, device="cuda"))
    elif kind == "propagate":
        s = kg.Sector(_case_model(case, seed))
        st.update(sector=s, x0=_vector(s.dim, seed), opts=kg.kg_opts_default(M=case["M"]))
        st["x"] = torch.empty_like(st["x0"])
    elif kind == "green":  # the ground state is in hand, as in a scan over orbitals and grids
        s = kg.Sector(_case_model(case, seed))
        s.ground_state()
        st.update(sector=s, orb=_orbitals(case), opts=kg.kg_opts_default(M=case["M"]))
    elif kind == "solve":
        st.update(model=_case_model(case, seed), orb=_orbitals(case), opts=kg.kg_opts_default(M=case["M"]))
    elif kind in ("keldysh", "staged"):
        a, b = _pair(case, seed)
        ini, fin = kg.Sector(a), kg.Sector(b)
        ini.ground_state()
        st.update(ini=ini, fin=fin, orb=_orbitals(case), opts=kg.kg_opts_default(M=case["M"]))
        if kind == "staged":
            st["K"] = kg.Keldysh(ini, fin, st["orb"], case["dt"], case["n_t"], st["opts"])
    elif kind == "batched":
        sectors = [kg.Sector(m) for m in _instances(case, seed)]
        for s in sectors:
            s.ground_state()
        st.update(sectors=sectors, opts=kg.kg_opts_default(M=case["M"]))
    elif kind == "gradient":
        m = _case_model(case, seed)
        st["params"] = [torch.from_numpy(np.ascontiguousarray(p)).cuda().requires_grad_()
                        for p in (m["h"].real, m["eps"], m["U"])]
        st.update(cot=_cotangents(case, seed), opts=kg.kg_opts_default(M=case["M"]))
    else:
        st["G"], st["omega"] = _series(case, seed)
    return st


def run(st):
    c, kind = st["case"], st["kind"]
    if kind == "hpsi":
        st["sector"].hpsi(st["x"], st["y"])
        return st["y"]
    if kind == "propagate":
        st["x"].copy_(st["x0"])
        st["sector"].propagate(st["x"], c["dt"], c["n_steps"], st["opts"])
        return st["x"]
    if kind == "green":
        return st["sector"].green_equilibrium(st["orb"], c["dt"], c["n_steps"], st["opts"])
    if kind == "solve":
        s = kg.Sector(st["model"])
        out = s.green_equilibrium(st["orb"], c["dt"], c["n_steps"], st["opts"])
        s.close()
        return out
    if kind == "keldysh":
        return kg.kg_green_keldysh(st["ini"].handle, st["fin"].handle, st["orb"], c["dt"], c["n_t"], st["opts"])
    if kind == "staged":
        for k in range(c["n_t"]):
            st["K"].row(k)
        return st["K"].gram()
    if kind == "batched":
        return kg.kg_green_equilibrium_batched([s.handle for s in st["sectors"]], [(0, 0)], c["dt"], c["n_steps"],
                                               st["opts"])
    if kind == "gradient":
        from paper_1109_1205_gb300.autograd import green_equilibrium
        h, eps, U = st["params"]
        Gg, Gl = green_equilibrium(h, eps, U, c["L"], c["n_up"], c["n_dn"], [(0, 0)], c["dt"], c["n_steps"],
                                   st["opts"])
        g = torch.autograd.grad([Gg, Gl], [h, eps, U], st["cot"])
        return [Gg.detach(), Gl.detach(), *g]
    return kg.kg_green_fourier(st["G"], c["dt"], st["omega"], c["eta"])


# ----------------------------------------------------------- what it must do
def _dim(L, nu, nd):
    return math.comb(L, nu) * math.comb(L, nd) if 0 <= nu <= L and 0 <= nd <= L else 0


def _h_flops(model, L, nu, nd):
    """Operations of one H*psi: the diagonal and every hop, real numbers."""
    bonds = {"ring": 2 * L, "chain": 2 * (L - 1), "star": 2 * (L - 1), "random": L * (L - 1)}[model]
    per = {"ring": 2, "chain": 2, "star": 4, "random": 8}[model]
    hop = lambda n: bonds * math.comb(L - 2, n - 1) / math.comb(L, n) if 0 < n < L else 0.0  # noqa: E731
    return _dim(L, nu, nd) * (4 + per * (hop(nu) + hop(nd)))


def _step_flops(model, L, nu, nd, M):
    """One Krylov step: M times H*psi and the three-term recurrence, the
    Gram-Schmidt dots and corrections against every vector, the combination."""
    d = _dim(L, nu, nd)
    return M * (_h_flops(model, L, nu, nd) + 16 * d) + 16 * d * M * (M + 1) / 2 + 8 * d * M


def _columns(L, nu, nd, orb):
    return [(nu + s * (sp == 0), nd + s * (sp == 1)) for _, sp in orb for s in (1, -1)
            if _dim(L, nu + s * (sp == 0), nd + s * (sp == 1))]


def work(case):
    kind = case["kind"]
    if kind == "fourier":
        n, t, w = case["n_series"], case["n_t"], case["n_omega"]
        return {"bytes": 16 * n * t + 8 * w + 16 * n * w, "flops": 8.0 * n * t * w}
    if kind == "batched":
        L = (case["L_min"] + case["L_max"]) // 2
        one = 2 * case["n_steps"] * _step_flops("star", L, L // 2, L // 2, case["M"])
        return {"bytes": case["n_inst"] * 48.0 * _dim(L, L // 2, L // 2), "flops": case["n_inst"] * one}
    m, L, nu, nd = case["model"], case["L"], case["n_up"], case["n_dn"]
    d = _dim(L, nu, nd)
    if kind == "hpsi":
        return {"bytes": 32.0 * d, "flops": _h_flops(m, L, nu, nd)}
    if kind == "propagate":
        return {"bytes": 32.0 * d, "flops": case["n_steps"] * _step_flops(m, L, nu, nd, case["M"])}
    orb = [(0, 0)] if kind == "gradient" else _orbitals(case)
    step = sum(_step_flops(m, L, a, b, case["M"]) for a, b in _columns(L, nu, nd, orb))
    if kind in ("keldysh", "staged"):
        n = case["n_t"]
        vec = sum(_dim(L, a, b) for a, b in _columns(L, nu, nd, orb))
        gram = 8.0 * vec * n * n * len(orb) / 2
        return {"bytes": 16.0 * d + 16.0 * n * n * len(orb) ** 2 * 2,
                "flops": step * n * (n - 1) / 2 + gram + (n - 1) * _step_flops(m, L, nu, nd, case["M"])}
    gs = _step_flops(m, L, nu, nd, 100) if kind == "solve" else 0.0
    back = 3.0 if kind == "gradient" else 1.0  # forward, recomputed segments and the adjoint sweep
    return {"bytes": 16.0 * d + 32.0 * case["n_steps"] * len(orb) ** 2, "flops": gs + back * case["n_steps"] * step}


# ---------------------------------------------------- the same in plain torch
class _Ham:
    """H of one sector on the states [i_dn][i_up] (strings in numeric order)."""

    def __init__(self, model, nu, nd):
        self.L, self.nu, self.nd, dev = model["L"], nu, nd, _device()
        L = self.L
        self.strings = [np.array([b for b in range(1 << L) if bin(b).count("1") == n], dtype=np.int64) for n in (nu, nd)]
        up, dn = self.strings
        bit = lambda s: (s[:, None] >> np.arange(L)) & 1  # noqa: E731
        eps = model["eps"] + np.real(np.diag(model["h"]))
        e_up, e_dn = bit(up) @ eps[0], bit(dn) @ eps[1]
        bu, bd = (torch.from_numpy(bit(s).astype(np.float64)).to(dev) for s in (up, dn))
        self.diag = ((bd * torch.from_numpy(model["U"]).to(dev)) @ bu.T + torch.from_numpy(e_dn).to(dev)[:, None]
                     + torch.from_numpy(e_up).to(dev)[None, :])
        self.hops = []
        for s in self.strings:
            rank = {int(b): i for i, b in enumerate(s)}
            rows = []
            for a in range(L):
                for b in range(L):
                    if a == b or model["h"][a, b] == 0:
                        continue
                    t = np.flatnonzero(((s >> a) & 1 == 1) & ((s >> b) & 1 == 0))  # targets of c^dag_a c_b
                    src = (s[t] & ~(1 << a)) | (1 << b)
                    lo, hi = min(a, b), max(a, b)
                    between = s[t] & (((1 << hi) - 1) & ~((2 << lo) - 1))
                    sign = np.array([1.0 - 2.0 * (bin(int(v)).count("1") & 1) for v in between])
                    amp = model["h"][a, b]
                    amp = sign * amp if amp.imag else sign * amp.real
                    rows.append((t, np.array([rank[int(v)] for v in src], dtype=np.int64), amp))
            if len(s) <= 300:  # one matrix per spin
                D = np.zeros((len(s), len(s)), dtype=np.complex128)
                for t, j, v in rows:
                    D[t, j] += v
                self.hops.append(torch.from_numpy(D).to(dev))
            else:
                self.hops.append([tuple(torch.from_numpy(x).to(dev) for x in r) for r in rows])
        self.shape = (len(dn), len(up))
        g = [np.abs(e_up).max(), np.abs(e_dn).max(), np.abs(model["U"]).sum(), 2 * np.abs(model["h"]).sum()]
        self.bound = float(sum(g))

    def __call__(self, x):
        """x: [..., D_dn, D_up]"""
        y = self.diag * x
        up, dn = self.hops
        if isinstance(up, torch.Tensor):
            y = y + x @ up.T
        else:
            for t, j, v in up:
                y[..., t] += v * x[..., j]
        if isinstance(dn, torch.Tensor):
            y = y + dn @ x
        else:
            for t, j, v in dn:
                y[..., t, :] += v[:, None] * x[..., j, :]
        return y

    def ground(self):
        d = self.shape[0] * self.shape[1]
        m = min(d, 120)
        g = torch.Generator(device=_device()).manual_seed(1)
        v = torch.randn(d, dtype=torch.float64, device=_device(), generator=g).to(torch.complex128)
        for _ in range(40):
            V = torch.zeros(m, d, dtype=torch.complex128, device=v.device)
            V[0] = v / torch.linalg.vector_norm(v)
            T = np.zeros((m, m))
            n = m
            for j in range(m):
                w = self(V[j].view(self.shape)).reshape(-1)
                T[j, j] = float(torch.vdot(V[j], w).real)
                for _ in range(2):
                    w = w - V[: j + 1].T @ (V[: j + 1].conj() @ w)
                b = float(torch.linalg.vector_norm(w))
                if j + 1 == m or b < 1e-11:
                    n = j + 1
                    break
                T[j, j + 1] = T[j + 1, j] = b
                V[j + 1] = w / b
            e, q = np.linalg.eigh(T[:n, :n])
            v = V[:n].T @ torch.from_numpy(q[:, 0].astype(np.complex128)).to(v.device)
            v = v / torch.linalg.vector_norm(v)
            hv = self(v.view(self.shape)).reshape(-1)
            E = float(torch.vdot(v, hv).real)
            if float(torch.linalg.vector_norm(hv - E * v)) < 2e-13 * max(1.0, abs(E)):
                break
        return E, v.view(self.shape)

    def evolve(self, x, t):
        """e^{-i H t} x by Taylor sub-steps."""
        n = max(1, int(math.ceil(abs(t) * self.bound / 2.0)))
        h = t / n
        for _ in range(n):
            term = y = x
            for k in range(1, 60):
                term = self(term) * (-1j * h / k)
                y = y + term
                if float(torch.linalg.vector_norm(term)) < 1e-18 * float(torch.linalg.vector_norm(y)):
                    break
            x = y
        return x


def _cop(src, dst, x, site, spin, dagger):
    """c or c^dag of (site, spin) from the states of src to those of dst."""
    s = dst.strings[spin]
    t = np.flatnonzero(((s >> site) & 1) == (1 if dagger else 0))
    rank = {int(b): i for i, b in enumerate(src.strings[spin])}
    j = np.array([rank[int(b) ^ (1 << site)] for b in s[t]], dtype=np.int64)
    sign = np.array([1.0 - 2.0 * (bin(int(b) & ((1 << site) - 1)).count("1") & 1) for b in s[t]])
    if spin == 1 and src.nu & 1:
        sign = -sign
    t, j, sign = (torch.from_numpy(v).to(x.device) for v in (t, j, sign))
    y = torch.zeros(dst.shape, dtype=x.dtype, device=x.device)
    if spin == 0:
        y[:, t] = sign * x[:, j]
    else:
        y[t, :] = sign[:, None] * x[j, :]
    return y


def _neighbour(model, nu, nd, spin, dagger):
    s = 1 if dagger else -1
    a, b = (nu + s, nd) if spin == 0 else (nu, nd + s)
    return _Ham(model, a, b) if 0 <= a <= model["L"] and 0 <= b <= model["L"] else None


def _green_exact(model, orb, dt, n_steps):
    H = _Ham(model, model["n_up"], model["n_dn"])
    E0, gs = H.ground()
    n = len(orb)
    G = {1: np.zeros((n_steps + 1, n, n), dtype=np.complex128), 0: np.zeros((n_steps + 1, n, n), dtype=np.complex128)}
    for spin in (0, 1):
        idx = [a for a in range(n) if orb[a][1] == spin]
        for dagger in (1, 0):
            N = _neighbour(model, H.nu, H.nd, spin, dagger) if idx else None
            if N is None:
                continue
            chi = torch.stack([_cop(H, N, gs, orb[a][0], spin, dagger) for a in idx])
            bra, psi = chi.reshape(len(idx), -1).conj(), chi
            got = []
            for k in range(n_steps + 1):
                if k:
                    psi = N.evolve(psi, dt if dagger else -dt)
                got.append(bra @ psi.reshape(len(idx), -1).T)  # [a][b] = <chi_a | psi_b>
            got = torch.stack(got).cpu().numpy()
            t = dt * np.arange(n_steps + 1)
            ph = (-1j * np.exp(1j * E0 * t) if dagger else 1j * np.exp(-1j * E0 * t))[:, None, None]
            got = ph * (got if dagger else got.transpose(0, 2, 1))
            G[dagger][np.ix_(range(n_steps + 1), idx, idx)] = got
    return G[1], G[0]


def _keldysh_exact(ini, fin, orb, dt, n_t):
    H = _Ham(fin, fin["n_up"], fin["n_dn"])
    _, phi0 = _Ham(ini, ini["n_up"], ini["n_dn"]).ground()
    n = len(orb)
    out = {0: np.zeros((n_t, n_t, n, n), dtype=np.complex128), 1: np.zeros((n_t, n_t, n, n), dtype=np.complex128)}
    phi = [phi0]
    for _ in range(n_t - 1):
        phi.append(H.evolve(phi[-1], dt))
    for spin in (0, 1):
        idx = [a for a in range(n) if orb[a][1] == spin]
        for dagger in (0, 1):
            N = _neighbour(fin, H.nu, H.nd, spin, dagger) if idx else None
            if N is None:
                continue
            # all later rows travel back together
            na = len(idx)
            psi = torch.zeros((0, *N.shape), dtype=torch.complex128, device=phi0.device)
            for k in range(n_t - 1, -1, -1):
                row = torch.stack([_cop(H, N, phi[k], orb[a][0], spin, dagger) for a in idx])
                psi = torch.cat([row, psi])
                if k:
                    psi = N.evolve(psi, -dt)
            X = psi.reshape(n_t * na, -1)
            g = (X.conj() @ X.T).cpu().numpy().reshape(n_t, na, n_t, na)  # <X_ka | X_lb>
            if dagger:
                g = -1j * g.transpose(0, 2, 1, 3)
            else:
                g = 1j * g.transpose(2, 0, 3, 1)
            out[dagger][np.ix_(range(n_t), range(n_t), idx, idx)] = g
    return out[0], out[1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "hpsi":
        H = _Ham(_case_model(case, seed), case["n_up"], case["n_dn"])
        return H(_vector(H.shape[0] * H.shape[1], seed).view(H.shape)).reshape(-1)
    if kind == "propagate":
        H = _Ham(_case_model(case, seed), case["n_up"], case["n_dn"])
        return H.evolve(_vector(H.shape[0] * H.shape[1], seed).view(H.shape), case["dt"] * case["n_steps"]).reshape(-1)
    if kind in ("green", "solve"):
        return _green_exact(_case_model(case, seed), _orbitals(case), case["dt"], case["n_steps"])
    if kind in ("keldysh", "staged"):
        return _keldysh_exact(*_pair(case, seed), _orbitals(case), case["dt"], case["n_t"])
    if kind == "batched":
        return None  # one evolution per instance and column: minutes
    if kind == "gradient":
        m = _case_model(case, seed)
        m = dict(m, h=m["h"].real.astype(np.complex128))
        return [*_green_exact(m, [(0, 0)], case["dt"], case["n_steps"]), None, None, None]
    g, w = _series(case, seed)
    dt, n, dev = case["dt"], case["n_t"], _device()
    wt = torch.full((n,), dt, dtype=torch.float64, device=dev)
    wt[0] = wt[-1] = dt / 2
    k = torch.arange(n, dtype=torch.float64, device=dev) * dt
    g = torch.from_numpy(g).to(dev) * wt * torch.exp(-case["eta"] * k)
    out = torch.empty((case["n_series"], len(w)), dtype=torch.complex128, device=dev)
    for j0 in range(0, len(w), 64):
        ph = torch.from_numpy(w[j0:j0 + 64]).to(dev)[:, None] * k
        out[:, j0:j0 + 64] = g @ torch.complex(torch.cos(ph), torch.sin(ph)).T
    return out.cpu().numpy()
