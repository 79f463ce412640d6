"""How far a wrong Gram-Schmidt dot moves the result that
tests/test_gpu_exact_dots.py compares: mistakes planted in a NumPy Lanczos
step with one classical pass."""
import numpy as np
import pytest

import oracle
import workloads as W


def lanczos(o, x, M, mistake=None):
    """T and the basis of M Lanczos vectors; mistake(j, k, products) returns
    the total of one dot."""
    V = [x / np.linalg.norm(x)]
    a, b = [], []
    for j in range(M):
        w = o.hpsi(V[j]) - (b[-1] * V[j - 1] if j else 0)
        alpha = np.vdot(V[j], w).real
        u = w - alpha * V[j]
        h = [mistake(j, k, v.conj() * u) if mistake else np.vdot(v, u) for k, v in enumerate(V)]
        for c, v in zip(h, V):
            u = u - c * v
        a.append(alpha + h[j].real)
        b.append(np.linalg.norm(u))
        if b[-1] < 1e-12:
            break
        V.append(u / b[-1])
    m = len(a)
    return np.diag(a) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1), np.array(V[:m])


def long_step(o, x, M):
    """A step so long that the last of M Lanczos vectors counts in e^{-iH tau} x:
    1.2 M over half the width of the spectrum (as 12 vectors show it)."""
    e = np.linalg.eigvalsh(lanczos(o, x, min(12, x.size))[0])
    return 1.2 * M / max(1.0, 0.5 * (e[-1] - e[0]))


def step(o, x, tau, M, mistake=None):
    T, V = lanczos(o, x, M, mistake)
    e, q = np.linalg.eigh(T)
    return np.linalg.norm(x) * V.T @ (q @ (np.exp(-1j * e * tau) * q[0]))


@pytest.mark.parametrize("L,nu,nd,M", [(2, 1, 0, 2), (9, 2, 0, 13), (8, 1, 1, 13), (17, 1, 1, 25), (11, 3, 2, 24),
                                       (11, 3, 2, 40)])
def test_a_wrong_total_shows(L, nu, nd, M):
    m = W.random_model(L, nu, nd, seed=L + 7 * M, complex_hopping=True)
    o = oracle.Sector(m)
    x = W.random_state(W.sector_dim(L, nu, nd), M)
    tau = long_step(o, x, M)
    good = step(o, x, tau, M)
    for name, f in {"an element left out": lambda p: p.sum() - p[-1], "an element twice": lambda p: p.sum() + p[0],
                    "half of them left out": lambda p: p[: p.size // 2].sum()}.items():
        for at in {min(1, M - 2), M // 2 - (M == 2), M - 2}:
            bad = step(o, x, tau, M, lambda j, k, p: f(p) if (j, k) == (at, at // 2) else p.sum())
            assert np.max(np.abs(bad - good)) > 1e-9, (name, at)
