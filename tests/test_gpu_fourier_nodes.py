"""The damped Fourier transform through Chebyshev nodes against the plain sum
in NumPy, at the shapes where its runs, windows and groups end unevenly, on
frequency lists of any order, spread and repetition.

Tolerance: 1e-12 of sum_k w_k e^{-eta t_k} |G_k|.  The interpolation error is below
1e-17 of that sum, its Lagrange factors amplify rounding about threefold, and
the arguments omega t of the rotations, up to 2e4, carry 2e-12 / 2 relative to
one term but add with random signs.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1109_1205_gb300 as kg  # noqa: E402


def plain(G, dt, omega, eta):
    n = G.shape[-1]
    w = np.full(n, dt)
    w[0] = w[-1] = 0.5 * dt
    t = dt * np.arange(n)
    out = np.empty((G.shape[0], len(omega)), dtype=complex)
    for j0 in range(0, len(omega), 64):
        out[:, j0:j0 + 64] = (G * (w * np.exp(-eta * t))) @ np.exp(1j * np.outer(t, omega[j0:j0 + 64]))
    return out, np.abs(G) @ (w * np.exp(-eta * t))


def grids():
    r = np.random.default_rng(5)
    return {"range": np.linspace(-10.0, 10.0, 701), "shuffled": r.permutation(np.linspace(-3.0, 40.0, 900)),
            "one": np.full(1500, 1.25), "pair": np.repeat([-2.0, 2.5], 800),
            "far": np.linspace(0.0, 0.5, 2000), "nodes": np.cos((2 * np.arange(1200) + 1) * np.pi / 48.0)}


@pytest.mark.parametrize("grid", ["range", "shuffled", "one", "pair", "far", "nodes"])
@pytest.mark.parametrize("n_t,dt,eta", [(20000, 0.05, 0.0), (30001, 0.01, 0.02), (16385, 0.002, 3.0), (40063, 0.5, 0.0)])
def test_fourier_through_nodes(grid, n_t, dt, eta):
    r = np.random.default_rng(n_t)
    G = r.standard_normal((2, n_t)) + 1j * r.standard_normal((2, n_t))
    omega = grids()[grid]
    if grid == "far":  # far from zero: arguments up to the 2e4 of the tolerance
        omega = 2e4 / (n_t * dt) - omega * min(1.0, 0.01 / dt)
    ref, scale = plain(G, dt, omega, eta)
    got = kg.kg_green_fourier(G, dt, omega, eta)
    assert np.all(np.max(np.abs(got - ref), axis=1) <= 1e-12 * scale)


def test_fourier_nodes_repeatable_and_nan():
    r = np.random.default_rng(1)
    G = r.standard_normal((1, 50001)) + 0j
    omega = np.linspace(-10, 10, 1001)
    a = kg.kg_green_fourier(G, 0.01, omega, 0.01)
    assert np.array_equal(a, kg.kg_green_fourier(G, 0.01, omega, 0.01))
    G[0, 31234] = np.nan
    assert np.all(np.isnan(kg.kg_green_fourier(G, 0.01, omega, 0.01)))
