"""The damped Fourier transform on frequencies so close together that their
spread is a few units in the last place, or tiny beside the frequencies, and on
samples near the top of FP64's range.

Tolerance: 1e-12 of sum_k w_k e^{-eta t_k} |G_k|, as in
tests/test_gpu_fourier_nodes.py: the arguments omega t stay below 2e4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1109_1205_gb300 as kg  # noqa: E402
from test_gpu_fourier_nodes import plain  # noqa: E402


@pytest.mark.parametrize("centre", [0.0, 1.0, -7.3, 1e-9])
@pytest.mark.parametrize("spread", [2.0 ** -52, 2.0 ** -51, 2.0 ** -50, 2.0 ** -46, 1e-12, 1e-9, 1e-5])
def test_close_frequencies(centre, spread):
    n_t = 20001
    r = np.random.default_rng(4)
    G = r.standard_normal((2, n_t)) + 1j * r.standard_normal((2, n_t))
    omega = centre + max(abs(centre), 1e-3) * spread * np.linspace(0.0, 1.0, 1500)
    ref, scale = plain(G, 0.05, omega, 0.01)
    got = kg.kg_green_fourier(G, 0.05, omega, 0.01)
    assert np.all(np.max(np.abs(got - ref), axis=1) <= 1e-12 * scale)


def test_large_frequencies():
    """Frequencies so large that a window of nodes around them is a few units in
    the last place wide: omega t is then uncertain by more than one, and only
    the size of the sum is defined."""
    n_t = 20001
    r = np.random.default_rng(6)
    G = r.standard_normal((1, n_t)) + 1j * r.standard_normal((1, n_t))
    omega = 1e15 * (1.0 + 2.0 ** -52 * np.arange(1500))
    got = kg.kg_green_fourier(G, 0.05, omega, 0.01)
    assert np.all(np.abs(got) <= np.abs(G[0]) @ np.full(n_t, 0.05))


def test_damping_of_large_samples():
    """Samples near the top of FP64's range under a damping that spans many
    powers of e within a run: nothing overflows on the way."""
    n_t = 16385
    r = np.random.default_rng(7)
    G = r.standard_normal((1, n_t)) + 1j * r.standard_normal((1, n_t))
    omega = np.linspace(-10.0, 10.0, 1201)
    ref, scale = plain(G, 0.002, omega, 75.0)
    got = kg.kg_green_fourier(G * 2.0 ** 1015, 0.002, omega, 75.0) * 2.0 ** -1015
    assert np.all(np.max(np.abs(got - ref), axis=1) <= 1e-12 * scale)
