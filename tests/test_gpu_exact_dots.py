"""The exact integer Gram-Schmidt dots on their own: one pass (reorth = 1), so
that nothing repairs a wrong total, at the vector counts and sizes where the
kernel changes its tiles, warps and rounds.

schedule = 2 keeps columns of any size in the streaming kernels with the
integer dots; schedule = 4 computes the same Krylov space with FP64 dots.  The
step is so long that every vector of the space counts in the result (which
then need not be converged); a dropped or doubled element then shifts it by
1e-8 or more (tests/test_dot_sensitivity.py plants such mistakes).

Tolerance 1e-11: both runs approximate e^{-iH tau} x in the same space; their
bases differ by rounding, a few 1e-16 per vector and at most 40 vectors, times
the loss of orthogonality of one classical pass (below 1e3 here).
"""
import numpy as np
import pytest

import oracle
import workloads as W
from test_dot_sensitivity import long_step

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1109_1205_gb300 as kg  # noqa: E402

TOL = 1e-11

# dimensions 1, 2, 36, 64, 65, 256, 257 x 1 .. and above: tiles of 64 to 256 elements, rounds of 256
SIZES = [(1, 1, 0), (2, 1, 0), (9, 2, 0), (8, 1, 1), (16, 1, 1), (17, 1, 1), (13, 1, 5), (11, 3, 2)]


def propagate(model, x, dt, **opts):
    xd = torch.from_numpy(x.copy()).cuda()
    kg.Sector(model).propagate(xd, dt, 1, kg.kg_opts_default(**opts))
    torch.cuda.synchronize()
    return xd.cpu().numpy()


@pytest.mark.parametrize("M", [1, 2, 3, 4, 6, 7, 12, 13, 18, 19, 24, 25, 26, 40])
@pytest.mark.parametrize("L,nu,nd", SIZES)
def test_one_pass_of_exact_dots(L, nu, nd, M):
    m = W.random_model(L, nu, nd, seed=L + 7 * M, complex_hopping=True)
    x = W.random_state(W.sector_dim(L, nu, nd), M)
    o = oracle.Sector(m)
    tau = long_step(o, x, M)
    y = propagate(m, x, tau, M=M, reorth=1, schedule=2)
    assert np.max(np.abs(y - propagate(m, x, tau, M=M, reorth=1, schedule=4))) < TOL
    if M >= 24:  # converged: |H| tau is below 2
        assert np.max(np.abs(propagate(m, x, 0.1, M=M, reorth=1, schedule=2) - o.propagate(x, 0.1))) < TOL


@pytest.mark.parametrize("M", [20, 30])
def test_images_made_again_near_a_breakdown(M):
    """A start vector that spans three eigenvectors to 1e-9, on a column of
    several rounds per block: the images of the vectors after the third are
    loose by many bits and re-made inside the dots, tile by tile."""
    rng = np.random.default_rng(2)
    m = W.siam_star(-1.5, 3.0, rng.uniform(-3, 3, 6), rng.uniform(0.2, 1.0, 6), 3, 3)
    o = oracle.Sector(m)
    d = W.sector_dim(7, 3, 3)
    e, v = np.linalg.eigh(np.array([o.hpsi(c) for c in np.eye(d, dtype=np.complex128)]).T)
    x = v[:, 2] + 0.5 * v[:, 40] - 1j * v[:, 777] + 1e-9 * W.random_state(d, 4)
    x /= np.linalg.norm(x)
    y = propagate(m, x, 0.15, M=M, reorth=1, schedule=2)
    assert np.max(np.abs(y - v @ (np.exp(-0.15j * e) * (v.conj().T @ x)))) < TOL
