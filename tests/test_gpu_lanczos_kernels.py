"""The Lanczos kernels at the sizes where their splits can go wrong: edges of
tiles and rounds, one element, vector counts at the edges of the dot kernels.

Tolerance 1e-11 on unit vectors, the bar of the propagation tests: a step's
rounding is a few 1e-16 per Lanczos vector and none of the runs has more than
200 of them, while a dropped or doubled element, vector or limb shifts the
result by its own size (components here are 1e-2 or larger).
"""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1109_1205_gb300 as kg  # noqa: E402

TOL = 1e-11


def propagate(model, x, dt, n, **opts):
    xd = torch.from_numpy(x.copy()).cuda()
    kg.Sector(model).propagate(xd, dt, n, kg.kg_opts_default(**opts))
    torch.cuda.synchronize()
    return xd.cpu().numpy()


# dimensions 1, 2, 63 .. 65, 255 .. 257 and above: tiles of 64 to 256 elements, rounds of 256
SIZES = [(1, 1, 0), (2, 1, 0), (9, 2, 0), (64, 0, 0), (8, 1, 1), (13, 1, 5), (16, 1, 1), (17, 1, 1), (11, 3, 2)]


@pytest.mark.parametrize("M", [1, 2, 3, 6, 7, 13, 24, 25, 40])
@pytest.mark.parametrize("L,nu,nd", [s for s in SIZES if s[0] <= 32])
def test_dot_splits(L, nu, nd, M):
    """Every count of vectors at which the dot kernel changes its tile or its
    warps, on columns of uneven size; the second pass (reorth = 2) keeps the
    streaming kernels on columns of any size."""
    m = W.random_model(L, nu, nd, seed=L + 7 * M, complex_hopping=True)
    x = W.random_state(W.sector_dim(L, nu, nd), M)
    y = propagate(m, x, 0.02, 3, M=M, reorth=2)
    if M >= 12 or M >= x.size:  # below, the step itself is not converged
        assert np.max(np.abs(y - oracle.Sector(m).propagate(x, 0.06))) < TOL
    fp64 = propagate(m, x, 0.02, 3, M=M, reorth=2, schedule=4)
    assert np.max(np.abs(y - fp64)) < TOL
