"""The adjoint's parameter sums and node vectors at the sizes where their
splits can go wrong: parameter counts (3 L + 4 bonds) at the edges of the
groups of 32 that a warp adds up together, sectors below, at and above one
block, one and several columns.

Tolerance 1e-8 of the largest gradient, the bar of the adjoint's tests against
the same oracle: a dropped or doubled state, parameter or node shifts a
gradient by its own share, 1e-3 or more here.
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

TOL = 1e-8


@pytest.mark.parametrize("L,nu,nd,bonds,orbs", [
    (2, 1, 1, 1, [(0, 0)]),             # 10 parameters, 4 states
    (4, 2, 1, 4, [(0, 0)]),             # 28
    (4, 2, 2, 5, [(1, 0), (2, 1)]),     # 32
    (4, 2, 2, 6, [(0, 0)]),             # 36
    (8, 2, 2, 9, [(3, 0)]),             # 60, 784 states
    (8, 2, 1, 10, [(0, 0), (5, 0)]),    # 64
    (6, 3, 3, 13, [(1, 1)]),            # 70
])
def test_parameter_sums(L, nu, nd, bonds, orbs):
    m = W.random_model(L, nu, nd, seed=L + bonds, complex_hopping=True)
    pairs = [(a, a + 1) for a in range(L - 1)] + [(a, b) for a in range(L) for b in range(a + 2, L)]
    for a, b in pairs[bonds:]:
        m["h"][a, b] = m["h"][b, a] = 0.0
    dt, n = 0.05, 7
    rng = np.random.default_rng(bonds)
    shape = (n + 1, len(orbs), len(orbs))
    A = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    B = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    ref = oracle.green_equilibrium_grad_dense(m, orbs, dt, n, A, B)
    s = kg.Sector(m)
    got = kg.kg_green_equilibrium_vjp(s.handle, L, orbs, dt, n, A, B, checkpoint=3)
    keep = (m["h"] != 0) | np.eye(L, dtype=bool)
    ref = (ref[0], np.where(keep, ref[1], 0.0), np.where(keep, ref[2], 0.0), ref[3])
    scale = max(1.0, max(float(np.max(np.abs(r))) for r in ref))
    for name, g, r in zip(("eps", "hre", "him", "U"), got, ref):
        assert np.max(np.abs(np.asarray(g) - r)) <= TOL * scale, name
