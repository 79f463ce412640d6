"""Overlaps of a vector with one dominant component and many small ones with a
vector that lives on the small ones only, where FP64 products lose nothing and
a fixed-point image on the largest component keeps no bit.

Phi(t_0) and Phi(t_1) are set by the caller and the time step is zero, so the
Keldysh columns are c Phi(t_k) themselves (up to the rounding of a Krylov
step, 1e-15 of each component for the flat vector) and G^< = i <c Phi|c Phi>.
Tolerance of an entry between two times: 2^-52 of the two norms, an FP64
sum's; of an equal-time entry 2^-50, its vector's norm being off by the step.
"""
import math

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1109_1205_gb300 as kg  # noqa: E402


def exact_sum(z):
    return complex(math.fsum(z.real), math.fsum(z.imag))


@pytest.mark.parametrize("L,nu,nd", [(6, 3, 3), (8, 4, 4), (10, 5, 5)])
@pytest.mark.parametrize("p2", [-60, -57, -54, -50, -30])
def test_peaked_against_flat(L, nu, nd, p2):
    m = W.siam_chain(L, 3.0, nu, nd, field=0.4)
    si, sf = kg.Sector(m), kg.Sector(m)
    K = kg.Keldysh(si, sf, [(0, 0)], 0.0, 2)
    up, dn = kg.kg_sector_strings(sf.handle)
    in_col = np.tile((up & 1).astype(bool), len(dn))  # states that c_{0,up} does not annihilate
    rng = np.random.default_rng(L)
    peaked = (2.0 ** p2 * (1.0 + rng.uniform(0, 0.5, sf.dim))).astype(np.complex128)
    flat = np.exp(0.1j * rng.standard_normal(sf.dim)) / np.sqrt(sf.dim)
    top = np.flatnonzero(in_col)[sf.dim // 5]
    peaked[top], flat[top] = 1.0, 0.0
    K.set_phi(0, peaked)
    K.set_phi(1, flat)
    diag = [K.row(k)[0][0, 0] for k in (0, 1)]
    G = K.gram()[0][:, :, 0, 0]
    phi = [peaked[in_col], flat[in_col]]
    norm = [np.linalg.norm(v) for v in phi]
    for k in (0, 1):
        assert abs(diag[k] - 1j * exact_sum(phi[k].conj() * phi[k])) < 2.0 ** -50 * norm[k] ** 2
        for l in (0, 1):
            ref = 1j * exact_sum(phi[l].conj() * phi[k])
            assert abs(G[k, l] - ref) < (2.0 ** -52 if k != l else 2.0 ** -50) * norm[k] * norm[l], (k, l)
    K.close()
