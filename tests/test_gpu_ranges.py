"""Start vectors and Hamiltonians far from one: what the kernels keep in FP32
may neither vanish nor overflow.

Everything is scaled by powers of two (x by 2^p; H by 2^q and the step by
2^-q), so exact arithmetic gives the unscaled result times 2^p, and FP64 at
these exponents the same roundings.  Tolerance 1e-13 on unit vectors: a term may
move between its FP32 and FP64 sums, which changes a few roundings of 1e-16
in each of the 40 to 80 Lanczos vectors of a run, while a lost FP32 term of
the combination is 1e-13 to 1e-10 of the result.
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

TOL = 1e-13


def model(name, q=0):
    if name == "star":
        rng = np.random.default_rng(6)
        m = W.siam_star(-1.5, 3.0, rng.uniform(-3, 3, 5), rng.uniform(0.2, 1.0, 5), 3, 3)
    elif name == "ring":
        m = W.hubbard_ring(8, 4.0, 4, 4)
    else:
        L = 8 if name == "random8" else 9
        m = W.random_model(L, 4, 4, seed=20, complex_hopping=True)
    return dict(m, h=np.asarray(m["h"]) * 2.0 ** q, eps=np.asarray(m["eps"]) * 2.0 ** q,
                U=np.asarray(m["U"]) * 2.0 ** q)


def run(name, p, q, schedule, M=20):
    s = kg.Sector(model(name, q))
    x = W.random_state(s.dim, 20)
    xd = torch.from_numpy(x * 2.0 ** p).cuda()
    s.propagate(xd, 0.02 * 2.0 ** -q, 2, kg.kg_opts_default(M=M, schedule=schedule))
    torch.cuda.synchronize()
    return xd.cpu().numpy() * 2.0 ** -p


# small columns (one cluster per column) of each kind of hop sum
@pytest.mark.parametrize("name", ["star", "ring", "random8"])
@pytest.mark.parametrize("p", [-400, -130, -100, -61, 61, 130, 161, 400])
def test_scaled_start_of_a_small_column(name, p):
    assert np.max(np.abs(run(name, p, 0, 0) - run(name, 0, 0, 0))) < TOL


@pytest.mark.parametrize("name,schedule", [("star", 0), ("ring", 0), ("random8", 0),
                                           ("random9", 2), ("random9", 4)])  # and the streaming kernels
@pytest.mark.parametrize("p,q", [(0, -70), (0, -40), (0, 58), (-58, 58), (-58, 55), (-60, 53), (58, -58), (0, 130),
                                 (30, -130)])
def test_scaled_hamiltonian(name, schedule, p, q):
    assert np.max(np.abs(run(name, p, q, schedule) - run(name, 0, 0, schedule))) < TOL


def outcome(name, p, q, schedule):
    try:
        return run(name, p, q, schedule)
    except kg.KGError as e:
        assert e.code == kg.KG_ENUMERIC
        return None


@pytest.mark.parametrize("name", ["star", "ring", "random8"])
@pytest.mark.parametrize("p,q", [(500, 3), (508, 0), (520, 0), (600, 0), (1000, 3), (1015, 3), (1022, 3), (0, 500), (0, 520),
                                 (0, 800), (0, 1010), (505, 515), (500, 500), (-500, 600)])
def test_what_is_out_of_range_is_refused(name, p, q):
    """Norms whose squares leave FP64's range are refused by the streaming
    kernels (schedule = 4), and so they are for a small column; anything else
    gives the scaled result."""
    y, z = outcome(name, p, q, 0), outcome(name, p, q, 4)
    assert (y is None) == (z is None)
    if y is not None:
        assert np.max(np.abs(y - run(name, 0, 0, 0))) < TOL


@pytest.mark.parametrize("L,nu,nd,M", [(5, 2, 2, 40), (6, 3, 3, 50), (6, 3, 3, 60)])
@pytest.mark.parametrize("q", [-40, -45, -63, -110])
@pytest.mark.parametrize("schedule", [0, 2])
def test_small_hamiltonian_is_still_orthogonalised(L, nu, nd, M, q, schedule):
    """Gram-Schmidt terms are 1e-16 of the Hamiltonian, so in FP32 they vanish
    first.  Steps so long that all M vectors count, and in which the basis
    loses orthogonality without those terms (the result then moves by 1e-5,
    1e-7 and 1e-4 of the vector).  Tolerance 1e-11 as for one pass in
    test_gpu_exact_dots: the same space, bases that differ by roundings."""
    m = W.random_model(L, nu, nd, seed=3, complex_hopping=True)
    if L == 6:
        r = np.random.default_rng(6)
        m = W.siam_star(-1.5, 3.0, r.uniform(-3, 3, 5), r.uniform(0.2, 1.0, 5), nu, nd)
    x = W.random_state(W.sector_dim(L, nu, nd), 20)
    tau = long_step(oracle.Sector(m), x, M)
    y = []
    for s in (0, q):
        xd = torch.from_numpy(x.copy()).cuda()
        scaled = dict(m, **{k: np.asarray(m[k]) * 2.0 ** s for k in ("h", "eps", "U")})
        kg.Sector(scaled).propagate(xd, tau * 2.0 ** -s, 1, kg.kg_opts_default(M=M, schedule=schedule))
        torch.cuda.synchronize()
        y.append(xd.cpu().numpy())
    assert np.max(np.abs(y[1] - y[0])) < 1e-11
