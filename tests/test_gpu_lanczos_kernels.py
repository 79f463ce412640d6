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
SIZES = [(1, 1, 0), (2, 1, 0), (9, 2, 0), (8, 1, 1), (13, 1, 5), (16, 1, 1), (17, 1, 1), (11, 3, 2)]


@pytest.mark.parametrize("M", [1, 2, 3, 6, 7, 13, 24, 25, 40])
@pytest.mark.parametrize("L,nu,nd", SIZES)
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


SMALL = [("random", 2, 1, 0, 8), ("random", 6, 3, 2, 20), ("random", 8, 4, 4, 20), ("random", 8, 4, 4, 63),
         ("star", 6, 4, 3, 40), ("star", 12, 1, 2, 33), ("ring", 9, 4, 4, 12), ("ring", 8, 3, 4, 24),
         ("chain", 10, 3, 2, 16), ("chain", 32, 1, 1, 14)]


def small_model(name, L, nu, nd):
    if name == "random":
        return W.random_model(L, nu, nd, seed=L + nu, complex_hopping=True)
    if name == "star":
        rng = np.random.default_rng(L)
        return W.siam_star(-1.5, 3.0, rng.uniform(-3, 3, L - 1), rng.uniform(0.2, 1.0, L - 1), nu, nd)
    return W.hubbard_ring(L, 4.0, nu, nd) if name == "ring" else W.siam_chain(L, 3.0, nu, nd, field=0.4)


@pytest.mark.parametrize("name,L,nu,nd,M", SMALL)
def test_small_columns_equal_streaming(name, L, nu, nd, M):
    """Columns that one cluster takes through a whole step, of one block to
    sixteen, against the streaming kernels (schedule = 4) and the oracle."""
    m = small_model(name, L, nu, nd)
    x = W.random_state(W.sector_dim(L, nu, nd), 3)
    y = propagate(m, x, 0.03, 4, M=M)
    assert np.max(np.abs(y - propagate(m, x, 0.03, 4, M=M, schedule=4))) < TOL
    if L <= 16:  # the oracle enumerates 2L-bit words
        assert np.max(np.abs(y - oracle.Sector(m).propagate(x, 0.12))) < TOL


@pytest.mark.parametrize("schedule", [2, 4])  # the streaming kernels, exact and FP64 dots
@pytest.mark.parametrize("p2", [-400, -130, -61, 61, 130, 400])
def test_scaled_start(p2, schedule):
    """A start vector scaled by a power of two, far enough to leave FP32's
    range in its coefficients and copies, gives the scaled result."""
    m = W.random_model(9, 4, 4, seed=20, complex_hopping=True)
    x = W.random_state(W.sector_dim(9, 4, 4), 20)
    y = propagate(m, x, 0.02, 2, M=20, schedule=schedule)
    z = propagate(m, x * 2.0 ** p2, 0.02, 2, M=20, schedule=schedule)
    assert np.max(np.abs(z * 2.0 ** -p2 - y)) < TOL


@pytest.mark.parametrize("L,n", [(4, 2), (8, 4), (10, 5), (12, 5)])  # 1, 20, 249 and 608 blocks of exponents
@pytest.mark.parametrize("where", [0, 0.5, 1])
def test_hpsi_largest_component(L, n, where):
    """H*psi of uniform hopping with one component 2^40 above the others, in
    the first, a middle and the last block: the image of x overflows if its
    exponent is missed.  1e-12 of the largest result: each of at most 2 L hops
    rounds to 2^-54 of the largest component, times |U| + |T| of order one."""
    m = W.hubbard_ring(L, 4.0, n, n)
    x = W.random_state(W.sector_dim(L, n, n), L)
    x[int(where * (x.size - 1))] *= 2.0 ** 40
    xd = torch.from_numpy(x.copy()).cuda()
    yd = torch.empty_like(xd)
    s = kg.Sector(m)
    s.hpsi(xd, yd, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    ref = oracle.Sector(m).hpsi(x)
    assert np.max(np.abs(yd.cpu().numpy() - ref)) < 1e-12 * np.max(np.abs(ref))


def test_small_column_near_breakdown():
    """A start vector that spans three eigenvectors to 1e-9: the space is
    nearly invariant after three vectors, so the images' exponent bounds are
    loose by many bits and have to be made again."""
    m = small_model("random", 6, 3, 2)
    o = oracle.Sector(m)
    d = W.sector_dim(6, 3, 2)
    e, v = np.linalg.eigh(np.array([o.hpsi(c) for c in np.eye(d, dtype=np.complex128)]).T)
    x = v[:, 2] + 0.5 * v[:, 40] - 1j * v[:, 77] + 1e-9 * W.random_state(d, 4)
    x /= np.linalg.norm(x)
    y = propagate(m, x, 0.05, 3, M=20)
    assert np.max(np.abs(y - v @ (np.exp(-0.15j * e) * (v.conj().T @ x)))) < TOL


@pytest.mark.parametrize("large", [False, True])
def test_small_columns_in_one_batch(large):
    """Columns of every cluster size in one batch (several launches side by
    side); with a large one among them, all in the streaming kernels."""
    sizes = [(6, 1, 5), (7, 3, 3), (8, 4, 4), (8, 2, 6), (7, 2, 2), (5, 2, 2)] + ([(10, 5, 5)] if large else [])
    models = [small_model("star", L, nu, nd) for L, nu, nd in sizes]
    secs = [kg.Sector(m) for m in models]
    gg, gl, st = kg.kg_green_equilibrium_batched([s.handle for s in secs], [(0, 0), (0, 1)], 0.05, 12)
    assert list(st) == [0] * len(models)
    for i, m in enumerate(models):
        ref = kg.Sector(m).green_equilibrium([(0, 0), (0, 1)], 0.05, 12, kg.kg_opts_default(schedule=4))
        assert np.max(np.abs(gg[i] - ref[0])) < TOL and np.max(np.abs(gl[i] - ref[1])) < TOL


@pytest.mark.parametrize("L,nu,nd", [(3, 1, 2), (5, 2, 2), (7, 3, 3)])
@pytest.mark.parametrize("n_orb,n_t", [(1, 1), (1, 2), (3, 1), (2, 8), (1, 31), (3, 11), (3, 16), (3, 22)])
def test_gram_tiles(L, nu, nd, n_orb, n_t):
    """G(t,t') whose Gram matrices have 1 to 66 vectors (one tile, a ragged
    second and third one, an odd count) of 3 to 1,225 states.  1e-10 is the bar
    of the Green's functions; a wrong tile shifts entries of order 0.1."""
    ini, fin = W.random_model(L, nu, nd, seed=5), W.random_model(L, nu, nd, seed=6)
    orbs = [(a, 0) for a in range(n_orb)]
    si, sf = kg.Sector(ini), kg.Sector(fin)
    gl, gg = kg.kg_green_keldysh(si.handle, sf.handle, orbs, 0.05, n_t)
    rl, rg = oracle.green_keldysh(ini, fin, orbs, 0.05, n_t)[:2]
    assert np.max(np.abs(gl - rl)) < 1e-10 and np.max(np.abs(gg - rg)) < 1e-10


@pytest.mark.parametrize("M_gs", [2, 3, 33, 64, 100, 255])
def test_lowest_ritz_pair(M_gs):
    """Ground states from restarts of every length class, against the oracle:
    energy 1e-12 relative, the vector to 1e-10 in overlap (its residual is
    1e-12 and the gap above 0.1)."""
    for m in (W.random_model(6, 3, 2, seed=9), W.siam_chain(7, 3.0, 3, 4, field=0.3)):
        s = kg.Sector(m)
        e, res, gap = s.ground_state(kg.kg_opts_default(M_gs=M_gs, max_restarts=4000, tol_resid=1e-11))
        e_ref, psi, _ = oracle.Sector(m).ground_state()
        assert abs(e - e_ref) < 1e-12 * max(1.0, abs(e_ref)) and gap > 0.0
        assert abs(abs(np.vdot(psi, s.ground_state_vector())) - 1.0) < 1e-10
