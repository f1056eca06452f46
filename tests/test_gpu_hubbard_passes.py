"""The kernels that only solves, ground states and Krylov recursions of the
matrix-free Hubbard operators run (a single apply has a kernel of its own): the
two passes of the two-orbital solve and the ring's real operator.

Two-orbital solves: numbers of up states (rows of pass 1, in pairs in compensated
vectors) odd and even, one and many; numbers of down states that leave a last
tile of 64 less than half full (6, 15, 18, 20, 25), more than half full (56) or
with one state; up to eight sites and more, where the neighbour counts take a
second word; hoppings that are FP32 values, whose products take a shorter form,
and others.  References: the oracle's CSR by sparse LU.  Bounds: a residual of tol leaves
|dG| <= tol / eta, 1e-12 (complex64: 1e-5); rounding u ||H|| N / eta with
||H|| < 42, N <= 800 iterations, eta = 1 and u = 1.1e-16, 2^-44 (compensated), 6e-8
(complex64, whose rounding acts as a change of H by u ||H||: u ||H|| / eta) adds
3.7e-12, 1.9e-9 and 2.5e-6.

Ring ground states: odd rings, whose hop lists are read singly, and sectors with
n_up != n_dn, whose diagonal table is not square; energies against dense
eigenvalues.  A residual of 1e-10 leaves |dE| <= 1e-10.
"""
import functools

import numpy as np
import pytest

from paper_0802_0748_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0802_0748_gb300 import scocg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return scocg


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def sparse(csr):
    import scipy.sparse as sp
    rp, c, v = csr
    return sp.csr_matrix((v, c, rp), shape=(rp.size - 1, rp.size - 1))


def two_orbital(sites, fp32):
    bonds = [(i, i + 1) for i in range(sites - 1)]
    vals = dict(U=3.1, Up=1.7, J=0.6, Jp=0.45, V=0.8)
    t = np.random.default_rng(sites).normal(size=(len(bonds), 2, 2))
    if fp32:
        t = t.astype(np.float32).astype(np.float64)
    m = inputs.eg_model(bonds=bonds, dirs=[0] * len(bonds), **vals)
    m["bond_t"] = t.tolist()
    return m


Z = np.array([-3.0, 2.0, 7.0]) + 1.0j


@functools.lru_cache(maxsize=None)
def reference(oracle_mod, sites, nu, nd, fp32):
    """Model, b and G of states 0, n / 2 and n - 1 at Z, [3][3]."""
    from scipy.sparse import identity
    from scipy.sparse.linalg import splu
    m = two_orbital(sites, fp32)
    H = sparse(oracle_mod.hubbard2_csr(m, nu, nd))
    n = H.shape[0]
    b = inputs.random_unit_complex(n, 11)
    idx = [0, n // 2, n - 1]
    return m, b, np.stack([splu((zk * identity(n) - H).tocsc()).solve(b)[idx] for zk in Z], axis=1)


SECTORS = [(3, 2, 0), (3, 0, 2), (3, 2, 3), (3, 3, 4), (3, 6, 2), (4, 1, 3), (4, 3, 4), (4, 4, 3), (9, 2, 1), (9, 1, 2)]


@pytest.mark.parametrize("prec,tol,bound", [(0, 1e-12, 5e-12), (2, 1e-12, 2e-9), (1, 1e-5, 2e-5)])
@pytest.mark.parametrize("fp32", [True, False])
@pytest.mark.parametrize("sites,nu,nd", SECTORS)
def test_two_orbital_solve_rows(S, oracle_mod, sites, nu, nd, fp32, prec, tol, bound):
    m, b, want = reference(oracle_mod, sites, nu, nd, fp32)
    h = S.scocg_create_hubbard2(m, nu, nd, opts=S.SolveOptions(precision=prec))
    try:
        for grid in (0, 2):
            S.scocg_set_opts(h, S.SolveOptions(precision=prec, grid=grid))
            G, info = S.scocg_solve(h, Z, cuda(b), proj_idx=[0, b.size // 2, b.size - 1], tol=tol)
            assert info["status"] == 0 and info["iters"] <= 800
            assert np.max(np.abs(G.cpu().numpy()[0] - want)) <= bound, grid
    finally:
        S.scocg_destroy(h)


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("sites,nu,nd", [(3, 2, 3), (4, 4, 3)])
def test_two_orbital_solve_continued(S, oracle_mod, sites, nu, nd, prec):
    """A solve stopped after 40 iterations and continued repeats its last apply's sums over the same rows:
    the same numbers as without the stop."""
    m = two_orbital(sites, True)
    h = S.scocg_create_hubbard2(m, nu, nd, opts=S.SolveOptions(precision=prec))
    try:
        b = cuda(inputs.random_unit_complex(S.scocg_dim(h), 11))
        z, tol = np.array([-3.0, 2.0, 7.0]) + 0.5j, 1e-4
        G, info = S.scocg_solve(h, z, b, proj_idx=[0], tol=tol)
        assert info["status"] == 0 and info["iters"] > 40
        S.scocg_set_opts(h, S.SolveOptions(precision=prec, max_iter=40))
        _, part = S.scocg_solve(h, z, b, proj_idx=[0], tol=tol)
        assert part["status"] == 1
        S.scocg_set_opts(h, S.SolveOptions(precision=prec))
        G2, info2 = S.scocg_solve_resume(h, z, b, proj_idx=[0], tol=tol)
        assert info2["status"] == 0 and torch.equal(G, G2)
    finally:
        S.scocg_destroy(h)


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("L,nu,nd", [(5, 1, 4), (5, 4, 2), (6, 2, 5), (7, 3, 4), (7, 5, 1)])
def test_ring_ground_energy(S, oracle_mod, L, nu, nd, periodic):
    H = sparse(oracle_mod.hubbard_csr(L, nu, nd, 1.0, 4.0, 1.0, periodic))
    e = np.linalg.eigvalsh(H.toarray())
    h = S.scocg_create_hubbard(L, nu, nd, 1.0, 4.0, 1.0, periodic)
    try:
        E, psi, info = S.scocg_ground_state(h, cuda(inputs.random_unit_real(H.shape[0], 5)), m=40, max_cycles=20,
                                            tol=1e-10)
    finally:
        S.scocg_destroy(h)
    assert info["status"] == 0
    assert abs(E - e[0]) <= 1e-10
    p = psi.cpu().numpy()
    assert np.linalg.norm(H @ p - E * p) <= 2e-10
