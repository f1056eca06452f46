"""Both sides of the rules that choose a form of a kernel by size: the grid
and with it the reduction between CTAs and the place of the shift scalars, the
full-vector item loop, the lanes per eigenvalue of the tridiagonal bisection,
and single applies of the matrix-free Hubbard operators.  (The place of q is in
test_gpu_waits.py, the Hubbard kernels that only solves and ground states run in
test_gpu_hubbard_passes.py.)

References: dense eigendecompositions, the oracle's CSR operators and closed
forms.  Bounds: a residual of tol leaves |dG| <= tol / eta (unit b and c; eta
the smallest Im z), 1e-11 below; the recurrences' rounding, u * iterations /
eta with u = 1.1e-16 (FP64), 2^-44 (compensated), 6e-8 (FP32) and at most 400
iterations, adds 4e-13, 2.3e-10 and 2.4e-4 at most.
"""
import math

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


def to_df(x):
    hi = np.stack([x.real, x.imag], axis=1).astype(np.float32)
    lo = (np.stack([x.real, x.imag], axis=1) - hi).astype(np.float32)
    return np.concatenate([hi, lo], axis=1)


def from_df(v):
    v = v.astype(np.float64)
    return (v[:, 0] + v[:, 2]) + 1j * (v[:, 1] + v[:, 3])


def shift_grid(K):
    return np.linspace(-3.0, 3.0, K) + 0.1j


# Grids of one CTA, around the two reductions' limit (32 CTAs: packets up to it,
# the counter barrier above) and beyond the units of work (the largest is
# clamped); 70 shifts give a CTA 70 of them (too many to keep), 24, 3, 3, 2 and
# fewer; 1 and 2 projections keep the shift scalars on the chip, 3 do not.
@pytest.mark.parametrize("prec,bound", [(0, 1e-10), (2, 1e-9), (1, 5e-4)])
@pytest.mark.parametrize("grid", [0, 1, 3, 31, 32, 33, 152])
@pytest.mark.parametrize("kind", ["blocks", "scalar"])
def test_solve_over_grids(S, kind, grid, prec, bound):
    h_csr = inputs.anderson_csr(6, seed=11) if kind == "blocks" else inputs.chain_csr(1037, t=-0.9)
    n = h_csr.n
    b = inputs.random_unit_complex(n, 3)
    H = h_csr.dense()
    e, U = np.linalg.eigh(H.astype(np.float32).astype(np.float64) if prec else H)   # H as the mode holds it
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val, opts=S.SolveOptions(precision=prec, grid=grid))
    try:
        for K, M in ((70, 1), (70, 3), (33, 2), (1, 1)):
            z = shift_grid(K)
            idx = [0, n - 1, n // 2][:M]
            G, info = S.scocg_solve(h, z, cuda(b), proj_idx=idx, tol=1e-5 if prec == 1 else 1e-12)
            assert info["status"] == 0
            want = np.einsum("mi,ki,i->mk", U[idx], 1.0 / (z[:, None] - e[None, :]), U.T @ b)
            got = G.cpu().numpy()[0]
            assert got.shape == want.shape
            assert np.max(np.abs(got - want)) <= bound, (K, M)
    finally:
        S.scocg_destroy(h)


# Full-vector items are (32 rows, a shift): one row, a ragged last chunk, odd
# numbers of shifts, one CTA and the default grid.
@pytest.mark.parametrize("grid", [0, 1])
@pytest.mark.parametrize("n,K", [(1, 3), (31, 1), (33, 7), (500, 5), (1037, 33)])
def test_full_vectors_ragged(S, n, K, grid):
    h_csr = inputs.anderson_csr(5, seed=5) if n == 500 else inputs.chain_csr(n, t=-0.9, onsite=0.2)
    assert h_csr.n == n
    b = inputs.random_unit_complex(n, 7)
    z = shift_grid(K)
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val, opts=S.SolveOptions(grid=grid))
    try:
        X, info = S.scocg_solve_full(h, z, cuda(b), tol=1e-12)
    finally:
        S.scocg_destroy(h)
    assert info["status"] == 0
    e, U = np.linalg.eigh(h_csr.dense())
    want = ((U.T @ b)[None, :] / (z[:, None] - e[None, :])) @ U.T
    assert np.max(np.abs(X.cpu().numpy().reshape(K, n) - want)) <= 1e-10


# 608 eigenvalues: 32 lanes each on 152 SMs, 609: eight; the ends of both forms.
@pytest.mark.parametrize("nu", [1, 2, 31, 608, 609, 1001])
def test_tridiagonal_eigenvalues(S, nu):
    h_csr = inputs.chain_csr(2048, t=-1.0)
    b = np.zeros(h_csr.n)
    b[0] = 1.0
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val)
    try:
        _, ritz, _, info = S.scocg_krylov_sd(h, cuda(b), nu, np.array([0.3 + 0.1j]), proj_idx=[0])
    finally:
        S.scocg_destroy(h)
    assert info["nu_used"] == nu
    ref = np.sort(-2.0 * np.cos(np.pi * np.arange(1, nu + 1) / (nu + 1)))
    assert np.max(np.abs(ritz.cpu().numpy()[:nu] - ref)) < 1e-13


# A single apply, one row per lane: odd and even numbers of up states (15, 20, 6)
# against ragged tiles of 32 down states; 9 sites take the cross-spin counts'
# second word.  Values in FP32 (exact amplitudes) and not.
@pytest.mark.parametrize("fp32", [True, False])
@pytest.mark.parametrize("sites,nu,nd", [(3, 2, 2), (3, 3, 4), (3, 6, 3), (3, 1, 0), (4, 3, 4), (4, 4, 2), (9, 2, 1), (9, 1, 2)])
def test_two_orbital_rows(S, oracle_mod, sites, nu, nd, fp32):
    import scipy.sparse as sp
    bonds = [(i, i + 1) for i in range(sites - 1)]
    vals = dict(U=3.1, Up=1.7, J=0.6, Jp=0.45, V=0.8)
    t = np.random.default_rng(sites).normal(size=(len(bonds), 2, 2))
    if fp32:
        vals = {k: float(np.float32(v)) for k, v in vals.items()}
        t = t.astype(np.float32).astype(np.float64)
    m = inputs.eg_model(bonds=bonds, dirs=[0] * len(bonds), **vals)
    m["bond_t"] = t.tolist()
    rp, c, v = oracle_mod.hubbard2_csr(m, nu, nd)
    n = rp.size - 1
    H = sp.csr_matrix((v, c, rp), shape=(n, n))
    x = inputs.random_unit_complex(n, 5)
    z = 0.3 + 0.2j
    want = z * x - H @ x
    scale = np.max(np.abs(want))
    h = S.scocg_create_hubbard2(m, nu, nd)
    try:
        assert S.scocg_dim(h) == n == math.comb(2 * sites, nu) * math.comb(2 * sites, nd)
        y = S.scocg_apply(h, z, cuda(x)).cpu().numpy()
        assert np.max(np.abs(y - want)) <= 1e-14 * scale
        y32 = S.scocg_apply(h, z, cuda(x.astype(np.complex64)), precision=S.MIXED).cpu().numpy()
        assert np.max(np.abs(y32 - want)) <= 1e-5 * scale
        ydf = from_df(S.scocg_apply(h, z, cuda(to_df(x)), precision=S.MIXED_DF).cpu().numpy())
        assert np.max(np.abs(ydf - want)) <= 1e-12 * scale
    finally:
        S.scocg_destroy(h)


# A single apply: in compensated vectors the hop lists of an even ring are read
# four entries at a time, of an odd one (or an open chain's) singly; complex128 reads
# them singly.  t, U, V and x are integers, so every form is exact.
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("L,nu,nd", [(3, 1, 2), (5, 2, 3), (6, 3, 3), (7, 3, 4), (8, 4, 4), (9, 4, 3)])
def test_ring_hop_lists(S, oracle_mod, L, nu, nd, periodic):
    import scipy.sparse as sp
    rp, c, v = oracle_mod.hubbard_csr(L, nu, nd, 1.0, 4.0, 1.0, periodic)
    n = rp.size - 1
    H = sp.csr_matrix((v, c, rp), shape=(n, n))
    rng = np.random.default_rng(L)
    x = (rng.integers(-8, 9, n) + 1j * rng.integers(-8, 9, n)).astype(np.complex128)
    z = 0.5 + 0.25j
    want = z * x - H @ x
    h = S.scocg_create_hubbard(L, nu, nd, 1.0, 4.0, 1.0, periodic)
    try:
        assert np.array_equal(S.scocg_apply(h, z, cuda(x)).cpu().numpy(), want)
        assert np.array_equal(from_df(S.scocg_apply(h, z, cuda(to_df(x)), precision=S.MIXED_DF).cpu().numpy()), want)
    finally:
        S.scocg_destroy(h)
