"""Both sides of every rule that chooses a form of a kernel by size: the grid
and with it the reduction between CTAs and the place of the shift scalars, the
full-vector item loop, the lanes per eigenvalue of the tridiagonal bisection,
and the row and hop-list forms of the matrix-free Hubbard operators.

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


# Rows in pairs: odd and even numbers of up states (15, 20, 6) against ragged
# tiles of 64 down states; 9 sites take the general cross-spin counts.  Values
# in FP32 (exact amplitudes) and not.
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
