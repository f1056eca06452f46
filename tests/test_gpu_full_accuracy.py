"""Full solution vectors are as accurate as the recurrences allow: the pi^k that
scales a step of x^k and the pi^k that the recurrence keeps are the same number.
Two expressions of it that round differently make x^k wrong by the relative
rounding error of pi^k times the step, which is large where pi^k comes out of a
cancellation; the systems below have such steps (rms errors of 3e-14 to 1.2e-13
with two expressions, 4e-15 to 7e-15 with one).

Bound on each x^k's error vector: the residual of tol that a shift is left with,
tol / eta, and the rounding of N steps of unit-sized recurrences, u N / eta; so
(tol + u N) / eta / sqrt(n) rms over its n entries.
"""
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


@pytest.mark.parametrize("norb,L,seed", [(1, 6, 64), (1, 6, 72), (1, 6, 44), (4, 4, 72), (3, 4, 65)])
def test_full_solutions_to_rounding(S, norb, L, seed):
    h_csr = inputs.anderson_csr(L, seed=seed + 1000, norb=norb)
    n, tol, eta = h_csr.n, 1e-13, 0.4
    H = h_csr.dense()
    e, U = np.linalg.eigh(H)
    b = inputs.random_unit_complex(n, seed + 7)
    z = np.linspace(-4, 4, 48) + 1j * eta
    def solve(B):
        return ((B @ U) / (z[:, None] - e[None, :])) @ U.T
    X = solve(b[None, :])
    X = X + solve(b[None, :] - (z[:, None] * X - X @ H))   # one step of refinement
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val)
    try:
        for grid in (0, 3, 7):
            S.scocg_set_opts(h, S.SolveOptions(grid=grid))
            got, info = S.scocg_solve_full(h, z, torch.from_numpy(b).cuda(), tol=tol)
            err = float(np.sqrt(np.mean(np.abs(got.cpu().numpy().reshape(z.size, n) - X) ** 2)))
            bound = (tol + 1.1e-16 * info["iters"]) / eta / np.sqrt(n)
            assert err <= bound, (grid, err, bound)
    finally:
        S.scocg_destroy(h)
