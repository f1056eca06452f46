"""Both waits between the CTAs of a solve give up after the handle's timeout: the
packets that grids of up to 32 CTAs exchange and the counter barrier of larger
ones.  One CTA withholds its part (a host-side option); the call reports it and
the handle solves afterwards.  And the two places of q: shared memory, or global
memory where a CTA's rows do not fit (7,168 FP64 or compensated rows, 14,336
complex64 rows).
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


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("grid", [2, 32, 33])
def test_wait_gives_up(S, grid, prec):
    h_csr = inputs.anderson_csr(4, seed=31)
    b = cuda(inputs.random_unit_complex(h_csr.n, 3))
    z = np.linspace(-2, 2, 8) + 0.5j
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val,
                           opts=S.SolveOptions(precision=prec, grid=grid, debug_inject=1, timeout_ms=300.0))
    try:
        with pytest.raises(S.ScocgError) as e:
            S.scocg_solve(h, z, b, proj_idx=[0], tol=1e-5)
        assert e.value.code == S.ERR_TIMEOUT
        S.scocg_set_opts(h, S.SolveOptions(precision=prec, grid=grid))
        G, info = S.scocg_solve(h, z, b, proj_idx=[0], tol=1e-5)
        assert info["status"] == 0
        x = [np.linalg.solve(zk * np.eye(h_csr.n) - h_csr.dense(), b.cpu().numpy())[0] for zk in z]
        # residual of 1e-5: |dG| <= 1e-5 / eta = 2e-5; complex64 rounding u ||H|| / eta = 8e-7
        assert np.max(np.abs(G.cpu().numpy()[0, 0] - np.array(x))) <= 3e-5
    finally:
        S.scocg_destroy(h)


# 16,384 rows: a CTA of one holds them all (q in global memory), two CTAs hold 8,192 each (complex64: shared
# memory), the default grid a few hundred each.  A residual of tol leaves |dG| <= tol / eta on either side; rounding
# u N / eta (N < 400; complex64 u ||H|| / eta) stays below 1e-13, 4e-11 and 8e-7.
@pytest.mark.parametrize("prec,tol,bound", [(0, 1e-11, 4e-11), (2, 1e-11, 1.2e-10), (1, 1e-5, 4e-5)])
@pytest.mark.parametrize("kind", ["blocks", "scalar"])
def test_q_in_shared_and_global_memory(S, kind, prec, tol, bound):
    h_csr = inputs.anderson_csr(16, seed=4) if kind == "blocks" else inputs.chain_csr(16384, t=-1.0, onsite=0.25)
    assert h_csr.n == 16384
    b = cuda(inputs.random_unit_complex(h_csr.n, 3))
    z = np.linspace(-3, 3, 7) + 0.6j
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val, opts=S.SolveOptions(precision=prec))
    try:
        G = []
        for grid in (0, 1, 2):
            S.scocg_set_opts(h, S.SolveOptions(precision=prec, grid=grid))
            g, info = S.scocg_solve(h, z, b, proj_idx=[0, 9999], tol=tol)
            assert info["status"] == 0 and info["iters"] < 400
            G.append(g.cpu().numpy())
        for g in G[1:]:
            assert np.max(np.abs(g - G[0])) <= bound
    finally:
        S.scocg_destroy(h)
