"""Full-vector solves on the matrix-free handles with as many shifts as one
launch takes (512), and with a number whose shift scalars pass the 48 KB that a
kernel may use without asking: each as the first full-vector solve of a fresh
process, since the limit, once raised, stays raised.

Bound: a residual of tol leaves |dx| <= tol / eta = 4e-12 (unit b, eta = 0.25);
1e-10 leaves room for the recurrences' rounding, u * iterations / eta < 1e-12.
"""
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parents[1]

CODE = """
import sys
import numpy as np, torch
import __graft_entry__
__graft_entry__.build()
import oracle
from paper_0802_0748_gb300 import inputs, scocg as S
oracle.build()
model, K = sys.argv[1], int(sys.argv[2])
if model == "ring":
    h = S.scocg_create_hubbard(6, 3, 3, 1.0, 4.0, 1.0, True)
    rp, c, v = oracle.hubbard_csr(6, 3, 3, 1.0, 4.0, 1.0, True)
else:
    m = inputs.eg_model()
    h = S.scocg_create_hubbard2(m, 1, 1)
    rp, c, v = oracle.hubbard2_csr(m, 1, 1)
n = rp.size - 1
assert S.scocg_dim(h) == n
H = np.zeros((n, n))
H[np.repeat(np.arange(n), np.diff(rp)), c] = v
e, U = np.linalg.eigh(H)
z = np.linspace(e[0] - 1.0, e[-1] + 1.0, K) + 0.25j
b = inputs.random_unit_complex(n, 3)
X, info = S.scocg_solve_full(h, z, torch.from_numpy(b).cuda(), tol=1e-12)
assert info["status"] == 0
want = ((U.T @ b)[None, :] / (z[:, None] - e[None, :])) @ U.T
err = float(np.max(np.abs(X.cpu().numpy().reshape(K, n) - want)))
assert err <= 1e-10, err
print("OK")
"""


@pytest.mark.parametrize("model,K", [("two-orbital", 400), ("two-orbital", 512), ("ring", 512)])
def test_full_solve_many_shifts_first(model, K):
    r = subprocess.run([sys.executable, "-c", CODE, model, str(K)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout + r.stderr[-2000:]
