"""The compensated apply's error against wider arithmetic is that of its steps as
stated: per term an exact product (FMA TwoProd), its remainder with the low
part's product, a TwoSum into the high part and one addition of the remainders
to the low part; then z x, normalised, and one compensated difference.  Forms
with more roundings of the low part are told apart: the remainders folded into
one fused operation have a 2 % larger rms error at 28 terms, z x accumulated
onto the negated sum a 4 to 20 % larger one.

The steps are restated here in NumPy (an FP32 FMA as FP64 arithmetic rounded once
more, which differs from a true FMA in one case in 2^29), a row's terms in the
layout's order (one lane a row, four lanes a row, 4x4 blocks).  Both errors are
rms values over the same N >= 2.5e5 rows and both parts of a complex x; the
relative spread of their ratio is below 1 / sqrt(N) = 0.2 % even if the orders
differed, so the kernel may be at most 1 % above the restatement.
"""
import numpy as np
import pytest

from paper_0802_0748_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
f32, f64, ld = np.float32, np.float64, np.longdouble


@pytest.fixture(scope="module")
def S():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0802_0748_gb300 import scocg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return scocg


def fma(a, b, c):
    return (a.astype(f64) * b.astype(f64) + c.astype(f64)).astype(f32)


def two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def norm(h, l):
    s = h + l
    return s, l - (s - h)


def row_sums(val, xh, xl, lanes):
    """Row sums of val * (xh + xl), [rows][terms], terms dealt to `lanes` accumulators: (hi, lo)."""
    acc = []
    for i in range(lanes):
        ah = np.zeros(val.shape[0], f32)
        al = np.zeros_like(ah)
        for j in range(i, val.shape[1], lanes):
            v, h, l = val[:, j], xh[:, j], xl[:, j]
            p = v * h
            e = fma(v, l, fma(v, h, -p))
            s, t = two_sum(ah, p)
            ah, al = s, al + (t + e)
        acc.append((ah, al))
    o = lanes // 2
    while o:
        n = [(norm(*a), norm(*acc[i ^ o])) for i, a in enumerate(acc)]
        acc = []
        for (ah, al), (bh, bl) in n:
            s, e = two_sum(ah, bh)
            acc.append(norm(s, e + (al + bl)))
        o //= 2
    return acc[0]


def add_product(h, l, a, b):
    (ah, al), (bh, bl) = a, b
    p = ah * bh
    e = fma(ah, bl, fma(al, bh, fma(ah, bh, -p)))
    s, t = two_sum(h, p)
    return s, l + (t + e)


def z_x_minus(terms, acc):
    """sum of the products minus acc, as the apply ends: (hi, lo)."""
    h = np.zeros_like(acc[0])
    l = np.zeros_like(h)
    for a, b in terms:
        h, l = add_product(h, l, a, b)
    h, l = norm(h, l)
    s, e = two_sum(h, -acc[0])
    return norm(s, e + (l - acc[1]))


def pair(x):
    hi = np.asarray(x).astype(f32)
    return hi, (x - hi).astype(f32)


def wide(p):
    return p[0].astype(ld) + p[1]


# 4x4 blocks (28 terms a row), four lanes a row (7 terms), one lane (3 terms)
@pytest.mark.parametrize("z", [0.0, 0.1 + 0.05j, 1.3 + 0.05j])
@pytest.mark.parametrize("norb,L,lanes", [(4, 40, 1), (1, 64, 4), (0, 262144, 1)])
def test_apply_error_is_that_of_its_steps(S, norb, L, lanes, z):
    if norb:
        h_csr = inputs.anderson_csr(L, seed=3, norb=norb)
    else:
        h_csr = inputs.chain_csr(L, t=float(f32(-0.9)), onsite=float(f32(0.37)))
    n = h_csr.n
    per_row = np.diff(h_csr.rowptr)
    m = int(per_row.max())
    rows = np.flatnonzero(per_row == m)
    at = h_csr.rowptr[rows][:, None] + np.arange(m)
    val, col = h_csr.val[at].astype(f32), h_csr.col[at]
    assert np.array_equal(val.astype(f64), h_csr.val[at])
    hi, lo = pair(np.random.default_rng(17).normal(size=(n, 2)))
    h = S.scocg_create_csr(h_csr.rowptr, h_csr.col, h_csr.val)
    try:
        y = S.scocg_apply(h, z, torch.from_numpy(np.concatenate([hi, lo], 1)).cuda(),
                          precision=S.MIXED_DF).cpu().numpy()[rows]
    finally:
        S.scocg_destroy(h)
    zz = [pair(np.full(rows.size, c)) for c in (complex(z).real, complex(z).imag)]
    minus_zi = tuple(-c for c in zz[1])
    x = [(hi[rows, c], lo[rows, c]) for c in range(2)]
    got, ref = [], []
    for part, terms in ((0, [(zz[0], x[0]), (minus_zi, x[1])]), (1, [(zz[0], x[1]), (zz[1], x[0])])):
        xh, xl = hi[col, part], lo[col, part]
        exact = sum(wide(a) * wide(b) for a, b in terms) - (val.astype(ld) * (xh.astype(ld) + xl)).sum(1)
        got.append(y[:, part].astype(ld) + y[:, 2 + part] - exact)
        ref.append(wide(z_x_minus(terms, row_sums(val, xh, xl, lanes))) - exact)
    rms = [float(np.sqrt(np.mean(np.concatenate(e) ** 2))) for e in (got, ref)]
    print(f"{norb} orbitals, z {z}: rms error {rms[0]:.4e}, restated {rms[1]:.4e}, ratio {rms[0] / rms[1]:.4f}")
    assert rms[0] <= 1.01 * rms[1]
