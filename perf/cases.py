"""The work a user of this library has it do, as measurable cases.

Every case goes through the public entry points of paper_0802_0748_gb300
(scocg.py, autograd.py).  The kinds, and what each stands for:

solve      scocg_solve on a tight-binding H in CSR form: Green's functions of
           one right-hand side (dense c = conj(b): a spectrum; unit c: G_ij or
           the local DOS) or of many unit right-hand sides together (G_jj of
           many sites, the block mode behind scocg_density too)
multi      scocg_solve_multi: independent clusters of uneven size in one launch
grad       autograd.shifted_green: G and dL/dH of a spectral loss, the matrix
           set up from the current values as in a training step
ring       scocg_solve on the matrix-free extended Hubbard ring
twoorb     scocg_solve on the matrix-free two-orbital Hubbard cluster
ground     scocg_ground_state of a Hubbard ring
krylov     scocg_krylov_sd_multi: broadened G_jj of many sites by subspace
           diagonalisation
apply      scocg_apply: one y = (z - H) x (a residual check)

Solves run to convergence with residual bounds tight enough that G is a
property of the problem and not of the rounding order.  Matrices, vectors and
shifts are made on the GPU from the seed, with the distributions of
paper_0802_0748_gb300/inputs.py: onsite blocks U[-1, 1], hopping blocks
N(0, 0.25), all rounded to FP32 values, normalised complex Gaussian b.
"""
import math

import numpy as np
import torch

from paper_0802_0748_gb300 import autograd, inputs, scocg

PREC = {"fp64": scocg.FP64, "mixed": scocg.MIXED, "df": scocg.MIXED_DF}
# half bandwidth of the lattices by orbitals per site (0: the chain with weak disorder)
HALF = {0: 2.2, 1: 3.5, 2: 4.6, 3: 5.5, 4: 6.3, 5: 7.0}


def listed():
    return [
        # one-orbital chain, 4096 sites, 64 energies at eta 0.01: launch- and latency-bound FP64 solve
        dict(name="chain4096_fp64", kind="solve", norb=0, L=4096, prec="fp64", nshift=64, eta=0.01, tol=1e-10,
             nrhs=1, nproj=1, dense=False),
        # the smallest solve: local DOS of a 5^3 cluster (500 rows), two projections
        dict(name="cluster5_fp64", kind="solve", norb=4, L=5, prec="fp64", nshift=24, eta=0.1, tol=1e-10, nrhs=1,
             nproj=2, dense=False),
        # the headline: 64^3 x 4 orbitals (1,048,576 rows), 512 energies, compensated FP32, spectrum of a random b
        dict(name="anderson64_df", kind="solve", norb=4, L=64, prec="df", nshift=512, eta=0.05, tol=1e-9, nrhs=1,
             nproj=1, dense=True),
        # the plain FP64 path on a medium lattice (256,000 rows)
        dict(name="anderson40_fp64", kind="solve", norb=4, L=40, prec="fp64", nshift=256, eta=0.05, tol=1e-9, nrhs=1,
             nproj=1, dense=True),
        # G_jj of 32 sites of the 32^3 x 4 lattice, 256 energies: many right-hand sides in one launch
        dict(name="sites32_df", kind="solve", norb=4, L=32, prec="df", nshift=256, eta=0.08, tol=1e-9, nrhs=32,
             nproj=1, dense=False),
        # nine clusters of uneven size (7,000 to 110,000 rows) solved together
        dict(name="clusters9_df", kind="multi", nsys=9, lmin=12, lmax=30, prec="df", nshift=128, eta=0.08, tol=1e-9),
        # one training step on a 16^3 x 4 lattice: sum_k w_k Im G_00(z_k), FP64
        dict(name="grad16_fp64", kind="grad", L=16, nshift=64, eta=0.1, tol=1e-10),
        # extended Hubbard ring, 12 sites at half filling (853,776 states)
        dict(name="ring12_df", kind="ring", L=12, up=6, dn=6, prec="df", nshift=128, eta=0.2, tol=1e-9),
        # two-orbital cluster of eight sites, 3 up and 4 down (1,019,200 states)
        dict(name="twoorb34_df", kind="twoorb", up=3, dn=4, prec="df", nshift=96, eta=0.4, tol=1e-9),
        # ground state of a 12-site ring
        dict(name="ground12_fp64", kind="ground", L=12, up=6, dn=6, m=80, cg=40, tol=1e-11),
        # broadened G_jj of 16 sites by Krylov subspace diagonalisation
        dict(name="krylov16_df", kind="krylov", L=32, prec="df", nrhs=16, nu=200, nshift=256, eta=0.5),
        # one complex64 residual check on the headline matrix
        dict(name="apply64_mixed", kind="apply", L=64, prec="mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes, precisions, shift counts and broadenings over what the listed cases span."""
    kind = rng.choice(["chain", "small", "lattice", "lattice", "lattice64", "sites", "multi", "grad", "ring", "twoorb",
                       "ground", "krylov", "apply"])
    eta = round(rng.uniform(0.06, 0.2), 3)
    if kind == "chain":
        return dict(kind="solve", norb=0, L=_log(rng, 300, 4096), prec=rng.choice(["fp64", "df"]),
                    nshift=_log(rng, 8, 64), eta=round(rng.uniform(0.01, 0.05), 4), tol=1e-10, nrhs=1, nproj=1,
                    dense=False)
    if kind == "small":
        return dict(kind="solve", norb=rng.choice([1, 3, 4, 4, 4]), L=rng.randint(3, 12),
                    prec=rng.choice(["fp64", "df"]), nshift=_log(rng, 8, 128), eta=eta, tol=1e-10, nrhs=1,
                    nproj=rng.randint(1, 4), dense=False)
    if kind == "lattice":
        return dict(kind="solve", norb=rng.choice([1, 4, 4, 4, 5]), L=rng.randint(13, 40),
                    prec=rng.choice(["df", "df", "fp64"]), nshift=_log(rng, 48, 512), eta=eta, tol=1e-9, nrhs=1,
                    nproj=1, dense=rng.random() < 0.7)
    if kind == "lattice64":
        return dict(kind="solve", norb=4, L=rng.randint(41, 64), prec="df", nshift=_log(rng, 64, 512), eta=eta,
                    tol=1e-9, nrhs=1, nproj=1, dense=True)
    if kind == "sites":
        prec = rng.choice(["df", "df", "fp64"])
        return dict(kind="solve", norb=4, L=rng.randint(8, 32 if prec == "df" else 18), prec=prec,
                    nshift=_log(rng, 24, 256), eta=max(eta, 0.08), tol=1e-9, nrhs=rng.randint(2, 32), nproj=1,
                    dense=False)
    if kind == "multi":
        return dict(kind="multi", nsys=rng.randint(2, 9), lmin=rng.randint(8, 14), lmax=rng.randint(18, 30),
                    prec=rng.choice(["df", "df", "fp64"]), nshift=_log(rng, 24, 128), eta=max(eta, 0.1), tol=1e-9)
    if kind == "grad":
        return dict(kind="grad", L=rng.randint(6, 16), nshift=_log(rng, 12, 64), eta=max(eta, 0.1), tol=1e-10)
    if kind == "ring":
        L = rng.randint(9, 12)
        return dict(kind="ring", L=L, up=L // 2 - rng.randint(0, 1), dn=L // 2, prec=rng.choice(["df", "df", "fp64"])
                    if L < 12 else "df", nshift=_log(rng, 24, 128), eta=round(rng.uniform(0.2, 0.4), 3), tol=1e-9)
    if kind == "twoorb":
        return dict(kind="twoorb", up=rng.randint(2, 3), dn=rng.randint(2, 4), prec="df", nshift=_log(rng, 24, 96),
                    eta=round(rng.uniform(0.4, 0.8), 3), tol=1e-9)
    if kind == "ground":
        L = rng.randint(9, 12)
        return dict(kind="ground", L=L, up=L // 2, dn=L // 2, m=rng.choice([60, 80]), cg=rng.choice([30, 40]),
                    tol=1e-11)
    if kind == "krylov":
        return dict(kind="krylov", L=rng.randint(14, 32), prec=rng.choice(["df", "fp64"]), nrhs=rng.randint(2, 16),
                    nu=rng.randint(160, 200), nshift=_log(rng, 32, 256), eta=round(rng.uniform(0.5, 0.7), 3))
    return dict(kind="apply", L=rng.randint(20, 64), prec=rng.choice(["mixed", "df", "fp64"]))


# ---------------------------------------------------------------- inputs
def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + salt)


def _lattice(L, norb, g):
    """CSR (int64 rowptr, int32 col, float64 val) of the periodic L^3 lattice of inputs.anderson_csr."""
    dev, ns = "cuda", L ** 3
    site = torch.arange(ns, device=dev)
    x, y, z = site % L, (site // L) % L, site // (L * L)
    fwd = [(x + 1) % L + L * (y + L * z), x + L * ((y + 1) % L + L * z), x + L * (y + L * ((z + 1) % L))]
    bwd = [(x - 1) % L + L * (y + L * z), x + L * ((y - 1) % L + L * z), x + L * (y + L * ((z - 1) % L))]
    on = torch.rand((ns, norb, norb), generator=g, device=dev, dtype=torch.float64) * 2 - 1
    on = torch.triu(on)
    on = on + torch.triu(on, 1).transpose(1, 2)
    hop = 0.5 * torch.randn((3, ns, norb, norb), generator=g, device=dev, dtype=torch.float64)
    dst = torch.stack([site] + fwd + bwd, 1)
    blk = torch.stack([on] + [hop[d] for d in range(3)] + [hop[d][bwd[d]].transpose(1, 2) for d in range(3)], 1)
    dst, order = dst.sort(1)
    blk = torch.gather(blk, 1, order[:, :, None, None].expand(-1, -1, norb, norb)).float().double()
    col = (dst[:, None, :, None] * norb + torch.arange(norb, device=dev)).expand(-1, norb, -1, -1)
    rowptr = torch.arange(ns * norb + 1, device=dev, dtype=torch.int64) * (7 * norb)
    return rowptr, col.reshape(-1).to(torch.int32).contiguous(), blk.transpose(1, 2).reshape(-1).contiguous()


def _chain(L, g):
    """Open chain with t = -1 and weak onsite disorder U[-0.1, 0.1] (FP32 values)."""
    e = ((torch.rand(L, generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.2).float().double()
    i = torch.arange(L, device="cuda")
    col = torch.stack([i - 1, i, i + 1], 1)
    val = torch.stack([torch.full_like(e, -1.0), e, torch.full_like(e, -1.0)], 1)
    keep = (col >= 0) & (col < L)
    rowptr = torch.zeros(L + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = keep.sum(1).cumsum(0)
    return rowptr, col[keep].to(torch.int32), val[keep]


def _matrix(case, seed, salt=0):
    g = _gen(seed, salt)
    return _chain(case["L"], g) if case.get("norb") == 0 else _lattice(case["L"], case.get("norb", 4), g)


def _unit_complex(n, g):
    v = torch.randn((n, 2), generator=g, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(v / v.norm())


def _energies(K, lo, hi, rs):
    return np.sort(rs.uniform(lo, hi, K))


def _rows(case):
    return case["L"] if case.get("norb") == 0 else case["L"] ** 3 * case.get("norb", 4)


def _solve_inputs(case, seed):
    """H, shifts, right-hand sides [nrhs][n] and projections (indices or vectors) of one lattice solve."""
    rs = np.random.RandomState((seed * 7919 + 13) % (1 << 31))
    H, n, nrhs = _matrix(case, seed), _rows(case), case["nrhs"]
    w = HALF[case["norb"]] if case["norb"] else 2.0
    z = _energies(case["nshift"], -w, w, rs) + 1j * case["eta"]
    if case["dense"]:
        b = _unit_complex(n, _gen(seed, 5))[None, :]
        return H, z, b, None, b.conj().resolve_conj().contiguous()
    j = rs.choice(n, size=nrhs * case["nproj"], replace=False).reshape(nrhs, case["nproj"])
    b = torch.zeros((nrhs, n), dtype=torch.complex128, device="cuda")
    b[torch.arange(nrhs), torch.as_tensor(j[:, 0])] = 1.0
    return H, z, b, j.astype(np.int64), None


def _cluster_sizes(case):
    """Edges spread evenly from lmin to lmax."""
    k = case["nsys"]
    return [round(case["lmin"] + (case["lmax"] - case["lmin"]) * s / max(1, k - 1)) for s in range(k)]


def _multi_inputs(case, seed):
    rs = np.random.RandomState((seed * 7919 + 17) % (1 << 31))
    out = []
    for s, L in enumerate(_cluster_sizes(case)):
        H = _lattice(L, 4, _gen(seed, 100 + s))
        b = _unit_complex(4 * L ** 3, _gen(seed, 200 + s))
        out.append((H, _energies(case["nshift"], -6.5, 6.5, rs) + 1j * case["eta"], b, b.conj().resolve_conj()))
    return out


def _grad_inputs(case, seed):
    rs = np.random.RandomState((seed * 7919 + 19) % (1 << 31))
    H = _lattice(case["L"], 4, _gen(seed))
    n = 4 * case["L"] ** 3
    j = int(rs.randint(n))
    b = torch.zeros(n, dtype=torch.complex128, device="cuda")
    b[j] = 1.0
    w = torch.as_tensor(rs.normal(size=case["nshift"]), device="cuda")
    return H, np.linspace(-6.0, 6.0, case["nshift"]) + 1j * case["eta"], b, j, w


def _hubbard_inputs(case, seed):
    n = _rows_hubbard(case)
    rs = np.random.RandomState((seed * 7919 + 23) % (1 << 31))
    b = _unit_complex(n, _gen(seed, 6))
    lo, hi = (-10.0, 20.0) if case["kind"] == "ring" else (-12.0, 48.0)
    return _energies(case["nshift"], lo, hi, rs) + 1j * case["eta"], b


def _rows_hubbard(case):
    sites = 16 if case["kind"] == "twoorb" else case["L"]
    return math.comb(sites, case["up"]) * math.comb(sites, case["dn"])


def _handle(case, H=None):
    opts = scocg.SolveOptions(precision=PREC[case.get("prec", "fp64")])
    if case["kind"] in ("ring", "ground"):
        return scocg.scocg_create_hubbard(case["L"], case["up"], case["dn"], 1.0, 4.0, 1.0, True, opts=opts)
    if case["kind"] == "twoorb":
        return scocg.scocg_create_hubbard2(inputs.eg_model(), case["up"], case["dn"], opts=opts)
    return scocg.scocg_create_csr(*H, opts=opts)


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "solve":
        H, s["z"], s["b"], s["idx"], s["c"] = _solve_inputs(case, seed)
        s["h"] = _handle(case, H)
    elif kind == "multi":
        sys = _multi_inputs(case, seed)
        s["h"] = [_handle(case, H) for H, _, _, _ in sys]
        s["z"], s["b"], s["c"] = ([q[i] for q in sys] for i in (1, 2, 3))
    elif kind == "grad":
        s["H"], s["z"], s["b"], s["j"], s["w"] = _grad_inputs(case, seed)
        s["val"] = s["H"][2].requires_grad_(True)
    elif kind in ("ring", "twoorb"):
        s["z"], s["b"] = _hubbard_inputs(case, seed)
        s["c"] = s["b"].conj().resolve_conj()[None, :]
        s["h"] = _handle(case)
    elif kind == "ground":
        v = torch.randn(_rows_hubbard(case), generator=_gen(seed, 7), device="cuda", dtype=torch.float64)
        s["v0"] = v / v.norm()
        s["h"] = _handle(case)
    elif kind == "krylov":
        H, s["z"], s["idx"], s["B"] = _krylov_inputs(case, seed)
        s["h"] = _handle(case, H)
    else:
        H, s["z"], s["x"] = _apply_inputs(case, seed)
        s["h"] = _handle(case, H)
    return s


def _krylov_inputs(case, seed):
    rs = np.random.RandomState((seed * 7919 + 29) % (1 << 31))
    H, n = _lattice(case["L"], 4, _gen(seed)), 4 * case["L"] ** 3
    j = rs.choice(n, size=case["nrhs"], replace=False).astype(np.int64)
    B = torch.zeros((case["nrhs"], n), dtype=torch.float64, device="cuda")
    B[torch.arange(case["nrhs"]), torch.as_tensor(j)] = 1.0
    return H, np.linspace(-6.5, 6.5, case["nshift"]) + 1j * case["eta"], j[:, None], B


def _apply_inputs(case, seed):
    rs = np.random.RandomState((seed * 7919 + 31) % (1 << 31))
    H = _lattice(case["L"], 4, _gen(seed))
    x = _unit_complex(4 * case["L"] ** 3, _gen(seed, 8))
    if case["prec"] == "mixed":
        x = x.to(torch.complex64)
    elif case["prec"] == "df":
        v = torch.view_as_real(x)
        hi = v.float()
        x = torch.cat([hi, (v - hi.double()).float()], 1).contiguous()
    return H, complex(rs.uniform(-6, 6), 0.05), x


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("solve", "ring", "twoorb"):
        G, _ = scocg.scocg_solve(s["h"], s["z"], s["b"], proj_idx=s.get("idx"), proj_vec=s.get("c"), tol=case["tol"])
        return G
    if kind == "multi":
        G, _ = scocg.scocg_solve_multi(s["h"], s["z"], s["b"], proj_vec=s["c"], tol=case["tol"])
        return G
    if kind == "grad":
        G = autograd.shifted_green(s["val"], s["H"][0], s["H"][1], s["z"], s["b"], proj_idx=[s["j"]], tol=case["tol"])
        loss = (s["w"] * G[0].imag).sum()
        (g,) = torch.autograd.grad(loss, s["val"])
        return {"G": G.detach(), "grad": g}
    if kind == "ground":
        E, psi, _ = scocg.scocg_ground_state(s["h"], s["v0"], m=case["m"], cg_steps=case["cg"], max_cycles=20,
                                             tol=case["tol"])
        return {"E": E, "psi": psi}
    if kind == "krylov":
        G, used, _ = scocg.scocg_krylov_sd_multi(s["h"], s["B"], case["nu"], s["z"], s["idx"])
        return {"G": G, "used": used}
    return scocg.scocg_apply(s["h"], s["z"], s["x"], PREC[case["prec"]])


# ---------------------------------------------------------------- what the path cannot do without
def _iterations(tol, eta, half):
    """Krylov steps that bring the residual of the least favourable shift down to tol (Chebyshev rate at distance eta)."""
    return math.log(1.0 / tol) / math.asinh(eta / half)


def _lattice_work(n, norb, prec, its, nrhs, nshift, nproj):
    """Per step: H read once (its values in the precision of the path, one index per block), four real operations per
    entry and right-hand side, and the recurrences (about 60 per row); the vectors stay on the chip between steps."""
    nnz = n * (3 if norb == 0 else 7 * norb)
    h = nnz * (8 if prec == "fp64" else 4) + 4 * nnz / max(1, norb * norb)
    vec = 16.0 * n * nrhs
    return {"bytes": its * h + 2 * vec + 16.0 * nrhs * nproj * nshift,
            "flops": its * nrhs * (4.0 * nnz + 60.0 * n)}


def work(case):
    kind = case["kind"]
    if kind == "solve":
        its = _iterations(case["tol"], case["eta"], HALF[case["norb"]])
        return _lattice_work(_rows(case), case["norb"], case["prec"], its, case["nrhs"], case["nshift"], case["nproj"])
    if kind == "multi":
        its = _iterations(case["tol"], case["eta"], HALF[4])
        each = [_lattice_work(4 * L ** 3, 4, case["prec"], its, 1, case["nshift"], 1) for L in _cluster_sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "grad":   # per step also p and x of every shift: 16 operations per row; then one product per entry and shift
        n, K = 4 * case["L"] ** 3, case["nshift"]
        its = _iterations(case["tol"], case["eta"], HALF[4])
        w = _lattice_work(n, 4, "fp64", its, 1, K, 1)
        return {"bytes": w["bytes"] + 16.0 * n * K + 28 * n * 20, "flops": w["flops"] + 16.0 * its * n * K + 112.0 * n * K}
    if kind in ("ring", "twoorb"):
        n = float(_rows_hubbard(case))
        its = _iterations(case["tol"], case["eta"], 15.0 if kind == "ring" else 30.0)
        hops = 13 if kind == "ring" else 60
        return {"bytes": 32.0 * n + (96.0 * n * its if 32.0 * n > 1.2e8 else 0.0) + 16.0 * case["nshift"],
                "flops": its * n * (4.0 * hops + 60.0)}
    if kind == "ground":
        n = float(_rows_hubbard(case))
        return {"bytes": 16.0 * n + 16.0 * n * case["m"], "flops": 2.0 * (case["m"] + case["cg"]) * n * 20.0}
    if kind == "krylov":
        n, nu, R = 4 * case["L"] ** 3, case["nu"], case["nrhs"]
        return {"bytes": nu * (28.0 * n * (4 if case["prec"] == "df" else 8)) + 16.0 * n * R + 16.0 * R * case["nshift"],
                "flops": nu * R * n * 66.0 + R * 60.0 * nu * nu}
    n = 4 * case["L"] ** 3
    v = {"mixed": 8, "df": 16, "fp64": 16}[case["prec"]]
    return {"bytes": 28.0 * n * (8 if case["prec"] == "fp64" else 4) + 7.0 * n + 2.0 * v * n, "flops": n * 120.0}


# ---------------------------------------------------------------- the same in 64 bits with plain torch and numpy
def _csr_apply(H, n):
    A = torch.sparse_csr_tensor(H[0], H[1].long(), H[2], size=(n, n))

    def mul(x):   # complex [n, T] or real [n, T]
        if not x.is_complex():
            return A @ x
        T = x.shape[1]
        return torch.view_as_complex((A @ torch.view_as_real(x).reshape(n, 2 * T)).reshape(n, T, 2).contiguous())
    return mul


def _cocg(mul, b, z, idx=None, c=None, tol=1e-13, full=False):
    """Shifted COCG in complex128: c^T (z - H)^{-1} b as [T][M][K] for the columns of b [n, T]; full: x [n, K] (T = 1)."""
    dev = b.device
    z = torch.as_tensor(z, dtype=torch.complex128, device=dev)
    n, T, K = b.shape[0], b.shape[1], z.numel()
    zs = z[int(np.argsort(z.real.cpu().numpy())[K // 2])]
    sigma = z - zs
    proj = (lambda r: r[idx, torch.arange(T, device=dev)[:, None]]) if idx is not None else (lambda r: (c @ r).T)
    one = torch.ones((T, K), dtype=torch.complex128, device=dev)
    pi, pi0, r, p = one.clone(), one.clone(), b.clone(), b.clone()
    rho, al0, be0 = (r * r).sum(0), one[:, 0].clone(), 0 * one[:, 0]
    bn = b.norm(dim=0)
    cr = proj(r)
    P = torch.zeros((T, cr.shape[1], K), dtype=torch.complex128, device=dev)
    X = P.clone()
    live = torch.ones((T, K), dtype=torch.bool, device=dev)
    if full:
        Pf = torch.zeros((n, K), dtype=torch.complex128, device=dev)
        Xf = Pf.clone()
    for it in range(60000):
        q = zs * p - mul(p)
        al = rho / (p * q).sum(0)
        bk = (pi0 / pi) ** 2 * be0[:, None]
        pin = (1 + al[:, None] * sigma) * pi + (al * be0 / al0)[:, None] * (pi - pi0)
        ak = pi / pin * al[:, None]
        Pn = cr[:, :, None] / pi[:, None, :] + bk[:, None, :] * P
        P = torch.where(live[:, None, :], Pn, P)
        X = torch.where(live[:, None, :], X + ak[:, None, :] * Pn, X)
        if full:
            Pf = r / pi + bk * Pf
            Xf = torch.where(live, Xf + ak * Pf, Xf)
        r = r - al * q
        rho, rho0 = (r * r).sum(0), rho
        be0, al0 = rho / rho0, al
        p = r + be0 * p
        cr = proj(r)
        pi0, pi = torch.where(live, pi, pi0), torch.where(live, pin, pi)
        live = live & (r.norm(dim=0)[:, None] / pi.abs() > tol * bn[:, None])
        if it % 32 == 31:
            if not bool(live.any()):
                break
            f = bn / r.norm(dim=0)   # the recurrences are homogeneous: keep a converged seed's r in range
            r, p, cr, rho = r * f, p * f, cr * f[:, None], rho * f * f
            pi, pi0 = pi * f[:, None], pi0 * f[:, None]
    return (X, Xf) if full else X


def _spin_states(modes, k):
    st = np.array([s for s in range(1 << modes) if bin(s).count("1") == k], dtype=np.int64)
    return st, {int(s): i for i, s in enumerate(st)}


def _spin_op(st, rank, terms):
    """Sparse matrix of sum t c+_i c_j over the terms (t, i, j) within one spin's states (Jordan-Wigner signs)."""
    r, c, v = [], [], []
    for col, s in enumerate(st):
        s = int(s)
        for t, i, j in terms:
            if not (s >> j) & 1 or (i != j and (s >> i) & 1):
                continue
            s1 = s ^ (1 << j)
            sg = bin(s & ((1 << j) - 1)).count("1") + bin(s1 & ((1 << i) - 1)).count("1")
            r.append(rank[s1 | (1 << i)]); c.append(col); v.append(-t if sg & 1 else t)
    A = torch.sparse_coo_tensor(torch.tensor([r, c], device="cuda"), torch.tensor(v, dtype=torch.float64, device="cuda"),
                                (len(st), len(st)))
    return A.coalesce().to_sparse_csr()


def _occ(st, modes):
    return torch.as_tensor(((st[:, None] >> np.arange(modes)) & 1).astype(np.float64), device="cuda")


def _hubbard_mul(case):
    """H x of the ring or the two-orbital cluster on x [n, T] (T = 1), from its definition: spin-wise hopping matrices,
    a diagonal, and (two orbitals) products of one orbital move of each spin."""
    pairs = []
    if case["kind"] == "twoorb":
        m = inputs.eg_model()
        modes = 16
        hops = [(m["bond_t"][k][a][b], p, q) for k, (i, j) in enumerate(m["bonds"]) for a in (0, 1) for b in (0, 1)
                for p, q in ((2 * i + a, 2 * j + b), (2 * j + b, 2 * i + a))]
    else:
        modes = case["L"]
        bonds = [(i, (i + 1) % modes) for i in range(modes)]
        hops = [(-1.0, p, q) for i, j in bonds for p, q in ((i, j), (j, i))]
    su, ru = _spin_states(modes, case["up"])
    sd, rd = _spin_states(modes, case["dn"])
    Hu, Hd = _spin_op(su, ru, hops), _spin_op(sd, rd, hops)
    nu, nd = _occ(su, modes), _occ(sd, modes)
    Du, Dd = len(su), len(sd)
    if case["kind"] == "twoorb":
        a, b = slice(0, None, 2), slice(1, None, 2)
        Nu, Nd = nu[:, a] + nu[:, b], nd[:, a] + nd[:, b]
        diag = m["U"] * nu @ nd.T + m["Up"] * (nu[:, a] @ nd[:, b].T + nu[:, b] @ nd[:, a].T)
        diag = diag + (m["Up"] - m["J"]) * ((nu[:, a] * nu[:, b]).sum(1)[:, None] + (nd[:, a] * nd[:, b]).sum(1)[None, :])
        for i, j in m["bonds"]:
            diag = diag + m["V"] * (Nu[:, i][:, None] + Nd[:, i][None, :]) * (Nu[:, j][:, None] + Nd[:, j][None, :])
        for i in range(8):
            mv = [[_spin_op(s, r, [(1.0, 2 * i + d, 2 * i + 1 - d)]) for d in (0, 1)] for s, r in ((su, ru), (sd, rd))]
            pairs += [(m["J"] if d != e else m["Jp"], mv[0][d], mv[1][e]) for d in (0, 1) for e in (0, 1)]
    else:
        diag = 4.0 * nu @ nd.T
        for i, j in bonds:
            diag = diag + (nu[:, i][:, None] + nd[:, i][None, :]) * (nu[:, j][:, None] + nd[:, j][None, :])

    def right(A, x):   # (1 x A) x
        return (A @ x.permute(1, 0, 2).reshape(Dd, -1)).reshape(Dd, Du, 2).permute(1, 0, 2)

    def left(A, x):
        return (A @ x.reshape(Du, -1)).reshape(Du, Dd, 2)

    def mul(x):
        v = torch.view_as_real(x).reshape(Du, Dd, 2)
        y = diag[:, :, None] * v + left(Hu, v) + right(Hd, v)
        for t, A, B in pairs:
            y = y + t * right(B, left(A, v))
        return torch.view_as_complex(y.reshape(-1, 1, 2).contiguous())
    return mul


def _lanczos(mul, v, m):
    """alpha, beta and the basis [m, n] of m fully reorthogonalised Lanczos steps from the unit vector v."""
    V = torch.zeros((m, v.numel()), dtype=torch.float64, device=v.device)
    al, be = torch.zeros(m, dtype=torch.float64), torch.zeros(m, dtype=torch.float64)
    V[0] = v
    for j in range(m):
        w = mul(V[j][:, None])[:, 0]
        al[j] = V[j] @ w
        for _ in range(2):
            w = w - V[:j + 1].T @ (V[:j + 1] @ w)
        be[j] = w.norm()
        if j + 1 < m:
            V[j + 1] = w / be[j]
    return al.numpy(), be.numpy(), V


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        H, z, b, idx, c = _solve_inputs(case, seed)
        return _cocg(_csr_apply(H, _rows(case)), b.T.contiguous(), z, None if idx is None else
                     torch.as_tensor(idx, device="cuda"), c)
    if kind == "multi":
        return [_cocg(_csr_apply(H, b.numel()), b[:, None], z, c=c[None, :])[0] for H, z, b, c in _multi_inputs(case, seed)]
    if kind == "grad":
        H, z, b, j, w = _grad_inputs(case, seed)
        n = b.numel()
        G, x = _cocg(_csr_apply(H, n), b[:, None], z, torch.as_tensor([[j]], device="cuda"), full=True)
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), H[0].diff())
        y = x * torch.conj(1j * w)[None, :]
        grad = torch.cat([(y[r] * x[k.long()]).sum(1).real for r, k in zip(row.split(1 << 18), H[1].split(1 << 18))])
        return {"G": G[0], "grad": grad}
    if kind in ("ring", "twoorb"):
        z, b = _hubbard_inputs(case, seed)
        return _cocg(_hubbard_mul(case), b[:, None], z, c=b.conj()[None, :].resolve_conj())
    if kind == "ground":   # the sign of psi is free
        v = torch.randn(_rows_hubbard(case), generator=_gen(seed, 7), device="cuda", dtype=torch.float64)
        f = _hubbard_mul(dict(case, kind="ring"))
        al, be, _ = _lanczos(lambda x: f(x.to(torch.complex128)).real, v / v.norm(), 160)
        return {"E": float(np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))[0]), "psi": None}
    if kind == "krylov":
        H, z, idx, B = _krylov_inputs(case, seed)
        mul, out = _csr_apply(H, B.shape[1]), []
        for k in range(case["nrhs"]):
            al, be, V = _lanczos(mul, B[k], case["nu"])
            e, s = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
            wt = (V[:, int(idx[k, 0])].cpu().numpy() @ s) * s[0]
            out.append([(wt[None, :] / (z[:, None] - e[None, :])).sum(1)])
        return {"G": np.array(out), "used": None}
    H, z, x = _apply_inputs(case, seed)
    if case["prec"] == "df":
        x = torch.view_as_complex((x[:, :2].double() + x[:, 2:].double()).contiguous())
    x = x.to(torch.complex128)
    y = z * x - _csr_apply(H, x.numel())(x[:, None])[:, 0]
    if case["prec"] == "df":   # the sum of the pairs is y; each pair's high part is its nearest FP32 value
        v = torch.view_as_real(y)
        return torch.cat([v.float().double(), v - v.float().double()], 1)
    return y
