"""Performance cases: what a user of this package has it do, and how long it takes.

A case is one call of a public entry point (or the few calls that belong
together) on one problem size.  The sizes are those of the configurations
this repository is measured and tested on (N = 16 Nk with Nv = Nc = 4 from 256
to 20000, nev 20 to 100, nex half of that, tol 1e-10, degree 20 in the first
filter and up to 36 after it), the serving mix between them (N = 1000 ..
16000, nev 10 .. 100) and ragged neighbours of both.

Matrices are exciton Hamiltonians of the shape the package is made for: a
diagonal of transition energies, a rank-8 exchange term and a screened direct
term that decays along a ring of k-points.  They are built here with torch,
so that the reference results need none of the package's code.
"""
import math

import numpy as np
import torch

import paper_2006_08498_gb300 as chase

PRECISION = {"fp64": chase.CHASE_FP64, "mixed": chase.CHASE_MIXED_FP32, "dfma": chase.CHASE_FP64_DFMA}


def listed():
    return [
        # one product H Y of a small problem: latency and launches
        dict(name="product_n256_w30", kind="product", Nk=16, Nv=4, Nc=4, n=30, precision="fp64", half=False),
        # the product of a late iteration: few columns left, a ragged size, memory rather than arithmetic
        dict(name="product_n10008_w24", kind="product", Nk=1251, Nv=4, Nc=2, n=24, precision="fp64", half=False),
        # the product on one triangle of H, for matrices that fit the device no other way
        dict(name="product_half_n6000_w70", kind="product", Nk=375, Nv=4, Nc=4, n=70, precision="fp64", half=True),
        # a later filter of the N = 2000 problem: a degree of its own for every column
        dict(name="filter_n2000_m75", kind="filter", Nk=125, Nv=4, Nc=4, m=75, deg_lo=8, deg_hi=36, precision="fp64"),
        # the first filter of the N = 20000 problem: all columns, one degree
        dict(name="filter_n20000_m140", kind="filter", Nk=1250, Nv=4, Nc=4, m=140, deg_lo=20, deg_hi=20, precision="fp64"),
        # the first filter of the mixed-precision mode at a serving size
        dict(name="filter_mixed_n8000_m96", kind="filter", Nk=500, Nv=4, Nc=4, m=96, deg_lo=20, deg_hi=20, precision="mixed"),
        # orthonormalisation of a block against the pairs that are locked already
        dict(name="qr_n20000_m100_k40", kind="qr", N=20000, m=100, k=40),
        # Rayleigh-Ritz: product, projected matrix, its eigenpairs, back-transformation, residuals
        dict(name="rr_n6006_m111", kind="rr", Nk=462, Nv=13, Nc=1, m=111, precision="fp64"),
        # a Gram product of two tall blocks in native FP64
        dict(name="gram_k20000_140x40", kind="gram", K=20000, m1=140, m2=40),
        # the spectral estimate before the first filter: narrow products one after another
        dict(name="lanczos_n8000", kind="lanczos", Nk=500, Nv=4, Nc=4, m=100, precision="fp64"),
        # whole solves: the smallest configuration and the N = 20000 one
        dict(name="solve_n2000", kind="solve", Nk=125, Nv=4, Nc=4, nev=50, nex=25, how="stored", precision="fp64", group=0),
        dict(name="solve_n20000", kind="solve", Nk=1250, Nv=4, Nc=4, nev=100, nex=40, how="stored", precision="fp64", group=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pairs(rng, lo, hi):
    """(Nk, Nv, Nc) with N = Nk Nv Nc between about lo and hi, ragged as a rule."""
    Nv, Nc = rng.choice([(4, 4), (4, 4), (3, 5), (4, 2), (2, 7), (13, 1)])
    return dict(Nk=max(3, _log(rng, lo, hi) // (Nv * Nc)), Nv=Nv, Nc=Nc)


def draw(rng):
    kind = rng.choice(["product", "product", "filter", "filter", "qr", "rr", "gram", "lanczos", "solve", "solve"])
    if kind == "product":
        p = rng.choice(["fp64", "fp64", "fp64", "mixed", "dfma"])
        return dict(kind=kind, n=_log(rng, 1, 300), precision=p, half=p == "fp64" and rng.random() < 0.3,
                    **_pairs(rng, 320, 4000 if p == "dfma" else 20000))
    if kind == "filter":
        lo = rng.randrange(2, 25)
        return dict(kind=kind, m=_log(rng, 8, 200), deg_lo=lo, deg_hi=rng.randrange(lo, 37),
                    precision=rng.choice(["fp64", "fp64", "mixed"]), **_pairs(rng, 320, 16000))
    if kind == "qr":
        return dict(kind=kind, N=_log(rng, 700, 20000), m=_log(rng, 10, 200), k=rng.choice([0, rng.randrange(1, 100)]))
    if kind == "rr":
        return dict(kind=kind, m=_log(rng, 15, 200), precision=rng.choice(["fp64", "fp64", "mixed"]), **_pairs(rng, 320, 16000))
    if kind == "gram":
        return dict(kind=kind, K=_log(rng, 300, 50000), m1=_log(rng, 1, 200), m2=_log(rng, 1, 200))
    if kind == "lanczos":
        return dict(kind=kind, m=rng.randrange(20, 150), precision="fp64", **_pairs(rng, 1000, 16000))
    nev = _log(rng, 10, 60)
    how = rng.choice(["stored", "stored", "half", "generated"])
    return dict(kind=kind, nev=nev, nex=max(10, nev // 2), how=how, precision=rng.choice(["fp64", "fp64", "mixed"]),
                group=rng.choice([0, 48]), Nk=_log(rng, 20, 600), Nv=4, Nc=4)


# ------------------------------------------------------------------ inputs

def _unif(seed, stream, idx):
    """Top 53 bits of SplitMix64(seed ^ stream << 56 ^ idx) as a number in [0, 1)."""
    def signed(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    def shifted(z, by):
        return (z >> by) & ((1 << (64 - by)) - 1)

    z = (idx ^ signed((seed ^ (stream << 56)) & ((1 << 64) - 1))) + signed(0x9E3779B97F4A7C15)
    z = (z ^ shifted(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shifted(z, 27)) * signed(0x94D049BB133111EB)
    z = z ^ shifted(z, 31)
    return shifted(z, 11).double() * 2.0 ** -53


def _hamiltonian(seed, Nk, Nv, Nc, gap=2.0, w0=0.3, x0=0.5, jitter=0.01, rank=8):
    """The seeded model Hamiltonian (default model of the package) as a column-major N x N complex128 tensor."""
    dev, N, nb = "cuda", Nk * Nv * Nc, Nv * Nc
    I = torch.arange(N, device=dev)
    c, v, k = I % Nc, (I // Nc) % Nv, I // nb
    s = (1.0 - torch.cos(2.0 * math.pi * k.double() / Nk)) / 2.0
    xi = 2.0 * _unif(seed, 1, k * Nc + c) - 1.0
    dE = (gap / 2.0 + c + 3.0 * s + jitter * xi) - (-gap / 2.0 - 0.5 * v - 2.0 * s)
    u = torch.polar(torch.ones(N, dtype=torch.float64, device=dev), 2.0 * math.pi * _unif(seed, 3, I))
    idx = 2 * (rank * I[:, None] + torch.arange(rank, device=dev)[None, :])
    amp = math.sqrt(3.0 * x0 / N) / math.sqrt(2.0)
    a = torch.complex(amp * (2.0 * _unif(seed, 2, idx) - 1.0), amp * (2.0 * _unif(seed, 2, idx + 1) - 1.0))
    T = torch.matmul(a.conj() * 2.0, a.T)        # row j of T is column j of H
    ks = torch.arange(Nk, device=dev)
    d = (ks[:, None] - ks[None, :]).abs()
    d = torch.minimum(d, Nk - d).double()
    W = w0 / (d * d + 0.5)
    for b in range(nb):
        ub = u[b::nb]
        T[b::nb, b::nb] -= W * torch.outer(ub.conj(), ub)
    i = torch.arange(N, device=dev)
    T[i, i] = torch.complex(T[i, i].real + dE, torch.zeros_like(dE))
    return T.T


def _block(seed, rows, cols, key=0):
    """Column-major block of independent normal entries."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * key + int(seed))
    return torch.randn((cols, rows), dtype=torch.complex128, device="cuda", generator=g).T


def _orthonormal(seed, rows, cols, key):
    q, _ = torch.linalg.qr(_block(seed, rows, cols, key))
    return q.T.contiguous().T


def _skewed(seed, rows, cols, L):
    """A block as the filter leaves it: columns of unequal length, leaning on each other and on L."""
    X = _block(seed, rows, cols, 5)
    if L is not None:
        X = X + L @ _block(seed, L.shape[1], cols, 6)
    X = X + 3.0 * X[:, :1]
    X = X * torch.logspace(0, -3, cols, dtype=torch.float64, device="cuda")[None, :]
    return X.T.contiguous().T


def _degrees(case):
    lo, hi, m = case["deg_lo"], case["deg_hi"], case["m"]
    return [lo + (hi - lo) * j // max(1, m - 1) for j in range(m)]


# The interval that the filter damps and the point that it is normalised at, as the N = 2000 problem's first iterations have them.
LOWER, ALPHA, BETA = 1.3, 3.2, 12.4


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, ctx=chase.Context(0), seed=int(seed))
    if kind == "qr":
        s["L"] = _orthonormal(seed, case["N"], case["k"], 4) if case["k"] else None
        s["X"] = _skewed(seed, case["N"], case["m"], s["L"])
        s["V"] = chase.colmajor_empty(case["N"], case["m"])
        return s
    if kind == "gram":
        s["A"], s["B"] = _block(seed, case["K"], case["m1"], 1), _block(seed, case["K"], case["m2"], 2)
        s["G"] = chase.colmajor_empty(case["m1"], case["m2"])
        return s
    N = case["Nk"] * case["Nv"] * case["Nc"]
    if kind != "solve" or case["how"] != "generated":
        s["H"] = _hamiltonian(seed, case["Nk"], case["Nv"], case["Nc"])
    if kind == "product":
        s["Y"] = _block(seed, N, case["n"], 1)
        s["C"] = chase.colmajor_empty(N, case["n"])
    elif kind == "filter":
        s["X"] = _block(seed, N, case["m"], 1)
        s["V"] = chase.colmajor_empty(N, case["m"])
        s["deg"] = np.array(_degrees(case), dtype=np.int32)
    elif kind == "rr":
        s["Q"] = _orthonormal(seed, N, min(case["m"], N), 1)
    elif kind == "solve":
        s["Z"] = chase.colmajor_empty(N, case["nev"])
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    prec = PRECISION[case.get("precision", "fp64")]
    if kind == "product":
        return ctx.hemm(s["H"], s["Y"], precision=prec, out=s["C"], half_storage=case["half"])
    if kind == "filter":                          # in place: a fresh block each time
        s["V"].copy_(s["X"])
        mv = ctx.filter(s["H"], s["V"], s["deg"], LOWER, (ALPHA + BETA) / 2, (BETA - ALPHA) / 2, precision=prec)
        return s["V"], mv
    if kind == "qr":
        s["V"].copy_(s["X"])
        return ctx.qr(s["V"], s["L"])
    if kind == "rr":
        theta, V, HV, resid = ctx.rayleigh_ritz(s["H"], s["Q"], norm=12.0, precision=prec)
        return theta, V, HV, resid
    if kind == "gram":
        return ctx.gram(s["A"], s["B"], out=s["G"])
    if kind == "lanczos":
        return ctx.lanczos(s["H"], case["m"], seed=s["seed"], precision=prec)
    # The eigenvectors and residuals are written to the caller's buffers too.  They are not among the outputs: tol = 1e-10 leaves the vectors
    # undetermined to about tol ||H|| / gap (1e-8 and more) and the residuals (below tol ||H||) wholly, so two correct solves differ by that much.
    kw = dict(tol=1e-10, deg_max=36, precision=prec, evecs=s["Z"], degree_group=case["group"])
    if case["how"] == "generated":
        return ctx.solve_bse(s["seed"], case["Nk"], case["Nv"], case["Nc"], case["nev"], case["nex"], **kw)[0]
    return ctx.solve(s["H"], case["nev"], case["nex"], half_storage=case["how"] == "half", **kw)[0]


def work(case):
    """Bytes that come in and go out once, and the flops of the complex FP64 arithmetic asked for (8 per multiply-add)."""
    z, kind = 16.0, case["kind"]
    if kind == "qr":
        N, m, k = case["N"], case["m"], case["k"]
        return dict(bytes=z * N * (2 * m + k), flops=8.0 * N * (2 * m * k + m * m))
    if kind == "gram":
        K, a, b = case["K"], case["m1"], case["m2"]
        return dict(bytes=z * (K * (a + b) + a * b), flops=8.0 * K * a * b)
    N = case["Nk"] * case["Nv"] * case["Nc"]
    H = z * N * N * (0.5 if case.get("half") or case.get("how") == "half" else 1.0)
    if kind == "product":
        return dict(bytes=H + 2 * z * N * case["n"], flops=8.0 * N * N * case["n"])
    if kind == "filter":
        return dict(bytes=H + 2 * z * N * case["m"], flops=8.0 * N * N * sum(_degrees(case)))
    if kind == "rr":
        m = min(case["m"], N)
        return dict(bytes=H + 3 * z * N * m, flops=8.0 * (N * N * m + 3.0 * N * m * m))
    if kind == "lanczos":
        return dict(bytes=H, flops=8.0 * N * N * 4 * 25)
    # a solve: at least one filter of degree 20 over the whole block, and one Rayleigh-Ritz product
    if case["how"] == "generated":
        H = 0.0
    return dict(bytes=H + z * N * case["nev"], flops=8.0 * N * N * (case["nev"] + case["nex"]) * 21)


# --------------------------------------------------------- reference results

def exact(case, seed):
    kind = case["kind"]
    if kind == "gram":
        return _block(seed, case["K"], case["m1"], 1).conj().T @ _block(seed, case["K"], case["m2"], 2)
    if kind == "qr":
        L = _orthonormal(seed, case["N"], case["k"], 4) if case["k"] else None
        X = _skewed(seed, case["N"], case["m"], L)
        for _ in range(2 if L is not None else 0):
            X = X - L @ (L.conj().T @ X)
        q, r = torch.linalg.qr(X)
        d = torch.diagonal(r)
        return q * (d / d.abs())[None, :]
    N = case["Nk"] * case["Nv"] * case["Nc"]
    if kind == "lanczos":
        return None
    if kind == "solve":
        if N > 2500:
            return None
        return torch.linalg.eigvalsh(_hamiltonian(seed, case["Nk"], case["Nv"], case["Nc"]))[:case["nev"]].cpu().numpy()
    H = _hamiltonian(seed, case["Nk"], case["Nv"], case["Nc"])
    if kind == "product":
        return H @ _block(seed, N, case["n"], 1)
    if kind == "filter":
        degs = _degrees(case)
        if 8.0 * N * N * sum(degs) > 1.2e13:
            return None
        c, e = (ALPHA + BETA) / 2, (BETA - ALPHA) / 2
        out = torch.empty((N, case["m"]), dtype=torch.complex128, device="cuda")
        s1 = e / (LOWER - c)
        prev, sig = _block(seed, N, case["m"], 1), s1
        cur = (s1 / e) * (H @ prev - c * prev)
        at = torch.tensor(degs, device="cuda")
        out[:, at == 1] = cur[:, at == 1]
        for t in range(1, max(degs)):
            new = 1.0 / (2.0 / s1 - sig)
            prev, cur = cur, (2.0 * new / e) * (H @ cur - c * cur) - (sig * new) * prev
            sig = new
            out[:, at == t + 1] = cur[:, at == t + 1]
        return out, None
    m = min(case["m"], N)                         # Rayleigh-Ritz: vectors up to a phase, so values and residuals only
    Q = _orthonormal(seed, N, m, 1)
    W = H @ Q
    G = Q.conj().T @ W
    th, Y = torch.linalg.eigh((G + G.conj().T) / 2)
    R = W @ Y - (Q @ Y) * th[None, :]
    return th.cpu().numpy(), None, None, (torch.linalg.norm(R, dim=0) / 12.0).cpu().numpy()
