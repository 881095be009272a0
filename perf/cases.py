"""What a user of the solver has it do, as cases that a timer can run.

Every case goes through the public Python entry points: a problem handle from
``SGProblem`` (kept, as a program keeps it), blocks on the GPU, one call.
Inputs follow the model problem of the package (Q1 elements on the unit
square, Karhunen-Loeve expansion of a coefficient with exponential covariance,
or its lognormal counterpart); the load, the coefficient blocks and the
parameters come from the seed.

A case is a dict: ``kind`` names the call, ``ne`` the elements per side, ``M``
and ``p`` the random variables and the chaos degree, and the rest its options.
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_1205_1864_gb300 as sg

F64 = torch.float64


# ------------------------------------------------------------------ cases ---

def listed():
    return [
        # The plain method in double precision on the smallest configuration: a call whose time is latency.
        dict(name="solve_16_fp64", kind="solve", ne=16, M=3, p=3, sigma=0.2, corr=0.5, prec="fp64"),
        # A row of the paper's convergence tables: 30 elements per side (no multigrid), diagonal inner preconditioner.
        dict(name="solve_30_diag", kind="solve", ne=30, M=4, p=4, sigma=0.3, corr=0.5, prec="diag"),
        # The mid-size mixed-precision solve.
        dict(name="solve_128", kind="solve", ne=128, M=6, p=4, sigma=0.3, corr=1.0, prec="mixed"),
        # The largest single system of the configurations, 261 million unknowns: the headline workload.
        dict(name="solve_512", kind="solve", ne=512, M=10, p=4, sigma=0.25, corr=0.5, prec="mixed"),
        # Many uneven systems solved by one call.
        dict(name="batch_10", kind="batch", count=10, pick=1864, top=256),
        # Quantity of interest and its gradient in the coefficient's parameters: forward and adjoint solve.
        dict(name="gradient_64", kind="gradient", ne=64, M=4, p=3, sigma=0.2, corr=0.5),
        # Lognormal coefficient (block-dense coupling, nested level solves), a row of the paper's second tables.
        dict(name="lognormal_10", kind="lognormal", ne=10, M=3, p=3, cov=1.0, corr=0.5),
        # The product alone, as a program with its own outer iteration calls it: double precision, ...
        dict(name="apply_128_fp64", kind="apply", ne=128, M=6, p=4, sigma=0.3, corr=1.0, dtype="fp64"),
        # ... single precision on an odd mesh and an odd block width (P = 495), ...
        dict(name="apply_201_fp32", kind="apply", ne=201, M=8, p=4, sigma=0.25, corr=0.5, dtype="fp32"),
        # ... and single-precision blocks with sums accurate to double precision, P = 1001.
        dict(name="apply_256_df64", kind="apply", ne=256, M=10, p=4, sigma=0.25, corr=0.5, dtype="df64"),
        # One off-diagonal block product of the hierarchy, single precision, 220 -> 55 columns.
        dict(name="level_257_fp32", kind="level", ne=257, M=10, p=4, sigma=0.25, corr=0.5, out=2, inp=3, dtype="fp32"),
        # The batched inner solve on the mean matrix: the columns of one degree level, an odd number of them.
        dict(name="inner_256_715", kind="inner", ne=256, w=715),
    ]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "apply", "apply", "apply", "level", "level", "inner", "inner", "batch",
                       "gradient", "lognormal"])
    sigma, corr = round(rng.uniform(0.1, 0.3), 3), round(rng.uniform(0.3, 1.5), 3)
    if kind == "solve":
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64", "diag"])
        most = {"mixed": 7e7, "fp64": 3e6, "diag": 4e5}[prec]
        while True:
            ne = rng.randint(5, 30) if prec == "diag" else rng.choice([16, 32, 64, 128, 256])
            M, p = rng.randint(2, 10), rng.randint(2, 4)
            if (ne - 1) ** 2 * math.comb(M + p, p) <= most:
                return dict(kind=kind, ne=ne, M=M, p=p, sigma=sigma, corr=corr, prec=prec)
    if kind in ("apply", "level"):
        dtype = rng.choice(["fp64", "fp32", "df64"])
        most = 2e7 if dtype == "fp64" else 7e7
        while True:
            ne = int(round(20 * (512 / 20) ** rng.random()))
            M, p = rng.randint(2, 10), rng.randint(2, 4)
            if (ne - 1) ** 2 * math.comb(M + p, p) <= most:
                break
        case = dict(kind=kind, ne=ne, M=M, p=p, sigma=sigma, corr=corr, dtype=dtype)
        if kind == "level":
            lo = p - 1 if dtype == "df64" else rng.randint(1, p - 1)
            case["out"], case["inp"] = (lo, lo + 1) if rng.random() < 0.5 else (lo + 1, lo)
        return case
    if kind == "inner":
        ne = rng.choice([64, 128, 256, 512])
        most = min(1000, 60_000_000 // (ne - 1) ** 2)
        return dict(kind=kind, ne=ne, w=int(round(math.exp(rng.uniform(0, math.log(most))))))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 10), pick=rng.randint(1, 9999), top=rng.choice([64, 128]))
    if kind == "gradient":
        return dict(kind=kind, ne=rng.choice([16, 32, 64, 128]), M=rng.randint(2, 5), p=rng.randint(2, 3), sigma=0.2, corr=corr)
    return dict(kind=kind, ne=rng.randint(5, 10), M=rng.randint(1, 3), p=rng.randint(1, 3),
                cov=round(rng.uniform(0.25, 1.0), 2), corr=corr)


# ------------------------------------------------- the model problem's data ---

def _modes(corr, count):
    """Eigenpairs of exp(-|s-t|/corr) on [0, 1]: (eigenvalue, frequency, odd, norm), largest first."""
    a, c = 0.5, 1.0 / corr
    out = []
    for i in range(count):
        for odd in (0, 1):
            lo, hi = ((i + 0.5 * odd) * math.pi / a + 1e-12, (i + 0.5 * odd + 0.5) * math.pi / a - 1e-12)
            f = (lambda w: w * math.cos(w * a) + c * math.sin(w * a)) if odd else \
                (lambda w: c * math.cos(w * a) - w * math.sin(w * a))
            up = f(lo) > 0
            for _ in range(200):
                w = 0.5 * (lo + hi)
                if (f(w) > 0) == up:
                    lo = w
                else:
                    hi = w
            w = 0.5 * (lo + hi)
            nrm = 1.0 / math.sqrt(a + (-1 if odd else 1) * math.sin(2 * w * a) / (2 * w))
            out.append((2 * c / (w * w + c * c), w, odd, nrm))
    return sorted(out, key=lambda t: -t[0])[:count]


def _fields(ne, M, corr):
    """sqrt(lambda_k) and phi_k at the Gauss points, (M, ne, ne, 4), of the M leading 2-D pairs."""
    g = 1.0 / math.sqrt(3.0)
    at = (np.arange(ne)[:, None] + (1 + np.array([-g, g])) / 2) / ne         # (ne, 2)
    one = _modes(corr, M + 2)
    pairs = [(one[i][0] * one[j][0], i + j, i, j) for i in range(M + 2) for j in range(M + 2)]
    pairs.sort(key=lambda t: (-round(t[0], 14), t[1], t[2]))
    val = [nrm * (np.sin(w * (at - 0.5)) if odd else np.cos(w * (at - 0.5))) for _, w, odd, nrm in one]
    phi = [(val[j][:, None, :, None] * val[i][None, :, None, :]).reshape(ne, ne, 4) for _, _, i, j in pairs[:M]]
    s = np.array([math.sqrt(lam) for lam, _, _, _ in pairs[:M]])
    return s, torch.tensor(np.array(phi).reshape(M, ne, ne, 4), dtype=F64, device="cuda")


@functools.lru_cache(None)
def _tables():
    """Gradient and mass products of the four bilinear functions at the four Gauss points, (4, 16)."""
    g = 1.0 / math.sqrt(3.0)
    B, N = np.zeros((4, 4, 4)), np.zeros((4, 4, 4))
    for q, (ey, ex) in enumerate(itertools.product((-g, g), (-g, g))):
        v = []
        for b, a in itertools.product((-1, 1), (-1, 1)):
            v.append(((1 + a * ex) * (1 + b * ey) / 4, a * (1 + b * ey) / 4, b * (1 + a * ex) / 4))
        for i in range(4):
            for j in range(4):
                B[q, i, j] = v[i][1] * v[j][1] + v[i][2] * v[j][2]
                N[q, i, j] = v[i][0] * v[j][0]
    return B.reshape(4, 16), N.reshape(4, 16)


def _stencils(ne, kappa, table):
    """(terms, ny, nx, 9) stencils, on the interior nodes, of element matrices kappa (terms, ne, ne, 4) @ table."""
    K = kappa.shape[0]
    e = (kappa.reshape(-1, 4) @ torch.tensor(table, dtype=F64, device="cuda")).reshape(K, ne, ne, 4, 4)
    S = torch.zeros(K, ne + 1, ne + 1, 9, dtype=F64, device="cuda")
    for i, j in itertools.product(range(4), range(4)):
        (yi, xi), (yj, xj) = divmod(i, 2), divmod(j, 2)
        S[:, yi:yi + ne, xi:xi + ne, (yj - yi + 1) * 3 + xj - xi + 1] += e[:, :, :, i, j]
    S = S[:, 1:ne, 1:ne].contiguous()
    S[:, 0, :, :3] = 0
    S[:, -1, :, 6:] = 0
    S[:, :, 0, ::3] = 0
    S[:, :, -1, 2::3] = 0
    return S


def _pattern(ne):
    m = ne - 1
    y, x = np.divmod(np.arange(m * m), m)
    dy, dx = np.divmod(np.arange(9), 3)
    yy, xx = y[:, None] + dy - 1, x[:, None] + dx - 1
    ok = (yy >= 0) & (yy < m) & (xx >= 0) & (xx < m)
    rowptr = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    return rowptr, (yy * m + xx)[ok].astype(np.int32), ok


def _kl(ne, M, sigma, corr, unit=False):
    """Stencils of A_0 .. A_M of the uniform coefficient (unit: sigma = sqrt(lambda_k) = 1)."""
    s, phi = _fields(ne, M, corr)
    scale = torch.ones(M, dtype=F64) if unit else torch.tensor(sigma * s)
    kap = torch.cat([torch.ones(1, ne, ne, 4, dtype=F64, device="cuda"), phi * scale.cuda()[:, None, None, None]])
    return s, _stencils(ne, kap, _tables()[0])


def _lognormal(ne, M, cov, corr, q):
    """Stencils of the Hermite expansion, to total degree q, of exp of the Gaussian field (mean 1, deviation cov)."""
    s, phi = _fields(ne, M, corr)
    var = math.log(1 + cov * cov)
    a = phi * torch.tensor(math.sqrt(var) * s).cuda()[:, None, None, None]
    mean = torch.exp(-0.5 * var + 0.5 * (a * a).sum(0))
    kap = []
    for g in _indices(M, q):
        v = mean.clone()
        for k, d in enumerate(g):
            v = v * a[k] ** d / math.sqrt(math.factorial(d))
        kap.append(v)
    return _stencils(ne, torch.stack(kap), _tables()[0])


def _handle(ne, M, p, S, mass=False, family=None, q=-1):
    rowptr, colidx, ok = _pattern(ne)
    pick = torch.tensor(ok.reshape(-1), device="cuda")
    vals = S.permute(1, 2, 3, 0).reshape(-1, S.shape[0])[pick].cpu().numpy()
    mv = None
    if mass:
        T = _stencils(ne, torch.ones(1, ne, ne, 4, dtype=F64, device="cuda"), _tables()[1] / (4.0 * ne * ne))
        mv = T.reshape(-1)[pick].cpu().numpy()
    return sg.SGProblem(ne, ne, M, p, rowptr, colidx, vals, mv, sg.SG_LEGENDRE if family is None else family, q)


def _indices(M, q):
    """Multi-indices of total degree <= q: degrees ascending, descending lexicographic inside a degree."""
    out = []
    for d in range(q + 1):
        out += _of_degree(d, M)
    return out


def _of_degree(d, m):
    if m == 1:
        yield (d,)
        return
    for a in range(d, -1, -1):
        for rest in _of_degree(d - a, m - 1):
            yield (a,) + rest


def _load(ne, rng):
    """A smooth positive source: 1 plus a few modes."""
    x = np.arange(1, ne) / ne
    f = np.ones((ne - 1, ne - 1))
    for i, j in itertools.product(range(1, 4), range(1, 4)):
        f += 0.1 * rng.uniform(-1, 1) * np.outer(np.cos(math.pi * i * x), np.cos(math.pi * j * x))
    return f.reshape(-1) / (ne * ne)


def _rhs(ne, P, rng):
    F = torch.zeros((ne - 1) ** 2, P, dtype=F64, device="cuda")
    F[:, 0] = torch.tensor(_load(ne, rng), device="cuda")
    return F


def _block(n, degrees, seed):
    """Seeded coefficients of degree d of size about 0.4^d, as those of a chaos expansion fall."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    U = torch.rand(n, len(degrees), generator=g, dtype=torch.float32, device="cuda") * 2 - 1
    return U * torch.tensor([0.4 ** d for d in degrees], dtype=torch.float32, device="cuda")


def _options(prec):
    if prec == "mixed":   # the options of the package's benchmark
        po = sg.prec_opts(precision=sg.SG_F32, top_level_f64=1, inner_tol=1e-2, df64=1)
    elif prec == "fp64":
        po = sg.prec_opts(precision=sg.SG_F64, inner_tol=1e-2)
    else:
        po = sg.prec_opts(precision=sg.SG_F64, m0=sg.SG_M0_DIAG, inner_tol=1e-8, inner_maxit=1000, level_tol=1e-8)
    return sg.solve_opts(po, precond=sg.SG_PREC_HSC, tol=1e-8, maxit=500, check_true_residual=0)


def _systems(case):
    """The systems of a batch: mesh, M, p, sigma and correlation length drawn as the package's batched workload does."""
    rng = np.random.Generator(np.random.PCG64(case["pick"]))
    meshes = [m for m in (32, 64, 128, 256) if m <= case["top"]]
    out = []
    for _ in range(case["count"]):
        ne = int(meshes[int(rng.integers(0, len(meshes)))])
        M, p = int(rng.integers(2, 9)), int(rng.integers(2, 5))
        out.append((ne, M, p, float(rng.uniform(0.1, 0.3)), float(rng.uniform(0.3, 1.5))))
    return out


def _theta(case, seed):
    rng = np.random.Generator(np.random.PCG64([4, seed]))
    s, _ = _fields(case["ne"], case["M"], case["corr"])
    return np.concatenate([[rng.uniform(0.8, 1.2), rng.uniform(0.1, 0.25)], s * rng.uniform(0.9, 1.1, size=case["M"])])


def prepare(case, seed):
    kind, rng = case["kind"], np.random.Generator(np.random.PCG64([7, seed]))
    st = {"kind": kind}
    if kind == "solve":
        ne, M, p = case["ne"], case["M"], case["p"]
        st["h"] = _handle(ne, M, p, _kl(ne, M, case["sigma"], case["corr"])[1])
        st["F"], st["o"] = _rhs(ne, st["h"].P, rng), _options(case["prec"])
    elif kind == "lognormal":
        ne, M, p = case["ne"], case["M"], case["p"]
        st["h"] = _handle(ne, M, p, _lognormal(ne, M, case["cov"], case["corr"], 2 * p), family=sg.SG_HERMITE, q=2 * p)
        st["F"], st["o"] = _rhs(ne, st["h"].P, rng), _options("diag")
    elif kind == "batch":
        hs = [_handle(ne, M, p, _kl(ne, M, s, c)[1]) for ne, M, p, s, c in _systems(case)]
        st["b"], st["o"] = sg.SGBatch(hs), _options("mixed")
        st["F"] = [_rhs(sy[0], h.P, rng) for sy, h in zip(_systems(case), hs)]
    elif kind == "gradient":
        ne, M, p = case["ne"], case["M"], case["p"]
        st["h"] = _handle(ne, M, p, _kl(ne, M, 1.0, case["corr"], unit=True)[1], mass=True)
        st["F"], st["o"] = _rhs(ne, st["h"].P, rng), _options("mixed")
        st["theta"] = torch.tensor(_theta(case, seed), device="cuda")
    elif kind == "inner":
        ne, w = case["ne"], case["w"]
        st["h"] = _handle(ne, 0, 0, _kl(ne, 0, 1.0, 1.0)[1])
        st["B"] = _block((ne - 1) ** 2, [0] * w, seed)
        st["o"] = sg.prec_opts(precision=sg.SG_F32, inner_fixed_iters=2)
    else:
        ne, M, p = case["ne"], case["M"], case["p"]
        st["h"] = _handle(ne, M, p, _kl(ne, M, case["sigma"], case["corr"])[1])
        st["df64"] = case["dtype"] == "df64"
        deg = [sum(a) for a in _indices(M, p)]
        t = F64 if case["dtype"] == "fp64" else torch.float32
        if kind == "apply":
            st["U"] = _block((ne - 1) ** 2, deg, seed).to(t)
        else:
            st["out"], st["inp"] = case["out"], case["inp"]
            st["X"] = _block((ne - 1) ** 2, [d for d in deg if d == case["inp"]], seed).to(t)
            st["Y"] = _block((ne - 1) ** 2, [d for d in deg if d == case["out"]], seed + 1_000_003)
            st["Y"] = st["Y"].to(torch.float32 if case["dtype"] == "fp32" else F64)
    return st


def run(st):
    kind = st["kind"]
    if kind in ("solve", "lognormal"):
        return sg.sg_solve(st["h"], st["F"], st["o"])[0]
    if kind == "batch":
        return st["b"].solve(st["F"], st["o"])[0]
    if kind == "gradient":
        th = st["theta"].clone().requires_grad_(True)
        q = sg.SGQoI.apply(th, st["h"], st["F"], st["o"])
        q.backward()
        return q.detach(), th.grad
    if kind == "inner":
        return sg.sg_inner_solve(st["h"], st["B"], st["o"])[0]
    if kind == "apply":
        return sg.sg_apply(st["h"], st["U"], df64=st["df64"])
    return sg.sg_level_apply(st["h"], st["out"], st["inp"], st["X"], st["Y"], df64=st["df64"])


# ------------------------------------------------------------------- work ---

def _edges(M, p):
    """Couplings between chaos polynomials, and distinct (direction, input) pairs among them."""
    c = math.comb
    if M == 0 or p == 0:
        return 0, 0
    n_m = 2 * M * c(M + p - 1, M)
    return n_m, M * (c(M + p - 1, M) + c(M + p - 1, M - 1) - (c(M + p - 2, M - 2) if M >= 2 else 0))


def work(case):
    """Inputs read once and outputs written once; multiply-adds of the sparse products (two operations each), a solve
    counted with seven outer steps of one product, the hierarchy's level products and two inner iterations each way."""
    kind = case["kind"]
    if kind == "batch":
        each = [work(dict(kind="solve", ne=ne, M=M, p=p, prec="mixed")) for ne, M, p, _, _ in _systems(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    n = (case["ne"] - 1) ** 2
    nnz = (3 * case["ne"] - 5) ** 2
    if kind == "inner":
        return {"bytes": 8.0 * n * case["w"], "flops": 2 * 110.0 * n * case["w"]}
    M, p = case["M"], case["p"]
    P = math.comb(M + p, p)
    if kind == "lognormal":
        terms = math.comb(M + 2 * p, M)
        return {"bytes": 8.0 * nnz * terms + 16.0 * n * P, "flops": 7 * 2.0 * nnz * P * terms}
    n_m, n_p = _edges(M, p)
    prod = 2.0 * nnz * (P + n_p) + 2.0 * n * n_m
    size = {"fp64": 8, "fp32": 4, "df64": 8}.get(case.get("dtype"), 8)
    vals = (size * (M + 1) + 4.0) * nnz
    if kind == "solve":
        return {"bytes": vals + 16.0 * n * P, "flops": 7 * (2 * prod + 2 * 2 * 110.0 * n * P)}
    if kind == "gradient":
        return {"bytes": vals + 24.0 * n * P, "flops": 10 * (2 * prod + 2 * 2 * 110.0 * n * P)}
    if kind == "apply":
        return {"bytes": vals + (4 if size == 4 or case["dtype"] == "df64" else 8) * n * P + size * n * P, "flops": prod}
    wi, wo = (math.comb(M + d - 1, d) for d in (case["inp"], case["out"]))
    cpl = M * math.comb(M + min(case["inp"], case["out"]) - 1, min(case["inp"], case["out"]))
    io = {"fp64": 8 * (wi + 2 * wo), "fp32": 4 * (wi + 2 * wo), "df64": 4 * wi + 12 * wo}[case["dtype"]]
    return {"bytes": vals + float(io) * n, "flops": 2.0 * (nnz + n) * cpl}


# --------------------------------------------- the same in plain 64 bits ---

def _stencil(S, V):
    """One stencil (ny, nx, 9) applied to V (ny, nx, w)."""
    ny, nx, w = V.shape
    Vp = torch.zeros(ny + 2, nx + 2, w, dtype=F64, device=V.device)
    Vp[1:-1, 1:-1] = V
    Y = torch.zeros_like(V)
    for s in range(9):
        Y.addcmul_(S[:, :, s:s + 1], Vp[s // 3:s // 3 + ny, s % 3:s % 3 + nx])
    return Y


@functools.lru_cache(8)
def _couplings(M, p):
    """Per direction k two lists (out, in, coefficient): E[xi_k psi_out psi_in], uniform variables of variance 1."""
    idx = _indices(M, p)
    at = {a: i for i, a in enumerate(idx)}
    got = []
    for k in range(M):
        lo, hi, c = [], [], []
        for i, a in enumerate(idx):
            b = a[:k] + (a[k] + 1,) + a[k + 1:]
            if b in at:
                m = a[k]
                lo.append(i)
                hi.append(at[b])
                c.append(math.sqrt(3.0) * (m + 1) / math.sqrt((2 * m + 1) * (2 * m + 3)))
        t = torch.tensor(c, dtype=F64, device="cuda")
        lo, hi = torch.tensor(lo, device="cuda"), torch.tensor(hi, device="cuda")
        got.append(((lo, hi, t), (hi, lo, t)))
    return got


def _coupled(V, M, p, k):
    W = torch.zeros_like(V)
    for o, i, c in _couplings(M, p)[k]:
        W[..., o] += V[..., i] * c
    return W


def _product(S, M, p, V):
    Y = _stencil(S[0], V)
    for k in range(M):
        Y += _stencil(S[k + 1], _coupled(V, M, p, k))
    return Y


def _solved(S, M, p, F, a0=1.0, tol=1e-14, most=120):
    """Conjugate gradients, preconditioned by the sine transform's exact inverse of a0 times the Laplacian."""
    m = F.shape[0]
    t = torch.arange(1, m + 1, dtype=F64, device="cuda") * (math.pi / (m + 1))
    Q = math.sqrt(2.0 / (m + 1)) * torch.sin(torch.outer(torch.arange(1, m + 1, dtype=F64, device="cuda"), t))
    k, ms = 2 - 2 * torch.cos(t), (4 + 2 * torch.cos(t)) / 6
    lam = (a0 * (k[:, None] * ms[None, :] + ms[:, None] * k[None, :]))[:, :, None]

    def both(V):
        w = V.shape[2]
        V = (Q @ V.reshape(m, -1)).reshape(m, m, w)
        return torch.matmul(Q, V)

    U, r, rho, p_ = torch.zeros_like(F), F.clone(), None, None
    stop = tol * float(F.norm())
    for _ in range(most):
        if float(r.norm()) <= stop:
            break
        z = both(both(r) / lam)
        new = float((z * r).sum())
        p_ = z if p_ is None else z + p_ * (new / rho)
        rho = new
        q = _product(S, M, p, p_)
        a = rho / float((p_ * q).sum())
        U += a * p_
        r -= a * q
    return U


def _hermite(M, p, q):
    """(terms, P, P) expectations of three normalised Hermite products."""
    def one(a, b, c):
        s = a + b + c
        if s % 2 or max(a, b, c) > s // 2:
            return 0.0
        s //= 2
        f = math.factorial
        return math.sqrt(f(a) * f(b) * f(c)) / (f(s - a) * f(s - b) * f(s - c))

    T = np.array([[[one(a, b, c) for c in range(p + 1)] for b in range(p + 1)] for a in range(q + 1)])
    g, u = np.array(_indices(M, q)), np.array(_indices(M, p))
    G = np.ones((len(g), len(u), len(u)))
    for k in range(M):
        G *= T[g[:, k][:, None, None], u[:, k][None, :, None], u[:, k][None, None, :]]
    return torch.tensor(G, device="cuda")


def _cycle(B, c0=8.0 / 3.0, omega=0.8):
    """One V-cycle for the Laplacian's 9-point stencil (8/3, -1/3), two sweeps each way, zero start."""
    m, w = B.shape[0], B.shape[2]
    if m == 1:
        return B / c0

    def A(V):
        Vp = torch.zeros(m + 2, m + 2, w, dtype=F64, device="cuda")
        Vp[1:-1, 1:-1] = V
        R = Vp[:-2] + Vp[1:-1] + Vp[2:]
        return 3.0 * V - (R[:, :-2] + R[:, 1:-1] + R[:, 2:]) / 3.0

    def sweep(V):
        return V + (omega / c0) * (B - A(V))

    X = sweep((omega / c0) * B)
    R = B - A(X)
    R = R[1::2] + 0.5 * (R[:-1:2] + R[2::2])
    R = R[:, 1::2] + 0.5 * (R[:, :-1:2] + R[:, 2::2])
    C = _cycle(R.contiguous(), c0, omega)
    half = torch.zeros(m, C.shape[1], w, dtype=F64, device="cuda")
    half[1::2] = C
    half[:-1:2] += 0.5 * C
    half[2::2] += 0.5 * C
    full = torch.zeros(m, m, w, dtype=F64, device="cuda")
    full[:, 1::2] = half
    full[:, :-1:2] += 0.5 * half
    full[:, 2::2] += 0.5 * half
    return sweep(sweep(X + full))


def _inner(B):
    """Two conjugate-gradient steps with the V-cycle, column by column."""
    S = torch.full((*B.shape[:2], 9), -1.0 / 3.0, dtype=F64, device="cuda")
    S[:, :, 4] = 8.0 / 3.0
    X, R, rho, D = torch.zeros_like(B), B.clone(), None, None
    for _ in range(2):
        Z = _cycle(R)
        new = (Z * R).sum((0, 1))
        D = Z if D is None else Z + D * (new / rho)
        rho = new
        Q = _stencil(S, D)
        a = rho / (D * Q).sum((0, 1))
        X += a * D
        R -= a * Q
    return X


def exact(case, seed):
    kind, rng = case["kind"], np.random.Generator(np.random.PCG64([7, seed]))
    if kind == "batch":
        got = []
        for ne, M, p, s, c in _systems(case):
            F = _rhs(ne, math.comb(M + p, p), rng).reshape(ne - 1, ne - 1, -1)
            small = F.numel() <= 4_000_000
            got.append(_solved(_kl(ne, M, s, c)[1], M, p, F).reshape((ne - 1) ** 2, -1) if small else None)
        return got
    ne = case["ne"]
    m, n = ne - 1, (ne - 1) ** 2
    if kind == "inner":
        B = _block(n, [0] * case["w"], seed)
        parts = [_inner(b.to(F64).reshape(m, m, -1)).reshape(n, -1) for b in B.split(64, 1)]
        return torch.cat(parts, 1)
    M, p = case["M"], case["p"]
    P = math.comb(M + p, p)
    if kind == "lognormal":
        S, G = _lognormal(ne, M, case["cov"], case["corr"], 2 * p), _hermite(M, p, 2 * p)
        rowptr, colidx, ok = _pattern(ne)
        rows, pick = torch.tensor(np.repeat(np.arange(n), np.diff(rowptr))).cuda(), torch.tensor(ok.reshape(-1)).cuda()
        A = torch.zeros(n, P, n, P, dtype=F64, device="cuda")
        for i in range(S.shape[0]):
            D = torch.zeros(n, n, dtype=F64, device="cuda")
            D[rows, torch.tensor(colidx).long().cuda()] = S[i].reshape(-1)[pick]
            A += D[:, None, :, None] * G[i][None, :, None, :]
        F = _rhs(ne, P, rng)
        return torch.linalg.solve(A.reshape(n * P, n * P), F.reshape(-1)).reshape(n, P)
    if kind == "solve":
        if n * P > 8_000_000:
            return None
        F = _rhs(ne, P, rng).reshape(m, m, P)
        return _solved(_kl(ne, M, case["sigma"], case["corr"])[1], M, p, F).reshape(n, P)
    if kind == "gradient":
        th = _theta(case, seed)
        unit = _kl(ne, M, 1.0, case["corr"], unit=True)[1]
        scale = torch.tensor(np.concatenate([[th[0]], th[1] * th[2:]]), device="cuda")
        S = unit * scale[:, None, None, None]
        T = _stencils(ne, torch.ones(1, ne, ne, 4, dtype=F64, device="cuda"), _tables()[1] / (4.0 * ne * ne))[0]
        U = _solved(S, M, p, _rhs(ne, P, rng).reshape(m, m, P), th[0])
        MU = _stencil(T, U)
        L = _solved(S, M, p, 2 * MU, th[0])
        hk = [float((L * _stencil(unit[0], U)).sum())]
        hk += [float((L * _stencil(unit[k + 1], _coupled(U, M, p, k))).sum()) for k in range(M)]
        g = [-hk[0], -sum(th[2 + k] * hk[k + 1] for k in range(M))] + [-th[1] * hk[k + 1] for k in range(M)]
        return (U * MU).sum(), torch.tensor(g, dtype=F64)
    S = _kl(ne, M, case["sigma"], case["corr"])[1]
    deg = torch.tensor([sum(a) for a in _indices(M, p)], device="cuda")
    if kind == "apply":
        U = _block(n, deg.tolist(), seed).to(F64)
        return _product(S, M, p, U.reshape(m, m, P)).reshape(n, P)
    at_in, at_out = (deg == case["inp"]).nonzero()[:, 0], (deg == case["out"]).nonzero()[:, 0]
    V = torch.zeros(m, m, P, dtype=F64, device="cuda")
    V[..., at_in] = _block(n, [case["inp"]] * len(at_in), seed).to(F64).reshape(m, m, -1)
    Y = _block(n, [case["out"]] * len(at_out), seed + 1_000_003).to(F64)
    return Y - _product(S, M, p, V)[..., at_out].reshape(n, -1)
