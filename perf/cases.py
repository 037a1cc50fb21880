"""The work a user of this library has it do, as cases that can be timed.

Each case is one pass through the library's public entry points (the Python
binding over the C ABI) at a size and on a matrix family this repository's own
benchmark and tests use: 2D / 3D stencils (banded rows), the power-law recipe
(very unbalanced rows, random columns), symmetric upper storage.  Kinds:

  spmv      y = alpha A x + beta y, FP64 or FP32
  step      one Arnoldi step: w = A v_k, then w orthogonalised against k rows
  ilu       one application of the ILU(0) preconditioner
  gmres     a whole GMRES(m) solve, FP64 or mixed FP32 / FP64
  bicgstab  a whole BiCGStab solve, plain or with ILU(0)
  batch     many uneven systems by GMRES(m) in one launch

Matrix entries and right-hand sides are multiples of a power of two wherever
sums are formed here, so that the inputs are the same bits whatever the order
of those sums.  Solves that run to convergence ask for 1e-12 and have a known
solution.
"""
import math

import numpy as np
import torch

import paper_2405_01599_gb300 as xb

DEV = "cuda"
ORTHO = {"mgs": xb.ORTHO_MGS, "cgs": xb.ORTHO_CGS, "dgks": xb.ORTHO_DGKS, "bcgs": xb.ORTHO_BCGS}
SPMV = {"default": None, "row": (xb.VAR_ROW, 256, 1), "segscan": (xb.VAR_SEGSCAN, 128, 8)}
PE = 10.0


def listed():
    return [
        # the smallest product: one 64 x 64 Poisson matrix (GMRES's small system)
        dict(name="spmv_poisson2d_n4096", kind="spmv", family="poisson2d", side=64, dtype="f64", choice="default", alpha=1.0, beta=0.0),
        # the benchmark's headline: power-law rows, 52M non-zeros, the tuned segmented scan
        dict(name="spmv_powerlaw_n4m", kind="spmv", family="powerlaw", n=4_000_000, dtype="f64", choice="segscan", alpha=1.0, beta=0.0),
        # the benchmark's symmetric product: upper storage of the 128^3 Laplacian
        dict(name="spmv_sym_n2m", kind="spmv", family="laplace3d_sym", side=128, dtype="f64", choice="default", alpha=1.0, beta=0.0),
        # Arnoldi inside GMRES(30) on a mid-size box with an odd row count, the default MGS
        dict(name="step_mgs_n104k", kind="step", family="convdiff3d", nx=47, ny=51, nz=43, k=20, ortho="mgs"),
        # Arnoldi / Lanczos inside an eigensolver (m = 40), twice-is-enough Gram-Schmidt
        dict(name="step_dgks_n2m", kind="step", family="convdiff3d", nx=120, ny=128, nz=136, k=40, ortho="dgks"),
        # Arnoldi inside the 256^3 solve under the accuracy policy: the largest basis
        dict(name="step_bcgs_n17m", kind="step", family="convdiff3d", nx=256, ny=256, nz=256, k=30, ortho="bcgs"),
        # the preconditioner on unbalanced rows: few dependency levels, long rows
        dict(name="ilu_powerlaw_n1m", kind="ilu", family="powerlaw", n=1_000_000),
        # a small linear solve, all launch and reduction latency
        dict(name="gmres_poisson2d_n4096", kind="gmres", family="poisson2d", side=64, m=30, ortho="mgs", precision="fp64"),
        # a mid-size nonsymmetric solve with every option at its default
        dict(name="gmres_convdiff_n262k", kind="gmres", family="convdiff3d", side=64, m=30, ortho="mgs", precision="fp64"),
        # the mixed FP32 / FP64 solve of a PDE with 2M unknowns
        dict(name="gmres_mixed_n2m", kind="gmres", family="convdiff3d", side=128, m=30, ortho="bcgs", precision="mixed"),
        # the preconditioned solve of a PDE: hundreds of dependency levels
        dict(name="bicgstab_ilu_n885k", kind="bicgstab", family="convdiff3d", side=96, precond=True),
        # many uneven systems at once, a fixed budget of steps each
        dict(name="batch_48_systems", kind="batch", count=48, nmin=1000, nmax=60_000, m=30, maxiter=150),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmv", "spmv", "step", "step", "ilu", "gmres", "bicgstab", "batch"])
    if kind == "spmv":
        family = rng.choice(["poisson2d", "powerlaw", "powerlaw", "laplace3d_sym", "convdiff3d"])
        c = dict(kind=kind, family=family, dtype=rng.choice(["f64", "f64", "f32"]))
        if family == "powerlaw":
            c.update(n=_logint(rng, 1000, 4_000_000), choice=rng.choice(["default", "segscan"]))
        elif family == "poisson2d":
            c.update(side=_logint(rng, 32, 2048), choice=rng.choice(["default", "row"]))
        elif family == "laplace3d_sym":
            c.update(side=_logint(rng, 10, 160), choice="default", dtype="f64")
        else:
            c.update(nx=_logint(rng, 10, 200), ny=_logint(rng, 10, 200), nz=_logint(rng, 10, 200), choice=rng.choice(["default", "row"]))
        c.update(rng.choice([dict(alpha=1.0, beta=0.0), dict(alpha=1.0, beta=0.0), dict(alpha=-1.0, beta=1.0), dict(alpha=0.5, beta=-2.0)]))
        return c
    if kind == "step":
        nx, ny, nz = (_logint(rng, 20, 220) for _ in range(3))
        k = rng.randint(2, 48)
        return dict(kind=kind, family="convdiff3d", nx=nx, ny=ny, nz=nz, k=min(k, max(2, 480_000_000 // (nx * ny * nz))), ortho=rng.choice(["mgs", "mgs", "cgs", "dgks", "bcgs"]))
    if kind == "ilu":
        if rng.random() < 0.5:
            return dict(kind=kind, family="powerlaw", n=_logint(rng, 20_000, 1_000_000))
        return dict(kind=kind, family="convdiff3d", nx=rng.randint(20, 120), ny=rng.randint(20, 120), nz=rng.randint(20, 120))
    if kind == "gmres":
        what = rng.choice(["small", "mid", "mixed"])
        m = rng.choice([20, 30, 40, 50])
        if what == "small":
            return dict(kind=kind, family="poisson2d", side=rng.randint(16, 80), m=m, ortho=rng.choice(["mgs", "bcgs"]), precision="fp64")
        if what == "mid":
            return dict(kind=kind, family="convdiff3d", side=rng.randint(22, 72), m=m, ortho=rng.choice(["mgs", "bcgs", "dgks"]), precision="fp64")
        return dict(kind=kind, family="convdiff3d", side=rng.randint(32, 120), m=m, ortho=rng.choice(["mgs", "bcgs"]), precision="mixed")
    if kind == "bicgstab":
        return dict(kind=kind, family="convdiff3d", side=rng.randint(20, 92), precond=rng.random() < 0.6)
    return dict(kind=kind, count=rng.randint(6, 48), nmin=1000, nmax=_logint(rng, 3000, 60_000), m=rng.choice([20, 30]), maxiter=150)


# ---- inputs ----------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _dyadic(g, n, lo, hi, bits):
    """n values of [lo, hi) that are multiples of 2^-bits."""
    s = 1 << bits
    return torch.randint(int(lo * s), int(hi * s), (n,), generator=g, device=DEV).double() / s


def _dims(case):
    if "nx" in case:
        return case["nx"], case["ny"], case["nz"]
    return (case["side"],) * (2 if case["family"] == "poisson2d" else 3)


def _rows(case):
    return case["n"] if case["family"] == "powerlaw" else math.prod(_dims(case))


def _coeffs(case):
    """Offset along each axis -> coefficient, the repository's stencils."""
    family, d = case["family"], len(_dims(case))
    ph = PE / (max(_dims(case)) + 1) if family == "convdiff3d" else 0.0
    co = {(0,) * d: 2.0 * d + 3.0 * ph}
    for a in range(d):
        for s in (-1, 1):
            co[tuple(s if b == a else 0 for b in range(d))] = -(1.0 + ph) if s < 0 else -1.0
    return co


def _stencil(case, upper=False):
    """CRS of a grid stencil with zero boundary, rows with x fastest."""
    dims, co = _dims(case), _coeffs(case)
    n = math.prod(dims)
    strides = [math.prod(dims[:a]) for a in range(len(dims))]
    at = torch.arange(n, device=DEV)
    offs = sorted((sum(o * s for o, s in zip(off, strides)), off, c) for off, c in co.items())
    offs = [t for t in offs if t[0] >= 0 or not upper]
    mask = torch.ones(n, len(offs), dtype=torch.bool, device=DEV)
    for j, (_, off, _) in enumerate(offs):
        for a, o in enumerate(off):
            if o:
                i = at // strides[a] % dims[a] + o
                mask[:, j] &= (i >= 0) & (i < dims[a])
    cols = at[:, None] + torch.tensor([t[0] for t in offs], device=DEV)
    vals = torch.tensor([t[2] for t in offs], dtype=torch.float64, device=DEV).expand(n, -1)
    return mask.sum(1), cols[mask], vals[mask]


def _powerlaw(n, g):
    """The power-law recipe: lognormal row lengths of mean 12, uniform columns,
    values in (-1, 1), diagonal twice the row's absolute sum."""
    mu = math.log(12.0) - 1.5 * 1.5 / 2
    length = torch.empty(n, dtype=torch.float64, device=DEV).log_normal_(mu, 1.5, generator=g)
    length = length.round().clamp(1, max(1, min(20_000, (n - 1) // 2))).long()
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), length)
    cols = torch.randint(0, n - 1, (rows.numel(),), generator=g, device=DEV)
    cols += cols >= rows
    key = torch.unique(rows * n + cols)
    rows, cols = key // n, key % n
    vals = _dyadic(g, key.numel(), -1, 1, 20) + 2.0 ** -21  # never zero
    total = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, rows, vals.abs())
    at = torch.arange(n, device=DEV)
    key, order = torch.sort(torch.cat([key, at * (n + 1)]))
    vals = torch.cat([vals, 2.0 * total])[order]
    return torch.bincount(rows, minlength=n) + 1, key % n, vals


def _matrix(case, g):
    if case["family"] == "powerlaw":
        counts, cols, vals = _powerlaw(case["n"], g)
    else:
        counts, cols, vals = _stencil(case, upper=case["family"] == "laplace3d_sym")
    rowptr = torch.zeros(counts.numel() + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = counts.cumsum(0)
    return rowptr, cols.int(), vals.contiguous()


def _solution(g, n):
    """A smooth solution with a little noise."""
    return 1.0 + _dyadic(g, n, -1, 1, 10) / 64


def _times(case, A, x):
    """A x formed here, in an order that does not change from run to run."""
    if case["family"] == "powerlaw":  # multiples of a power of two: exact sums
        rowptr, col, val = A
        rows = torch.repeat_interleave(torch.arange(x.numel(), device=DEV), rowptr.diff().long())
        return torch.zeros_like(x).index_add_(0, rows, val * x[col.long()])
    dims = _dims(case)
    u = x.view(dims[::-1])
    y = torch.zeros_like(u)
    for off, c in sorted(_coeffs(case).items()):
        to = tuple(slice(max(0, -o), d - max(0, o)) for o, d in zip(off[::-1], u.shape))
        of = tuple(slice(max(0, o), d - max(0, -o)) for o, d in zip(off[::-1], u.shape))
        y[to] += c * u[of]
    return y.reshape(-1)


def _orthonormal(seed, k, n):
    """k orthonormal rows of length n: distinct rows of the cosine transform,
    turned by a random rotation."""
    r = np.random.default_rng(seed)
    freq = torch.from_numpy(1 + r.choice(n - 1, size=k, replace=False)).to(DEV)
    Q = torch.from_numpy(np.linalg.qr(r.standard_normal((k, k)))[0]).to(DEV)
    odd = 2 * torch.arange(n, device=DEV) + 1
    C = torch.empty(k, n, dtype=torch.float64, device=DEV)
    for i in range(k):
        C[i] = torch.cos((odd * freq[i] % (4 * n)).double() * (math.pi / (2 * n))) * math.sqrt(2 / n)
    return Q @ C


def _batch_specs(case, seed):
    r = np.random.default_rng(seed)
    ns = np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["count"]))
    specs = []
    for i, n in enumerate(ns):
        if i % 3 == 0:
            specs.append(dict(family="poisson2d", side=max(2, round(n ** 0.5))))
        elif i % 3 == 1:
            specs.append(dict(family="laplace3d", side=max(2, round(n ** (1 / 3)))))
        else:
            specs.append(dict(family="powerlaw", n=int(n)))
    return specs


def _batch_systems(case, seed):
    # sizes are the case's, values the seed's
    g, systems = _gen(seed), []
    for spec in _batch_specs(case, case["count"]):
        A = _matrix(spec, g)
        systems.append((spec, A, _times(spec, A, _solution(g, _rows(spec)))))
    return systems


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        systems = [dict(rowptr=A[0], col=A[1], val=A[2], b=b, x=torch.zeros_like(b), m=case["m"], mode=1 if spec["family"] == "powerlaw" else 0)
                   for spec, A, b in _batch_systems(case, seed)]
        return dict(case=case, systems=systems, batch=xb.Batch(systems, tol=1e-12, maxiter=case["maxiter"]))
    g = _gen(seed)
    A = _matrix(case, g)
    n = _rows(case)
    s = dict(case=case, plan=xb.Plan(*A, sym_upper=case["family"] == "laplace3d_sym"))
    if kind == "spmv":
        dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        if SPMV[case["choice"]]:
            s["plan"].set_choice(*SPMV[case["choice"]])
        s["x"] = torch.rand(n, dtype=torch.float64, generator=g, device=DEV).mul_(2).sub_(1).to(dtype)
        s["y0"] = torch.rand(n, dtype=torch.float64, generator=g, device=DEV).to(dtype)
        s["y"] = torch.zeros_like(s["y0"])
    elif kind == "step":
        s["V"] = _orthonormal(seed, case["k"], n)
        s["w"] = torch.empty(n, dtype=torch.float64, device=DEV)
    elif kind == "ilu":
        s["plan"].ilu0_setup()
        s["r"] = torch.rand(n, dtype=torch.float64, generator=g, device=DEV).sub_(0.5)
        s["z"] = torch.empty_like(s["r"])
    else:
        s["b"] = _times(case, A, _solution(g, n))
        s["x"] = torch.zeros_like(s["b"])
        if case.get("precond"):
            s["plan"].ilu0_setup()
    return s


# ---- one pass --------------------------------------------------------------------


def run(state):
    case, plan = state["case"], state.get("plan")
    kind = case["kind"]
    if kind == "spmv":
        y = state["y"]
        if case["beta"] != 0.0:
            y.copy_(state["y0"])
        call = plan.spmv if case["dtype"] == "f64" else plan.spmv_f32
        return call(state["x"], y, alpha=case["alpha"], beta=case["beta"])
    if kind == "step":
        V, w = state["V"], state["w"]
        plan.spmv(V[-1], w)
        return dict(w=w, h=plan.orth(V, w, ORTHO[case["ortho"]]))
    if kind == "ilu":
        return plan.ilu0_apply(state["r"], state["z"])
    if kind == "batch":
        state["batch"].run()
        return [q["x"] for q in state["systems"]]
    x = state["x"].zero_()
    if kind == "gmres":
        plan.gmres(state["b"], x, m=case["m"], tol=1e-12, ortho=ORTHO[case["ortho"]], maxiter=20_000,
                   precision=xb.PREC_MIXED if case["precision"] == "mixed" else xb.PREC_FP64)
    else:
        plan.bicgstab(state["b"], x, tol=1e-12, maxiter=20_000, precond=xb.PRECOND_ILU0 if case["precond"] else xb.PRECOND_NONE)
    return x


# ---- what a pass cannot do without -------------------------------------------------


def _entries(case):
    if case["family"] == "powerlaw":
        return 13.0 * case["n"]
    dims = _dims(case)
    n = math.prod(dims)
    full = (2 * len(dims) + 1) * n - 2 * sum(n // d for d in dims)
    return (full + n) / 2 if case["family"] == "laplace3d_sym" else full


def work(case):
    kind = case["kind"]
    if kind == "batch":
        one = [work(dict(spec, kind="gmres", precision="fp64", m=case["m"], steps=case["maxiter"])) for spec in _batch_specs(case, case["count"])]
        return {k: sum(o[k] for o in one) for k in ("bytes", "flops")}
    n, nnz = _rows(case), _entries(case)
    vb = 4 if case.get("dtype") == "f32" else 8
    A = (vb + 4) * nnz + 4 * n
    terms = 2 * nnz - n if case["family"] == "laplace3d_sym" else nnz
    if kind == "spmv":
        return {"bytes": A + (3 if case["beta"] else 2) * vb * n, "flops": 2 * terms}
    if kind == "step":  # the basis once, w out; every projection is a dot and an update
        k, passes = case["k"], 2 if case["ortho"] == "dgks" else 1
        return {"bytes": A + 8 * n * (k + 1), "flops": 2 * nnz + 4 * n * k * passes + 2 * n}
    if kind == "ilu":
        return {"bytes": A + 16 * n, "flops": 2 * nnz}
    # a solve: its inputs and output once; the products and vector work of the
    # steps that it takes (a step count of the problem's size where none is given)
    if kind == "bicgstab":
        steps = case["side"] * (0.5 if case["precond"] else 2.5)
        return {"bytes": A + 16 * n, "flops": steps * ((8 if case["precond"] else 4) * nnz + 20 * n)}
    steps = case.get("steps") or 6 * case["side"]
    return {"bytes": A + 16 * n, "flops": steps * (2 * nnz + 2 * (case["m"] + 1) * n)}


# ---- the same in plain torch, 64 bits ------------------------------------------------


def _product(A, n):
    rowptr, col, val = A
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), rowptr.diff().long())
    col = col.long()
    return lambda x: torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, rows, val * x[col])


def _gram_schmidt(V, w, method):
    """Coefficients of w against the orthonormal rows of V, and what is left."""
    k = V.shape[0]
    block = {"mgs": 1, "bcgs": 4}.get(method, k)
    h = torch.zeros(k + 1, dtype=torch.float64, device=DEV)
    w = w.clone()
    for _ in range(2 if method == "dgks" else 1):
        for i in range(0, k, block):
            c = V[i:i + block] @ w
            w -= c @ V[i:i + block]
            h[i:i + c.numel()] += c
    h[k] = w.norm()
    return w, h


def _ilu_apply(A, n, r):
    """ILU(0) and its two substitutions by fixed-point sweeps, which are exact
    after as many as the longest chain of dependencies."""
    rowptr, col, val = A
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), rowptr.diff().long())
    col = col.long()
    key = rows * n + col
    low = (col < rows).nonzero().squeeze(1)
    at = torch.arange(n, device=DEV)
    diag = torch.searchsorted(key, at * (n + 1))
    # triples (entry (i, k), entry (k, j), entry (i, j)) with k < i, k < j
    k, first = col[low], diag[col[low]] + 1
    cnt = rowptr.long()[k + 1] - first
    upd = [[], [], []]
    for a in range(0, low.numel(), 4_000_000):
        c, e, f = cnt[a:a + 4_000_000], low[a:a + 4_000_000], first[a:a + 4_000_000]
        e, f = torch.repeat_interleave(e, c), torch.repeat_interleave(f, c)
        f = f + torch.arange(f.numel(), device=DEV) - torch.repeat_interleave(c.cumsum(0) - c, c)
        want = rows[e] * n + col[f]
        p = torch.searchsorted(key, want).clamp_(max=key.numel() - 1)
        ok = key[p] == want
        for u, v in zip(upd, (e, f, p)):
            u.append(v[ok])
    e, f, p = (torch.cat(u) for u in upd)
    # an entry (i, j) takes the products with k < min(i, j): all the triples above
    ok = torch.minimum(rows[p], col[p]) > col[e]
    e, f, p = e[ok], f[ok], p[ok]
    def levels(tri):
        lev = torch.zeros(n, dtype=torch.long, device=DEV)
        while True:
            new = torch.zeros_like(lev).scatter_reduce_(0, rows[tri], lev[col[tri]] + 1, "amax")
            if bool((new == lev).all()):
                return int(lev.max()) + 1
            lev = new

    up = (col > rows).nonzero().squeeze(1)
    nl, nu = levels(low), levels(up)
    lu = val.clone()
    for _ in range(2 * nl + 2):
        lu = val.clone().index_add_(0, p, -lu[e] * lu[f])
        lu[low] = lu[low] / lu[diag[col[low]]]
    z = r
    for tri, d, depth in ((low, None, nl), (up, lu[diag], nu)):
        rhs, cols_, vals_, rows_ = z, col[tri], lu[tri], rows[tri]
        for _ in range(depth):
            t = rhs - torch.zeros_like(rhs).index_add_(0, rows_, vals_ * z[cols_])
            z = t if d is None else t / d
    return z


def _gmres(A, n, b, m, steps):
    """x after `steps` steps of GMRES(m) from zero."""
    mul = _product(A, n)
    x = torch.zeros_like(b)
    while steps > 0:
        r = b - mul(x)
        beta = float(r.norm())
        if beta <= 1e-12 * float(b.norm()):
            break
        V = torch.zeros(m + 1, n, dtype=torch.float64, device=DEV)
        H = torch.zeros(m + 1, m, dtype=torch.float64, device=DEV)
        V[0] = r / beta
        k = min(m, steps)
        for j in range(k):
            w, h = _gram_schmidt(V[:j + 1], mul(V[j]), "dgks")
            H[:j + 2, j] = h
            V[j + 1] = w / h[j + 1]
        rhs = np.zeros(k + 1)
        rhs[0] = beta
        y = np.linalg.lstsq(H[:k + 1, :k].cpu().numpy(), rhs, rcond=None)[0]
        x = x + torch.from_numpy(y).to(DEV) @ V[:k]
        steps -= k
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_gmres(A, _rows(spec), b, case["m"], case["maxiter"]) for spec, A, b in _batch_systems(case, seed)]
    g = _gen(seed)
    A = _matrix(case, g)
    n = _rows(case)
    if kind == "spmv":
        dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        x = torch.rand(n, dtype=torch.float64, generator=g, device=DEV).mul_(2).sub_(1).to(dtype).double()
        y = torch.rand(n, dtype=torch.float64, generator=g, device=DEV).to(dtype).double()
        s = _product(A, n)(x)
        if case["family"] == "laplace3d_sym":
            rows = torch.repeat_interleave(torch.arange(n, device=DEV), A[0].diff().long())
            off = A[1] != rows
            s.index_add_(0, A[1][off].long(), A[2][off] * x[rows[off]])
        return case["alpha"] * s + case["beta"] * y
    if kind == "step":
        V = _orthonormal(seed, case["k"], n)
        w, h = _gram_schmidt(V, _product(A, n)(V[-1]), case["ortho"])
        return dict(w=w, h=h)
    if kind == "ilu":
        return _ilu_apply(A, n, torch.rand(n, dtype=torch.float64, generator=g, device=DEV).sub_(0.5))
    return _solution(g, n)
