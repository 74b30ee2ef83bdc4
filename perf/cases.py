"""The work this library is used for, as cases that can be timed and compared.

A case is one call sequence of a user's program on one HSS matrix (or a batch
of them).  ``op`` names the sequence:

* ``matvec``   y = A x with the generators of a resident object (FP64);
* ``noalloc``  the same through the entry point that allocates nothing;
* ``solve``    x = A^-1 b with a factor that the program keeps;
* ``loglik``   factorize, log-determinant and solve (a Gaussian-process
               likelihood evaluation, FP64);
* ``mixed``    factorize in lower precision and solve with iterative refinement
               (the log-determinant of a lower-precision factor is not refined,
               so x is what such a program takes from it);
* ``batch``    many matrices of uneven shapes factored and solved together.

Sizes are those of the repository's workloads (cube_inv_4k, grid_exp_64k,
sphere_yukawa_256k, the leaf 1024 / rank 256 shape of cube_exp_2m, the batched
uneven mix) and of its tests.
"""
import math
import random

import numpy as np
import torch

from paper_2311_00921_gb300 import hss, inputs

F64 = torch.float64


# ------------------------------------------------------------------ the cases
def _case(name, op, kind, leaf, rank, levels, nrhs, **more):
    c = {"name": name, "op": op, "kind": kind, "leaf": leaf, "rank": rank, "levels": levels,
         "nrhs": nrhs, "n": leaf << levels, "precision": "fp64", "residual": "fp64"}
    c.update(more)
    return c


def listed():
    return [
        # one product with a small operator, e.g. inside a Krylov loop: latency only
        _case("matvec_cube_1k", "matvec", "inv", 128, 32, 3, 1),
        # one right-hand side against a kept factor, the smallest workload's shape
        _case("solve_cube_4k", "solve", "inv", 256, 32, 4, 1),
        # one likelihood evaluation at that shape: a chain of small launches
        _case("loglik_cube_4k", "loglik", "inv", 256, 32, 4, 1),
        # covariance product of the geostatistics grid by a host that owns all device memory
        _case("noalloc_grid_64k", "noalloc", "exp", 512, 128, 7, 8),
        # likelihood evaluation of the geostatistics grid
        _case("loglik_grid_64k", "loglik", "exp", 512, 128, 7, 8),
        # the 16-column FP64 product of the headline workload (its refinement residual)
        _case("matvec_sphere_256k", "matvec", "yukawa", 512, 128, 9, 16),
        # time stepping with a kept FP64 factor of the headline workload
        _case("solve_sphere_256k", "solve", "yukawa", 512, 128, 9, 16),
        # the headline workload in FP64 throughout
        _case("loglik_sphere_256k", "loglik", "yukawa", 512, 128, 9, 16),
        # the headline workload: BF16 x3 tensor-core factor, refined to 1e-12
        _case("mixed_sphere_256k", "mixed", "yukawa", 512, 128, 9, 16, precision="bf16"),
        # points that divide by nothing (an uneven tree), FP32 factor, a ragged block of columns
        _case("mixed_uneven_50k", "mixed", "inv", 391, 96, 7, 3, n=49999, precision="fp32"),
        # the largest leaf and rank (the shape of the two-million-point workload, fewer leaves)
        _case("mixed_leaf1024_128k", "mixed", "inv", 1024, 256, 7, 4, precision="tf32"),
        # independent matrices of uneven order, leaf and rank in one batch
        {"name": "batch_10", "op": "batch", "count": 10, "mix": 1003, "n_min": 2048,
         "n_max": 16384, "nrhs": 1},
    ]


def draw(rng):
    """One more case of these ranges: any leaf and rank, odd ones too, sizes
    spread over their logarithm, and a size that stays below the largest listed
    case's work."""
    op = rng.choice(["matvec", "noalloc", "solve", "loglik", "mixed", "mixed", "batch"])
    if op == "batch":
        n_min = int(math.exp(rng.uniform(math.log(512), math.log(4096))))
        return {"op": op, "count": rng.randint(2, 12), "mix": rng.randrange(1 << 20),
                "n_min": n_min, "n_max": int(n_min * rng.uniform(1.5, 6.0)),
                "nrhs": rng.choice([1, 1, 2, 5])}
    leaf = int(round(math.exp(rng.uniform(math.log(40), math.log(600)))))
    if rng.random() < 0.5:
        leaf = rng.choice([64, 128, 256, 512])
    rank = max(4, min(160, int(leaf * rng.uniform(0.12, 0.55))))
    if rng.random() < 0.5:
        rank = max(8, rank & ~15)
    n = math.exp(rng.uniform(math.log(1024), math.log(180000)))
    levels = max(2, int(math.log2(n / leaf)))
    if op == "noalloc":   # its fixed scratch: 2 (2^(levels+1) - 2) rank <= 2^21 doubles
        while 2 * ((2 << levels) - 2) * rank > 1 << 21:
            levels -= 1
    nrhs = min(40, int(round(math.exp(rng.uniform(0.0, math.log(40.0))))))
    # refinement to 1e-12 needs a moderate condition number: not the covariance with a
    # small nugget, where a program factors in FP64
    kinds = ["inv", "yukawa"] + (["exp"] if op != "mixed" else [])
    c = _case("", op, rng.choice(kinds), leaf, rank, levels, nrhs)
    del c["name"]
    if op == "mixed":
        c["precision"] = rng.choice(["fp32", "tf32", "bf16"])
        c["residual"] = rng.choice(["fp64", "fp64", "pair32"])
    if op != "noalloc" and leaf > rank + 1 and rng.random() < 0.3:
        # not every leaf is full
        c["n"] -= rng.randint(1, (1 << levels) - 1)
    return c


# ------------------------------------------------------------------ inputs
def _orth(y):
    """Orthonormal columns of a batch of tall blocks (Cholesky QR, twice)."""
    for _ in range(2):
        c = torch.linalg.cholesky(y.mT @ y)
        y = torch.linalg.solve_triangular(c, y.mT, upper=False).mT
    return y


def _points(kind, n, g):
    if kind == "inv":      # electrostatics: the unit cube
        return torch.rand(n, 3, generator=g, dtype=F64, device="cuda")
    if kind == "yukawa":   # the unit sphere's surface
        p = torch.randn(n, 3, generator=g, dtype=F64, device="cuda")
        return p / p.norm(dim=1, keepdim=True)
    sx = 1 << int(math.ceil(math.log2(n) / 2))   # geostatistics: a jittered grid
    k = torch.arange(n, device="cuda")
    jit = 0.5 * torch.rand(n, 2, generator=g, dtype=F64, device="cuda") - 0.25
    return (torch.stack([k % sx, k // sx], 1) + 0.5 + jit) / sx


def _kernel(kind, a, b):
    d = torch.cdist(a, b, compute_mode="donot_use_mm_for_euclid_dist")
    if kind == "inv":
        return 1.0 / (d + 1e-3)
    if kind == "yukawa":
        return torch.exp(-d) / (d + 1e-3)
    return torch.exp(-d / 0.1)


def _generators(kind, n, leaf, rank, levels, seed):
    """D, U, {E_l}, {S_l} of an SPD HSS matrix of kernel type, batched per level
    on the GPU, in a uniform (leaf, rank) layout.  Leaf blocks are the shifted
    kernel on median-bisection clusters; bases are whitened by the blocks'
    Cholesky factors and couplings have norm below one, which keeps the matrix
    SPD at any rank.  Where n < leaf 2^levels the tree is uneven: the last row of
    the short leaves is taken out (identity in D, zero in U)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    randn = lambda *s: torch.randn(*s, generator=g, dtype=F64, device="cuda")
    nl = 1 << levels
    full = leaf * nl
    p = _points(kind, full, g)
    far = p[torch.randint(0, full, (rank + 8,), generator=g, device="cuda")]
    p = p[None]
    for _ in range(levels):   # halve every cluster along its longest axis
        ax = (p.amax(1) - p.amin(1)).argmax(1)
        key = p.gather(2, ax[:, None, None].expand(-1, p.shape[1], 1))[..., 0]
        p = p.gather(1, key.argsort(1)[..., None].expand_as(p))
        p = p.reshape(2 * p.shape[0], p.shape[1] // 2, p.shape[2])
    shift = {"inv": float(full) ** (1.0 / 3.0), "yukawa": 64.0, "exp": 1e-3}[kind]
    D = _kernel(kind, p, p)
    D.diagonal(dim1=1, dim2=2).add_(shift)
    lam = torch.linalg.cholesky(D)
    w = _kernel(kind, p, far.expand(nl, -1, -1))   # far field of the leaf, plus noise
    w = w @ randn(rank + 8, rank) / math.sqrt(rank)
    w = w / w.norm(dim=(1, 2), keepdim=True) * math.sqrt(rank) + 0.05 * randn(nl, leaf, rank)
    U = lam @ _orth(torch.linalg.solve_triangular(lam, w, upper=False))
    decay = torch.exp(-4.0 * torch.arange(rank, dtype=F64, device="cuda") / rank)
    E, S = {}, {}
    for l in range(levels, 0, -1):
        s = randn(1 << (l - 1), rank, rank) * decay
        S[l] = 0.5 * s / s.norm(dim=(1, 2), keepdim=True)
        if l >= 2:
            h = torch.eye(2 * rank, dtype=F64, device="cuda").repeat(1 << (l - 1), 1, 1)
            h[:, rank:, :rank] = S[l]
            h[:, :rank, rank:] = S[l].mT
            E[l - 1] = torch.linalg.cholesky(h) @ _orth(randn(1 << (l - 1), 2 * rank, rank))
    if n < full:
        # short leaves spread over the tree, as median bisection leaves them
        k = torch.arange(nl, device="cuda")
        short = (k + 1) * (full - n) // nl != k * (full - n) // nl
        D[short, -1, :] = 0.0
        D[short, :, -1] = 0.0
        D[short, -1, -1] = 1.0
        U[short, -1, :] = 0.0
        sizes = leaf - short.to(torch.int64)
    else:
        sizes = torch.full((nl,), leaf, device="cuda")
    return D, U, E, S, sizes


def _packed(D, U, E, S, levels):
    """The packed column-major layout of the library."""
    cm = lambda t: t.mT.reshape(-1)
    e = [cm(E[l]) for l in range(1, levels)] or [torch.zeros(1, dtype=F64, device="cuda")]
    return cm(D), cm(U), torch.cat(e), torch.cat([cm(S[l]) for l in range(1, levels + 1)])


def _host_matrix(D, U, E, S, sizes, levels, rank):
    """The same matrix as host blocks."""
    b = [int(v) for v in sizes.tolist()]
    d, u = D.cpu().numpy(), U.cpu().numpy()
    return inputs.HSSMatrix(
        levels=levels, sizes=np.array(b), ranks={l: np.full(1 << l, rank) for l in range(1, levels + 1)},
        D=[d[i, :m, :m] for i, m in enumerate(b)], U=[u[i, :m] for i, m in enumerate(b)],
        E={l: list(E[l].cpu().numpy()) for l in E}, S={l: list(S[l].cpu().numpy()) for l in S})


def _rhs(n, nrhs, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 77)
    return torch.randn(nrhs, n, generator=g, dtype=F64, device="cuda").t()   # column-major


def _members(case):
    """Shapes of a batch's matrices: order log-uniform, leaf and rank from the
    batched workload's choices, every third tree uneven."""
    rng = random.Random(case["mix"])
    out = []
    for i in range(case["count"]):
        leaf, rank = rng.choice([128, 256, 512]), rng.choice([32, 64, 128])
        n = math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
        levels = max(1, int(round(math.log2(n / leaf))))
        rank = min(rank, leaf // 2)
        n = (leaf << levels) - (rng.randint(1, (1 << levels) - 1) if i % 3 == 2 else 0)
        out.append((rng.choice(["inv", "exp"]), n, leaf, rank, levels))
    return out


def prepare(case, seed):
    if case["op"] == "batch":
        mats, bs = [], []
        for i, (kind, n, leaf, rank, levels) in enumerate(_members(case)):
            gen = _generators(kind, n, leaf, rank, levels, 1000 * seed + i)
            mats.append(_host_matrix(*gen, levels, rank))
            bs.append(_rhs(n, case["nrhs"], 1000 * seed + i))
        return {"op": "batch", "batch": hss.HSSBatch(mats), "b": bs}
    n, leaf, rank, levels = case["n"], case["leaf"], case["rank"], case["levels"]
    gen = _generators(case["kind"], n, leaf, rank, levels, seed)
    st = {"op": case["op"], "b": _rhs(n, case["nrhs"], seed)}
    if case["op"] == "noalloc":
        st["shape"], st["gen"] = (n, leaf, rank, levels), _packed(*gen[:4], levels)
        st["y"] = torch.empty_like(st["b"].t()).t()
        return st
    if n < leaf << levels:
        dev = hss.HSS(_host_matrix(*gen, levels, rank))
    else:
        dev = hss.HSS.from_device((n, leaf, rank, levels), *_packed(*gen[:4], levels))
    if case["op"] == "solve":
        dev.factorize("fp64")
    st.update(dev=dev, precision=case["precision"], residual=case["residual"])
    return st


def run(state):
    op, b = state["op"], state["b"]
    if op == "batch":
        state["batch"].factorize()
        x = state["batch"].solve(b)
        return {"x": x, "logdet": state["batch"].logdet()}
    if op == "noalloc":
        return {"y": hss.matvec_noalloc(state["shape"], *state["gen"], b, state["y"])}
    dev = state["dev"]
    if op == "matvec":
        return {"y": dev.matvec(b)}
    if op == "solve":
        return {"x": dev.solve(b)}
    if op == "loglik":
        dev.factorize("fp64")
        return {"x": dev.solve(b), "logdet": dev.logdet()}
    dev.factorize(state["precision"], residual=state["residual"])
    return {"x": dev.solve(b)}


# ------------------------------------------------------------------ work
def _generator_bytes(leaf, rank, levels):
    nl = 1 << levels
    return 8.0 * (nl * (leaf * leaf + leaf * rank) + (nl - 2) * 2 * rank * rank + (nl - 1) * rank * rank)


def _factor_flops(leaf, rank, levels):
    f = (2.0 * rank) ** 3 / 3
    for l in range(1, levels + 1):
        b, r = (leaf if l == levels else 2 * rank), rank
        c = b - r
        f += (1 << l) * (3.0 * b * r * r - 2.0 * r ** 3 / 3      # basis completion
                         + 4.0 * b * b * r + 4.0 * b * r * r     # Q^T A Q
                         + c ** 3 / 3.0 + c * c * r + c * r * r  # partial Cholesky
                         + 4.0 * r ** 3)                         # merge
    return f


def _factor_size(leaf, rank, levels):
    s = 2.0 * rank * rank
    for l in range(1, levels + 1):
        b = leaf if l == levels else 2 * rank
        s += (1 << l) * (b * (b + 1) / 2.0 + b * rank + rank * rank / 2.0)
    return s


def _solve_flops(leaf, rank, levels):
    f = 2.0 * (2 * rank) ** 2
    for l in range(1, levels + 1):
        b = leaf if l == levels else 2 * rank
        c = b - rank
        f += (1 << l) * (2.0 * c * c + 4.0 * c * rank + 2 * (4.0 * b * rank + rank * rank))
    return f


def _one_work(op, n, leaf, rank, levels, nrhs, precision):
    gen, vec = _generator_bytes(leaf, rank, levels), 16.0 * n * nrhs
    fac = _factor_size(leaf, rank, levels) * (8.0 if precision == "fp64" else 4.0)
    mv, sv = 2.0 * gen / 8.0 * nrhs, _solve_flops(leaf, rank, levels) * nrhs
    if op in ("matvec", "noalloc"):
        return gen + vec, mv
    if op == "solve":
        return fac + vec, sv
    ff = _factor_flops(leaf, rank, levels)
    if op == "loglik":
        return gen + fac + vec, ff + sv
    return gen + fac + vec, ff + 2 * sv + 2 * mv   # at least one refinement step


def work(case):
    if case["op"] == "batch":
        w = [_one_work("loglik", n, leaf, rank, levels, case["nrhs"], "fp64")
             for _, n, leaf, rank, levels in _members(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    b, f = _one_work(case["op"], case["n"], case["leaf"], case["rank"], case["levels"],
                     case["nrhs"], case["precision"])
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit values
def _pairs(t):
    """Blocks of siblings one above the other: (2k, m, j) -> (k, 2m, j)."""
    return t.reshape(t.shape[0] // 2, 2 * t.shape[1], t.shape[2])


def _coupling(s):
    k, r, _ = s.shape
    c = torch.zeros(k, 2 * r, 2 * r, dtype=F64, device="cuda")
    c[:, r:, :r] = s
    c[:, :r, r:] = s.mT
    return c


def _parts(t, dim):
    """t as a sum of three parts of 21 bits each, scaled along ``dim``."""
    out, top = [], torch.frexp(t.abs().amax(dim, keepdim=True))[1]
    for k in (1, 2, 3):
        q = torch.ldexp(torch.ones_like(t), top - 21 * k)
        out.append(torch.round(t / q) * q)
        t = t - out[-1]
    return out


def _mm(*ab):
    """The sum of products a @ b of a list of pairs: every partial product is
    exact in 64 bits, so only their final sum rounds."""
    terms = []
    for a, b in zip(ab[0::2], ab[1::2]):
        pa, pb = _parts(a, 2), _parts(b, 1)
        terms += [(i + j, pa[i] @ pb[j]) for i in range(3) for j in range(3)]
    return sum(t for _, t in sorted(terms, key=lambda t: -t[0]))


def _exact_matvec(gen, x):
    D, U, E, S, _ = gen
    L = max(S)
    h = {L: _mm(U.mT, x)}
    for l in range(L - 1, 0, -1):
        h[l] = _mm(E[l].mT, _pairs(h[l + 1]))
    y = None
    for l in range(1, L + 1):
        c = (_coupling(S[l]), _pairs(h[l]))
        y = _mm(*c) if y is None else _mm(*c, E[l - 1], y)
        y = y.reshape(h[l].shape)
    return _mm(D, x, U, y)


def _exact_solve(gen, b):
    """x and log det A by the Woodbury identity, sibling pair by sibling pair."""
    D, U, E, S, _ = gen
    L, r = max(S), U.shape[2]
    lam = torch.linalg.cholesky(D)
    logdet = 2.0 * lam.diagonal(dim1=1, dim2=2).log().sum()
    yb, yu = torch.cholesky_solve(b, lam), torch.cholesky_solve(U, lam)
    G, h, kept = U.mT @ yu, U.mT @ yb, {}
    for l in range(L, 0, -1):
        C, h = _coupling(S[l]), _pairs(h)
        G2 = torch.zeros_like(C)
        G2[:, :r, :r] = G[0::2]
        G2[:, r:, r:] = G[1::2]
        M = torch.eye(2 * r, dtype=F64, device="cuda") + C @ G2
        logdet = logdet + torch.linalg.slogdet(M)[1].sum()
        kept[l] = (M, C, h)
        if l > 1:
            K = torch.linalg.solve(M, C)
            G = E[l - 1].mT @ (G2 - G2 @ K @ G2) @ E[l - 1]
            h = E[l - 1].mT @ (h - G2 @ (K @ h))
    w = None
    for l in range(1, L + 1):
        M, C, h = kept[l]
        v = C @ h
        if w is not None:
            v = v + E[l - 1] @ w
        w = torch.linalg.solve(M, v)
        w = w.reshape(2 * w.shape[0], r, w.shape[2])
    return yb - yu @ w, float(logdet)


def _exact_one(op, gen, b):
    D, sizes = gen[0], gen[4]
    keep = (torch.arange(D.shape[1], device="cuda") < sizes[:, None]).reshape(-1)
    full = torch.zeros(keep.numel(), b.shape[1], dtype=F64, device="cuda")
    full[keep] = b
    full = full.reshape(D.shape[0], D.shape[1], b.shape[1])
    if op in ("matvec", "noalloc"):
        y, logdet = _exact_matvec(gen, full), None
    else:
        y, logdet = _exact_solve(gen, full)
        y = y + _exact_solve(gen, full - _exact_matvec(gen, y))[0]
    return y.reshape(-1, b.shape[1])[keep], logdet


def exact(case, seed):
    if case["op"] == "batch":
        xs, lds = [], []
        for i, (kind, n, leaf, rank, levels) in enumerate(_members(case)):
            gen = _generators(kind, n, leaf, rank, levels, 1000 * seed + i)
            x, ld = _exact_one("loglik", gen, _rhs(n, case["nrhs"], 1000 * seed + i))
            xs.append(x)
            lds.append(ld)
        return {"x": xs, "logdet": np.array(lds)}
    gen = _generators(case["kind"], case["n"], case["leaf"], case["rank"], case["levels"], seed)
    v, logdet = _exact_one(case["op"], gen, _rhs(case["n"], case["nrhs"], seed))
    if case["op"] in ("matvec", "noalloc"):
        return {"y": v}
    return {"x": v, "logdet": logdet} if case["op"] == "loglik" else {"x": v}
