"""The work a user of this framework has it do, as measurable cases.

Every case goes through the public entry points of ``paper_1503_07152_gb300``:

* ``train``     the fused training step of the factored HODLR layer
                (loss ||H x - b||^2: forward, residual, every gradient)
* ``autograd``  the same layer as a torch.autograd.Function, forward and backward
* ``gemm``      the dense black box: one sampling product A X or A^T X
* ``compress``  one whole compression (HODLR or HBS-ID) of a dense or matrix-free
                black box, then the compressed operator and its transpose applied
                to a block of vectors
* ``batch``     many operators of uneven size and rank compressed in one call
* ``apply``     a compressed handle and its transpose applied to a block of vectors
* ``solve``     the fast direct solver: factorization, then a solve and a
                transposed solve

Matrices of vectors are (ncols, n) tensors: the column-major n x ncols blocks
that the library takes.
"""
import math

import torch

import paper_1503_07152_gb300 as hm
from paper_1503_07152_gb300.autograd import HodlrApply

DEV = "cuda:0"
PREC = {"fp64": hm.HM_FP64, "a32": hm.HM_A32, "mixed": hm.HM_MIXED}
BLOCK = {"fp64": torch.float64, "a32": torch.float64, "mixed": torch.float32}
VECTORS = 16  # vectors that a compression's result is applied to


def listed():
    return [
        # a training step of the largest factored layer: bandwidth
        {"name": "train_n262144_k32", "kind": "train", "n": 262144, "leaf": 256, "k": 32},
        # forward and backward of a small layer inside a model: latency and launches
        {"name": "autograd_n4096_k32", "kind": "autograd", "n": 4096, "leaf": 256, "k": 32},
        # one transposed product of the black box with an FP32 operator and FP64 vectors
        # (what every level of a compression asks for, r = 60 columns)
        {"name": "gemm_a32_t_n32768_c60", "kind": "gemm", "prec": "a32", "n": 32768, "cols": 60, "trans": 1},
        # the FP32 black box at a ragged size and more columns than a tile holds
        {"name": "gemm_mixed_n10000_c130", "kind": "gemm", "prec": "mixed", "n": 10000, "cols": 130, "trans": 0},
        # the smallest compression: FP64, exact rank, a small operator
        {"name": "hodlr_fp64_n1024_k10", "kind": "compress", "fmt": "hodlr", "source": "lowrank",
         "prec": "fp64", "n": 1024, "leaf": 64, "k": 10},
        # HODLR of a kernel matrix with adaptive ranks
        {"name": "hodlr_a32_n16384", "kind": "compress", "fmt": "hodlr", "source": "log",
         "prec": "a32", "n": 16384, "leaf": 128, "r": 60},
        # HBS-ID of the large kernel matrix: the headline compression
        {"name": "hbsid_a32_n65536", "kind": "compress", "fmt": "hbsid", "source": "log",
         "prec": "a32", "n": 65536, "leaf": 256, "r": 60},
        # HBS-ID of a black box that stores no matrix, at an odd size
        {"name": "hbsid_free_n20001", "kind": "compress", "fmt": "hbsid", "source": "free",
         "prec": "a32", "n": 20001, "leaf": 256, "r": 60},
        # twelve operators of uneven size and rank in one call
        {"name": "batch_a32_12ops", "kind": "batch", "ops": 12, "low": 2048, "high": 8192, "spec": 4},
        # the large compressed kernel matrix applied to a few vectors (error estimates, iterations)
        {"name": "apply_hbsid_n65536_c10", "kind": "apply", "fmt": "hbsid", "prec": "a32",
         "n": 65536, "leaf": 256, "r": 60, "cols": 10},
        # a compressed HODLR operator applied to a block of vectors
        {"name": "apply_hodlr_n16384_c37", "kind": "apply", "fmt": "hodlr", "prec": "a32",
         "n": 16384, "leaf": 128, "r": 60, "cols": 37},
        # factorization and solves of a compressed operator, uneven leaves
        {"name": "solve_fp64_n3000_k8", "kind": "solve", "prec": "fp64", "n": 3000, "leaf": 100, "k": 8,
         "cols": 5},
    ]


def _log(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["train", "autograd", "gemm", "compress", "compress", "compress", "batch",
                       "apply", "solve"])
    if kind in ("train", "autograd"):
        n = _log(rng, 2048, 262144)
        return {"kind": kind, "n": n, "leaf": rng.choice([64, 100, 128, 256] if n < 65536 else [128, 256]),
                "k": rng.randint(4, 32 if n > 131072 else 64)}
    if kind == "gemm":
        prec = rng.choice(["a32", "a32", "mixed", "fp64"])
        n = _log(rng, 512, 4096 if prec == "fp64" else 32768)
        return {"kind": kind, "prec": prec, "n": n, "cols": _log(rng, 1, 130), "trans": rng.randint(0, 1)}
    if kind == "batch":
        return {"kind": kind, "ops": rng.randint(2, 12), "low": 2048, "high": 8192,
                "spec": rng.randint(5, 1 << 20)}
    if kind == "apply":
        fmt = rng.choice(["hodlr", "hbsid"])
        return {"kind": kind, "fmt": fmt, "prec": "a32",
                "n": _log(rng, 2048, 16384 if fmt == "hodlr" else 65536),
                "leaf": 128 if fmt == "hodlr" else 256, "r": 60, "cols": _log(rng, 1, 150)}
    if kind == "solve":
        return {"kind": kind, "prec": rng.choice(["fp64", "a32", "mixed"]), "n": _log(rng, 1024, 6000),
                "leaf": rng.choice([64, 100, 128]), "k": rng.randint(4, 16), "cols": _log(rng, 1, 64)}
    form = rng.choice(["lowrank", "log", "hbsid", "free"])
    if form == "lowrank":
        prec = rng.choice(["fp64", "a32", "mixed"])
        return {"kind": kind, "fmt": "hodlr", "source": "lowrank", "prec": prec,
                "n": _log(rng, 512, 2048 if prec == "fp64" else 8192), "leaf": rng.choice([64, 100]),
                "k": rng.randint(5, 30)}
    if form == "log":
        return {"kind": kind, "fmt": "hodlr", "source": "log", "prec": "a32", "n": _log(rng, 2048, 24000),
                "leaf": rng.choice([100, 128]), "r": 60}
    return {"kind": kind, "fmt": "hbsid", "source": "free" if form == "free" else "log", "prec": "a32",
            "n": _log(rng, 4096, 24000 if form == "free" else 49152), "leaf": 256, "r": 60}


# ------------------------------------------------------------------ inputs ---
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(shape, g, dtype=torch.float32):
    return torch.randn(shape, device=DEV, dtype=dtype, generator=g)


def _depth(n, leaf):
    d = 0
    while -(-n // 2 ** d) > leaf:
        d += 1
    return d


def _levels(n, leaf):
    """[(start, size) of every node] per level, root first; a node splits into floor and rest."""
    lv = [[(0, n)]]
    for _ in range(_depth(n, leaf)):
        lv.append([x for s, z in lv[-1] for x in ((s, z // 2), (s + z // 2, z - z // 2))])
    return lv


def _lda(n):
    return -(-n // 4) * 4


def _lowrank(n, leaf, k, seed, dtype):
    """Row-major (n, lda) operator with off-diagonal blocks of exact rank k, leaf blocks N(0,1) + n I."""
    g = _gen(seed)
    A = torch.zeros((n, _lda(n)), device=DEV, dtype=dtype)
    lv = _levels(n, leaf)
    for nodes in lv[1:]:
        U, V = _randn((n, k), g, dtype), _randn((n, k), g, dtype)
        for (sa, za), (sb, zb) in zip(nodes[0::2], nodes[1::2]):
            torch.matmul(U[sa:sa + za], V[sb:sb + zb].T, out=A[sa:sa + za, sb:sb + zb])
            torch.matmul(U[sb:sb + zb], V[sa:sa + za].T, out=A[sb:sb + zb, sa:sa + za])
    D = _randn((n, max(z for _, z in lv[-1])), g, dtype)
    for s, z in lv[-1]:
        A[s:s + z, s:s + z] = D[s:s + z, :z]
    A.diagonal().add_(float(n))
    return A


def _log_rows(n, i0, i1, shift):
    """Rows i0:i1 of log|x_i - x_j| in FP64, 1 on the diagonal, for the points (cos t, sin t / 2),
    t_i = 2 pi (i + shift) / n: with d = pi (i - j) / n and f = pi (i + j + 2 shift) / n,
    |x_i - x_j|^2 = sin^2(d) (1 + 3 sin^2(f)), a Toeplitz and a Hankel term."""
    m = torch.arange(n, device=DEV, dtype=torch.float64)
    S = torch.log(torch.sin(math.pi * m / n))
    s = torch.arange(2 * n - 1, device=DEV, dtype=torch.float64)
    P = 0.5 * torch.log1p(3.0 * torch.sin(math.pi * (s + 2.0 * shift) / n) ** 2)
    toe = torch.cat([S.flip(0), S[1:]])  # toe[n - 1 + j - i] = S[|i - j|]
    A = toe.unfold(0, n, 1)[n - i1:n - i0].flip(0)
    A += P.unfold(0, n, 1)[i0:i1]
    A.diagonal(i0).fill_(1.0)
    return A


def _shift(seed):
    return float(torch.rand((), generator=torch.Generator().manual_seed(int(seed)), dtype=torch.float64))


def _log_operator(n, seed):
    A = torch.zeros((n, _lda(n)), device=DEV, dtype=torch.float32)
    for i in range(0, n, 4096):
        A[i:min(n, i + 4096), :n] = _log_rows(n, i, min(n, i + 4096), _shift(seed))
    return A


def _dense_box(A, prec):
    if prec == "a32":
        return hm.hm_dense_operator_create(A, fp64_blocks=True, tensor_cores=True)
    return hm.hm_dense_operator_create(A)


def _matrix(case, seed):
    """The dense operator of a compression case (None: it is never stored)."""
    if case.get("source") == "lowrank":
        return _lowrank(case["n"], case["leaf"], case["k"], seed,
                        torch.float64 if case["prec"] == "fp64" else torch.float32)
    return None if case.get("source") == "free" else _log_operator(case["n"], seed)


def _options(case, seed):
    o = {"seed": int(seed) + 2, "prec": PREC[case["prec"]]}
    o.update({"k": case["k"], "p": 10} if "k" in case else {"tol": 1e-7, "r": case["r"]})
    return o


def _compress(case, op, tree, opts):
    if case["fmt"] == "hodlr":
        return hm.hm_compress_hodlr(op, tree, **opts)
    return hm.hm_compress_hbs(op, tree, **opts)


def _batch_specs(case):
    g = torch.Generator().manual_seed(case["spec"])
    u = torch.rand((case["ops"], 2), generator=g, dtype=torch.float64).tolist()
    low, high = math.log(case["low"]), math.log(case["high"])
    return [(64 * round(math.exp(low + a * (high - low)) / 64), 8 + int(33 * b)) for a, b in u]


def _factors(case, seed):
    g = _gen(seed)
    n, k, leaf = case["n"], case["k"], case["leaf"]
    depth = _depth(n, leaf)
    nmax = -(-n // 2 ** depth)
    s = {"case": case, "tree": hm.Tree(n, leaf)}
    s["U"], s["V"] = _randn((depth, k, n), g), _randn((depth, k, n), g)
    s["D"] = _randn((2 ** depth, nmax, nmax), g)
    s["x"], s["b"] = _randn((n,), g), _randn((n,), g)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("train", "autograd"):
        s = _factors(case, seed)
        if kind == "train":
            s["out"] = {"y": torch.empty_like(s["x"]), "r": torch.empty_like(s["x"]),
                        "gx": torch.empty_like(s["x"]), "gU": torch.empty_like(s["U"]),
                        "gV": torch.empty_like(s["V"]), "gD": torch.empty_like(s["D"])}
        else:
            for name in ("x", "U", "V", "D"):
                s[name].requires_grad_()
        return s
    if kind == "gemm":
        g = _gen(seed)
        n = case["n"]
        A = _randn((n, _lda(n)), g, torch.float64 if case["prec"] == "fp64" else torch.float32)
        X = _randn((case["cols"], n), g, BLOCK[case["prec"]])
        return {"case": case, "op": _dense_box(A, case["prec"]), "X": X, "Y": torch.empty_like(X), "A": A}
    if kind == "batch":
        s = {"case": case, "ops": [], "trees": [], "opts": [], "X": []}
        for i, (n, k) in enumerate(_batch_specs(case)):
            A = _lowrank(n, 64, k, 1000 * int(seed) + i, torch.float32)
            s["ops"].append(_dense_box(A, "a32"))
            s["trees"].append(hm.Tree(n, 64))
            s["opts"].append({"k": k, "p": 10, "seed": int(seed) + 2000 + i, "prec": hm.HM_A32})
            s["X"].append(_randn((VECTORS, n), _gen(1000 * int(seed) + 500 + i), torch.float64))
        return s
    n, dtype = case["n"], BLOCK[case["prec"]]
    s = {"case": case, "tree": hm.Tree(n, case["leaf"])}
    if kind == "compress":
        A = _matrix(case, seed)
        s["op"] = hm.hm_log_kernel_operator_create(n) if A is None else _dense_box(A, case["prec"])
        s["opts"] = _options(case, seed)
        s["X"] = _randn((VECTORS, n), _gen(int(seed) + 1), dtype)
        return s
    if kind == "apply":
        op = hm.hm_log_kernel_operator_create(n)
        s["h"] = _compress(case, op, s["tree"], _options(case, seed))
    else:
        A = _lowrank(n, case["leaf"], case["k"], seed, torch.float64 if case["prec"] == "fp64" else torch.float32)
        s["h"] = hm.hm_compress_hodlr(_dense_box(A, case["prec"]), s["tree"], **_options(case, seed))
    s["X"] = _randn((case["cols"], n), _gen(int(seed) + 1), dtype)
    return s


# --------------------------------------------------------------------- run ---
def _both(call, h, X):
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    call(h, 0, X, Y)
    call(h, 1, X, Z)
    return [Y, Z]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        hm.hm_hodlr_factored_loss_grad(s["tree"], case["k"], s["U"], s["V"], s["D"], s["x"], s["b"],
                                       2.0, **s["out"])
        return dict(s["out"])
    if kind == "autograd":
        y = HodlrApply.apply(s["x"], s["U"], s["V"], s["D"], s["tree"], case["k"])
        return [y, *torch.autograd.grad(y, (s["x"], s["U"], s["V"], s["D"]), s["b"])]
    if kind == "gemm":
        hm.hm_dense_apply(s["op"], case["trans"], s["X"], s["Y"])
        return s["Y"]
    if kind == "compress":
        h = _compress(case, s["op"], s["tree"], s["opts"])
        return _both(hm.hm_apply, h, s["X"])
    if kind == "batch":
        hs = hm.hm_compress_batched(s["ops"], s["trees"], "hodlr", s["opts"])
        return [_both(hm.hm_apply, h, X) for h, X in zip(hs, s["X"])]
    if kind == "apply":
        return _both(hm.hm_apply, s["h"], s["X"])
    hm.hm_hodlr_factorize(s["h"])
    return _both(hm.hm_solve, s["h"], s["X"])


# -------------------------------------------------------------------- work ---
def _compress_work(n, leaf, r, source, prec, vectors):
    depth = _depth(n, leaf)
    nmax = -(-n // 2 ** depth)
    size = 8 if prec == "fp64" else 4
    # the operator once (formed on the fly: its tables), the vectors once each way
    read = 24 * n if source == "free" else size * n * n
    block = 4 if prec == "mixed" else 8
    # 2 r columns per level and side, each nonzero on half of the rows; the leaf probe
    # has one nonzero per leaf and column
    flops = depth * 2 * 2 * r * n * n + 2 * n * 2 ** depth * nmax
    held = 2 * depth * n * r + n * nmax
    return {"bytes": read + block * 3 * vectors * n, "flops": flops + 2 * 2 * held * vectors}


def work(case):
    kind, n = case["kind"], case.get("n")
    if kind in ("train", "autograd"):
        depth = _depth(n, case["leaf"])
        nmax = -(-n // 2 ** depth)
        held = 2 * depth * case["k"] * n + 2 ** depth * nmax * nmax
        # factors once, their gradients once, the vectors x, b, y, (r,) gx
        return {"bytes": 4 * (2 * held + (5 if kind == "train" else 4) * n), "flops": 6 * held}
    if kind == "gemm":
        size = 8 if case["prec"] == "fp64" else 4
        block = 4 if case["prec"] == "mixed" else 8
        return {"bytes": size * n * n + 2 * block * n * case["cols"], "flops": 2 * n * n * case["cols"]}
    if kind == "compress":
        r = case["r"] if "r" in case else case["k"] + 10
        return _compress_work(n, case["leaf"], r, case["source"], case["prec"], VECTORS)
    if kind == "batch":
        each = [_compress_work(m, 64, k + 10, "lowrank", "a32", VECTORS) for m, k in _batch_specs(case)]
        return {w: sum(e[w] for e in each) for w in ("bytes", "flops")}
    depth = _depth(n, case["leaf"])
    nmax = -(-n // 2 ** depth)
    c = case["cols"]
    if kind == "apply":
        r = case["r"]
        # HODLR: two factors of n x r per level; HBS-ID: nested, about two of n x r in all
        held = n * nmax + 2 * n * r * (depth if case["fmt"] == "hodlr" else 1)
        return {"bytes": 2 * 8 * (held + 2 * n * c), "flops": 2 * 2 * held * c}
    block = 4 if case["prec"] == "mixed" else 8
    k = case["k"]
    held = n * nmax + 2 * depth * n * k
    factor = 2 * n * nmax * nmax + 2 * n * k * k * depth * depth
    return {"bytes": block * (3 * held + 2 * 2 * n * c), "flops": factor + 2 * 2 * held * c}


# ------------------------------------------------------------------- exact ---
def _exact_layer(case, s, g):
    """[y, H^T g, and the gradients of <g, H x>] at the factors, in 64 bits; g from y if callable."""
    n, leaf = case["n"], case["leaf"]
    lv = _levels(n, leaf)
    with torch.no_grad():
        x, U, V, D = (s[name].double() for name in ("x", "U", "V", "D"))
        y = torch.zeros_like(x)
        for i, (a, z) in enumerate(lv[-1]):
            y[a:a + z] = D[i, :z, :z].T @ x[a:a + z]
        proj = []
        for j, nodes in enumerate(lv[1:]):
            p = [V[j, :, a:a + z] @ x[a:a + z] for a, z in nodes]
            proj.append(p)
            for i, (a, z) in enumerate(nodes):
                y[a:a + z] += U[j, :, a:a + z].T @ p[i ^ 1]
        r = g(y)
        gx = torch.zeros_like(x)
        gU, gV, gD = torch.zeros_like(U), torch.zeros_like(V), torch.zeros_like(D)
        for i, (a, z) in enumerate(lv[-1]):
            gx[a:a + z] = D[i, :z, :z] @ r[a:a + z]
            gD[i, :z, :z] = torch.outer(x[a:a + z], r[a:a + z])
        for j, nodes in enumerate(lv[1:]):
            q = [U[j, :, a:a + z] @ r[a:a + z] for a, z in nodes]
            for i, (a, z) in enumerate(nodes):
                gx[a:a + z] += V[j, :, a:a + z].T @ q[i ^ 1]
                gU[j, :, a:a + z] = torch.outer(proj[j][i ^ 1], r[a:a + z])
                gV[j, :, a:a + z] = torch.outer(q[i ^ 1], x[a:a + z])
    return y, r, gx, gU, gV, gD


def _products(rows, n, X):
    """[(A X)^T, (A^T X)^T] for X given as a (c, n) block, A from rows(i0, i1), in 64 bits."""
    X = X.double()
    Y, Z = torch.empty_like(X), torch.zeros_like(X)
    for i in range(0, n, 4096):
        e = min(n, i + 4096)
        A = rows(i, e)
        Y[:, i:e] = X @ A.T
        Z += X[:, i:e] @ A
    return [Y, Z]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "autograd"):
        s = _factors(case, seed)
        if kind == "autograd":
            y, _, gx, gU, gV, gD = _exact_layer(case, s, lambda y: s["b"].double())
            return [y, gx, gU, gV, gD]
        y, r, gx, gU, gV, gD = _exact_layer(case, s, lambda y: y - s["b"].double())
        return {"y": y, "r": r, "gx": 2 * gx, "gU": 2 * gU, "gV": 2 * gV, "gD": 2 * gD}
    if kind == "gemm":
        s = prepare(case, seed)
        n = case["n"]
        return _products(lambda i, e: s["A"][i:e, :n].double(), n, s["X"])[case["trans"]]
    if kind == "batch":
        out = []
        for i, (n, k) in enumerate(_batch_specs(case)):
            A = _lowrank(n, 64, k, 1000 * int(seed) + i, torch.float32)
            X = _randn((VECTORS, n), _gen(1000 * int(seed) + 500 + i), torch.float64)
            out.append(_products(lambda a, e: A[a:e, :n].double(), n, X))
        return out
    n = case["n"]
    X = _randn((case.get("cols", VECTORS), n), _gen(int(seed) + 1), BLOCK[case["prec"]])
    if kind == "solve":
        A = _lowrank(n, case["leaf"], case["k"], seed,
                     torch.float64 if case["prec"] == "fp64" else torch.float32)[:, :n].double()
        return [torch.linalg.solve(A, X.double().T).T.contiguous(),
                torch.linalg.solve(A.T, X.double().T).T.contiguous()]
    A = _matrix(case, seed) if kind == "compress" else None
    if A is None:  # the matrix-free kernel: its points are not shifted
        return _products(lambda i, e: _log_rows(n, i, e, 0.0), n, X)
    return _products(lambda i, e: A[i:e, :n].double(), n, X)
