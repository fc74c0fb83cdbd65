"""The workloads whose speed is tracked, each run through the public Python binding.

A case is one whole call as a user's program makes it: a batched GDA run on a problem handle the
program keeps (``Problem.gda``: start, iterations, evaluations) followed by the read-back it needs,
a grouped run over instances of uneven size, or the Lagrangian's value and gradients through
``torch.autograd``.  Kinds:

* ``qubo``    dense QUBO, integer entries in [-100, 100] (BF16 tensor-core problems, FP32 problems,
  and the tiny FP32 problems with n <= 64)
* ``graph``   Max-Cut as a sparse QUBO: Erdos-Renyi and torus graphs with +-1 weights, random
  4-regular graphs with unit weights, in each weight precision
* ``maxk``    Max-k-Cut on the same graphs
* ``group``   several dense BF16 instances of uneven n advanced together
* ``lagr``    Lagrangian value and gradients (forward and backward) at a batch of points

Runs whose state is small enough to be read back on every call return the iterates X and Y; the
larger ones return what such programs read: every restart's best objective and the trace.
"""
import math

import numpy as np
import torch

from paper_2509_21064_gb300 import sbo as S
from paper_2509_21064_gb300.autograd import lagrangian

STATE_LIMIT = 6_000_000          # n * restarts up to which a run returns its iterates
PREC = {"fp32": S.SBO_FP32, "bf16": S.SBO_BF16, "e4m3": S.SBO_FP8_E4M3}


def listed():
    return [
        # plain method on a small QUBO (the brute-forced configuration): pure latency
        {"name": "tiny_n20_fp32", "kind": "qubo", "n": 20, "B": 32, "T": 1000, "K": 10, "prec": "fp32"},
        # small dense instance at ragged sizes, as one member of a sweep
        {"name": "dense_n1003_bf16", "kind": "qubo", "n": 1003, "B": 200, "T": 100, "K": 10, "prec": "bf16"},
        # the plain FP32 form, used where a run is compared with full-precision arithmetic
        {"name": "dense_n1500_fp32", "kind": "qubo", "n": 1500, "B": 130, "T": 50, "K": 50, "prec": "fp32"},
        # dense QUBO n = 5,000 of the benchmark
        {"name": "dense_n5000_bf16", "kind": "qubo", "n": 5000, "B": 256, "T": 200, "K": 50, "prec": "bf16"},
        # the headline: dense QUBO n = 20,000, 1,024 restarts, one step of 50 iterations + evaluation
        {"name": "dense_n20000_bf16", "kind": "qubo", "n": 20000, "B": 1024, "T": 50, "K": 50, "prec": "bf16"},
        # Max-Cut on a sparse random graph, the small sparse configuration
        {"name": "er_n2000_fp32", "kind": "graph", "family": "er", "n": 2000, "B": 256, "T": 400, "K": 10,
         "prec": "fp32"},
        # Max-Cut on the 100 x 100 torus with E4M3 weights
        {"name": "torus_n10000_e4m3", "kind": "graph", "family": "torus", "n": 10000, "B": 512, "T": 400, "K": 10,
         "prec": "e4m3"},
        # Max-Cut on a random 4-regular graph, the largest sparse configuration
        {"name": "regular_n20000_fp32", "kind": "graph", "family": "regular", "n": 20000, "B": 512, "T": 300,
         "K": 10, "prec": "fp32"},
        # Max-3-Cut on the torus with the paper's B = 100
        {"name": "max3cut_n10000", "kind": "maxk", "family": "torus", "n": 10000, "k": 3, "B": 100, "T": 200,
         "K": 10},
        # a heterogeneous batch of dense instances in one grouped run
        {"name": "group_8x_bf16", "kind": "group", "count": 8, "n_lo": 500, "n_hi": 3000, "B": 128, "T": 30,
         "K": 10},
        # value and gradients of the Lagrangian inside a torch program: dense and sparse problems
        {"name": "lagr_dense_n5000_bf16", "kind": "lagr", "family": "dense", "n": 5000, "B": 256, "prec": "bf16"},
        {"name": "lagr_regular_n20000_fp32", "kind": "lagr", "family": "regular", "n": 20000, "B": 512,
         "prec": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph_n(rng, family, lo, hi):
    n = _log(rng, lo, hi)
    return max(5, round(math.sqrt(n))) ** 2 if family == "torus" else n


def draw(rng):
    kind = rng.choice(["tiny", "dense", "fp32", "graph", "graph", "graph", "maxk", "group", "lagr", "lagr"])
    if kind == "tiny":
        return {"kind": "qubo", "n": rng.randint(4, 64), "B": _log(rng, 1, 300), "T": _log(rng, 50, 1000),
                "K": rng.choice([1, 10, 50]), "prec": "fp32"}
    if kind == "dense":
        n = _log(rng, 200, 8000)
        return {"kind": "qubo", "n": n, "B": _log(rng, 10, 512), "T": rng.choice([50, 100]),
                "K": rng.choice([10, 50]), "prec": "bf16"}
    if kind == "fp32":
        return {"kind": "qubo", "n": _log(rng, 65, 3000), "B": _log(rng, 8, 256), "T": 50,
                "K": rng.choice([10, 50]), "prec": "fp32"}
    if kind == "graph":
        family = rng.choice(["er", "torus", "regular"])
        return {"kind": "graph", "family": family, "n": _graph_n(rng, family, 300, 20000), "B": _log(rng, 8, 512),
                "T": _log(rng, 50, 400), "K": rng.choice([5, 10, 25]), "prec": rng.choice(["fp32", "bf16", "e4m3"])}
    if kind == "maxk":
        family = rng.choice(["er", "torus", "regular"])
        return {"kind": "maxk", "family": family, "n": _graph_n(rng, family, 300, 10000), "k": rng.choice([2, 3, 4, 5]),
                "B": _log(rng, 8, 128), "T": rng.choice([50, 100, 200]), "K": 10}
    if kind == "group":
        return {"kind": "group", "count": rng.randint(2, 8), "n_lo": rng.randint(200, 600),
                "n_hi": rng.randint(800, 3000), "B": rng.choice([64, 100, 128]), "T": 30, "K": 10}
    family = rng.choice(["dense", "torus", "er", "regular"])
    if family == "dense":
        prec = rng.choice(["bf16", "fp32"])
        return {"kind": "lagr", "family": "dense", "n": _log(rng, 100, 5000 if prec == "bf16" else 2000),
                "B": _log(rng, 4, 256), "prec": prec}
    return {"kind": "lagr", "family": family, "n": _graph_n(rng, family, 300, 20000), "B": _log(rng, 4, 256),
            "prec": rng.choice(["fp32", "bf16"])}


# ---- inputs ------------------------------------------------------------------------------------
def _dense(n, seed):
    """Symmetric integer Q in [-100, 100] (int8, host) with its diagonal moved into c."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    q = torch.randint(-100, 101, (n, n), generator=g, device="cuda", dtype=torch.int8)
    c = torch.diagonal(q).to(torch.int32).cpu().numpy()
    u = torch.triu(q, 1)
    del q
    return (u + u.T).cpu().numpy(), c


def _edges(family, n, seed):
    rng = np.random.default_rng(seed)
    if family == "torus":
        side = math.isqrt(n)
        v = np.arange(n).reshape(side, side)
        a = np.concatenate([v.ravel(), v.ravel()])
        b = np.concatenate([np.roll(v, -1, 1).ravel(), np.roll(v, -1, 0).ravel()])
    elif family == "regular":        # two random Hamiltonian cycles
        p, q = rng.permutation(n), rng.permutation(n)
        a, b = np.concatenate([p, q]), np.concatenate([np.roll(p, -1), np.roll(q, -1)])
    else:                            # mean degree 6
        a, b = rng.integers(0, n, 3 * n), rng.integers(0, n, 3 * n)
        a, b = a[a != b], b[a != b]
    key = np.unique(np.minimum(a, b).astype(np.int64) * n + np.maximum(a, b))
    a, b = (key // n).astype(np.int32), (key % n).astype(np.int32)
    w = np.ones(a.size, np.int32) if family == "regular" else rng.choice(np.array([-1, 1], np.int32), a.size)
    return a, b, w


def _csr(n, a, b, w):
    r, c, v = np.concatenate([a, b]), np.concatenate([b, a]), np.concatenate([w, w])
    o = np.lexsort((c, r))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int64)
    lin = -np.bincount(r, weights=v, minlength=n).astype(np.int32)
    return rowptr, c[o].astype(np.int32), v[o].astype(np.int32), lin


def _group_ns(case, seed):
    rng = np.random.default_rng(seed)
    # the sizes belong to the case (every seed has the same amount of work); the entries to the seed
    span = np.linspace(case["n_lo"], case["n_hi"], case["count"]).round().astype(int)
    return [int(v) for v in span], [int(v) for v in rng.integers(1, 2**31, case["count"])]


def _lam(n):
    """Semicircle estimate of |lambda_min| of Q with entries uniform in [-100, 100]."""
    return 2.0 * math.sqrt((201**2 - 1) / 12.0) * math.sqrt(n)


def _hyper(case, n):
    """The paper's Max-Cut step sizes, rescaled to a dense instance's spectrum; Max-k-Cut's table."""
    if case["kind"] == "graph":
        return {"alpha": 0.025, "beta": 0.025, "ybar": 6.0, "grad_tol": 0.02}
    if case["kind"] == "maxk":
        return {"alpha": 0.1, "beta": 0.01, "ybar": 6.0, "grad_tol": 0.02}
    s = _lam(n) / 4.0
    return {"alpha": 0.025 / s, "beta": 0.025 * s, "ybar": 6.0 * s, "grad_tol": 0.02 * s}


def _params(case, n, seed):
    return S.params(restarts=case["B"], iters=case["T"], eval_every=case["K"], delta=0.01, seed=seed,
                    **_hyper(case, n))


def _points(n, B, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand(B, n, generator=g, device="cuda")
    Y = 6.0 * torch.rand(B, n, generator=g, device="cuda")
    return X, Y, 0.5 + torch.rand(B, generator=g, device="cuda")


def prepare(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "group":
        ns, seeds = _group_ns(case, seed)
        probs = [S.Problem.dense(*_dense(m, s)) for m, s in zip(ns, seeds)]
        return {"kind": kind, "G": S.Group(probs), "P": probs, "T": case["T"],
                "prm": [_params(case, m, s) for m, s in zip(ns, seeds)]}
    if kind == "qubo" or case.get("family") == "dense":
        Q, c = _dense(n, seed)
        P = S.Problem.dense(Q, c, precision=PREC[case["prec"]])
    elif kind == "maxk":
        P = S.Problem.maxkcut(n, *_edges(case["family"], n, seed), case["k"])
    else:
        P = S.Problem.csr(n, *_csr(n, *_edges(case["family"], n, seed)), precision=PREC[case["prec"]])
    state = {"kind": kind, "P": P}
    if kind == "lagr":
        X, Y, g = _points(n, case["B"], seed)
        state.update(X=X.requires_grad_(), Y=Y.requires_grad_(), g=g)
    else:
        state.update(prm=_params(case, n, seed), iterates=n * case["B"] * case.get("k", 1) <= STATE_LIMIT)
    return state


def _records(P):
    F, _ = P.restart_best()
    return {"F": F.astype(np.float64), "trace": P.trace(4096).astype(np.float64)}


def run(state):
    kind, P = state["kind"], state["P"]
    if kind == "lagr":
        L = lagrangian(state["X"], state["Y"], P)
        gx, gy = torch.autograd.grad(L, (state["X"], state["Y"]), grad_outputs=state["g"])
        return {"L": L.detach(), "GX": gx, "GY": gy}
    if kind == "group":
        state["G"].start(state["prm"])
        state["G"].run(state["T"])
        state["G"].sync()
        out = []
        for p in P:
            X, Y = p.state()
            out.append({"X": X, "Y": Y, **_records(p)})
        return out
    P.gda(state["prm"])
    out = _records(P)
    if state["iterates"]:
        out["X"], out["Y"] = P.state()
    return out


# ---- amounts and accuracy ----------------------------------------------------------------------
def _shape(case):
    """(variables, entries of A, entries of the state) of one restart's iteration."""
    kind, n = case["kind"], case.get("n", 0)
    if kind == "group":
        ns, _ = _group_ns(case, 0)
        return sum(ns), sum(m * m for m in ns), sum(ns)
    if kind == "qubo" or case.get("family") == "dense":
        return n, n * n, n
    return n, (6 if case["family"] == "er" else 4) * n, n * case.get("k", 1)


def work(case):
    n, nnz, per = _shape(case)
    B, k = case["B"], case.get("k", 1)
    a_bytes = nnz * ({"bf16": 2, "fp32": 4}.get(case.get("prec", "bf16"), 4)
                     if case["kind"] in ("qubo", "group") or case.get("family") == "dense" else 8)
    if case["kind"] == "lagr":
        # x and y in, both gradients out; one contraction forward and one backward
        return {"bytes": a_bytes + 16 * n * B, "flops": 2 * (2 * nnz + 8 * n) * B}
    evals = -(-case["T"] // case["K"])
    return {"bytes": a_bytes + 8 * per * B, "flops": (case["T"] * (2 * nnz * k + 12 * per) + evals * 2 * nnz) * B}


def tolerance(case):
    """About four times what the sums in another order (other tile widths) change, measured; where
    a candidate bit of one restart flips with them, its objective moves by up to 1e-3 of itself."""
    if case["kind"] == "lagr":
        return {"rel": 5e-6}
    if case["kind"] == "maxk" or case.get("prec") == "fp32":
        return {"rel": 1e-4, "max": 5e-3}
    return {"rel": 8e-4, "max": 6e-3}


def _splitmix(seed, r, i):
    """x^0 of restart r, coordinate i: the top 24 bits of the SplitMix64 output number r 2^32 + i."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + ((r << np.uint64(32)) + i + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(40)).astype(np.float64) / float(1 << 24)


def _exact_matrix(case, seed):
    n = case["n"]
    if case["kind"] == "qubo" or case.get("family") == "dense":
        Q, c = _dense(n, seed)
        A = torch.from_numpy(Q).cuda().double()
        return (A + A.T).fill_diagonal_(0.0), torch.from_numpy(c).cuda().double()
    a, b, w = _edges(case["family"], n, seed)
    idx = torch.from_numpy(np.stack([np.concatenate([a, b]), np.concatenate([b, a])]).astype(np.int64)).cuda()
    val = torch.from_numpy(np.concatenate([w, w])).cuda().double()
    W = torch.sparse_coo_tensor(idx, val, (n, n)).coalesce()
    lin = torch.zeros(n, dtype=torch.double, device="cuda").index_add_(0, idx[0], val)
    return (W, lin) if case["kind"] == "maxk" else (2.0 * W, -lin)


def _exact_qubo(A, c, x0, h, T):
    X = torch.from_numpy(x0).cuda()                      # n x B
    Y = torch.full_like(X, h["ybar"])
    c = c[:, None]
    for _ in range(T):
        D = A @ X + c + Y * (2.0 * X - 1.0)
        stuck = ((X - 0.5).abs() <= 0.01) & (D.abs() <= h["grad_tol"]) & (Y <= 0)
        Z = (X - h["alpha"] * D).clamp(0.0, 1.0)
        Y = Y + h["beta"] * (X * X - X)
        X = torch.where(stuck, torch.where(X <= 0.5, 0.49, 0.51).to(X.dtype), Z)
    return {"F": None, "trace": None, "X": X.T.cpu().numpy(), "Y": Y.T.cpu().numpy()}


def _exact_maxk(W, z0, n, k, B, h, T):
    Z = torch.from_numpy(z0).cuda().reshape(B, n, k)
    Y = torch.full((B, n), h["ybar"], dtype=torch.double, device="cuda")
    for _ in range(T):
        X = torch.softmax(Z, 2)
        G = (W @ X.permute(1, 0, 2).reshape(n, B * k)).reshape(n, B, k).permute(1, 0, 2)
        H = 2.0 * (G + Y[:, :, None] * X)
        Z = Z - h["alpha"] * X * (H - (X * H).sum(2, keepdim=True))
        Y = Y + h["beta"] * ((X * X).sum(2) - 1.0)
    return {"F": None, "trace": None, "X": torch.softmax(Z, 2).cpu().numpy(), "Y": Y.cpu().numpy()}


def exact(case, seed):
    """The same outputs in 64 bits (None where they are whole numbers or the run is too long for it)."""
    n, B, kind = case.get("n", 0), case["B"], case["kind"]
    if kind == "group":
        ns, seeds = _group_ns(case, seed)
        return [exact({**case, "kind": "qubo", "n": m}, s) for m, s in zip(ns, seeds)]
    if kind == "lagr":
        A, c = _exact_matrix(case, seed)
        X, Y, g = (t.double() for t in _points(n, B, seed))
        G = (A @ X.T).T
        return {"L": 0.5 * (X * G).sum(1) + X @ c + (Y * (X * X - X)).sum(1),
                "GX": g[:, None] * (G + c + Y * (2.0 * X - 1.0)), "GY": g[:, None] * (X * X - X)}
    if n * B * case.get("k", 1) > STATE_LIMIT:
        return None
    if kind == "qubo" and float(n) * n * B * case["T"] > 4e12:
        return None
    A, c = _exact_matrix(case, seed)
    h = _hyper(case, n)
    r = np.arange(B, dtype=np.uint64)
    i = np.arange(n * case.get("k", 1), dtype=np.uint64)
    if kind == "maxk":
        return _exact_maxk(A, _splitmix(seed, r[:, None], i[None, :]), n, case["k"], B, h, case["T"])
    return _exact_qubo(A, c, _splitmix(seed, r[None, :], i[:, None]), h, case["T"])
