"""The work that a user of this library has it do, as cases that can be measured one by one.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (the handle
on its matrix, the starting vectors, result buffers), ``run`` makes one call through the public
binding, ``work`` counts the bytes and operations that the call cannot do without, and ``exact``
gives the outputs in 64 bits from plain torch.

Solves run a fixed number of sweeps (a negative tolerance), so that a case is the same work whatever
the data.  A component is defined up to its sign, which depends on the winning start: ``run`` fixes it
as programs that compare components do (the largest loading is positive).
"""
import math

import numpy as np
import torch

from paper_1212_4137_gb300 import spca

STORAGE = {"f32": spca.SPCA_F32, "fp16": spca.SPCA_FP16, "fp8": spca.SPCA_FP8_E4M3_COLSCALED,
           "resident16": spca.SPCA_FP16_RESIDENT}


def listed():
    return [
        # the small dense problem: latency of one call, 16 starts
        {"name": "small_dense", "kind": "solve", "data": "gauss", "n": 100, "p": 500, "r": 16, "form": 1, "s": 10,
         "calib": 0, "sweeps": 40, "storage": "f32"},
        # a batch of 16 starts of the economies-of-scale experiment (n = p / 10, 10 nonzeros, 10 sweeps)
        {"name": "economies_batch16", "kind": "solve", "data": "gauss", "n": 400, "p": 4000, "r": 16, "form": 5,
         "s": 10, "calib": 5, "sweeps": 10, "storage": "f32"},
        # the wide shape of the L1-variance comparison (n = p / 200): few samples, many variables
        {"name": "wide_l1", "kind": "solve", "data": "gauss", "n": 500, "p": 100000, "r": 16, "form": 8, "s": 10,
         "calib": 10, "sweeps": 16, "storage": "f32"},
        # the benchmark's spiked matrix from 1024 starts: the largest batches of one problem
        {"name": "spiked_many", "kind": "solve", "data": "spiked", "n": 5000, "p": 20000, "r": 1024, "form": 1,
         "s": 50, "calib": 0, "sweeps": 10, "storage": "f32"},
        # the same matrix from one start: a warm-started or single solve, bound by reading A
        {"name": "spiked_one", "kind": "solve", "data": "spiked", "n": 5000, "p": 20000, "r": 1, "form": 3,
         "s": 50, "calib": 0, "sweeps": 16, "storage": "f32"},
        # a request to the serving layer's resident 16-bit matrices
        {"name": "resident_request", "kind": "solve", "data": "spiked", "n": 9001, "p": 17003, "r": 16, "form": 7,
         "s": 40, "calib": 10, "sweeps": 16, "storage": "resident16"},
        # a dozen problems of uneven sizes and all formulations solved together
        {"name": "group_mixed", "kind": "group", "count": 12, "nmax": 4000, "pmax": 20000, "r": 64, "sweeps": 8},
        # word counts in compressed sparse rows with the text corpora's settings (s = 5, 20 starts)
        {"name": "corpus", "kind": "corpus", "n": 40000, "p": 20000, "per_doc": 120, "r": 20, "form": 1, "s": 5,
         "calib": 0, "sweeps": 20},
        # one sweep's two contractions with FP32 accuracy, 1024 starts, ragged sizes
        {"name": "products_f32", "kind": "products", "data": "spiked", "n": 5003, "p": 20011, "r": 1024, "form": 1,
         "engine": "auto", "storage": "f32"},
        # the precision layer's large matrix: the two contractions of a low-precision sweep
        {"name": "products_fp8", "kind": "products", "data": "spiked", "n": 20000, "p": 50000, "r": 1024, "form": 1,
         "engine": "lowp", "storage": "fp8"},
        # the x-step alone on given v (the L1-ball operator of formulation 3)
        {"name": "xstep_l1ball", "kind": "xstep", "p": 20011, "r": 1024, "form": 3, "s": 50, "calib": 0},
        # objectives of given sparse x without allocating, as a latency-critical loop evaluates them
        {"name": "objective", "kind": "objective", "n": 5000, "p": 20000, "r": 64, "form": 5, "s": 50},
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["solve"] * 5 + ["group", "corpus", "products", "products", "xstep", "xstep", "objective"])
    form = rng.randint(1, 8)
    if kind == "group":
        return {"kind": "group", "count": rng.randint(2, 12), "nmax": log(400, 4000), "pmax": log(1000, 20000),
                "r": log(16, 64), "sweeps": rng.randint(6, 8)}
    if kind == "corpus":
        return {"kind": "corpus", "n": log(2000, 40000), "p": log(1000, 20000), "per_doc": rng.randint(30, 120),
                "r": log(5, 64), "form": rng.choice([1, 3]), "s": rng.randint(3, 10), "calib": 0, "sweeps": 20}
    if kind == "xstep":
        return {"kind": "xstep", "p": log(500, 40000), "r": log(1, 512), "form": form, "s": rng.randint(5, 100),
                "calib": 1 if form >= 5 else 0}
    if kind == "objective":
        return {"kind": "objective", "n": log(300, 5000), "p": log(1000, 20000), "r": log(1, 64), "form": form,
                "s": rng.randint(5, 60)}
    if kind == "products":
        # L2 variance: a sign of L1 variance at u = 0 is decided by the last bit of u
        return {"kind": "products", "data": "spiked", "n": log(300, 5000), "p": log(1000, 20000), "r": log(1, 1024),
                "form": rng.choice([1, 3, 5, 7]), "engine": "auto", "storage": "f32"}
    what = rng.choice(["small", "economies", "wide", "many", "few", "resident"])
    c = {"kind": "solve", "data": "gauss", "form": form, "calib": 5 if form >= 5 else 0, "storage": "f32"}
    if what == "small":
        c.update(n=log(40, 250), p=log(150, 1000), r=log(2, 32), s=rng.randint(5, 12), sweeps=rng.randint(10, 40))
    elif what == "economies":
        p = log(1000, 32000)
        c.update(n=p // 10, p=p, r=log(1, 256), s=10, sweeps=10)
    elif what == "wide":
        p = log(4000, 100000)
        c.update(n=p // 200, p=p, r=log(1, 256), s=10, sweeps=12)
    elif what == "many":
        c.update(data="spiked", n=log(1000, 5000), p=log(4000, 20000), r=log(128, 1000), s=rng.randint(20, 60),
                 form=rng.choice([1, 3, 5, 7]), sweeps=rng.randint(8, 10))
    elif what == "few":
        c.update(data="spiked", n=log(1000, 5000), p=log(4000, 20000), r=rng.randint(1, 8), s=rng.randint(20, 60),
                 form=rng.choice([1, 3, 5, 7]), sweeps=rng.randint(8, 16))
    else:
        c.update(data="spiked", n=log(1000, 9001), p=log(2000, 17003), r=rng.choice([1, 16, 16, 256]),
                 s=rng.randint(10, 100), form=rng.choice([3, 7]), sweeps=rng.randint(8, 16), storage="resident16")
    c["calib"] = 5 if c["form"] >= 5 else 0
    return c


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _generator(seed, stream):
    return torch.Generator(device=_device()).manual_seed((int(seed) * 1000003 + stream) % (1 << 62))


def _matrix(data, n, p, seed, spikes=5, nnz=50):
    """N(0,1) entries, plus (spiked) a few rank-one terms with sparse loadings."""
    g = _generator(seed, 1)
    A = torch.randn(n, p, generator=g, device=_device())
    if data == "spiked":
        nnz = min(nnz, p)
        for k, base in enumerate((40.0, 30.0, 20.0, 15.0, 10.0)[:spikes]):
            u = torch.randn(n, generator=g, device=_device())
            at = torch.randperm(p, generator=g, device=_device())[:nnz]
            v = torch.randn(nnz, generator=g, device=_device())
            A[:, at] += base * math.sqrt(n / p) * torch.outer(u / u.norm(), v / v.norm())
    return A


def _starts(p, r, seed):
    return torch.randn(r, p, generator=_generator(seed, 2), device=_device())


def _corpus(case, seed):
    """Documents x words counts in compressed sparse rows: Zipf word popularity, log-normal document
    lengths, and topics whose words occur together in a share of the documents."""
    n, p, dev = case["n"], case["p"], _device()
    g = _generator(seed, 3)
    m = (1.35 * case["per_doc"] * torch.exp(0.5 * torch.randn(n, generator=g, device=dev) - 0.125)).round().long() + 1
    word = torch.randperm(p, generator=g, device=dev)
    cdf = torch.cumsum(1.0 / torch.arange(1, p + 1, device=dev, dtype=torch.float64), 0)
    doc = torch.repeat_interleave(torch.arange(n, device=dev), m)
    u = torch.rand(doc.numel(), generator=g, device=dev, dtype=torch.float64) * cdf[-1]
    keys = [doc * p + word[torch.searchsorted(cdf, u).clamp_(max=p - 1)]]
    member = torch.randint(0, 12, (n,), generator=g, device=dev)   # topics 0..4, else none
    extra = torch.where(member < 5, m // 4, torch.zeros_like(m))
    doc = torch.repeat_interleave(torch.arange(n, device=dev), extra)
    pick = torch.randint(0, 10, (doc.numel(),), generator=g, device=dev)
    keys.append(doc * p + word[50 + member[doc] * 10 + pick])
    key, count = torch.unique(torch.cat(keys), return_counts=True)
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    indptr[1:] = torch.cumsum(torch.bincount(key // p, minlength=n), 0)
    return indptr, (key % p).int(), count.float()


def _group_sizes(case):
    """(n, p, form, s) of each problem: sizes spread over the logarithm of their ranges."""
    out = []
    for i in range(case["count"]):
        a, b, c = (i * 0.6180339887 + 0.31) % 1.0, (i * 0.7548776662 + 0.77) % 1.0, (i * 0.5698402910) % 1.0
        out.append((int(200 * (case["nmax"] / 200) ** a), int(500 * (case["pmax"] / 500) ** b), 1 + i % 8,
                    5 + int(45 * c)))
    return out


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "group":
        problems = []
        for i, (n, p, form, s) in enumerate(_group_sizes(case)):
            h = spca.Handle(_matrix("spiked", n, p, seed + 7919 * i, 3, 20))
            x0 = _starts(p, case["r"], seed + 7919 * i)
            kw = dict(s=float(s), max_iter=case["sweeps"], tol=-1.0, x0=x0.data_ptr(), x0_device=True)
            if form >= 5:
                kw.update(gamma_target=True, calib=5)
            problems.append((h, form, case["r"], kw, x0))
        return {"kind": kind, "group": spca.Group(), "problems": [q[:4] for q in problems],
                "keep": [q[4] for q in problems]}
    if kind in ("solve", "corpus"):
        if kind == "corpus":
            indptr, col, val = (t.cpu().numpy() for t in _corpus(case, seed))
            h = spca.Handle((indptr, col, val, (case["n"], case["p"])))
        else:
            h = spca.Handle(_matrix(case["data"], case["n"], case["p"], seed), storage=STORAGE[case["storage"]])
        x0 = _starts(case["p"], case["r"], seed)
        kw = dict(s=float(case["s"]), max_iter=case["sweeps"], tol=-1.0, x0=x0.data_ptr(), x0_device=True)
        if case["form"] >= 5:
            kw.update(gamma_target=True, calib=case["calib"])
        return {"kind": "solve", "h": h, "form": case["form"], "r": case["r"], "kw": kw, "x0": x0}
    p, r, dev = case["p"], case["r"], _device()
    if kind == "products":
        n = case["n"]
        h = spca.Handle(_matrix(case["data"], n, p, seed), storage=STORAGE[case["storage"]])
        engine = spca.SPCA_ENGINE_TC_LOWP if case["engine"] == "lowp" else spca.SPCA_ENGINE_AUTO
        X = _starts(p, r, seed)
        X /= X.norm(dim=1, keepdim=True)
        return {"kind": kind, "h": h, "form": case["form"], "engine": engine, "X": X,
                "U": torch.empty(r, n, device=dev), "V": torch.empty(r, p, device=dev)}
    if kind == "xstep":
        h = spca.Handle(_matrix("gauss", 16, p, seed))   # the handle gives p and the stream
        return {"kind": kind, "h": h, "form": case["form"], "s": float(case["s"]), "calib": case["calib"],
                "V": _given_v(case, seed), "X": torch.empty(r, p, device=dev),
                "F": torch.empty(r, dtype=torch.float64, device=dev),
                "nnz": torch.empty(r, dtype=torch.int32, device=dev),
                "thr": torch.empty(r, dtype=torch.float64, device=dev)}
    spca.load()
    return {"kind": kind, "form": case["form"], "A": _matrix("gauss", case["n"], p, seed), "X": _sparse_x(case, seed),
            "f": torch.empty(r, dtype=torch.float64, device=dev), "ev": torch.empty(r, dtype=torch.float64, device=dev)}


def _given_v(case, seed):
    """v = A^T y of a spiked matrix: noise, and a few hundred entries that stand out."""
    V = _starts(case["p"], case["r"], seed) * 70.0
    V[:, ::97] *= 2.5
    return V


def _sparse_x(case, seed):
    """Unit vectors with s nonzeros each, as a solve returns them."""
    g = _generator(seed, 4)
    r, p, s = case["r"], case["p"], case["s"]
    at = torch.rand(r, p, generator=g, device=_device()).topk(s, dim=1).indices
    X = torch.zeros(r, p, device=_device())
    X.scatter_(1, at, torch.randn(r, s, generator=g, device=_device()))
    return X / X.norm(dim=1, keepdim=True)


def _component(out):
    """The result of a solve with the component's sign fixed: its largest loading is positive."""
    sign = math.copysign(1.0, out["x"][np.argmax(np.abs(out["x"]))])
    return {"objective": out["objective"], "explained_variance": out["explained_variance"],
            "x": out["x"] * np.float32(sign), "y": out["y"] * np.float32(sign), "nnz": out["nnz"]}


def run(state):
    kind = state["kind"]
    if kind == "solve":
        return _component(state["h"].solve(state["form"], state["r"], **state["kw"]))
    if kind == "group":
        return [_component(out) for out in state["group"].solve(state["problems"])]
    if kind == "products":
        X, U, V = state["X"], state["U"], state["V"]
        _ok(spca.spca_products(state["h"].h, state["form"], state["engine"], X.data_ptr(), X.stride(0), X.shape[0],
                               U.data_ptr(), U.stride(0), V.data_ptr(), V.stride(0)))
        return {"U": U, "V": V}
    if kind == "xstep":
        V, X = state["V"], state["X"]
        _ok(spca.spca_xstep(state["h"].h, state["form"], state["s"], 0.0, state["calib"], V.data_ptr(), V.stride(0),
                            V.shape[0], X.data_ptr(), X.stride(0), state["F"].data_ptr(), state["nnz"].data_ptr(),
                            state["thr"].data_ptr()))
        # F and the threshold are FP32 sums in 64-bit cells: they go on with the FP32 iterates
        return {"X": X, "F": state["F"].float(), "nnz": state["nnz"], "thr": state["thr"].float()}
    A, X = state["A"], state["X"]
    _ok(spca.spca_objective_noalloc(state["form"], 1.0, A.data_ptr(), A.shape[0], A.shape[1], A.stride(0),
                                    X.data_ptr(), X.stride(0), X.shape[0], state["f"].data_ptr(),
                                    state["ev"].data_ptr(), torch.cuda.current_stream().cuda_stream))
    return {"f": state["f"], "ev": state["ev"]}


def _ok(status):
    if status != spca.SPCA_OK:
        raise RuntimeError(spca.spca_strerror(status))


# ------------------------------------------------------------------ the work of one pass
def _solve_work(n, p, r, s, sweeps, entries, entry_bytes):
    """A read once, the starts read, x and y written; per sweep and start v = A^T y over every entry
    of A, u = A x over every entry in the first sweep and over the support afterwards."""
    per_column = entries / p
    flops = 2.0 * r * entries * (sweeps + 1) + 2.0 * r * s * per_column * (sweeps - 1)
    return {"bytes": entry_bytes * entries + 4.0 * (r * p + n + p), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "group":
        parts = [_solve_work(n, p, case["r"], s, case["sweeps"], n * p, 4) for n, p, _, s in _group_sizes(case)]
        return {"bytes": sum(w["bytes"] for w in parts), "flops": sum(w["flops"] for w in parts)}
    p, r = case["p"], case["r"]
    if kind == "corpus":
        return _solve_work(case["n"], p, r, case["s"], case["sweeps"], case["n"] * case["per_doc"], 8)
    if kind == "solve":
        n = case["n"]
        return _solve_work(n, p, r, case["s"], case["sweeps"], n * p, 2 if case["storage"] == "resident16" else 4)
    if kind == "products":
        n = case["n"]
        size = {"f32": 4, "fp16": 2, "fp8": 1}[case["storage"]]
        return {"bytes": size * n * p + 4.0 * r * (2 * p + n), "flops": 4.0 * n * p * r}
    if kind == "xstep":
        return {"bytes": 4.0 * r * (2 * p) + 20.0 * r, "flops": 4.0 * r * p}
    columns = min(p, r * case["s"])
    return {"bytes": 4.0 * case["n"] * columns + 4.0 * r * p + 16.0 * r, "flops": 2.0 * case["n"] * r * case["s"]}


# ------------------------------------------------------------------ the same in 64 bits
def _keep_largest(V, s):
    W = torch.zeros_like(V)
    at = V.abs().topk(min(s, V.shape[1]), dim=1).indices
    return W.scatter_(1, at, V.gather(1, at))


def _soft(V, t):
    return torch.sign(V) * (V.abs() - t).clamp_(min=0.0)


def _lambda(V, s):
    """The root of s ||V_lambda||_2^2 = ||V_lambda||_1^2 (0 where the L1 ball does not bind)."""
    a = V.abs().sort(dim=1, descending=True).values
    S1, S2 = a.cumsum(1), (a * a).cumsum(1)
    k = torch.arange(1, a.shape[1] + 1, dtype=a.dtype, device=a.device)
    lam = (S1 - (s * (k * S2 - S1 * S1) / (k - s)).clamp(min=0.0).sqrt()) / k
    below = torch.cat([a[:, 1:], torch.zeros_like(a[:, :1])], 1)
    right = (k > s) & (lam >= below) & (lam < a)      # the piece with k active entries
    at = right.int().argmax(1, keepdim=True)
    lam = lam.gather(1, at)
    free = s * S2[:, -1:] >= S1[:, -1:] ** 2
    return torch.where(free | ~right.any(1, keepdim=True), torch.zeros_like(lam), lam)


def _operator(V, form, s, calibrate, thr):
    """(W, threshold): the x-step's result before it is normalised."""
    if form <= 2:
        return _keep_largest(V, s), None
    if form <= 4:
        thr = _lambda(V, float(s))
        return _soft(V, thr), thr
    if calibrate:
        thr = V.abs().topk(s + 1, dim=1).values[:, -1:]
    return (torch.where(V.abs() > thr, V, torch.zeros_like(V)) if form <= 6 else _soft(V, thr)), thr


def _y(U, form):
    return torch.where(U >= 0, 1.0, -1.0).to(U.dtype) if form % 2 == 0 else U / U.norm(dim=1, keepdim=True)


def _times(X, M):
    """X M^T for a dense or a sparse M."""
    return (M @ X.T).T.contiguous() if M.layout != torch.strided else X @ M.T


def _exact_solve(A, At, X0, form, s, calib, sweeps):
    X = X0.double()
    X = X / X.norm(dim=1, keepdim=True)
    thr = None
    for k in range(1, sweeps + 1):
        V = _times(_y(_times(X, A), form), At)
        W, thr = _operator(V, form, s, k <= calib, thr)
        X = W / W.norm(dim=1, keepdim=True)
    U = _times(X, A)
    l1, l2 = U.abs().sum(1), U.norm(dim=1)
    ev = l1 if form % 2 == 0 else l2 * l2
    f = l1 if form % 2 == 0 else l2
    if form in (5, 6):
        f = f * f - thr[:, 0] ** 2 * (X != 0).sum(1)
    elif form >= 7:
        f = f - thr[:, 0] * X.abs().sum(1)
    best = int((ev if form >= 5 else f).argmax())
    x = X[best]
    return _component({"objective": float(f[best]), "explained_variance": float(ev[best]), "x": x.cpu().numpy(),
                       "y": _y(U[best:best + 1], form)[0].cpu().numpy(), "nnz": int((x != 0).sum())})


def exact(case, seed):
    kind = case["kind"]
    if kind == "group":
        out = []
        for i, (n, p, form, s) in enumerate(_group_sizes(case)):
            A = _matrix("spiked", n, p, seed + 7919 * i, 3, 20).double()
            out.append(_exact_solve(A, A.T, _starts(p, case["r"], seed + 7919 * i), form, s, 5, case["sweeps"]))
        return out
    p, r = case["p"], case["r"]
    form = case["form"]
    if kind == "corpus":
        indptr, col, val = _corpus(case, seed)
        A = torch.sparse_csr_tensor(indptr, col.long(), val.double(), (case["n"], p))
        At = A.to_sparse_coo().t().coalesce().to_sparse_csr()
        return _exact_solve(A, At, _starts(p, r, seed), form, case["s"], case["calib"], case["sweeps"])
    if kind == "solve":
        A = _matrix(case["data"], case["n"], p, seed).double()
        return _exact_solve(A, A.T, _starts(p, r, seed), form, case["s"], case["calib"], case["sweeps"])
    if kind == "products":
        A = _matrix(case["data"], case["n"], p, seed).double()
        X = _starts(p, r, seed)
        X /= X.norm(dim=1, keepdim=True)
        U = X.double() @ A.T
        return {"U": U, "V": _y(U, form) @ A}
    if kind == "xstep":
        V = _given_v(case, seed).double()
        W, thr = _operator(V, form, case["s"], True, None)
        nrm = W.norm(dim=1)
        F = nrm
        if form in (3, 4):
            F = nrm + thr[:, 0] * math.sqrt(case["s"])
        elif form in (5, 6):
            F = nrm * nrm - thr[:, 0] ** 2 * (W != 0).sum(1)
        gamma = torch.zeros(r, device=V.device) if thr is None else thr[:, 0] ** 2 if form in (5, 6) else thr[:, 0]
        return {"X": W / nrm[:, None], "F": F, "nnz": (W != 0).sum(1), "thr": gamma}
    A, X = _matrix("gauss", case["n"], p, seed).double(), _sparse_x(case, seed).double()
    U = X @ A.T
    l1, l2 = U.abs().sum(1), U.norm(dim=1)
    f = l1 if form % 2 == 0 else l2
    if form in (5, 6):
        f = f * f - (X != 0).sum(1)
    elif form >= 7:
        f = f - X.abs().sum(1)
    return {"f": f, "ev": l1 if form % 2 == 0 else l2 * l2}
