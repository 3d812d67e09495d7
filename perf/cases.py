"""Measured cases of the library, each through the entry points a program calls.

``listed()`` names the standing cases, ``draw(rng)`` gives one more of the same
ranges, ``prepare(case, seed)`` makes what a program holds before the call (the
data set on the GPU, the run with its windows), ``run(state)`` makes one pass,
``work(case)`` counts the bytes and operations a pass cannot do without, and
``exact(case, seed)`` gives a pass's outputs in plain FP64 torch.

The data are isotropic Gaussian mixtures (unit variance, means ~ N(0, 4 I)) and
image-like rows (values in [0, 1], about 80 % zeros), the generators of
``paper_2410_05902_gb300.inputs`` restated on the GPU; bandwidths follow the
median heuristic in closed form. A run starts from full windows (what a run
holds after its first few dozen iterations), put in place with ``set_state``:
every center's blocks are rows of one mixture component, its weights follow the
beta rate, and its norm is w' K w in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_05902_gb300 import kkm as K
from paper_2410_05902_gb300.autograd import objective
from paper_2410_05902_gb300.group import Group
from paper_2410_05902_gb300.kkm import KKM, Lloyd

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # PenDigits/Letters scale: a batch of host indices in, assignments out, 16
        # iterations a call. Launches and latency are all there is.
        dict(name="host_steps_small", kind="host_steps", data="mixture", n=2000, d=16, c=10, k=10, b=256, tau=200,
             kernel="gaussian", precision="tf32", iters=16),
        # The headline workload's iteration loop with the built-in sampler, then
        # held-out points scored against the centers it left.
        dict(name="steps_headline", kind="steps", data="mixture", n=1_000_000, d=128, c=100, k=100, b=4096, tau=200,
             kernel="gaussian", precision="bf16", iters=16, queries=1024),
        # One iteration on MNIST-shaped data with the batch and the outputs on the device.
        dict(name="step_image", kind="step", data="image", n=70_000, d=784, c=10, k=10, b=1024, tau=200,
             kernel="gaussian", precision="bf16"),
        # The split form and the Laplacian kernel at ragged sizes.
        dict(name="step_laplacian_split", kind="step", data="mixture", n=200_000, d=61, c=37, k=37, b=1500, tau=150,
             kernel="laplacian", precision="bf16x3"),
        # FP32 products, for callers who want no tensor-core rounding.
        dict(name="step_fp32", kind="step", data="mixture", n=200_000, d=64, c=50, k=50, b=2048, tau=200,
             kernel="gaussian", precision="fp32"),
        # A sweep over k and the bandwidth, its runs stepped together and checked every few iterations.
        dict(name="sweep_8_runs", kind="sweep", data="mixture", runs=8, iters=4, queries=256, shapes=777),
        # Every point of a data set assigned, and the objective over it.
        dict(name="score_dataset", kind="score", data="mixture", n=100_000, d=256, c=64, k=64, b=2048, tau=200,
             kernel="gaussian", precision="tf32"),
        # Kernel k-means++ seeding of a run.
        dict(name="seeding", kind="seeding", data="mixture", n=200_000, d=64, c=50, k=50, kernel="gaussian"),
        # One full-batch iteration at MNIST's shape (the baseline the method is compared with).
        dict(name="lloyd_image", kind="lloyd", data="image", n=70_000, d=784, c=10, k=10, kernel="gaussian",
             precision="bf16x3"),
        # A training step of an encoder against fixed centers: objective, gradient of the rows and of the bandwidth.
        dict(name="gradient", kind="gradient", data="mixture", n=200_000, d=64, c=50, k=50, b=2048, tau=200,
             kernel="gaussian", precision="bf16", m=2048),
        # A serving process that scores a few queries against centers it holds itself.
        dict(name="serve_queries", kind="serve", data="mixture", d=64, c=50, k=50, tau=200, m=64,
             kernel="gaussian"),
        # Two iterations of the untruncated table form at MNIST's shape.
        dict(name="table_image", kind="table", data="image", n=70_000, d=784, c=10, k=10, b=1024,
             kernel="gaussian", precision="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _kernel(rng):
    return rng.choice(["gaussian"] * 6 + ["laplacian"] * 2 + ["linear", "poly"])


def draw(rng):
    kind = rng.choice(["host_steps", "steps", "step", "step", "step", "sweep", "score", "seeding", "lloyd",
                       "gradient", "serve", "table"])
    if kind == "sweep":
        return dict(kind=kind, data="mixture", runs=rng.randint(2, 8), iters=rng.randint(1, 4),
                    queries=_log(rng, 64, 1024), shapes=rng.randint(1000, 999_999))
    d = rng.choice([_log(rng, 3, 784), _log(rng, 3, 784), 16, 64, 128, 256, 784])
    c = _log(rng, 2, 128)
    case = dict(kind=kind, data="image" if d >= 256 and rng.random() < 0.5 else "mixture", d=d, c=c,
                kernel=_kernel(rng), precision=rng.choice(["fp32", "bf16", "bf16", "bf16x3", "tf32", "tf32"]))
    if kind in ("seeding", "serve"):
        case.pop("precision")
    if kind == "serve":
        k = _log(rng, 2, 128)
        case.update(k=k, tau=_log(rng, 16, min(1000, 40_000 // k)), m=_log(rng, 1, 4096))
        return case
    n = _log(rng, 2000, min(1_000_000, 100_000_000 // d))
    case.update(n=n, k=min(n, _log(rng, 2, 128)))
    if kind == "seeding":
        case["n"] = min(n, 12_000_000 // (d * case["k"]) * 50 + 2000, 200_000)
        return case
    if kind == "lloyd":
        case["n"] = min(n, 70_000 if case["precision"] != "fp32" else 12_000)
        if case["kernel"] == "poly":   # a degree-2 mean of 70000 rows: keep its sums in FP32 range
            case["kernel"] = "gaussian"
        return case
    case["b"] = _log(rng, 64, 4096)
    if kind == "table":
        case["n"] = min(n, 70_000)
        if case["precision"] == "fp32":
            case["b"] = min(case["b"], 1024)
        return case
    case["tau"] = _log(rng, 16, min(1000, 40_000 // case["k"]))
    if kind == "gradient":
        case["kernel"] = rng.choice(["gaussian", "gaussian", "laplacian"])
        case["m"] = _log(rng, 64, 4096)
    if kind == "score":
        case["n"] = min(n, 100_000 if case["precision"] != "fp32" else 20_000)
    if kind in ("steps", "host_steps"):
        case["iters"] = rng.choice([1, 5, 16, 16, 21, 32])
        if kind == "steps":
            case["queries"] = _log(rng, 64, 2048)
    return case


# ------------------------------------------------------------ data and windows
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _data(case, seed):
    """(X float32 (n, d), rows i, i + c, i + 2c, ... of one component)."""
    n, d, c = case["n"], case["d"], case["c"]
    g = _gen(seed)
    lab = torch.arange(n, device=DEV) % c
    if case["data"] == "mixture":
        X = torch.randn(n, d, generator=g, device=DEV)
        means = 2.0 * torch.randn(c, d, generator=g, device=DEV)
        for s in range(0, n, 131072):
            X[s:s + 131072] += means[lab[s:s + 131072]]
        return X
    masks = torch.rand(c, d, generator=g, device=DEV) < 0.25
    X = torch.empty(n, d, device=DEV)
    for s in range(0, n, 16384):
        e = min(n, s + 16384)
        v = torch.rand(3, e - s, d, generator=g, device=DEV).median(0).values   # Beta(2, 2)
        keep = masks[lab[s:e]] & (torch.rand(e - s, d, generator=g, device=DEV) < 0.8)
        X[s:e] = torch.where(keep, v, torch.zeros_like(v))
    return X


def _kernel_args(case, X):
    """(kernel, param, coef0, degree): the bandwidth from the mean squared pair distance 2 tr Cov(X)."""
    name = case["kernel"]
    sub = X[:8192].double()
    sigma2 = 2.0 * float(sub.var(0).sum())
    if name == "gaussian":
        return name, 2.0 * sigma2, 0.0, 2
    if name == "laplacian":
        return name, math.sqrt(sigma2), 0.0, 2
    return name, 1.0, (float(sub.square().sum(1).mean()) if name == "poly" else 0.0), 2


def _pair(kern, A, B):
    """Kernel matrix in the dtype of A and B."""
    name, param, coef0, degree = kern
    G = A @ B.T
    if name in ("gaussian", "laplacian"):
        d2 = ((A * A).sum(1)[:, None] + (B * B).sum(1)[None, :] - 2.0 * G).clamp_min(0.0)
        return torch.exp(-d2 / param) if name == "gaussian" else torch.exp(-torch.sqrt(d2) / param)
    return G if name == "linear" else (G + coef0) ** degree


def _self(kern, A):
    name, _, coef0, degree = kern
    if name in ("gaussian", "laplacian"):
        return torch.ones(A.shape[0], dtype=A.dtype, device=A.device)
    s = (A * A).sum(1)
    return s if name == "linear" else (s + coef0) ** degree


def _windows(case, X, kern, seed):
    """Full windows as set_state takes them: newest blocks of about b / k rows until they hold tau."""
    n, k, b, tau, c = case["n"], case["k"], case["b"], case["tau"], case["c"]
    rng = np.random.default_rng([seed, 1])
    mean = max(1.0, b / k)
    rows, idx, w, nblk, cnts, cn = [], [], [], [], [], []
    for j in range(k):
        counts, total = [], 0
        while total < tau:                      # newest to oldest
            m = int(min(b, max(1, rng.poisson(mean))))
            counts.append(m)
            total += m
        f, wj = 1.0, []
        for m in counts:
            a = math.sqrt(m / b)
            wj.append(np.full(m, f * a / m))
            f *= 1.0 - a
        q = j % min(c, n)
        idx.append(q + c * rng.integers(0, (n - q - 1) // c + 1, size=total))
        w.append(np.concatenate(wj[::-1]))
        rows.append(total)
        nblk.append(len(counts))
        cnts.append(np.asarray(counts[::-1], np.int32))
    it = max(nblk) + 1
    for j in range(k):
        Y = X[torch.from_numpy(idx[j]).to(DEV)].double()
        wt = torch.from_numpy(w[j]).to(DEV)
        cn.append(wt @ _pair(kern, Y, Y) @ wt)
    return dict(iteration=it, rows_per_center=np.asarray(rows, np.int32), row_idx=np.concatenate(idx),
                row_w=np.concatenate(w), blocks_per_center=np.asarray(nblk, np.int32),
                block_iter=np.concatenate([np.arange(it - m, it) for m in nblk]), block_count=np.concatenate(cnts),
                c1_kept=np.zeros(k, np.uint8), cnorm=torch.stack(cn).cpu().numpy())


def _inner(kern, A, Y, w, off):
    """<phi(a), C_j> in FP64 for every row a and center j."""
    out = torch.empty(A.shape[0], len(off) - 1, dtype=torch.float64, device=DEV)
    j = 0
    while j < len(off) - 1:                     # a few thousand support rows at a time
        e = j + 1
        while e < len(off) - 1 and off[e + 1] - off[j] <= 8192:
            e += 1
        sl = slice(off[j], off[e])
        P = _pair(kern, A, Y[sl]) * w[sl]
        for q in range(j, e):
            out[:, q] = P[:, off[q] - off[j]:off[q + 1] - off[j]].sum(1)
        j = e
    return out


def _state_distances(kern, X, st, A):
    off = np.concatenate([[0], np.cumsum(st["rows_per_center"])]).tolist()
    Y = X[torch.from_numpy(st["row_idx"]).to(DEV)].double()
    w = torch.from_numpy(st["row_w"]).to(DEV)
    cn = torch.from_numpy(st["cnorm"]).to(DEV)
    out = [(_self(kern, A[s:s + 4096].double())[:, None] - 2.0 * _inner(kern, A[s:s + 4096].double(), Y, w, off)
            + cn[None, :]) for s in range(0, A.shape[0], 4096)]
    return torch.cat(out)


def _make_run(case, seed):
    """(X, kernel arguments, window state, run) of a windows-form case."""
    X = _data(case, seed)
    kern = _kernel_args(case, X)
    st = _windows(case, X, kern, seed)
    run = KKM(X, case["k"], case["b"], kernel=kern[0], param=kern[1], coef0=kern[2], degree=kern[3],
              tau=case["tau"], precision=case["precision"], seed=seed,
              init_idx=np.arange(case["k"], dtype=np.int64))
    run.set_state(st)
    return X, kern, st, run


def _queries(case, X, m, seed):
    """m held-out points: the mean of two rows of one component plus noise of its own."""
    g = _gen(seed * 7 + 3)
    n, c = X.shape[0], case["c"]
    q = torch.arange(m, device=DEV) % min(c, n)
    span = (n - q - 1) // c + 1
    i = q + c * (torch.rand(m, generator=g, device=DEV) * span).long()
    j = q + c * (torch.rand(m, generator=g, device=DEV) * span).long()
    return (0.5 * (X[i] + X[j]) + 0.1 * torch.randn(m, X.shape[1], generator=g, device=DEV)).contiguous()


def _batches(n, b, iters, seed):
    return np.random.default_rng([seed, 2]).integers(0, n, size=(iters, b)).astype(np.int32)


def _sweep_cases(case):
    """The runs of a sweep: the batched workload's ranges, every one with its own k, d and batch size."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["runs"]):
        k = int(rng.integers(5, 101))
        out.append(dict(data="mixture", n=int(rng.integers(5000, 50_001)), d=int(rng.choice([16, 64, 256])), c=k, k=k,
                        b=int(rng.choice([256, 512, 1024, 2048])), tau=200, kernel="gaussian", precision="tf32"))
    return out


def _serve_inputs(case, seed):
    """Support rows, weights, offsets, norms and queries that a serving process holds."""
    big = dict(case, n=max(2000, 40 * case["c"]), b=max(64, 16 * case["k"]))
    X = _data(big, seed)
    kern = _kernel_args(case, X)
    st = _windows(big, X, kern, seed)
    Y = X[torch.from_numpy(st["row_idx"]).to(DEV)].contiguous()
    off = np.concatenate([[0], np.cumsum(st["rows_per_center"])]).astype(np.int32)
    return dict(kern=kern, Y=Y, w=torch.from_numpy(st["row_w"].astype(np.float32)).to(DEV),
                off=torch.from_numpy(off).to(DEV), cnorm=torch.from_numpy(st["cnorm"]).to(DEV),
                Q=_queries(case, X, case["m"], seed))


def _assignments(case, m):
    """Query row i belongs to component i mod c, held by center i mod c (mod k)."""
    return (torch.arange(m, device=DEV) % case["c"] % case["k"]).to(torch.int32)


# ------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, kind=kind)
    if kind == "sweep":
        runs, qs = [], []
        for i, sub in enumerate(_sweep_cases(case)):
            X, _, _, run = _make_run(sub, seed * 100 + i)
            runs.append(run)
            qs.append(_queries(sub, X, case["queries"], seed * 100 + i))
        torch.cuda.synchronize()
        return dict(s, runs=runs, group=Group(runs), Q=qs)
    if kind == "serve":
        s.update(_serve_inputs(case, seed))
        name, param, coef0, degree = s["kern"]
        s["kernel"] = K.kkm_kernel(K.KERNELS[name], param, coef0, degree)
        s["dist"] = torch.empty(case["m"], case["k"], device=DEV)
        s["assign"] = torch.empty(case["m"], dtype=torch.int32, device=DEV)
        return s
    if kind in ("seeding", "lloyd", "table"):
        X = _data(case, seed)
        name, param, coef0, degree = _kernel_args(case, X)
        s.update(X=X, kw=dict(kernel=name, param=param, coef0=coef0, degree=degree), seed=seed)
        init = np.arange(case["k"], dtype=np.int64)
        if kind == "lloyd":
            s["run"] = Lloyd(X, case["k"], init, precision=case["precision"], **s["kw"])
        if kind == "table":
            s["run"] = KKM(X, case["k"], case["b"], tau=0, algo="table", precision=case["precision"], seed=seed,
                           init_idx=init, **s["kw"])
            s["batches"] = torch.from_numpy(_batches(case["n"], case["b"], 2, seed)).to(DEV)
            s["dist"] = torch.empty(case["b"], case["k"], device=DEV)
            s["assign"] = torch.empty(case["b"], dtype=torch.int32, device=DEV)
        return s
    X, kern, _, run = _make_run(case, seed)
    s.update(X=X, run=run)
    if kind in ("steps", "host_steps", "step"):
        run.graph(True)
    if kind == "host_steps":
        s["batches"] = _batches(case["n"], case["b"], case["iters"], seed)
    if kind == "steps":
        s["Q"] = _queries(case, X, case["queries"], seed)
    if kind == "step":
        s["batch"] = torch.from_numpy(_batches(case["n"], case["b"], 1, seed)[0]).to(DEV)
        s["dist"] = torch.empty(case["b"], case["k"], device=DEV)
        s["assign"] = torch.empty(case["b"], dtype=torch.int32, device=DEV)
    if kind == "gradient":
        # the module's own parameters are FP32: the rows it encodes and the log bandwidth
        s["Q"] = _queries(case, X, case["m"], seed)
        param = kern[1]
        s["ls"] = torch.tensor(0.5 * math.log(param / 2.0) if kern[0] == "gaussian" else math.log(param),
                               dtype=torch.float32, device=DEV)
        s["assign"] = _assignments(case, case["m"])
    return s


# ----------------------------------------------------------------------- run
def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "host_steps":
        assign, f_b = s["run"].steps_host(s["batches"])
        return assign, f_b.astype(np.float32)   # a mean of FP32 distances
    if kind == "steps":
        s["run"].steps(case["iters"])
        return s["run"].assign(s["Q"], want_dist=True)
    if kind == "step":
        s["run"].step(s["batch"], None, s["assign"], s["dist"], None)
        return s["assign"], s["dist"]
    if kind == "sweep":
        for _ in range(case["iters"]):
            s["group"].step()
        s["group"].sync()
        return [r.assign(q, want_dist=True)[2] for r, q in zip(s["runs"], s["Q"])]
    if kind == "score":
        assign, mind, _ = s["run"].assign(s["X"])
        return assign, mind, s["run"].objective()
    if kind == "seeding":
        return K.kmeanspp(s["X"], case["k"], seed=s["seed"], **s["kw"])
    if kind == "lloyd":
        s["run"].iterate(1)
        return s["run"].assignments()
    if kind == "gradient":
        Q = s["Q"].detach().requires_grad_(True)
        ls = s["ls"].detach().requires_grad_(True)
        loss = objective(s["run"], Q, ls.double(), s["assign"]).float()
        loss.backward()
        return loss.detach(), Q.grad, ls.grad
    if kind == "serve":
        Q, Y = s["Q"], s["Y"]
        K.kkm_distances_noalloc(Q.data_ptr(), Q.shape[0], Q.stride(0), Q.shape[1], Y.data_ptr(), Y.shape[0],
                                Y.stride(0), s["w"].data_ptr(), s["off"].data_ptr(), s["cnorm"].data_ptr(), case["k"],
                                s["kernel"], s["dist"].data_ptr(), s["assign"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        return s["assign"], s["dist"]
    # table: two iterations, the second on centers the first has moved
    for i in range(2):
        s["run"].step(s["batches"][i], None, s["assign"], s["dist"], None)
    return s["assign"], s["dist"]


# ---------------------------------------------------------------------- work
def _esize(precision):
    return {"fp32": 4, "tf32": 4, "bf16": 2, "bf16x3": 4}[precision]


def _step_work(c):
    S = c["k"] * c["tau"] + c["b"] / 2.0
    return dict(bytes=4.0 * c["b"] * c["d"] + S * c["d"] * _esize(c["precision"]) + 4.0 * c["b"] * c["k"],
                flops=2.0 * c["b"] * S * c["d"])


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        w = [_step_work(c) for c in _sweep_cases(case)]
        return {q: case["iters"] * sum(x[q] for x in w) for q in ("bytes", "flops")}
    if kind in ("host_steps", "steps", "step"):
        w = _step_work(case)
        return {q: case.get("iters", 1) * w[q] for q in w}
    k, d = case["k"], case["d"]
    if kind == "serve":
        S, m = k * case["tau"], case["m"]
        return dict(bytes=4.0 * (S * (d + 1) + m * (d + k + 1)), flops=2.0 * m * S * d)
    n = case["n"]
    if kind == "seeding":       # every draw reads the points and their D^2 once
        return dict(bytes=(k - 1.0) * n * (4.0 * d + 16.0), flops=3.0 * (k - 1) * n * d)
    if kind == "lloyd":
        return dict(bytes=4.0 * n * d + 8.0 * n, flops=2.0 * n * n * d)
    if kind == "table":         # the table read and written, and X against the batch
        return dict(bytes=2.0 * (8.0 * n * k + n * d * _esize(case["precision"])), flops=4.0 * n * case["b"] * d)
    S = k * case["tau"]
    if kind == "score":         # the points go through twice: the assignment and the objective
        return dict(bytes=2.0 * (4.0 * n * d) + 8.0 * n, flops=4.0 * n * S * d)
    # gradient: each row against its own center's window, the window's pairs once
    m, t = case["m"], case["tau"]
    return dict(bytes=4.0 * (S * d + 2.0 * m * d), flops=2.0 * d * (3.0 * m * t + k * t * t / 2.0))


# --------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        X = _data(case, seed)
        kern = _kernel_args(case, X)
        st = _windows(case, X, kern, seed)
        B = torch.from_numpy(_batches(case["n"], case["b"], 1, seed)[0].astype(np.int64)).to(DEV)
        return None, _state_distances(kern, X, st, X[B])
    if kind == "score" and case["n"] * case["k"] * case["tau"] * case["d"] < 2e12:
        X = _data(case, seed)
        kern = _kernel_args(case, X)
        st = _windows(case, X, kern, seed)
        mind = torch.cat([_state_distances(kern, X, st, X[s:s + 4096]).min(1).values
                          for s in range(0, case["n"], 4096)])
        return None, mind, float(mind.mean())
    if kind == "serve":
        s = _serve_inputs(case, seed)
        off, Q = s["off"].cpu().tolist(), s["Q"].double()
        inner = _inner(s["kern"], Q, s["Y"].double(), s["w"].double(), off)
        return None, _self(s["kern"], Q)[:, None] - 2.0 * inner + s["cnorm"][None, :]
    if kind == "gradient":
        X = _data(case, seed)
        kern = _kernel_args(case, X)
        st = _windows(case, X, kern, seed)
        Q = _queries(case, X, case["m"], seed).double().requires_grad_(True)
        ls = 0.5 * math.log(kern[1] / 2.0) if kern[0] == "gaussian" else math.log(kern[1])
        ls = torch.tensor(np.float32(ls), dtype=torch.float64, device=DEV).requires_grad_(True)
        a = _assignments(case, case["m"]).cpu().numpy()
        off = np.concatenate([[0], np.cumsum(st["rows_per_center"])])
        total = 0.0
        for j in range(case["k"]):
            rows = np.flatnonzero(a == j)
            if not len(rows):
                continue
            Y = X[torch.from_numpy(st["row_idx"][off[j]:off[j + 1]]).to(DEV)].double()
            w = torch.from_numpy(st["row_w"][off[j]:off[j + 1]]).to(DEV)
            q = Q[torch.from_numpy(rows).to(DEV)]

            def val(A):
                d2 = (A[:, None, :] - Y[None, :, :]).square().sum(2)
                if kern[0] == "gaussian":
                    return torch.exp(-d2 / (2.0 * torch.exp(2.0 * ls)))
                return torch.exp(-torch.where(d2 > 0, d2, torch.ones_like(d2)).sqrt() * (d2 > 0) / torch.exp(ls))
            norm = w @ torch.cat([val(Y[s:s + 64]) for s in range(0, Y.shape[0], 64)]) @ w
            part = sum((1.0 - 2.0 * val(q[s:s + 64]) @ w + norm).sum() for s in range(0, len(rows), 64))
            (part / case["m"]).backward()
            total += float(part.detach()) / case["m"]
        return torch.tensor(total, dtype=torch.float64), Q.grad, ls.grad
    if kind == "table":
        X = _data(case, seed)
        kern = _kernel_args(case, X)
        k, b = case["k"], case["b"]
        B = torch.from_numpy(_batches(case["n"], b, 2, seed).astype(np.int64)).to(DEV)
        C, B1, B2 = X[:k].double(), X[B[0]].double(), X[B[1]].double()
        cn = _self(kern, C)
        d1 = _self(kern, B1)[:, None] - 2.0 * _pair(kern, B1, C) + cn[None, :]
        a = d1.argmin(1)
        K1, K2, P, P2 = _pair(kern, B1, C), _pair(kern, B2, C), _pair(kern, B1, B1), _pair(kern, B2, B1)
        for j in range(k):
            at = (a == j).nonzero().flatten()
            if not len(at):
                continue
            al = math.sqrt(len(at) / b)
            cn[j] = (1 - al) ** 2 * cn[j] + 2 * al * (1 - al) * K1[at, j].mean() + al * al * P[at][:, at].mean()
            K2[:, j] = (1 - al) * K2[:, j] + al * P2[:, at].mean(1)
        return None, _self(kern, B2)[:, None] - 2.0 * K2 + cn[None, :]
    return None     # free-running iterations, whole numbers, or n^2 work
