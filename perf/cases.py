"""The work that this framework is timed on, as a user's program has it done.

A case names one call of the public interface and the matrix it is made on. The matrices are drawn on the GPU from
the seed alone, in the shapes that the framework is written for: a small banded system, a Holstein-Hubbard-like
matrix (seven diagonals and symmetric off-band entries, 15 a row), the 27-point stencil with a tenth of its couplings
dropped (symmetric, positive definite), dense 4x4 blocks near the diagonal (144 a row) and power-law (Zipf) row
lengths. `exact` computes the same results in 64 bits with torch alone.
"""
import math

import numpy as np
import torch

DEV = "cuda"
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}
VECTOR = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32}
DIAGONALS = (1, 64, 4096)
ZIPF_MAX = 512
# the learned tuner's network: 15 inputs, two hidden layers of 64, one output
IN, HID = 15, 64


def listed():
    return [
        # one product on a small system that fits in L2: a call's latency is all there is
        {"name": "spmv banded 20k f64", "call": "spmv", "matrix": "banded", "n": 20000, "dtype": "f64", "permuted": False},
        # the product on the largest physics matrix, vectors in the caller's own numbering
        {"name": "spmv hmep 6.2M f64", "call": "spmv", "matrix": "hmep", "n": 6200000, "dtype": "f64", "permuted": False},
        # an inner solver step's product: permuted basis, values at reduced storage precision
        {"name": "spmv stencil 4.5M bf16", "call": "spmv", "matrix": "stencil", "n": 165 ** 3, "dtype": "bf16", "permuted": True},
        # row lengths from 1 to several hundred, as of an algebraic multigrid or a graph
        {"name": "spmv zipf 1M f64", "call": "spmv", "matrix": "zipf", "n": 1000003, "dtype": "f64", "s": 2.0, "permuted": False},
        # ELLPACK-R, the simpler format, on an ordinary matrix of an odd size in single precision
        {"name": "ellr hmep 300k f32", "call": "ellr", "matrix": "hmep", "n": 300001, "dtype": "f32"},
        # block solvers and eigensolvers: one matrix of dense blocks and 32 vectors
        {"name": "spmm blocks 280k f32 k32", "call": "spmm", "matrix": "blocks", "n": 280000, "dtype": "f32", "k": 32},
        # the same with few vectors on a stencil in double precision
        {"name": "spmm stencil 512k f64 k8", "call": "spmm", "matrix": "stencil", "n": 80 ** 3, "dtype": "f64", "k": 8},
        # many uneven systems at once (subdomains, ensembles) in one launch
        {"name": "batch 64 zipf f64", "call": "batch", "count": 64, "lo": 10000, "hi": 500000, "dtype": "f64", "s": 2.0},
        # a small linear system solved to full precision, single-precision inner steps: launches and latency
        {"name": "cg stencil 20k f32", "call": "cg", "n": 27 ** 3, "dtype": "f32", "outer": 6, "inner": 50},
        # a large one, solved in double precision throughout
        {"name": "cg stencil 2M f64", "call": "cg", "n": 126 ** 3, "dtype": "f64", "outer": 4, "inner": 50},
        # a short Lanczos run that keeps its basis for the Ritz vectors
        {"name": "lanczos stencil 1M f32", "call": "lanczos", "n": 100 ** 3, "dtype": "f32", "steps": 24},
        # fitting the tuner's cost model to one machine's timings (600 matrices, 36 candidates each)
        {"name": "train tuner 21600", "call": "train", "samples": 21600, "batch": 1024, "epochs": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["spmv", "spmv", "spmv", "ellr", "spmm", "spmm", "batch", "cg", "cg", "lanczos", "train"])
    dtype = rng.choice(["f64", "f32", "bf16"])
    if call in ("spmv", "ellr", "spmm"):
        matrix = rng.choice(["banded", "hmep", "stencil", "blocks"] + (["zipf"] if call != "ellr" else []))
        most = {"spmv": 4000000, "ellr": 1500000, "spmm": 400000}[call]
        n = _log(rng, 2000, most // 6 if matrix == "blocks" else most)
        c = {"call": call, "matrix": matrix, "n": _size(matrix, n), "dtype": dtype}
        if matrix == "zipf":
            c["s"] = round(rng.uniform(1.6, 3.0), 2)
        if call == "spmv":
            c["permuted"] = rng.random() < 0.4
        if call == "spmm":
            c["k"] = rng.choice([2, 4, 6, 8, 16, 24, 32, 64] if dtype == "f64" else [4, 8, 12, 16, 24, 32, 64, 128])
        return c
    if call == "batch":
        lo = _log(rng, 1000, 20000)
        return {"call": call, "count": rng.randint(3, 64), "lo": lo, "hi": lo * rng.randint(2, 25), "dtype": dtype,
                "s": round(rng.uniform(1.6, 3.0), 2)}
    if call == "cg":
        g = _log(rng, 10, 110)
        return {"call": call, "n": g ** 3, "dtype": dtype, "outer": {"f64": 4, "f32": 6, "bf16": 8}[dtype],
                "inner": rng.randint(40, 60)}
    if call == "lanczos":
        g = _log(rng, 12, 110)
        return {"call": call, "n": g ** 3, "dtype": dtype, "steps": rng.randint(12, 24)}
    return {"call": call, "samples": _log(rng, 500, 40000), "batch": rng.choice([256, 1000, 1024, 4096]),
            "epochs": rng.randint(1, 3)}


def _size(matrix, n):
    if matrix == "stencil":
        return max(10, round(n ** (1 / 3))) ** 3
    return n // 4 * 4 if matrix == "blocks" else n


# ---------------------------------------------------------------------------------------------------- matrices (CRS)


def _generator(seed, more=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + more) % (1 << 60))


def _values(n, g):
    """Uniform in [-1, 1), exact in 32 bits."""
    return (torch.rand(n, generator=g, device=DEV) * 2 - 1).double()


def _crs(n, keys, g):
    """CRS arrays of the pattern that the keys row * n + column give, columns ascending, repeats dropped."""
    keys = torch.unique(keys)
    ptr = torch.searchsorted(keys, torch.arange(n + 1, device=DEV, dtype=torch.int64) * n)
    return n, ptr, (keys % n).int(), _values(keys.numel(), g)


def _pairs(counts):
    """The row of each entry, for rows of these lengths."""
    return torch.repeat_interleave(torch.arange(counts.numel(), device=DEV), counts)


def _draws(n, rows, half, g):
    """One column for each of `rows`, uniform within `half` of the row."""
    lo, hi = (rows - half).clamp_(min=0), (rows + half).clamp_(max=n - 1)
    u = torch.rand(rows.numel(), generator=g, device=DEV, dtype=torch.float64)
    return torch.minimum(lo + (u * (hi - lo + 1)).long(), hi)


def _banded(n, g):
    rows = _pairs(torch.randint(4, 40, (n,), generator=g, device=DEV))
    i = torch.arange(n, device=DEV)
    return _crs(n, torch.cat([i * n + i, rows * n + _draws(n, rows, max(40, n // 10), g)]), g)


def _hmep(n, g):
    i = torch.arange(n, device=DEV)
    rows = _pairs(torch.randint(1, 8, (n,), generator=g, device=DEV))
    cols = _draws(n, rows, n // 8, g)
    keys = [i * (n + 1), rows * n + cols, cols * n + rows]
    for d in DIAGONALS:
        keys += [i[d:] * (n + 1) - d, i[: max(0, n - d)] * (n + 1) + d]
    return _crs(n, torch.cat(keys), g)


def _blocks(n, g):
    nb = n // 4
    rows = _pairs(torch.full((nb,), 36, device=DEV))
    block = torch.unique(rows * nb + _draws(nb, rows, max(40, nb // 20), g))
    r, c = torch.div(block, nb, rounding_mode="floor"), block % nb
    four = torch.arange(4, device=DEV)
    return _crs(n, ((r[:, None, None] * 4 + four[:, None]) * n + c[:, None, None] * 4 + four).reshape(-1), g)


def _zipf_weights(s):
    w = np.arange(1, ZIPF_MAX + 1, dtype=np.float64) ** -s
    return w / w.sum()


def _zipf(n, s, g):
    edges = torch.from_numpy(np.cumsum(_zipf_weights(s))).to(DEV)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    lengths = (torch.searchsorted(edges, u) + 1).clamp_(max=min(ZIPF_MAX, n))
    rows = _pairs(lengths)
    return _crs(n, rows * n + torch.randint(0, n, (rows.numel(),), generator=g, device=DEV), g)


def _stencil(n, g):
    m = round(n ** (1 / 3))
    i = torch.arange(n, device=DEV)
    z, y, x = torch.div(i, m * m, rounding_mode="floor"), torch.div(i, m, rounding_mode="floor") % m, i % m
    keys, vals = [], []
    total = torch.ones(n, dtype=torch.float64, device=DEV)
    for off in range(14, 27):  # the upper half of the 26 neighbours; each coupling is drawn once
        dz, dy, dx = off // 9 - 1, off // 3 % 3 - 1, off % 3 - 1
        inside = (z + dz >= 0) & (z + dz < m) & (y + dy >= 0) & (y + dy < m) & (x + dx >= 0) & (x + dx < m)
        a = i[inside & (torch.rand(n, generator=g, device=DEV) >= 0.1)]
        b = a + (dz * m + dy) * m + dx
        # multiples of 2^-12: their sums, the diagonal, are exact in any order and in 32 bits
        v = -torch.randint(1, 4096, (a.numel(),), generator=g, device=DEV).double() / 4096
        total.index_add_(0, a, -v)
        total.index_add_(0, b, -v)
        keys += [a * n + b, b * n + a]
        vals += [v.float(), v.float()]
    keys, at = torch.sort(torch.cat(keys + [i * (n + 1)]))
    val = torch.cat(vals + [total.float()])[at].double()
    ptr = torch.searchsorted(keys, torch.arange(n + 1, device=DEV, dtype=torch.int64) * n)
    return n, ptr, (keys % n).int(), val


def _matrix(case, seed):
    g, n = _generator(seed), case["n"]
    kind = case.get("matrix", "stencil")
    if kind == "zipf":
        return _zipf(n, case["s"], g)
    return {"banded": _banded, "hmep": _hmep, "blocks": _blocks, "stencil": _stencil}[kind](n, g)


def _vector(n, dtype, seed, k=None):
    g = _generator(seed, 7)
    x = torch.rand((n,) if k is None else (n, k), generator=g, device=DEV, dtype=VECTOR[dtype])
    return x * 2 - 1


def _batch_sizes(case):
    """Sizes spread evenly over the logarithm, the same for every seed."""
    lo, hi, m = math.log(case["lo"]), math.log(case["hi"]), case["count"]
    return [int(math.exp(lo + (hi - lo) * ((q * 0.618034) % 1.0))) for q in range(1, m + 1)]


def _samples(case, seed):
    """Features of matrices and candidates and the logarithm of their times: smooth, with noise, as timings are."""
    g, n = _generator(seed), case["samples"]
    X = torch.randn((n, IN), generator=g, device=DEV, dtype=torch.float64) * 1.5 + 2.0
    y = X[:, 1] + 0.3 * (X[:, 2] - X[:, 9]).abs() + 0.1 * X[:, 3] * X[:, 13]
    y = y + 0.05 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    return X.float().cpu().numpy(), y.float().cpu().numpy()


# ------------------------------------------------------------------------------------------------- prepare and run


def _device(crs, dtype, permuted=False):
    from paper_1112_5588_gb300 import pjds

    n, ptr, col, val = crs
    return pjds.pjds_create(n, n, ptr.cpu().numpy(), col.cpu().numpy(), val.cpu().numpy(), b=32, dtype=dtype,
                            permute_cols=permuted).to_device(DEV)


def prepare(case, seed):
    from paper_1112_5588_gb300 import batch, krylov, learned, pjds

    call, s = case["call"], {"case": case}
    if call == "train":
        s["X"], s["y"] = _samples(case, seed)
        s["model"] = bytes(learned.fit_scaling(learned.init(5), s["X"], s["y"]))
        return s
    dtype = case["dtype"]
    if call == "batch":
        mats, xs, ys = [], [], []
        for q, n in enumerate(_batch_sizes(case)):
            mats.append(_device(_zipf(n, case["s"], _generator(seed, 100 + q)), dtype))
            xs.append(_vector(n, dtype, seed * 64 + q))
            ys.append(torch.empty_like(xs[-1]))
        s["batch"], s["ys"] = batch.Batch(mats, xs, ys), ys
        return s
    crs, n = _matrix(case, seed), case["n"]
    if call == "ellr":
        s["A"] = pjds.ellr_create(n, n, crs[1].cpu().numpy(), crs[2].cpu().numpy(), crs[3].cpu().numpy(),
                                  dtype=dtype).to_device(DEV)
        s["x"] = _vector(n, dtype, seed)
        s["out"] = torch.empty_like(s["x"])
    elif call in ("spmv", "spmm"):
        s["A"] = _device(crs, dtype, case.get("permuted", False))
        s["x"] = _vector(n, dtype, seed, case.get("k"))
        s["out"] = torch.empty_like(s["x"])
        if case.get("permuted"):
            s["x"] = pjds.pjds_permute(s["A"], s["x"], torch.empty_like(s["x"]))
    elif call == "cg":
        s["A"] = _device(crs, "f64", True)
        s["low"] = _device(crs, dtype, True) if dtype != "f64" else None
        b = _vector(n, "f64", seed)
        s["b"] = pjds.pjds_permute(s["A"], b, torch.empty_like(b))
        need = krylov.cg_workspace_bytes(s["A"].n_rows, s["A"].n_pad, 0 if dtype == "f64" else 1)
        s["work"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    else:
        s["A"] = _device(crs, dtype, True)
        v = _vector(n, dtype, seed)
        s["v"] = pjds.pjds_permute(s["A"], v, torch.empty_like(v))
    return s


def run(state):
    from paper_1112_5588_gb300 import batch, krylov, learned, pjds

    case = state["case"]
    call = case["call"]
    if call == "spmv":
        return pjds.pjds_spmv(state["A"], state["x"], state["out"])
    if call == "ellr":
        return pjds.ellr_spmv(state["A"], state["x"], state["out"])
    if call == "spmm":
        return batch.spmm(state["A"], state["x"], state["out"])
    if call == "batch":
        state["batch"].run()
        return state["ys"]
    if call == "cg":
        x = torch.zeros_like(state["b"])
        r = krylov.cg_solve(state["A"], state["low"], state["b"], x, max_outer=case["outer"],
                            inner_iters=case["inner"], work=state["work"])
        return {"x": x, "steps": r["inner_total"]}
    if call == "lanczos":
        alpha, beta, basis = krylov.lanczos(state["A"], state["v"], case["steps"], keep_basis=True)
        return {"alpha": alpha, "beta": beta, "basis": basis}
    m = learned.Mlp.from_buffer_copy(state["model"])
    loss = learned.train(m, state["X"], state["y"], epochs=case["epochs"], batch=case["batch"], lr=2e-3, seed=1)
    return {"loss": loss, **{k: np.ctypeslib.as_array(getattr(m, k)).copy() for k in ("w1", "b1", "w2", "b2", "w3")},
            "b3": float(m.b3)}


# ------------------------------------------------------------------------------------------ work, tolerance, exact


def _row_length(case):
    kind = case.get("matrix", "stencil")
    if kind == "zipf":
        return float((np.arange(1, ZIPF_MAX + 1) * _zipf_weights(case["s"])).sum())
    return {"banded": 22.4, "hmep": 15.0, "blocks": 144.0 if case["n"] > 20000 else 125.0, "stencil": 24.0}[kind]


def work(case):
    call = case["call"]
    if call == "train":
        weights = IN * HID + HID * HID + HID
        steps = case["epochs"] * math.ceil(case["samples"] / case["batch"])
        # the samples are read once an epoch and the parameters and their two moments updated once a step
        return {"bytes": 4.0 * (case["samples"] * (IN + 1) * case["epochs"] + steps * 7 * weights),
                "flops": 6.0 * weights * case["samples"] * case["epochs"]}
    vb = VALUE_BYTES[case["dtype"]]
    xb = 8 if case["dtype"] == "f64" else 4
    if call == "batch":
        rows = float(sum(_batch_sizes(case)))
        nnz = rows * float((np.arange(1, ZIPF_MAX + 1) * _zipf_weights(case["s"])).sum())
        return {"bytes": nnz * (vb + 4) + rows * (2 * xb + 4), "flops": 2 * nnz}
    n = case["n"]
    nnz = n * _row_length(case)
    matrix = nnz * (vb + 4)
    if call in ("spmv", "ellr", "spmm"):
        k = case.get("k", 1)
        index = 0 if case.get("permuted") else 4 * n
        return {"bytes": matrix + 2.0 * k * n * xb + index, "flops": 2 * k * nnz}
    if call == "cg":
        # an inner step reads the matrix and p, writes q; reads q and r, writes r; reads and writes d and p
        steps = case["outer"] * case["inner"]
        outer = (case["outer"] + 1) * (nnz * 12 + 3.0 * 8 * n) + case["outer"] * n * (8 + 2 * xb + 16)
        return {"bytes": steps * (matrix + 9.0 * n * xb) + outer, "flops": steps * (2 * nnz + 10.0 * n) + 2 * nnz}
    # a Lanczos step reads the matrix and v, writes w; reads w, v and the v before, writes the next into the basis
    return {"bytes": case["steps"] * (matrix + 6.0 * n * xb), "flops": case["steps"] * (2 * nnz + 8.0 * n)}


def tolerance(case):
    """About four times what the path is off the same results in 64 bits, where that is summed in another order."""
    call, wide = case["call"], case.get("dtype") == "f64"
    if call in ("spmv", "ellr", "spmm", "batch"):
        # sums of up to a few hundred products in the vectors' type
        return {"rel": 1e-15, "max": 1e-13} if wide else {"rel": 1e-6, "max": 5e-5}
    if call == "cg":
        # refined until the residual in 64 bits is at its rounding
        return {"rel": 5e-15, "max": 5e-13}
    if call == "lanczos":
        # differences of rounding grow from step to step
        return {"rel": 1e-12, "max": 1e-10} if wide else {"rel": 5e-5, "max": 5e-3}
    return {"rel": 1e-5, "max": 1e-3}


def _sparse(crs, dtype="f64"):
    """The matrix with its values as they are stored at dtype, in 64 bits."""
    n, ptr, col, val = crs
    if dtype != "f64":
        val = (val.float() if dtype == "f32" else val.float().bfloat16()).double()
    return torch.sparse_csr_tensor(ptr, col.long(), val, size=(n, n), check_invariants=False)


def _times(A, x):
    return torch.mv(A, x) if x.dim() == 1 else torch.mm(A, x)


def _permutation(crs):
    """Rows by falling length, equal lengths in their order."""
    lengths = crs[1][1:] - crs[1][:-1]
    return torch.sort(-lengths, stable=True).indices


def _exact_cg(A, b):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), torch.dot(r, r)
    for _ in range(220):
        q = _times(A, p)
        a = torch.where(rr > 0, rr / torch.dot(p, q).clamp(min=1e-300), torch.zeros_like(rr))
        x, r = x + a * p, r - a * q
        new = torch.dot(r, r)
        p, rr = r + torch.where(rr > 0, new / rr.clamp(min=1e-300), torch.zeros_like(rr)) * p, new
    return x


def _exact_lanczos(A, v, steps):
    alpha, beta, basis = [], [torch.zeros((), dtype=torch.float64, device=DEV)], []
    before, v = torch.zeros_like(v), v / torch.linalg.vector_norm(v)
    for _ in range(steps):
        basis.append(v)
        w = _times(A, v)
        alpha.append(torch.dot(v, w))
        w = w - alpha[-1] * v - beta[-1] * before
        beta.append(torch.linalg.vector_norm(w))
        before, v = v, w / beta[-1]
    return {"alpha": torch.stack(alpha), "beta": torch.stack(beta), "basis": torch.stack(basis)}


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _order(n, epoch, seed=1):
    """The order of the samples in an epoch that the training call documents: a shuffle by a counter's hash."""
    with np.errstate(over="ignore"):
        base = _mix(np.array(seed + 0x51ED2701 * (epoch + 1), np.uint64))
        r = _mix(base + np.arange(n, dtype=np.uint64)) % np.arange(1, n + 1, dtype=np.uint64)
    o, r = list(range(n)), r.tolist()
    for i in range(n - 1, 0, -1):
        o[i], o[r[i]] = o[r[i]], o[i]
    return o


def _first_weights(seed=5):
    """The weights before the first step: uniform, by a counter's hash."""
    with np.errstate(over="ignore"):
        base = _mix(np.array((seed * 0x9E3779B97F4A7C15 + 77) % (1 << 64), np.uint64))
        n = HID * IN + HID * HID + HID
        r = _mix(base + np.arange(n, dtype=np.uint64) * np.uint64(0xD1B54A32D192ED03))
    u = (r >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 * 2 - 1
    lim = np.repeat([np.float32(math.sqrt(6 / IN)), np.float32(math.sqrt(6 / HID))], [HID * IN, n - HID * IN])
    w = (u * lim.astype(np.float64)).astype(np.float32).astype(np.float64)
    return w[: HID * IN].reshape(HID, IN), w[HID * IN: HID * IN + HID * HID].reshape(HID, HID), w[-HID:]


def _exact_train(case, seed):
    X, y = _samples(case, seed)
    n, B = case["samples"], min(case["batch"], case["samples"])

    def standard(a):
        a = a.astype(np.float64)
        return torch.from_numpy((a - a.mean(0)) / a.std(0)).to(DEV)

    X, y = standard(X), standard(y)
    P = [torch.from_numpy(np.ascontiguousarray(w)).to(DEV) for w in _first_weights()]
    P = [P[0], torch.zeros(HID, dtype=torch.float64, device=DEV), P[1],
         torch.zeros(HID, dtype=torch.float64, device=DEV), P[2], torch.zeros((), dtype=torch.float64, device=DEV)]
    P = [p.requires_grad_() for p in P]
    M, V, t, loss = [torch.zeros_like(p) for p in P], [torch.zeros_like(p) for p in P], 0, []

    def out(x):
        z = torch.relu(x @ P[0].T + P[1])
        return torch.relu(z @ P[2].T + P[3]) @ P[4] + P[5]

    for epoch in range(case["epochs"]):
        o = torch.tensor(_order(n, epoch) if B < n else list(range(n)), device=DEV)
        for at in range(0, n, B):
            s, t = o[at: at + B], t + 1
            grads = torch.autograd.grad((out(X[s]) - y[s]).square().mean(), P)
            with torch.no_grad():
                for p, q, m, v in zip(P, grads, M, V):
                    m.mul_(0.9).add_(q, alpha=0.1)
                    v.mul_(0.999).addcmul_(q, q, value=0.001)
                    p -= 2e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        with torch.no_grad():
            loss.append((out(X) - y).square().mean())
    P = [p.detach() for p in P]
    return {"loss": torch.stack(loss), "w1": P[0].reshape(-1), "b1": P[1], "w2": P[2].reshape(-1), "b2": P[3],
            "w3": P[4], "b3": P[5]}


def exact(case, seed):
    call = case["call"]
    if call == "train":
        return _exact_train(case, seed)
    dtype = case["dtype"]
    if call == "batch":
        return [_times(_sparse(_zipf(n, case["s"], _generator(seed, 100 + q)), dtype),
                       _vector(n, dtype, seed * 64 + q).double()) for q, n in enumerate(_batch_sizes(case))]
    crs, n = _matrix(case, seed), case["n"]
    if call in ("spmv", "ellr", "spmm"):
        y = _times(_sparse(crs, dtype), _vector(n, dtype, seed, case.get("k")).double())
        return y[_permutation(crs)] if case.get("permuted") else y
    perm = _permutation(crs)
    if call == "cg":
        return {"x": _exact_cg(_sparse(crs), _vector(n, "f64", seed))[perm], "steps": None}
    found = _exact_lanczos(_sparse(crs, dtype), _vector(n, dtype, seed).double(), case["steps"])
    return {**found, "basis": found["basis"][:, perm]}
