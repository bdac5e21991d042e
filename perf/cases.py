"""Performance cases of the library: what a program that uses it computes, over the sizes, orders,
precision forms and entry points in real use. Inputs are synthetic systems of the shapes of the
benchmark and the tests: real state matrices with conjugate mode pairs in blocks of four states and
sparse coupling, and packed Taylor tensors with 30% nonzero entries N(0, 1)."""
import math

import numpy as np
import torch

import paper_2509_08968_gb300 as npf
from paper_2509_08968_gb300.mlp import Mlp, param_layout


def listed():
    return [
        # a small system studied interactively: latency and launches are all that counts
        {"name": "small_n10_o3", "kind": "npf", "n": 10, "orders": "2,3", "precision": "split_bf16"},
        # one operating point of a mid-size system at every order: the ordinary call
        {"name": "medium_n60_o4", "kind": "npf", "n": 60, "orders": "2,3,4", "precision": "split_bf16"},
        # a large system at the order most studies stop at
        {"name": "large_n120_o3", "kind": "npf", "n": 120, "orders": "3", "precision": "split_bf16"},
        # the largest call: the benchmark's system at orders 3 and 4, under a memory budget
        {"name": "largest_n120_o4", "kind": "npf", "n": 120, "orders": "3,4", "precision": "split_bf16",
         "budget_gb": 66.0},
        # the FP32 form (accuracy 1e-5 asked for) of a system of odd size
        {"name": "fp32_n75_o4", "kind": "npf", "n": 75, "orders": "3,4", "precision": "fp32",
         "budget_gb": 48.0},
        # the native FP64 form, the library's own reference on the GPU
        {"name": "fp64_n60_o3", "kind": "npf", "n": 60, "orders": "2,3", "precision": "fp64"},
        # many systems of uneven size and order in one call
        {"name": "batch_64_systems", "kind": "batch", "count": 64, "lo": 20, "hi": 80},
        # a new operating point in a kept plan: modal data and tensors replaced, then one call
        {"name": "point_n40_o3", "kind": "point", "n": 40, "orders": "2,3", "precision": "split_bf16"},
        # only the critical modes of a large system, of odd number
        {"name": "subset_n100_m31_o4", "kind": "subset", "n": 100, "m": 31, "orders": "3,4",
         "precision": "split_bf16", "budget_gb": 48.0},
        # mode-interaction participation factors of a mid-size system
        {"name": "interaction_n60_o3", "kind": "interaction", "n": 60, "orders": "2,3",
         "precision": "split_bf16", "delta": 0.05},
        # the surrogate's training: two passes over 4096 points
        {"name": "train_4096x256", "kind": "train", "rows": 4096, "batch": 256, "epochs": 2, "members": 5,
         "hidden": 256, "outputs": 64},
        # the surrogate's gated queries
        {"name": "predict_512", "kind": "predict", "rows": 512, "members": 5, "hidden": 256, "outputs": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["npf", "npf", "npf", "npf", "npf", "fp64", "batch", "point", "subset", "interaction",
                       "train", "predict"])
    if kind == "npf":
        top = rng.choice([2, 3, 3, 4, 4])
        n = _log_int(rng, 4, 128 if top < 4 else 100)
        orders = [k for k in range(2, top + 1) if k == top or rng.random() < 0.5]
        case = {"kind": "npf", "n": n, "orders": ",".join(map(str, orders)),
                "precision": rng.choice(["split_bf16", "split_bf16", "fp32"])}
        if top == 4 and n > 64:
            case["budget_gb"] = 48.0
        return case
    if kind == "fp64":
        top = rng.choice([2, 3])
        return {"kind": "npf", "n": _log_int(rng, 5, 70), "orders": "2" if top == 2 else "2,3",
                "precision": "fp64"}
    if kind == "batch":
        lo = rng.randint(4, 40)
        return {"kind": "batch", "count": _log_int(rng, 3, 64), "lo": lo, "hi": rng.randint(lo, 80)}
    if kind == "point":
        return {"kind": "point", "n": _log_int(rng, 6, 90), "orders": rng.choice(["2", "3", "2,3"]),
                "precision": rng.choice(["split_bf16", "fp32"])}
    if kind == "subset":
        top = rng.choice([3, 4])
        n = _log_int(rng, 12, 120 if top == 3 else 100)
        case = {"kind": "subset", "n": n, "m": rng.randint(2, max(3, n // 2)),
                "orders": "3" if top == 3 else "3,4", "precision": "split_bf16"}
        if top == 4 and n > 64:
            case["budget_gb"] = 48.0
        return case
    if kind == "interaction":
        precision = rng.choice(["split_bf16", "split_bf16", "fp64"])
        return {"kind": "interaction", "n": _log_int(rng, 5, 70 if precision == "fp64" else 120),
                "orders": rng.choice(["2", "2,3"]), "precision": precision,
                "delta": rng.choice([0.02, 0.05, 0.1])}
    if kind == "train":
        return {"kind": "train", "rows": _log_int(rng, 300, 4096), "batch": _log_int(rng, 32, 256),
                "epochs": rng.randint(1, 2), "members": rng.randint(1, 5), "hidden": 16 * rng.randint(2, 16),
                "outputs": rng.randint(8, 64)}
    return {"kind": "predict", "rows": _log_int(rng, 1, 4096), "members": rng.randint(2, 5),
            "hidden": 16 * rng.randint(2, 16), "outputs": rng.randint(8, 64)}


# ------------------------------------------------------------------------------------------- inputs
def _orders(case):
    return [int(x) for x in case["orders"].split(",")]


def _modes(n, rng):
    """(lam, U, V): conjugate pairs sigma +- i omega (one real mode when n is odd), sigma in
    [-2, -0.05], omega in [0.5, 15]; right eigenvectors from a real, block-structured similarity."""
    pairs = n // 2
    s, w = rng.uniform(-2.0, -0.05, n - pairs), rng.uniform(0.5, 15.0, pairs)
    lam = np.empty(n, np.complex128)
    lam[0:2 * pairs:2] = s[:pairs] + 1j * w
    lam[1:2 * pairs:2] = s[:pairs] - 1j * w
    W = np.zeros((n, n), np.complex128)
    for b in range(pairs):
        W[2 * b, 2 * b:2 * b + 2] = 1.0
        W[2 * b + 1, 2 * b:2 * b + 2] = [1j, -1j]
    if n % 2:
        lam[-1], W[-1, -1] = s[-1], 1.0
    block = np.arange(n) // 4
    same = block[:, None] == block[None, :]
    for _ in range(1000):
        P = np.where(same, np.eye(n) + 0.3 * rng.standard_normal((n, n)), 0.0)
        P = P + np.where(~same & (rng.random((n, n)) < 0.1), 0.1 * rng.standard_normal((n, n)), 0.0)
        if np.linalg.cond(P) < 200.0:
            break
    U = P.astype(np.complex128) @ W
    return lam, U, np.linalg.inv(U)


def _tensor(n, N, seed):
    """Packed symmetric order-N tensor [n, C(n+N-1, N)] on the GPU, 30% nonzero N(0, 1)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    count = math.comb(n + N - 1, N)
    out = torch.empty((n, count), dtype=torch.float64, device="cuda")
    rows = max(1, min(n, (1 << 27) // count))
    for j in range(0, n, rows):
        part = out[j:j + rows]
        part.normal_(generator=g)
        part.masked_fill_(torch.rand(part.shape, generator=g, device="cuda") >= 0.3, 0.0)
    return out


def _system(n, orders, seed):
    lam, U, V = _modes(n, np.random.default_rng(seed))
    return lam, U, V, {N: _tensor(n, N, seed * 16 + N) for N in orders}


def _plan(lam, U, V, tensors, precision, budget_gb=0.0):
    p = npf.Plan(lam, U, V, max(tensors), mem_budget=int(budget_gb * 1e9), precision=precision)
    for N, t in tensors.items():
        p.set_tensor(N, t)
    return p


def _batch(case, seed):
    """(n, order, seed) of every system: the sizes are the case's own, the data the seed's."""
    rng = np.random.default_rng([case["count"], case["lo"], case["hi"]])
    for b in range(case["count"]):
        yield int(rng.integers(case["lo"], case["hi"] + 1)), int(rng.integers(2, 4)), seed * 1000 + b


def _subset(case, seed):
    return np.sort(np.random.default_rng(seed + 7).permutation(case["n"])[:case["m"]]).astype(np.int32)


def _widths(case):
    return [4, case["hidden"], case["hidden"], case["hidden"], case["outputs"]]


def _net(case, seed):
    """He-uniform weights; for queries the members differ as trained ones do (by a few percent)."""
    rng = np.random.default_rng(seed)
    widths, members = _widths(case), []
    base = None
    for _ in range(case["members"]):
        parts = []
        for r, c in param_layout(widths):
            W = np.zeros((r, c), np.float32)
            b = math.sqrt(6.0 / (c - 1))
            W[:, :-1] = rng.uniform(-b, b, (r, c - 1))
            parts.append(W.ravel())
        flat = np.concatenate(parts)
        base = flat if base is None else base
        members.append(base + 0.02 * flat if case["kind"] == "predict" else flat)
    return widths, np.stack(members).astype(np.float32)


def _points(case, seed):
    """Features in [-1, 1] and smooth standardised targets of them."""
    rng = np.random.default_rng(seed + 1)
    X = rng.uniform(-1.0, 1.0, (case["rows"], 4)).astype(np.float32)
    A = rng.standard_normal((4, case["outputs"]))
    T = np.sin(X @ A) + 0.3 * (X ** 2) @ A
    mu = rng.uniform(-3.0, 1.0, case["outputs"]).astype(np.float32)
    sigma = rng.uniform(0.05, 0.3, case["outputs"]).astype(np.float32)
    return X, ((T - T.mean(0)) / T.std(0)).astype(np.float32), mu, sigma


# -------------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("train", "predict"):
        widths, weights = _net(case, seed)
        X, T, mu, sigma = _points(case, seed)
        return {"case": case, "net": Mlp(widths, weights), "X": X, "T": T, "mu": mu, "sigma": sigma}
    if kind == "batch":
        plans, orders, outs = [], [], []
        for n, N, s in _batch(case, seed):
            plans.append(_plan(*_system(n, [N], s), "split_bf16"))
            orders.append(N)
            outs.append(np.empty((n, n), np.complex128))
        return {"case": case, "plans": plans, "orders": orders, "outs": outs}
    lam, U, V, tensors = _system(case["n"], _orders(case), seed)
    p = _plan(lam, U, V, tensors, case["precision"], case.get("budget_gb", 0.0))
    state = {"case": case, "plan": p, "order": max(tensors)}
    if kind == "point":   # the plan comes from another operating point; these are the new one's data
        state.update(lam=lam, U=U, V=V, tensors=tensors)
    if kind == "subset":
        p.set_mode_subset(_subset(case, seed))
    if kind != "point":
        del tensors
        torch.cuda.empty_cache()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        hist = state["net"].train(state["X"], state["T"], case["epochs"], case["batch"], 1e-3, seed=3)
        return hist, state["net"].weights()
    if kind == "predict":
        return state["net"].predict(state["X"], state["mu"], state["sigma"], 0.05)
    if kind == "batch":
        outs = npf.batch_compute(state["plans"], state["orders"], state["outs"])
        return np.concatenate([o.ravel() for o in outs])
    p = state["plan"]
    if kind == "point":
        p.set_modes(state["lam"], state["U"], state["V"])
        for N, t in state["tensors"].items():
            p.set_tensor(N, t)
    if kind == "interaction":
        return p.interaction(state["order"], case["delta"])
    return p.compute(state["order"])


# ---------------------------------------------------------------------------- work and tolerances
def _npf_work(n, m, orders, pairs, interaction=False):
    """Each packed tensor read once and the result written once; the products over sorted index
    tuples (the tensors are symmetric), a real multiply and add per slice pair."""
    size, flops = 16 * n * n * 4, 0.0
    for N in orders:
        tuples = math.comb(n + N - 1, N)
        size += 8 * n * tuples
        per = 4.0 * n * m * tuples                                    # upper index, real tensor
        for c in range(1, N + 1):                                     # lower indices, one after another
            per += 8.0 * n * m * math.comb(m + c - 1, c) * math.comb(n + N - c - 1, N - c)
        red = 8.0 * m * n * math.comb(m + N - 1, N)                   # divided entries into Psi_N
        flops += (per + red) * pairs * (2 if interaction else 1)
    return size, flops


def work(case):
    kind = case["kind"]
    if kind in ("train", "predict"):
        widths = _widths(case)
        params = sum(r * c for r, c in param_layout(widths)) * case["members"]
        if kind == "predict":
            rows = case["rows"]
            return {"bytes": 4 * params + 4 * rows * (4 + widths[-1] + 2), "flops": 2.0 * rows * params}
        steps = case["rows"] // case["batch"] * case["epochs"]
        return {"bytes": 4 * 6 * params + 4 * case["rows"] * (4 + widths[-1]),
                "flops": 6.0 * steps * case["batch"] * params}
    if kind == "batch":
        n = 0.5 * (case["lo"] + case["hi"])
        n = int(round(n))
        size, flops = _npf_work(n, n, [2], 21)
        more, most = _npf_work(n, n, [3], 21)
        return {"bytes": case["count"] * (size + more) // 2, "flops": case["count"] * (flops + most) / 2}
    pairs = {"split_bf16": 21, "fp32": 10, "fp64": 1}[case["precision"]]
    size, flops = _npf_work(case["n"], case.get("m", case["n"]), _orders(case), pairs, kind == "interaction")
    return {"bytes": size, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "train":
        return {"rel": 2e-2, "max": 0.9}
    if kind == "predict":
        return {"rel": 2e-2, "max": 0.9, "differ": 0.01}
    # four times the largest error seen against `exact`
    return {"split_bf16": {"rel": 1.6e-10, "max": 1.6e-8}, "fp32": {"rel": 4e-7, "max": 4e-5},
            "fp64": {"rel": 1e-13, "max": 1e-11}}[case.get("precision", "split_bf16")]


# --------------------------------------------------------------------------------- exact (64 bits)
def _sorted_rank(n, N):
    """Packed rank of every index tuple [n, .., n] (N of them) on the GPU."""
    cnt = torch.tensor([[math.comb(n - v + r - 1, r) if r else 1 for v in range(n + 1)] for r in range(N + 1)],
                       device="cuda")
    idx = torch.stack(torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.int16)] * N, indexing="ij"), -1)
    idx = idx.reshape(-1, N).sort(dim=1).values
    rank = torch.zeros(idx.shape[0], dtype=torch.int64, device="cuda")
    prev = torch.zeros_like(rank)
    for k in range(N):
        cur = idx[:, k].long()
        rank += cnt[N - k][prev] - cnt[N - k][cur]
        prev = cur
    return rank


def _reduce(h, W, N):
    """sum over p_1..p_N of h[p_1, .., p_N] prod W[p_m, k], per k."""
    n = W.shape[1]
    g = h.reshape(-1, W.shape[0]) @ W
    for _ in range(N - 1):
        g = (g.reshape(-1, W.shape[0], n) * W).sum(1)
    return g.reshape(n)


def _terms(lam, U, V, tensors, modes, weights=None):
    """{N: -sum_p h^i_p prod W[p_m, k]} with modal indices in `modes`, rows of other modes zero."""
    dev = {"device": "cuda", "dtype": torch.complex128}
    n = len(lam)
    lam, U, V = (torch.as_tensor(x).to(**dev) for x in (lam, U, V))
    keep = torch.as_tensor(np.asarray(modes), device="cuda").long()
    ls, Us = lam[keep], U[:, keep].contiguous()
    Wsel = (V if weights is None else weights)[keep].contiguous()
    out = {}
    for N, A in tensors.items():
        rank = _sorted_rank(n, N)
        sums = torch.zeros((), **dev)
        for k in range(N):
            sums = sums + ls.reshape([-1 if d == k else 1 for d in range(N)])
        res = torch.zeros((n, n), **dev)
        for i in keep.tolist():
            s = (V[i].real @ A) + 1j * (V[i].imag @ A)
            h = s[rank].reshape([n] * N)
            for _ in range(N):          # contract the first index, put the new one last
                h = (h.reshape(n, -1).T @ Us).reshape(list(h.shape[1:]) + [len(keep)])
            den = sums - lam[i]
            den = torch.where(den.abs() < 1e-8, torch.full_like(den, 1e-8), den)
            res[i] = -_reduce(h / den / math.factorial(N), Wsel, N)
            del h, den, s
        out[N] = res
        del rank, sums
    return out, U, V


def _exact_system(case, seed):
    n, orders = case["n"], _orders(case)
    lam, U, V, tensors = _system(n, orders, seed)
    modes = _subset(case, seed) if case["kind"] == "subset" else np.arange(n)
    terms, Ut, Vt = _terms(lam, U, V, tensors, modes)
    if case["kind"] != "interaction":
        return (Ut * (Vt + sum(terms.values())).T).cpu().numpy()
    top, d = max(orders), case["delta"]
    z = d * Vt + sum(d ** N * t for N, t in terms.items())
    res = np.zeros((top, n, n), np.complex128)
    res[0] = (Ut * z.T).cpu().numpy()
    again, _, _ = _terms(lam, U, V, tensors, modes, z)
    for N, t in again.items():
        res[N - 1] = (-Ut * t.T).cpu().numpy()
    return res


def _layers(flat, widths):
    out, o = [], 0
    for r, c in param_layout(widths):
        out.append(torch.as_tensor(flat[:, o:o + r * c].reshape(-1, r, c).astype(np.float64), device="cuda"))
        o += r * c
    return out


def _forward(layers, X):
    hs, ones = [X], torch.ones(X.shape[:-1] + (1,), dtype=torch.float64, device="cuda")
    for k, W in enumerate(layers):
        z = torch.cat([hs[-1], ones], -1) @ W.transpose(1, 2)
        hs.append(torch.relu(z) if k + 1 < len(layers) else z)
    return hs


def _shuffles(rows, members, epochs, seed):
    """The documented permutations: Fisher-Yates drawn from splitmix64(seed + 7919 e)."""
    mask = (1 << 64) - 1
    states = [(seed + 7919 * e) & mask for e in range(members)]
    for _ in range(epochs):
        perms = []
        for e in range(members):
            p = list(range(rows))
            for r in range(rows - 1, 0, -1):
                states[e] = s = (states[e] + 0x9E3779B97F4A7C15) & mask
                s = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & mask
                s = ((s ^ (s >> 27)) * 0x94D049BB133111EB) & mask
                j = (s ^ (s >> 31)) % (r + 1)
                p[r], p[j] = p[j], p[r]
            perms.append(p)
        yield torch.tensor(perms, device="cuda")


def _exact_net(case, seed):
    widths, flat = _net(case, seed)
    X, T, mu, sigma = _points(case, seed)
    layers = _layers(flat, widths)
    Xd = torch.as_tensor(X.astype(np.float64), device="cuda")
    if case["kind"] == "predict":
        y = _forward(layers, Xd.expand(case["members"], -1, -1))[-1].cpu().numpy()
        v = np.exp(mu.astype(np.float64) + sigma.astype(np.float64) * y)
        return v.mean(0), (v.std(0) / v.mean(0)).max(1), None
    Td = torch.as_tensor(T.astype(np.float64), device="cuda")
    m1 = [torch.zeros_like(W) for W in layers]
    m2 = [torch.zeros_like(W) for W in layers]
    hist, step, B = [], 0, case["batch"]
    for perm in _shuffles(case["rows"], case["members"], case["epochs"], 3):
        total, steps = 0.0, case["rows"] // B
        for k in range(steps):
            idx = perm[:, k * B:(k + 1) * B]
            leaves = [W.requires_grad_(True) for W in layers]
            loss = ((_forward(leaves, Xd[idx])[-1] - Td[idx]) ** 2).mean((1, 2))
            grads = torch.autograd.grad(loss.sum(), leaves)
            total += float(loss.sum().detach())
            step += 1
            with torch.no_grad():
                for j, g in enumerate(grads):
                    m1[j] = 0.9 * m1[j] + 0.1 * g
                    m2[j] = 0.999 * m2[j] + 0.001 * g * g
                    up = (m1[j] / (1 - 0.9 ** step)) / ((m2[j] / (1 - 0.999 ** step)).sqrt() + 1e-8)
                    layers[j] = (leaves[j] - 1e-3 * up).detach()
        hist.append(total / (case["members"] * steps))
    weights = torch.cat([W.reshape(case["members"], -1) for W in layers], 1)
    return np.array(hist), weights.cpu().numpy()


def exact(case, seed):
    if case["kind"] in ("train", "predict"):
        return _exact_net(case, seed)
    if case["kind"] == "batch":
        parts = []
        for n, N, s in _batch(case, seed):
            parts.append(_exact_system({"kind": "npf", "n": n, "orders": str(N)}, s).ravel())
        return np.concatenate(parts)
    if max(_orders(case)) >= 4 and case.get("m", case["n"]) > 80:
        return None
    return _exact_system(case, seed)
