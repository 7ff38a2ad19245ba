"""Timed cases of the bucket-level resolve, through the package's public entry points.

The gradients stand for K per-language gradients of one model on one GPU: a shared direction plus a
language-specific one, with the share drawn per bucket and the scale per tensor (see `prepare`).  Sizes are
those of this repository's workloads (the tensor lists of GPT-2 small, Llama-3.2-1B and Qwen3-8B layers, the
flat sweep vectors) or generic ones around them.
"""
import math

import numpy as np
import torch

from paper_2606_05613_gb300 import inputs, native

DEV = "cuda:0"
MIB = 1 << 20
WINDOW = 1 << 26      # elements generated at a time


def _case(name, entry, K, dtype, out, model, n, bucket_kib, rule):
    return {"name": name, "entry": entry, "K": K, "dtype": dtype, "out": out, "model": model, "n": n,
            "bucket_kib": bucket_kib, "rule": rule}


def listed():
    return [
        # A small adapter's gradients: one call, four buckets; launches and latency are what it costs.
        _case("tiny-k2-f32", "resolve", 2, "f32", "f32", "flat", 1 << 20, 1024, "mgda"),
        # A small model of odd tensor sizes, bucket starts off the vector grid, mixed precision out.
        _case("ragged-k3-bf16-f32", "resolve", 3, "bf16", "f32", "ragged", 3_300_001, 1024, "pcgrad"),
        # One fine-tuning step of GPT-2 small: every bucket at the step's end.
        _case("gpt2-k4-f32", "resolve", 4, "f32", "f32", "gpt2", 0, 25 * 1024, "mgda"),
        # The same step resolved bucket by bucket, as the backward pass fills them.
        _case("gpt2-k4-f32-buckets", "buckets", 4, "f32", "f32", "gpt2", 0, 25 * 1024, "pcgrad"),
        # One step of Llama-3.2-1B in eight languages.
        _case("llama1b-k8-bf16", "resolve", 8, "bf16", "bf16", "llama", 0, 25 * 1024, "mgda"),
        # Decoder layers of Qwen3-8B, the benchmark's model: the two rules it is run with.
        _case("qwen-4layers-k4-bf16-cagrad", "resolve", 4, "bf16", "bf16", "qwen", 4, 25 * 1024, "cagrad"),
        _case("qwen-8layers-k4-bf16", "resolve", 4, "bf16", "bf16", "qwen", 8, 25 * 1024, "mgda"),
        # The bucket-size sweep: small and mid-sized buckets, few and many languages, one flat vector.
        _case("sweep-k2-f32-4mib", "resolve", 2, "f32", "f32", "flat", 500_000_000, 4 * 1024, "mgda"),
        _case("sweep-k4-f32-1mib", "resolve", 4, "f32", "f32", "flat", 250_000_000, 1024, "mgda"),
        _case("sweep-k16-f32-25mib", "resolve", 16, "f32", "f32", "flat", 100_000_001, 25 * 1024, "mgda"),
        # Conflict diagnostics of a step: Gram matrices and cosine statistics, no update.
        _case("conflicts-k8-bf16", "conflicts", 8, "bf16", "f32", "flat", 200_000_000, 4 * 1024, "mean"),
        # Gradients kept in host memory: in over the link, resolved, the direction back to the host.
        _case("host-k4-bf16", "host", 4, "bf16", "bf16", "flat", 64_000_000, 25 * 1024, "mgda"),
    ]


def draw(rng):
    def log_between(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    entry = rng.choice(["resolve"] * 6 + ["buckets", "conflicts", "host"])
    K = rng.choice([2, 3, 4, 4, 5, 6, 8, 8, 12, 16])
    dtype = rng.choice(["f32", "bf16"])
    out = rng.choice([dtype, dtype, "f32"])
    e = 4 if dtype == "f32" else 2
    most = (6e8 if entry == "host" else 6e9) / (K * e)
    n = int(log_between(1 << 18, most)) | rng.choice([0, 1])
    # at most 1200 buckets (a call each in the bucket-by-bucket entry: 100)
    kib = max(log_between(256, 100 * 1024), n * e / 1024 / (100 if entry == "buckets" else 1200))
    rule = rng.choice(["mgda", "mgda", "pcgrad", "cagrad"]) if entry != "conflicts" else "mean"
    c = _case("", entry, K, dtype, out, rng.choice(["flat", "ragged"]), n, int(math.ceil(kib)), rule)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------
# Plans and inputs
# ---------------------------------------------------------------------------------------------------

def _sizes(case):
    """Tensor sizes in registration order."""
    m, n = case["model"], case["n"]
    if m == "gpt2":
        return inputs.gpt2_small_sizes()
    if m == "llama":
        return inputs.llama32_1b_sizes()
    if m == "qwen":
        return list(inputs.qwen3_8b_layers(n).param_sizes)
    if m == "flat":
        return [n]
    # ragged: large odd tensors with small ones between, n elements in all
    rng, sizes, left = np.random.default_rng(n), [], n
    while left > 0:
        t = int(min(left, rng.integers(1, 200) if len(sizes) % 3 else rng.integers(n // 40 + 1, n // 12 + 2)))
        sizes.append(t)
        left -= t
    return sizes


def _elem(dtype):
    return 4 if dtype == "f32" else 2


def _torch(dtype):
    return torch.float32 if dtype == "f32" else torch.bfloat16


def _total(case):
    return case["n"] if case["model"] in ("flat", "ragged") else int(sum(_sizes(case)))


def _bucket_bounds(case):
    """Buckets filled from the last tensor on; one that does not fit closes the open bucket, one larger than a
    bucket is cut into whole buckets."""
    cap = case["bucket_kib"] * 1024 // _elem(case["dtype"])
    bounds, end, fill = [0], 0, 0
    for s in reversed(_sizes(case)):
        if fill and fill + s > cap:
            bounds.append(end)
            fill = 0
        while s > cap:
            end += cap
            bounds.append(end)
            s -= cap
        fill += s
        end += s
    if fill:
        bounds.append(end)
    return np.array(bounds, dtype=np.int64)


def _gradients(case, seed):
    """K flat gradients on the GPU: sigma_t (eps_k rho_b s + sqrt(1 - rho_b^2) u_k), rho_b per bucket in
    [-0.3, 0.95] (a negative one flips the shared part on odd languages), 5 % of the buckets at -0.7 or with
    one language negated, sigma_t lognormal per tensor."""
    K, n = case["K"], _total(case)
    bounds, sizes = _bucket_bounds(case), np.array(list(reversed(_sizes(case))), dtype=np.int64)
    B = len(bounds) - 1
    rng = np.random.default_rng([seed, 17])
    rho = rng.uniform(-0.3, 0.95, B)
    rho = np.where(rng.random(B) < 0.05, -0.7, rho)
    sign = np.where((rho[None, :] < 0) & (np.arange(K)[:, None] % 2 == 1), -1.0, 1.0)
    sign *= np.where((rng.random(B) < 0.05)[None, :] & (rng.integers(0, K, B)[None, :] == np.arange(K)[:, None]), -1.0, 1.0)
    sigma = np.exp(rng.standard_normal(len(sizes)))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    grads = [torch.empty(n, dtype=_torch(case["dtype"]), device=DEV) for _ in range(K)]

    def spread(values, edges, lo, hi):  # one value per element of [lo, hi), from values per interval of edges
        i0, i1 = np.searchsorted(edges, lo, side="right") - 1, np.searchsorted(edges, hi, side="left")
        e = np.clip(edges[i0:i1 + 1], lo, hi)
        return torch.repeat_interleave(torch.tensor(values[i0:i1], dtype=torch.float32, device=DEV),
                                       torch.tensor(np.diff(e), device=DEV), output_size=int(hi - lo))

    ends = np.concatenate([[0], np.cumsum(sizes)])
    for lo in range(0, n, WINDOW):
        hi = min(n, lo + WINDOW)
        m = hi - lo
        scale = spread(sigma, ends, lo, hi)
        s = torch.randn(m, generator=gen, device=DEV).mul_(scale)
        own = spread(np.sqrt(1 - rho ** 2), bounds, lo, hi).mul_(scale)
        for k in range(K):
            u = torch.randn(m, generator=gen, device=DEV).mul_(own)
            grads[k][lo:hi] = u.addcmul_(s, spread(np.abs(rho) * sign[k], bounds, lo, hi))
    return grads


def prepare(case, seed):
    K, n = case["K"], _total(case)
    grads = _gradients(case, seed)
    offsets = native.bkmoo_plan(_sizes(case), _elem(case["dtype"]), case["bucket_kib"] * 1024)
    B = len(offsets) - 1
    state = {"case": case, "grads": grads, "resolver": native.Resolver(K, _torch(case["dtype"]), offsets, DEV)}
    if case["entry"] == "conflicts":
        state["gram"] = torch.empty(B, K, K, dtype=torch.float64, device=DEV)
        state["cos"] = torch.empty(B, K, K, device=DEV)
        state["stats"] = torch.empty(B, 3, device=DEV)
        state["flag"] = torch.empty(B, dtype=torch.int32, device=DEV)
        return state
    state["weights"] = torch.empty(B, K, device=DEV)
    state["status"] = torch.empty(B, dtype=torch.int32, device=DEV)
    state["params"] = native.bkmoo_default_params()
    if case["model"] == "llama":
        state["params"].max_iter = 20
    if case["entry"] == "host":
        host = [torch.empty(n, dtype=_torch(case["dtype"]), pin_memory=True) for _ in range(K)]
        for h, g in zip(host, grads):
            h.copy_(g)
        state["grads"] = host
        state["direction"] = torch.empty(n, dtype=_torch(case["out"]), pin_memory=True)
        code = native.BKMOO_F32 if case["out"] == "f32" else native.BKMOO_BF16
        state["staging"] = torch.empty(state["resolver"].staging_size(code), dtype=torch.uint8, device=DEV)
    else:
        state["direction"] = torch.empty(n, dtype=_torch(case["out"]), device=DEV)
    return state


def run(state):
    case, r = state["case"], state["resolver"]
    if case["entry"] == "conflicts":
        r.gram(state["grads"], state["gram"])
        native.bkmoo_conflicts(state["gram"], state["cos"], state["stats"], state["flag"])
        return {"gram": state["gram"], "cos": state["cos"], "stats": state["stats"], "flag": state["flag"]}
    kw = {"params": state["params"], "out_weights": state["weights"], "out_status": state["status"]}
    if case["entry"] == "host":
        r.resolve_host(state["grads"], case["rule"], state["direction"], state["staging"], **kw)
        torch.cuda.current_stream().synchronize()   # the direction is read on the host
    elif case["entry"] == "buckets":
        for b in range(r.n_buckets):
            r.resolve_buckets(state["grads"], b, b + 1, case["rule"], state["direction"], **kw)
    else:
        r.resolve(state["grads"], case["rule"], state["direction"], **kw)
    return {"direction": state["direction"], "weights": state["weights"], "status": state["status"]}


def work(case):
    K, n, e = case["K"], _total(case), _elem(case["dtype"])
    B = len(_bucket_bounds(case)) - 1
    if case["entry"] == "conflicts":
        return {"bytes": K * e * n + B * (K * K * 12 + 16), "flops": K * (K + 1) * n}
    return {"bytes": (K * e + _elem(case["out"])) * n + B * (4 * K + 4), "flops": (K * (K + 1) + 2 * K) * n}


def tolerance(case):
    # 32-bit results: fp32 products summed in another order and fp32 combinations of them.  bf16 results: one
    # rounding to 8 bits.  A conflict flag may differ where the smallest cosine is a rounding error from 0.
    if case["entry"] == "conflicts":
        return {"rel": 1e-5, "differ": 0.005}
    return {"rel": 1e-5} if case["out"] == "f32" else {"rel": 7e-3}


# ---------------------------------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------------------------------

def _mgda(G):
    """Min-norm point of the hull: w / sum(w) for the w >= 0 with G w >= 1, equal where w > 0 (active sets)."""
    K = len(G)
    s = np.sqrt(np.diag(G))
    A, one = G / np.outer(s, s), 1.0 / s          # scaled to a unit diagonal
    w, P = np.zeros(K), np.zeros(K, bool)
    for _ in range(200):
        g = one - A @ w
        if P.all() or np.max(np.where(P, -np.inf, g / one)) <= 1e-13:
            break
        P[np.argmax(np.where(P, -np.inf, g / one))] = True
        while True:
            z = np.zeros(K)
            z[P] = np.linalg.solve(A[np.ix_(P, P)], one[P])
            if (z[P] > 0).all():
                w = z
                break
            t = min(w[i] / (w[i] - z[i]) for i in np.flatnonzero(P) if z[i] <= 0)
            w = w + t * (z - w)
            P &= w > 1e-15
            w[~P] = 0
    w = w / s
    return w / w.sum()


def _cagrad(G, c=0.5):
    """min over the simplex of <g0, g_w> + c |g0| |g_w|: stationary points of every support, in closed form."""
    K = len(G)
    b = G.mean(axis=1)
    n0 = math.sqrt(b.mean())
    c0, best, w_best = c * n0, math.inf, None
    for mask in range(1, 1 << K):
        S = [i for i in range(K) if mask >> i & 1]
        A = G[np.ix_(S, S)]
        u, v = np.linalg.solve(A, np.stack([np.ones(len(S)), b[S]], 1)).T
        p, q, r = u.sum(), v.sum(), b[S] @ v       # c0^2 = p x^2 - 2 q x + r for the multiplier x
        disc = q * q - p * (r - c0 * c0)
        if disc < 0:
            continue
        for x in ((q + math.sqrt(disc)) / p, (q - math.sqrt(disc)) / p):
            y = x * u - v
            if y.sum() <= 0:
                continue
            w = y / y.sum()
            if (w < -1e-12).any():
                continue
            F = b[S] @ w + c0 * math.sqrt(max(w @ A @ w, 0.0))
            if F < best:
                best, w_best = F, np.zeros(K)
                w_best[S] = w
    return 1.0 / K + c0 * w_best / math.sqrt(w_best @ G @ w_best)


M64 = (1 << 64) - 1
GOLD = 0x9E3779B97F4A7C15


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def _pcgrad(G, bucket):
    """Sequential projections off the original gradients, task t's order a keyed shuffle (include/bkmoo.h)."""
    K = len(G)
    beta = np.zeros(K)
    for t in range(K):
        k3 = _mix((_mix((_mix(GOLD) + (bucket + 1) * GOLD) & M64) + (t + 1) * GOLD) & M64)
        order = [j for j in range(K) if j != t]
        for m, i in enumerate(range(len(order) - 1, 0, -1)):
            j = _mix((k3 + (m + 1) * GOLD) & M64) % (i + 1)
            order[i], order[j] = order[j], order[i]
        x = np.zeros(K)
        x[t] = 1.0
        for j in order:
            dot = x @ G[:, j]
            if dot < 0 and G[j, j] > 0:
                x[j] -= dot / G[j, j]
        beta += x
    return beta


def exact(case, seed):
    K, n = case["K"], _total(case)
    if case["rule"] == "cagrad" and K > 6:
        return None                                # too many supports
    grads, bounds = _gradients(case, seed), _bucket_bounds(case)
    B = len(bounds) - 1
    gram = np.zeros((B, K, K))
    for b in range(B):
        G = torch.zeros(K, K, dtype=torch.float64, device=DEV)
        for lo in range(int(bounds[b]), int(bounds[b + 1]), WINDOW):
            x = torch.stack([g[lo:min(lo + WINDOW, int(bounds[b + 1]))] for g in grads]).double()
            G += x @ x.T
        gram[b] = G.cpu().numpy()
    if case["entry"] == "conflicts":
        d = np.sqrt(np.einsum("bkk->bk", gram))
        cos = gram / (d[:, :, None] * d[:, None, :])
        pairs = cos[:, np.triu_indices(K, 1)[0], np.triu_indices(K, 1)[1]]
        stats = np.stack([pairs.mean(1), pairs.std(1), pairs.min(1)], 1)
        return {"gram": gram, "cos": cos, "stats": stats, "flag": None}
    rule = {"mgda": lambda b: _mgda(gram[b]), "cagrad": lambda b: _cagrad(gram[b]), "pcgrad": lambda b: _pcgrad(gram[b], b)}[case["rule"]]
    beta = np.stack([rule(b) for b in range(B)])
    out = torch.empty(n, dtype=torch.float64, device=DEV)
    for b in range(B):
        for lo in range(int(bounds[b]), int(bounds[b + 1]), WINDOW):
            hi = min(lo + WINDOW, int(bounds[b + 1]))
            torch.mul(grads[0][lo:hi].double(), float(beta[b, 0]), out=out[lo:hi])
            for k in range(1, K):
                out[lo:hi].add_(grads[k][lo:hi].double(), alpha=float(beta[b, k]))
    return {"direction": out, "weights": torch.tensor(beta), "status": None}
