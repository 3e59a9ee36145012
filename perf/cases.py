"""The folded-MoE layer's working range as a set of measurable cases.

A case is one call of the library on one layer: a prefill of T tokens (Top-K folding), a decode step of B tokens
(expert-pool folding, dynamic or static pool) or the offline calibration of m tokens, on a layer of the shapes that
the repository's configurations name (`tiny`, `mixtral`, `qwen3`, `glm45air`) or of a generic shape. `listed()` names
the ones that stand for typical use, `draw()` gives more of the same ranges, `prepare()` builds what a serving process
holds before the call (weights, tables, workspace, this step's activations and router scores), `run()` makes the one
call and returns what it computes.
"""
import math

import numpy as np
import torch

from paper_2608_24938_b200 import binding as ex

# routed experts, shared experts, hidden, intermediate, Top-K, dtype, distribution of the router scores
SHAPES = {
    "tiny": (8, 0, 128, 256, 2, "f32", "normal"),
    "mixtral": (8, 0, 4096, 14336, 2, "bf16", "normal"),
    "qwen3": (128, 0, 2048, 768, 8, "bf16", "zipf"),
    "glm45air": (128, 1, 4096, 1408, 8, "bf16", "normal"),
}
FIELDS = ("experts", "shared", "hidden", "inter", "top_k", "dtype", "scores")
ZIPF_S = 1.1
MAX_WEIGHT_BYTES = 4_600_000_000  # the largest listed layer's 4.5 GB


def _case(op, shape, **kw):
    c = {"op": op, "router": False, "guard": False, "static": False}
    c.update(zip(FIELDS, SHAPES[shape] if isinstance(shape, str) else shape))
    c.update(kw)
    return c


def listed():
    return [
        # the smallest calls: an fp32 layer small enough that latency and launches are the whole cost
        _case("prefill", "tiny", name="f32_prefill_t64", tokens=64, budget=1),
        _case("decode", "tiny", name="f32_decode_b16", tokens=16, budget=4),
        # one user's generation: a single token, every one of its experts read once
        _case("decode", "qwen3", name="qwen3_decode_b1", tokens=1, budget=16),
        # an ordinary decode batch with a small pool: the weights stream in little more time than the fixed costs
        _case("decode", "qwen3", name="qwen3_decode_b64_m16", tokens=64, budget=16),
        # the largest decode batch, router included, through a large pool
        _case("decode", "qwen3", name="qwen3_decode_layer_b256_m64", tokens=256, budget=64, router=True),
        # a server's usual decode step on a large layer with a shared expert
        _case("decode", "glm45air", name="glm_decode_b128_m32", tokens=128, budget=32),
        # few, wide experts: the most bytes per decode step
        _case("decode", "mixtral", name="mixtral_decode_b32_m4", tokens=32, budget=4),
        # a short ragged prompt with the router and the safeguards on (loss threshold 0.99, per-token rescale)
        _case("prefill", "qwen3", name="qwen3_prefill_guard_t777_k6", tokens=777, budget=6, router=True, guard=True),
        # a long prompt on many small experts of very uneven popularity
        _case("prefill", "qwen3", name="qwen3_prefill_t8192_k4", tokens=8192, budget=4),
        # a long prompt on few wide experts
        _case("prefill", "mixtral", name="mixtral_prefill_t4096_k1", tokens=4096, budget=1),
        # the largest prefill: eight prompts of 2048 tokens, shared expert
        _case("prefill", "glm45air", name="glm_prefill_t16384_k4", tokens=16384, budget=4),
        # a layer's offline calibration
        _case("calibrate", "qwen3", name="qwen3_calibrate_m8192", tokens=8192, budget=8),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _weight_bytes(c):
    return (c["experts"] + c["shared"]) * 3 * c["hidden"] * c["inter"] * (4 if c["dtype"] == "f32" else 2)


def _generic(rng, dtype):
    """A layer of no particular model: any size that the library takes, up to the listed ones."""
    while True:
        n = _log_int(rng, 4, 256)
        unit = 64 if dtype == "bf16" else 32
        d = unit * _log_int(rng, 2, 64 if dtype == "bf16" else 24)
        i = unit * _log_int(rng, 2, 40 if dtype == "bf16" else 32)
        k = rng.randint(1, min(n, 10))
        s = (n, rng.randint(0, 1), d, i, k, dtype, rng.choice(("normal", "zipf")))
        c = dict(zip(FIELDS, s))
        if _weight_bytes(c) <= (MAX_WEIGHT_BYTES if dtype == "bf16" else 256_000_000):
            return s


def draw(rng):
    kind = rng.choice(("prefill", "prefill", "prefill", "decode", "decode", "decode", "f32", "f32", "calibrate"))
    if kind == "f32":
        op = rng.choice(("prefill", "decode"))
        shape = rng.choice(("tiny", None)) or _generic(rng, "f32")
    else:
        op = kind
        shape = rng.choice(("mixtral", "qwen3", "glm45air", None)) or _generic(rng, "bf16")
    c = _case(op, shape)
    n, k = c["experts"], c["top_k"]
    if op == "decode":
        c["tokens"] = _log_int(rng, 1, 256)
        c["budget"] = _log_int(rng, 1, n)
        c["static"] = rng.random() < 0.2
        c["router"] = not c["static"] and rng.random() < 0.4
    elif op == "prefill":
        c["tokens"] = _log_int(rng, 1, 16384 if kind != "f32" else 1024)
        c["budget"] = rng.randint(1, k)
        c["router"] = rng.random() < 0.4
        c["guard"] = rng.random() < 0.25
    else:
        c["tokens"] = _log_int(rng, 64, 8192)
        c["budget"] = k
    # no case costs more than the largest listed one
    limit = work(listed()[10])["flops"] if kind != "f32" else 2e9
    while op != "decode" and c["tokens"] > 1 and work(c)["flops"] > limit:
        c["tokens"] = max(1, c["tokens"] * 3 // 4)
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _tables(n, rng):
    """Calibrated tables of the geometry real layers show: norms spread over a factor of three, S = similarity times the
    norm ratio, a tenth of the scalars negative, 2 % of the pairs never observed."""
    h = np.exp(rng.uniform(0.0, np.log(3.2), size=n))
    c = np.triu(rng.uniform(0.2, 0.9, size=(n, n)), 1)
    c = c + c.T
    S = np.clip(c * h[:, None] / h[None, :], -4.0, 4.0)
    S = np.where(rng.uniform(size=(n, n)) < 0.10, -S, S)
    L = 1.0 - c * c
    unseen = rng.uniform(size=(n, n)) < 0.02
    S, L = np.where(unseen, 0.0, S), np.where(unseen, 1e30, L)
    np.fill_diagonal(S, 1.0)
    np.fill_diagonal(L, 0.0)
    h = h.astype(np.float32)
    return S.astype(np.float32), L.astype(np.float32), h, np.log(h.astype(np.float64)).astype(np.float32)


def _popularity(c, rng):
    """ln p(e) of the experts: p_k ~ k^-1.1 over a random order of the experts, or even."""
    n = c["experts"]
    if c["scores"] != "zipf":
        return np.zeros(n)
    p = np.arange(1, n + 1, dtype=np.float64) ** -ZIPF_S
    return np.log(p / p.sum())[rng.permutation(n)]


def prepare(case, seed):
    n, s, d, i, k = (case[f] for f in FIELDS[:5])
    t, dtype, op = case["tokens"], torch.float32 if case["dtype"] == "f32" else torch.bfloat16, case["op"]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    rng = np.random.default_rng([seed, 7])

    def normal(shape, std, dt=dtype):
        a = torch.empty(shape, dtype=dt, device=dev)
        return a.normal_(0.0, std, generator=g)

    st = {"case": dict(case), "layer": ex.make_layer(n, s, d, i, k, dtype)}
    st["x"] = normal((t, d), 1.0)
    std = 0.02 if d >= 1024 else 0.05
    st["w"] = [normal((n + s, i, d), std), normal((n + s, i, d), std), normal((n + s, d, i), std)]
    if case["router"]:  # the scores come from the router matrix
        st["w_router"] = normal((n, d), d ** -0.5)
        st["logits"] = torch.empty((t, n), dtype=torch.float32, device=dev)
    else:
        pop = torch.from_numpy(_popularity(case, rng).astype(np.float32)).to(dev)
        st["logits"] = normal((t, n), 1.0, torch.float32) + pop
    if op == "calibrate":
        st["out"] = [torch.empty(sh, dtype=dt, device=dev) for sh, dt in (
            ((n, n), torch.float32), ((n, n), torch.float32), ((n,), torch.float32), ((n,), torch.float32),
            ((n, n), torch.int32))]
        st["tables"] = ex.make_tables(*st["out"])
    else:
        st["tabs"] = [torch.from_numpy(a).to(dev) for a in _tables(n, rng)]
        st["tables"] = ex.make_tables(*st["tabs"])
        st["y"] = torch.empty((t, d), dtype=dtype, device=dev)
    if case["static"]:
        st["pool_t"] = [torch.empty(m, dtype=dt, device=dev) for m, dt in (
            (case["budget"], torch.int32), (n, torch.int32), (n, torch.float32))]
        st["pool"] = ex.exfold_static_pool_build(st["layer"], st["tables"], case["budget"], *st["pool_t"])
    st["ws"] = ex.alloc_workspace(st["layer"], t, case["budget"] if op == "prefill" else k, device=dev)
    return st


def run(st):
    c, layer, x, logits, ws = st["case"], st["layer"], st["x"], st["logits"], st["ws"]
    wg, wu, wd = st["w"]
    if c["op"] == "calibrate":
        ex.exfold_calibrate(layer, x, logits, wg, wu, wd, st["tables"], ws)
        return dict(zip(("S", "L", "h", "lnh", "n_obs"), st["out"]))
    y, tables, budget = st["y"], st["tables"], c["budget"]
    if c["op"] == "decode":
        if c["static"]:
            ex.exfold_moe_decode_static(layer, x, logits, wg, wu, wd, st["pool"], y, ws)
        elif c["router"]:
            ex.exfold_moe_decode_layer(layer, x, st["w_router"], wg, wu, wd, tables, budget, y, ws, logits)
        else:
            ex.exfold_moe_decode(layer, x, logits, wg, wu, wd, tables, budget, y, ws)
    elif c["guard"]:
        if c["router"]:
            ex.exfold_router_logits(layer, x, st["w_router"], logits, ws)
        ex.exfold_moe_prefill_ex(layer, x, logits, wg, wu, wd, tables, budget, y, ws, loss_threshold=0.99, rescale=True)
    elif c["router"]:
        ex.exfold_moe_prefill_layer(layer, x, st["w_router"], wg, wu, wd, tables, budget, y, ws, logits)
    else:
        ex.exfold_moe_prefill(layer, x, logits, wg, wu, wd, tables, budget, y, ws)
    return (y, logits) if c["router"] else y


# ------------------------------------------------------------------------------------------------ accounting
def _executed(c):
    """(experts whose weights are read, executed routed rows) of one call, from scores of the case's distribution."""
    n, k, t = c["experts"], c["top_k"], c["tokens"]
    rng = np.random.default_rng(11)
    sample = min(t, 2048)
    z = rng.standard_normal((sample, n)) + (0 if c["router"] else _popularity(c, rng)[None, :])
    _, L, h, lnh = _tables(n, rng)
    top = np.argsort(-z, axis=1)[:, :k]
    r = np.take_along_axis(z, top, 1)
    if c["op"] == "calibrate":
        kept = top
    elif c["op"] == "prefill":
        order = np.argsort(-(r + lnh[top]), axis=1)[:, :c["budget"]]
        kept = np.take_along_axis(top, order, 1)
    else:
        w = np.exp(r - r[:, :1])
        w /= w.sum(1, keepdims=True)
        score = np.zeros(n)
        np.add.at(score, top, w)
        union = np.flatnonzero(score) if not c["static"] else np.arange(n)
        rank = h if c["static"] else score * h
        pool = union[np.argsort(-rank[union])][:c["budget"]]
        target = np.where(np.isin(np.arange(n), pool), np.arange(n), pool[np.argmin(L[:, pool], axis=1)])
        kept = target[top]
    rows = sum(len(set(q)) for q in kept.tolist())
    hit = np.bincount(kept.ravel(), minlength=n)
    if t > sample:  # the rest of a long prompt reaches experts that the sample did not
        seen = np.where(hit > 0, 1.0, 0.0)
        p = 1.0 / (sample * k)
        touched = seen.sum() + (1.0 - seen).sum() * (1.0 - (1.0 - p) ** ((t - sample) * k))
        rows = rows * t // sample
    else:
        touched = np.count_nonzero(hit)
    return float(touched), int(rows)


def work(case):
    """Bytes and operations of one call that no implementation can do without: the weights of the experts that serve a
    token (and the shared expert's), x, the router scores and the result once each; 6 d I operations per executed row."""
    n, s, d, i, k = (case[f] for f in FIELDS[:5])
    t, el = case["tokens"], 4 if case["dtype"] == "f32" else 2
    touched, rows = _executed(case)
    if case["op"] == "calibrate":
        s = 0  # the shared expert is not calibrated
    flops = 6.0 * d * i * (rows + s * t)
    nbytes = (touched + s) * 3 * d * i * el + t * d * el + t * n * 4
    if case["op"] == "calibrate":  # inner products of every token's expert outputs; S, L, n_obs
        flops += t * k * (k + 1) / 2 * 2 * d
        nbytes += 3 * n * n * 4
    else:
        nbytes += t * d * el
    if case["router"]:
        flops += 2.0 * t * n * d
        nbytes += n * d * el
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Measured against the same path in 64-bit arithmetic (rel, max): fp32 layers 2.1e-7, 1.1e-6; calibration tables
    # 2.1e-4, 2.3e-3 (the diagonal and unobserved pairs are exact; the other scalars carry the bf16 rounding of H);
    # bf16 layers 2.9e-3, 1.6e-2 (H and the rows that are summed are bf16). About four times that is stated.
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 8e-6}
    if case["op"] == "calibrate":
        return {"rel": 2e-3, "max": 2e-2}
    return {"rel": 1e-2, "max": 6e-2}
