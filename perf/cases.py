"""Performance cases of the library: calls a user's program makes, through the package's public entry points.

Sizes are those of `workloads.CONFIGS` (the five benchmark configurations), of the sequence-length sweep, of the ragged
full-size tests and of the paper's own forward + backward sweep (12 heads, d = 64).  Inputs are synthetic, drawn on the GPU
with the distributions of `workloads.py`: "gaussian" (i.i.d. N(0,1)), "clustered" (64 centres per head, queries at three
times their centre: large entries for the hash to find, many equal bucket ids), "student_t" (3 degrees of freedom, clipped
at 20: heavy tails).

A case names its entry point: "forward" (device tensors), "train" (forward, then backward of its result: a training step's
two calls), "host" (host buffers in pinned memory, copies included)."""
import math

import torch

import paper_2310_05869_b200 as ha


def _case(entry, B, H, n, d, b, m, r, kind, causal=False, n0=0, n_k=0, dtype="bf16", option=""):
    return {"entry": entry, "B": B, "H": H, "n": n, "n_k": n_k or n, "d": d, "dtype": dtype, "b": b, "m": m, "r": r,
            "causal": causal, "n0": n0, "kind": kind, "option": option}


def listed():
    named = {
        # One small fp32 head: a unit test, a notebook, one decoder step of a prototype.  All latency.
        "fp32_1k": _case("forward", 1, 1, 1024, 64, 128, 128, 7, "gaussian", dtype="fp32"),
        # The short end of the sequence sweep: a layer at an ordinary context length; launches and the tail count.
        "sweep_4k": _case("forward", 1, 32, 4096, 64, 256, 256, 7, "clustered"),
        # A ChatGLM2-6B-32k-like layer at its full context.
        "layer_32k": _case("forward", 1, 32, 32768, 128, 256, 256, 7, "gaussian"),
        # The long end of the sweep, the paper's non-causal headline length.
        "sweep_131k": _case("forward", 1, 32, 131072, 64, 256, 256, 7, "clustered"),
        # The causal headline: recursion from 131072 rows down to exact leaves of 4096.
        "causal_131k": _case("forward", 1, 32, 131072, 64, 256, 256, 7, "gaussian", causal=True, n0=4096),
        # A batch of heavy-tailed causal layers; values of up to 20 need the split weights.
        "heavy_tail_16k": _case("forward", 4, 32, 16384, 128, 128, 512, 8, "student_t", causal=True, n0=2048, option="precise"),
        # A prompt of a length that nothing divides, few heads (one GPU's share of a layer split over several).
        "ragged_causal_100003": _case("forward", 1, 4, 100003, 64, 256, 256, 7, "gaussian", causal=True, n0=4096),
        # Cross attention, queries and keys of different number, columns sampled by value norms.
        "cross_50000x131072": _case("forward", 1, 4, 50000, 64, 256, 256, 7, "gaussian", n_k=131072, option="value_norms"),
        # The paper's forward + backward sweep: short end (12 heads) ...
        "train_4k": _case("train", 1, 12, 4096, 64, 256, 256, 7, "gaussian"),
        # ... a full-context layer with wide heads ...
        "train_32k": _case("train", 1, 32, 32768, 128, 256, 256, 7, "gaussian"),
        # ... and the causal headline length, the largest call of all.
        "train_causal_131k": _case("train", 1, 32, 131072, 64, 256, 256, 7, "gaussian", causal=True, n0=4096),
        # Inputs and results in host memory (activations offloaded between layers): the copies are part of the call.
        "host_32k": _case("host", 1, 8, 32768, 128, 256, 256, 7, "gaussian"),
    }
    return [dict(c, name=name) for name, c in named.items()]


_MAX_ROWS = 32 * 131072            # rows (B H n) of the largest listed case


def draw(rng):
    def span(lo, hi):              # log-uniform, both ends included
        return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))

    def heads(lo, hi, n):
        return max(1, min(span(lo, hi), _MAX_ROWS // n))

    family = rng.choice(["fp32", "sweep", "layer", "causal", "heavy", "cross", "train", "train_causal", "host"])
    if family == "fp32":
        return _case("forward", 1, rng.randint(1, 4), span(256, 4096), rng.choice([64, 128]), rng.choice([64, 128]), 128, 7,
                     "gaussian", dtype="fp32")
    if family == "sweep":
        n = span(4096, 131072)
        return _case("forward", 1, heads(8, 32, n), n, 64, 256, 256, 7, "clustered")
    if family == "layer":
        n = span(4096, 32768)
        return _case("forward", 1, heads(8, 32, n), n, 128, 256, 256, 7, "gaussian")
    if family == "causal":
        n = span(4096, 131072)
        return _case("forward", 1, heads(4, 32, n), n, 64, 256, 256, 7, "gaussian", causal=True, n0=4096)
    if family == "heavy":
        n = span(4096, 16384)
        return _case("forward", rng.randint(1, 4), heads(8, 32, n), n, 128, 128, 512, 8, "student_t", causal=True, n0=2048,
                     option="precise")
    if family == "cross":
        return _case("forward", 1, rng.randint(2, 8), span(8192, 65536), 64, 256, 256, 7, "gaussian", n_k=span(16384, 131072),
                     option="value_norms")
    if family == "train":
        n = span(4096, 32768)
        return _case("train", 1, heads(8, 32, n), n, rng.choice([64, 128]), 256, 256, 7, "gaussian")
    if family == "train_causal":
        leaf, halvings = rng.randint(2049, 4096), rng.randint(0, 5)     # the backward pass takes lengths that the halvings divide
        n = leaf << halvings
        return _case("train", 1, heads(4, 32, n), n, 64, 256, 256, 7, "gaussian", causal=True, n0=4096)
    n = span(1024, 8192) * 4           # host buffers go through in groups of heads: every head's rows start on 16 bytes
    return _case("host", 1, heads(4, 16, n), n, 128, 256, 256, 7, "gaussian")


def _inputs(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, H, d, kind = c["B"], c["H"], c["d"], c["kind"]
    dtype = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    def one(rows, side):
        if kind == "student_t":
            chi2 = sum(normal(B, H, rows, d).square_() for _ in range(3))
            return (normal(B, H, rows, d) / (chi2 / 3).sqrt_()).clamp_(-20.0, 20.0).to(dtype)
        if kind == "clustered" and side < 2:
            pick = torch.randint(0, 64, (B * H, rows), generator=gen, device="cuda")
            base = (3.0 if side == 0 else 1.0) * centres
            rows_of = torch.gather(base, 1, pick[..., None].expand(-1, -1, d)).view(B, H, rows, d)
            return (rows_of + 0.1 * normal(B, H, rows, d)).to(dtype)
        return normal(B, H, rows, d).to(dtype)

    centres = normal(B * H, 64, d)
    return [one(c["n"], 0), one(c["n_k"], 1), one(c["n_k"], 2)]


def prepare(case, seed):
    q, k, v = _inputs(case, seed)
    args = (case["b"], case["m"], case["r"])
    kw = {"causal": case["causal"], "n0": case["n0"], "seed": 0}
    state = {"entry": case["entry"], "q": q, "k": k, "v": v, "args": args, "kw": kw}
    if case["entry"] == "forward":
        if case["option"] == "precise":
            kw["precise"] = True
        elif case["option"] == "value_norms":
            kw["value_norm_sampling"] = True
    elif case["entry"] == "train":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + (1 << 40))
        state["dout"] = torch.randn(q.shape, generator=gen, device="cuda").to(q.dtype)
    else:
        for name in ("q", "k", "v"):
            pinned = torch.empty(state[name].shape, dtype=state[name].dtype, pin_memory=True)
            pinned.copy_(state[name])
            state[name] = pinned
        state["out"] = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
        state["lse"] = torch.empty(q.shape[:3], dtype=torch.float32, pin_memory=True)
    return state


def run(state):
    q, k, v = state["q"], state["k"], state["v"]
    if state["entry"] == "host":
        ha.forward_host(q, k, v, state["out"], state["lse"], *state["args"], **state["kw"])
        return {"out": state["out"], "lse": state["lse"]}
    out, lse = ha.forward(q, k, v, *state["args"], **state["kw"])
    if state["entry"] == "forward":
        return {"out": out, "lse": lse}
    dq, dk, dv = ha.backward(q, k, v, out, lse, state["dout"], *state["args"], **state["kw"])
    return {"out": out, "lse": lse, "dq": dq, "dk": dk, "dv": dv}


def _scores(c):
    """Query-key pairs one head evaluates (the method's own count: blocks, sampled columns, causal leaves)."""
    n, n_k, b, m = c["n"], c["n_k"], c["b"], c["m"]

    def node(n_q, keys):           # every query meets the keys of its block and the samples, or all keys of a small node
        return n_q * (b + m) if b < keys else n_q * keys

    if not c["causal"]:
        return node(n, n_k)
    levels = 0
    while -(-n >> levels) > c["n0"]:
        levels += 1
    leaf = -(-n >> levels)
    total = 0
    for i in range(1 << levels):
        rows = max(0, min(leaf, n - i * leaf))
        total += rows * (rows + 1) // 2
    for level in range(levels):
        s = (leaf << levels) >> (level + 1)
        for j in range(1 << level):
            total += node(max(0, min(s, n - (2 * j + 1) * s)), s)
    return total


def work(case):
    G, d, e = case["B"] * case["H"], case["d"], 4 if case["dtype"] == "fp32" else 2
    rows, rows_k = G * case["n"], G * case["n_k"]
    nbytes = (2 * rows + 2 * rows_k) * d * e + 4 * rows                       # q, out; k, v; lse
    flops = 4.0 * d * G * _scores(case) + 2.0 * d * case["r"] * (rows + rows_k)  # two products per pair; hashing
    if case["entry"] == "train":
        nbytes += 2 * rows * d * e + 2 * rows_k * d * e                       # dout, dq; dk, dv
        flops += 10.0 * d * G * _scores(case)                                 # five products per pair
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Softmax weights and outputs are rounded to bf16 (2^-9 each, partial results of the causal recursion once more);
    # gradients carry one more rounded factor.  fp32 calls keep fp32 logits and outputs, weights and values in bf16.
    if case["entry"] == "train":
        return {"rel": 1e-2}
    if case["dtype"] == "fp32":
        return {"rel": 4e-3}
    return {"rel": 6e-3}
