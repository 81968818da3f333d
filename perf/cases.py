"""The workloads whose speed this library is measured by, as a user's program calls it.

Four kinds of pass, all through the public Python entry points:

  step      compress(K, V), then attend(Q, ...) over the coreset: one layer of a prompt.  With ``ragged`` the
            sequence has any length and keeps its first and last 32 rows exactly (compress_ragged).
  decode    attend() of one or a few new tokens over a coreset that is already there.
  stream    a generation from its first token on: a Stream over K and V and T tokens through it.
  prefill   express_prefill(): every token of a prompt over the Express cache as of its own position.

Inputs are drawn on the GPU by the recipes of the package's ``workloads`` module (clustered, low-rank, rotary and
heavy-tailed keys).
"""
import functools
import math

import torch

import paper_2606_10944_b200 as elm

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "e4m3": torch.float8_e4m3fn}
ITEM = {"f32": 4, "bf16": 2, "e4m3": 1}
KEPT_ROWS = 32                                  # sink rows and window rows of the ragged steps


def listed():
    return [
        # One new token of a long-context chat over the coreset of its prompt: the latency of a single call.
        dict(name="decode_1x2048", kind="decode", batch=1, q_heads=32, kv_heads=8, n=131072, n_q=1, d=128,
             dtype="bf16", n_core=2048, recipe="mixture64_t3"),
        # A batch of four sequences, each over a multi-level cache (unequal weights, odd length).
        dict(name="decode_4x5193", kind="decode", batch=4, q_heads=32, kv_heads=8, n=32768, n_q=1, d=128,
             dtype="bf16", n_core=5193, recipe="rope"),
        # A generation of 2496 tokens (half of them a prompt known beforehand) with the cache thinned as it grows.
        dict(name="stream_2496", kind="stream", batch=1, q_heads=32, kv_heads=8, n=2496, d=128, dtype="bf16",
             log2_nout=8, mbar=6, known=1248, recipe="mixture64_t3"),
        # The package's five workloads: the smallest step (launches and latency) ...
        dict(name="step_1024_f32", kind="step", batch=1, q_heads=1, kv_heads=1, n=1024, n_q=1024, d=64, dtype="f32",
             log2_nout=5, m=5, ragged=False, recipe="iid"),
        # ... a batch of short fp32 sequences (an encoder layer) ...
        dict(name="step_4x1024_f32", kind="step", batch=4, q_heads=12, kv_heads=12, n=1024, n_q=1024, d=64,
             dtype="f32", log2_nout=7, m=3, ragged=False, recipe="mixture16"),
        # ... ordinary prompts ...
        dict(name="step_2x8192", kind="step", batch=2, q_heads=32, kv_heads=32, n=8192, n_q=8192, d=128, dtype="bf16",
             log2_nout=8, m=5, ragged=False, recipe="lowrank8"),
        dict(name="step_32768", kind="step", batch=1, q_heads=32, kv_heads=32, n=32768, n_q=32768, d=128,
             dtype="bf16", log2_nout=10, m=5, ragged=False, recipe="rope"),
        # ... and the long-context prompt with grouped queries, in both storage types it is kept in.
        dict(name="step_131072", kind="step", batch=1, q_heads=32, kv_heads=8, n=131072, n_q=131072, d=128,
             dtype="bf16", log2_nout=11, m=6, ragged=False, recipe="mixture64_t3"),
        dict(name="step_131072_e4m3", kind="step", batch=1, q_heads=32, kv_heads=8, n=131072, n_q=131072, d=128,
             dtype="e4m3", log2_nout=11, m=6, ragged=False, recipe="mixture64_t3"),
        # A prompt of no special length: sink and window rows kept, leftovers in every level.
        dict(name="step_121673_ragged", kind="step", batch=1, q_heads=32, kv_heads=8, n=121673, n_q=121673, d=128,
             dtype="bf16", log2_nout=11, m=6, ragged=True, recipe="mixture64_t3"),
        # Causal prefill: a short prompt, and the long one at the published setting of 512 cache points.
        dict(name="prefill_16384", kind="prefill", batch=1, q_heads=32, kv_heads=8, n=16384, n_q=16384, d=128,
             dtype="bf16", log2_nout=8, mbar=6, recipe="rope"),
        dict(name="prefill_131072", kind="prefill", batch=1, q_heads=32, kv_heads=8, n=131072, n_q=131072, d=128,
             dtype="bf16", log2_nout=9, mbar=7, recipe="mixture64_t3"),
    ]


def draw(rng):
    """One more case of the same ranges; none costs more than the longest listed step."""
    kind = rng.choice(["step", "step", "step", "ragged", "decode", "decode", "stream", "prefill"])
    kv_heads = rng.choice([1, 2, 4, 8])
    rep = rng.choice([1, 2, 4])
    d = rng.choice([64, 128, 128])
    recipe = rng.choice(["iid", "mixture16", "lowrank8", "rope", "mixture64_t3"])
    c = dict(batch=1, q_heads=kv_heads * rep, kv_heads=kv_heads, d=d, dtype="bf16", recipe=recipe)
    if kind == "step":
        k = rng.randint(10, 17)
        c["dtype"] = rng.choice(["f32", "bf16"]) if k <= 12 else "bf16"
        if d == 128 and k >= 13 and rng.random() < 0.25:
            c["dtype"] = "e4m3"
        g = rng.randint(0, 2) if k <= 12 else rng.randint(1, 3)
        if k <= 13:
            c["batch"] = rng.randint(1, 4)
        n = 1 << k
        c.update(kind="step", n=n, n_q=rng.randint(max(64, n // 4), n), log2_nout=k // 2 + g,
                 m=k - (k // 2 + g), ragged=False)
    elif kind == "ragged":
        n = int(math.exp(rng.uniform(math.log(3000), math.log(121672)))) // 8 * 8 + rng.randint(0, 1)
        k = max(12, (n - 2 * KEPT_ROWS - 1).bit_length())           # n_out 2^m >= the middle rows
        g = rng.randint(1, 3 if n < 50000 else 2)                   # (several times n_out entries are left at the end)
        c.update(kind="step", n=n, n_q=n, log2_nout=k // 2 + g, m=k - (k // 2 + g), ragged=True)
    elif kind == "decode":
        n_core = int(math.exp(rng.uniform(math.log(100), math.log(12288))))
        c["batch"] = rng.randint(1, 8)
        c["n_q"] = rng.randint(1, 2)
        c["dtype"] = rng.choice(["f32", "bf16", "bf16"])
        c.update(kind="decode", n=rng.randint(n_core, 32768), n_core=n_core)
    elif kind == "stream":
        log2_nout = rng.randint(6, 9)
        n = 8 * rng.randint(40, 375)
        c.update(kind="stream", n=n, log2_nout=log2_nout, mbar=log2_nout - 2, known=rng.randint(0, n))
    else:
        log2_nout = rng.randint(7, 10)
        rounds = rng.randint(2, 4 if log2_nout < 9 else 3)
        n = 4 ** rounds << log2_nout
        c.update(kind="prefill", n=n, n_q=n, log2_nout=log2_nout, mbar=rng.randint(2, log2_nout - 2))
    return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _keys_values(g, recipe, heads, n, d):
    """float32 K, V [heads, n, d] (heads drawn from the same recipe, each with its own parameters)."""
    if recipe == "iid":
        std = d ** -0.25
        return _randn(g, heads, n, d) * std, _randn(g, heads, n, d) * std
    if recipe == "lowrank8":
        def factor():
            w = _randn(g, heads, 8, d) * 8 ** -0.5
            return _randn(g, heads, n, 8) @ w + _randn(g, heads, n, d) * 0.1 ** 0.5
        return factor(), factor()
    if recipe == "rope":
        x = _randn(g, heads, n, d)
        ang = (torch.arange(n, device="cuda", dtype=torch.float64)[:, None]
               * 10000.0 ** (-2.0 * torch.arange(d // 2, device="cuda", dtype=torch.float64) / d))
        c, s = ang.cos().float(), ang.sin().float()
        k = torch.empty_like(x)
        k[..., 0::2] = x[..., 0::2] * c - x[..., 1::2] * s
        k[..., 1::2] = x[..., 0::2] * s + x[..., 1::2] * c
        return k, _randn(g, heads, n, d)
    parts = 16 if recipe == "mixture16" else 64
    mu = _randn(g, heads, parts, d)
    comp = torch.randint(parts, (heads, n, 1), generator=g, device="cuda")
    k = torch.gather(mu, 1, comp.expand(-1, -1, d)) + _randn(g, heads, n, d) * 0.3
    if recipe == "mixture64_t3":
        # Student-t norms with 3 degrees of freedom: normal over the root of a chi-square over 3
        k *= (_randn(g, heads, n) / (_randn(g, heads, n, 3).square().sum(-1) / 3).sqrt()).abs()[..., None]
    return k, _randn(g, heads, n, d)


def _store(x, dtype):
    if dtype == "e4m3":
        x = x.clamp(-448.0, 448.0)              # the largest finite E4M3 value
    return x.to(DTYPES[dtype])


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": c, "seed": seed}
    k, v = _keys_values(g, c["recipe"], c["batch"] * c["kv_heads"], c["n"], c["d"])
    shape = (c["batch"], c["kv_heads"], c["n"], c["d"])
    s["K"], s["V"] = _store(k, c["dtype"]).view(shape), _store(v, c["dtype"]).view(shape)
    del k, v
    q_std = c["d"] ** -0.25
    if c["kind"] == "stream":
        s["Q"] = _store(_randn(g, c["n"], c["batch"], c["q_heads"], 1, c["d"]) * q_std, c["dtype"])
    else:
        s["Q"] = _store(_randn(g, c["batch"], c["q_heads"], c["n_q"], c["d"]) * q_std, c["dtype"])
    if c["kind"] == "decode":
        # a coreset as compression leaves it: one row of every stretch of the sequence, weights that are powers of
        # two over the length
        n, nc = c["n"], c["n_core"]
        edge = (torch.arange(nc + 1, device="cuda") * n) // nc
        u = torch.rand(c["batch"], c["kv_heads"], nc, generator=g, device="cuda")
        width = edge[1:] - edge[:-1]
        s["idx"] = torch.minimum(edge[:-1] + (u * width).long(), edge[1:] - 1).to(torch.int32)
        level = (torch.arange(nc, device="cuda") * 6) // nc
        s["w"] = (2.0 ** level.float() / n).expand(c["batch"], c["kv_heads"], nc).contiguous()
    return s


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def run(state):
    c = state["case"]
    Q, K, V = state["Q"], state["K"], state["V"]
    if c["kind"] == "decode":
        return elm.attend(Q, K, V, state["idx"], state["w"])
    if c["kind"] == "stream":
        stream = elm.Stream(K, V, c["q_heads"], c["log2_nout"], c["mbar"], seed=state["seed"], n_known=c["known"])
        out = stream.steps(Q)
        idx, w = stream.cache()
        return out, idx, w
    if c["kind"] == "prefill":
        return elm.express_prefill(Q, K, V, c["log2_nout"], c["mbar"], seed=state["seed"])
    if c["ragged"]:
        idx, w = elm.compress_ragged(K, V, c["log2_nout"], c["m"], KEPT_ROWS, KEPT_ROWS, seed=state["seed"])
    else:
        idx, w = elm.compress(K, V, c["log2_nout"], c["m"], seed=state["seed"])
    return elm.attend(Q, K, V, idx, w), idx, w


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _express_counts(n, log2_nout, mbar):
    """(cache entries seen, summed over the n tokens of a run; sum over its Halve calls of points squared)."""
    n_out = 1 << log2_nout
    m = q = b = ell = t = n_e = 0
    level = [0] * 40
    seen = halved = 0
    while t < n:
        # a token sees E, every level, and itself
        seen += n_e + sum(level[:q + 1]) + 1
        t += 1
        if t <= n_out:
            n_e += 1
            continue
        ell += 1
        if ell % (1 << (m - q)) == 0:                       # one point kept per stratum
            level[0] += 1
            for i in range(q):
                points = ((n_out << q) << i) >> (2 * (q - 1))
                if level[i] < points:
                    break
                halved += points * points
                level[i + 1] += points // 2
                level[i] = 0
        if ell == n_out << m:
            n_e += level[q]
            level[q], ell, b = 0, 0, b + 1
        if t == 4 * (n_out << m):
            halved += (4 * n_out) ** 2 + (2 * n_out) ** 2
            n_e, m, b = n_out, m + 2, 0
        if ell == 0:
            q = min(m, mbar)
    return seen, halved


def work(case):
    c = case
    item = ITEM[c["dtype"]]
    out_item = 2 if c["dtype"] == "e4m3" else item
    problems, heads, d, n = c["batch"] * c["kv_heads"], c["batch"] * c["q_heads"], c["d"], c["n"]
    n_q = n if c["kind"] == "stream" else c["n_q"]
    bytes_qo = heads * n_q * d * (item + out_item)
    if c["kind"] == "decode":
        return {"bytes": bytes_qo + problems * c["n_core"] * (2 * d * item + 8), "flops": 4.0 * d * heads * n_q * c["n_core"]}
    bytes_kv = 2 * problems * n * d * item
    if c["kind"] in ("stream", "prefill"):
        seen, halved = _express_counts(n, c["log2_nout"], c["mbar"])
        # a Halve call of s points: keys and values against each other, one triangle of each product
        return {"bytes": bytes_qo + bytes_kv, "flops": 4.0 * d * heads * seen + 2.0 * d * problems * halved}
    n_out = 1 << c["log2_nout"]
    if c["ragged"]:
        a, n_core, halved = n - 2 * KEPT_ROWS, 2 * KEPT_ROWS, 0
        for i in range(c["m"]):
            points = (n_out << (i + 2)) >> c["m"]
            calls = a // points
            halved += calls * points * points
            n_core += a - calls * points
            a = calls * points // 2
        n_core += a
    else:
        n_core, halved = n_out, 4 * n_out * n_out * c["m"]
    bytes_core = problems * n_core * 8
    return {"bytes": bytes_qo + bytes_kv + bytes_core,
            "flops": 4.0 * d * heads * n_q * n_core + 2.0 * d * problems * halved}


def tolerance(case):
    # Measured against the library's fp64 mode on the same inputs: outputs 2.5e-7 (fp32 storage) and 1.2e-3 .. 2.6e-3
    # (bf16 O: its rounding, and that of the probabilities); the limits are about four times that, with room for
    # longer lists than the measured ones in fp32.  The selected rows were the same in every case; a decision can
    # differ only where a uniform falls within rounding distance of its probability.  The weights are powers of two
    # over a count.
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "differ": 0.01}
    return {"rel": 1e-2, "differ": 0.01}
