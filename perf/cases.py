"""The work this library is measured on: windowed attention calls as a serving program makes them.

Every case is one call pattern through the public binding (`paper_2608_02947_b200`): a prefill of a prompt, rows
appended to a context, a split-precision prefill, a decode step on one of the K-cache layouts, or a whole layer
step (RoPE, prefill that writes the decode cache, decode on it).  Shapes are the attention layers the repository
is configured for (14/2 heads of 64; 24/8 and 28/4 heads of 128) and the small 2/1-head shape of its tests.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a program holds before the
call, run() is one pass, work() is what the pass cannot do without, tolerance() what two correct implementations
may differ by.
"""
import math

import torch

import paper_2608_02947_b200 as atf

# attention layers: query heads, KV heads, head dimension, RoPE base, llama3 frequency scaling
LAYERS = {
    "small": (2, 1, 64, 1e6, False),
    "h14d64": (14, 2, 64, 1e6, False),
    "h24d128": (24, 8, 128, 5e5, True),
    "h28d128": (28, 4, 128, 1e7, False),
}
K_WINDOW = 2.0


def listed():
    return [
        # One decode step of a short chat turn on the small layer, default (row) cache: pure latency.
        {"name": "decode rows d64 L1000", "op": "decode", "layer": "h14d64", "B": 1, "L": 1000, "cache": "rows", "mode": "exact"},
        # A decode step after a medium prompt on the cache the prefill writes, LSE asked for (a later merge needs it).
        {"name": "decode groups L8201", "op": "decode", "layer": "h24d128", "B": 1, "L": 8201, "cache": "groups", "mode": "exact"},
        # The plain atf_decode call (row cache, no options) at an ordinary long context, two sequences.
        {"name": "decode rows B2 L32768", "op": "decode", "layer": "h24d128", "B": 2, "L": 32768, "cache": "rows", "mode": "exact"},
        # Batched serving: eight sequences on group-major caches, coarse granularity.
        {"name": "decode groups B8 L32768 coarse", "op": "decode", "layer": "h24d128", "B": 8, "L": 32768, "cache": "groups", "mode": "coarse"},
        # A position-independent cache that is rotated as it is read (prefix reuse) at 128K.
        {"name": "decode unrotated L131072", "op": "decode", "layer": "h24d128", "B": 1, "L": 131072, "cache": "unrotated", "mode": "exact"},
        # One sequence at a million tokens: the largest decode step.
        {"name": "decode groups L1048576", "op": "decode", "layer": "h28d128", "B": 1, "L": 1048576, "cache": "groups", "mode": "exact"},
        # A short prompt on the small layer: launches and latency.
        {"name": "prefill small N2048", "op": "prefill", "layer": "small", "B": 1, "N": 2048, "Nq": 2048, "mode": "exact"},
        # A whole layer step at an ordinary prompt length: RoPE of Q and K, prefill that writes the decode cache, one decode.
        {"name": "layer step N8192", "op": "layer", "layer": "h24d128", "B": 1, "N": 8192, "mode": "exact"},
        # A long prompt at head dimension 64.
        {"name": "prefill d64 N32768", "op": "prefill", "layer": "h14d64", "B": 1, "N": 32768, "Nq": 32768, "mode": "exact"},
        # A chunk of a chunked prefill: 4000 rows appended to a ragged 61003-key context, coarse granularity.
        {"name": "chunk 4000 of N61003 coarse", "op": "prefill", "layer": "h24d128", "B": 1, "N": 61003, "Nq": 4000, "mode": "coarse"},
        # Scores of more than bf16 input precision, ragged length.
        {"name": "split N10001", "op": "split", "layer": "h24d128", "B": 1, "N": 10001, "Nq": 10001, "mode": "exact"},
        # The headline: a 128K prompt in one shot.
        {"name": "prefill N131072", "op": "prefill", "layer": "h24d128", "B": 1, "N": 131072, "Nq": 131072, "mode": "exact"},
    ]


def _log_size(rng, lo, hi):
    """A length spread over the logarithm of [lo, hi]; every third one a multiple of 128, the others as they fall."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.randrange(3) == 0:
        n = max(128, n // 128 * 128)
    return min(max(n, lo), hi)


def draw(rng):
    op = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "chunk", "layer", "split"])
    mode = rng.choice(["exact", "exact", "exact", "coarse", "full"])  # "full": no table, every term
    if op == "decode":
        layer = rng.choice(["h14d64", "h24d128", "h24d128", "h28d128"])
        cache = rng.choice(["rows", "groups", "groups", "unrotated"])
        B = rng.choice([1, 1, 2, 4, 8])
        return {"op": op, "layer": layer, "B": B, "L": _log_size(rng, 300, 1048576 // B), "cache": cache, "mode": mode}
    layer = rng.choice(["small", "h14d64", "h24d128", "h24d128"])
    B = rng.choice([1, 1, 1, 2])
    if op == "layer":
        return {"op": op, "layer": layer, "B": B, "N": _log_size(rng, 300, 65536 // B), "mode": mode}
    if op == "chunk":
        N = _log_size(rng, 1024, 131072 // B)
        return {"op": "prefill", "layer": layer, "B": B, "N": N, "Nq": _log_size(rng, 128, min(N, 16384)), "mode": mode}
    N = _log_size(rng, 300, (65536 if op == "split" else 98304) // B)
    case = {"op": op, "layer": layer, "B": B, "N": N, "Nq": N, "mode": mode}
    if op == "prefill" and rng.randrange(5) == 0:
        # outlier channels: the four lowest-frequency pairs of Q and K times 8 (logits in the hundreds)
        case["outlier"] = True
    return case


def _length(case):
    return case["L"] if case["op"] == "decode" else case["N"]


def _window(case):
    """(window widths or None for full attention, angular frequencies)"""
    _, _, d, base, scaled = LAYERS[case["layer"]]
    W, theta = atf.atf_window_table(base, d, K_WINDOW, _length(case), atf.llama3_scaling() if scaled else None)
    return (None if case["mode"] == "full" else W), theta


def _inputs(case, seed):
    """What the case draws: queries, keys and values before any rotation (a decode's are what its cache holds)."""
    Hq, Hkv, d, _, _ = LAYERS[case["layer"]]
    B, N = case["B"], _length(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(shape, dtype=torch.bfloat16):
        # head by head: the fp32 draws of a long prompt need not be on the card together
        out = torch.empty(shape, dtype=dtype, device="cuda")
        for b in range(shape[0]):
            for h in range(shape[1]):
                out[b, h] = torch.randn(shape[2:], generator=gen, dtype=torch.float32, device="cuda")
        return out

    if case["op"] == "decode":
        # keys and values of the context; the query has been rotated by the program
        K = normal((B, Hkv, N, d))
        return normal((B, Hq, d)), K, normal((B, Hkv, N, d))
    kind = torch.float32 if case["op"] == "split" else torch.bfloat16
    Q, K, V = normal((B, Hq, case.get("Nq", N), d), kind), normal((B, Hkv, N, d), kind), normal((B, Hkv, N, d))
    if case.get("outlier"):
        h = d // 2
        for t in (Q, K):
            t[..., h - 4:h] *= 8
            t[..., d - 4:] *= 8
    return Q, K, V


def prepare(case, seed):
    _, Hkv, d, _, _ = LAYERS[case["layer"]]
    B, N = case["B"], _length(case)
    W, theta = _window(case)
    Q, K, V = _inputs(case, seed)
    state = {"case": case, "theta": theta, "V": V,
             "table": None if W is None else atf.WindowTable(W),
             "mode": atf.ATF_MODE_COARSE if case["mode"] == "coarse" else atf.ATF_MODE_EXACT}
    if case["op"] == "decode":
        state["q"] = Q
        if case["cache"] == "rows":
            state["K"] = K
        else:
            # a serving cache has room for tokens to come
            state["K"] = atf.atf_kcache_pack(K, Kg=atf.new_kcache_groups(B, Hkv, N + 512, d, "cuda"))
            if case["cache"] == "unrotated":
                state["tables"] = atf.atf_rope_tables(theta, d, N + 512)
        return state
    if case["op"] == "layer":
        # fresh projections: the step itself rotates them
        state["cache"] = atf.new_kcache_groups(B, Hkv, N + 512, d, "cuda")
    else:
        rope = atf.atf_rope_f32 if case["op"] == "split" else atf.atf_rope
        rope(Q, theta, pos0=N - Q.shape[2])
        rope(K, theta)
    state["Q"], state["K"] = Q, K
    return state


def run(state):
    case, table, mode = state["case"], state["table"], state["mode"]
    if case["op"] == "decode":
        if case["cache"] == "rows":
            return atf.atf_decode(state["q"], state["K"], state["V"], table=table, mode=mode)
        return atf.atf_decode(state["q"], state["K"], state["V"], table=table, mode=mode, return_lse=True,
                              rope_tables=state.get("tables"))
    if case["op"] == "layer":
        Q, K, V, cache = state["Q"], state["K"], state["V"], state["cache"]
        atf.atf_rope(Q, state["theta"])
        atf.atf_rope(K, state["theta"])
        O, lse = atf.atf_prefill(Q, K, V, table=table, mode=mode, kcache_groups=cache)
        o = atf.atf_decode(Q[:, :, -1].contiguous(), cache, V, table=table, mode=mode)
        return O, lse, o, cache
    if case["op"] == "split":
        return atf.atf_prefill_split(state["Q"], state["K"], state["V"], table=table, mode=mode)
    return atf.atf_prefill(state["Q"], state["K"], state["V"], table=table, mode=mode)


def _kept_terms(W, n0, n1):
    """Sum over rows n0..n1-1 and pairs of min(W_r, n) + 1: the (cell, pair) terms of one head."""
    total = 0
    for w in W:
        w = int(w)
        a, b = min(n0, w), min(n1, w)                       # rows below the width keep n + 1 terms
        total += (b * (b + 1) - a * (a + 1)) // 2
        total += (max(n1, w) - max(n0, w)) * (w + 1)        # the others w + 1
    return total


def work(case):
    Hq, Hkv, d, _, _ = LAYERS[case["layer"]]
    B, N = case["B"], _length(case)
    W, _ = _window(case)
    W = [N] * (d // 2) if W is None else W.tolist()
    if case["op"] == "decode":
        live = sum(min(int(w) + 1, N) for w in W)           # live (key, pair) terms of the row
        k_bytes = 4 * live if case["cache"] != "rows" else 2 * N * d
        return {"bytes": B * (Hkv * (k_bytes + 2 * N * d) + 2 * 2 * Hq * d), "flops": B * Hq * (4 * live + 2 * N * d)}
    Nq = case.get("Nq", N)
    cells = Nq * (N - Nq) + Nq * (Nq + 1) // 2
    flops = B * Hq * (4 * _kept_terms(W, N - Nq, N) + 2 * d * cells)
    size = 4 if case["op"] == "split" else 2
    moved = B * (Hq * Nq * (d * (size + 2) + 4) + Hkv * N * d * (size + 2))
    if case["op"] == "split":
        flops += 2 * B * Hq * 4 * _kept_terms(W, N - Nq, N)  # three products for every score term
    if case["op"] == "layer":
        # Q and K are read and written by the rotation, the cache is written, then the decode step
        moved += B * (Hq * N * d * 4 + Hkv * N * d * 4 + Hkv * N * d * 2)
        step = work({"op": "decode", "layer": case["layer"], "B": B, "L": N, "cache": "groups", "mode": case["mode"]})
        moved, flops = moved + step["bytes"], flops + step["flops"]
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # P is rounded to bf16 before the product with V and O once at the end.  Measured against the definition in fp64 on
    # prompts of 4000 to 8000 tokens: 2.1e-3 (split precision, d = 128) to 2.4e-3 (decode) in the 2-norm, largest element
    # 0.025 of the output's root mean square; LSE 4e-7.  Four times that.
    return {"rel": 9e-3, "max": 0.1}


def _frequencies(case):
    """Angular frequencies and window widths of the layer, from their formulas."""
    _, _, d, base, scaled = LAYERS[case["layer"]]
    N, theta, W = _length(case), [], []
    for r in range(d // 2):
        f = base ** (-2.0 * r / d)
        if scaled:  # llama3 rule: factor 32, low 1, high 4, original context 8192
            lam = 2.0 * math.pi / f
            if lam > 8192.0:
                f /= 32.0
            elif lam >= 8192.0 / 4.0:
                t = (8192.0 / lam - 1.0) / 3.0
                f = (1.0 - t) * f / 32.0 + t * f
        w = K_WINDOW * (2.0 * math.pi / f)
        theta.append(f)
        W.append(int(w) if case["mode"] != "full" and w < N else N)
    if case["mode"] == "coarse":  # groups of eight pairs live as long as their widest window
        W = [W[r // 8 * 8 + 7] for r in range(d // 2)]
    return torch.tensor(theta, dtype=torch.float64, device="cuda"), W


def _rotated(X, theta, pos0):
    """Half-split rotation in 64 bits, rounded to what X holds (that is what attention is given)."""
    h = X.shape[-1] // 2
    out = torch.empty_like(X)
    ang = torch.arange(pos0, pos0 + X.shape[-2], dtype=torch.float64, device="cuda")[:, None] * theta
    c, s = ang.cos(), ang.sin()
    for b in range(X.shape[0]):
        for i in range(X.shape[1]):
            x, y = X[b, i, :, :h].double(), X[b, i, :, h:].double()
            out[b, i, :, :h], out[b, i, :, h:] = (x * c - y * s).to(X.dtype), (y * c + x * s).to(X.dtype)
    return out


def _attend(Q, K, V, W, n0, coarse):
    """One (batch, KV head) in 64 bits: rows n0.. of the heads Q [g, Nq, d] on keys K, V [N, d]; O and LSE."""
    g, Nq, d = Q.shape
    h, blk = d // 2, 512
    O = torch.empty((g, Nq, d), dtype=torch.float64, device="cuda")
    lse = torch.empty((g, Nq), dtype=torch.float64, device="cuda")
    K, V = K.double(), V.double()
    a = n0
    while a < n0 + Nq:
        b = min(a // blk * blk + blk, n0 + Nq)
        q = Q[:, a - n0:b - n0].double() / math.sqrt(d)
        S = torch.full((g, b - a, b), -math.inf, dtype=torch.float64, device="cuda")
        n = torch.arange(a, b, device="cuda")[:, None]
        for m0 in range(0, b, blk):
            m1 = min(m0 + blk, b)
            m = torch.arange(m0, m1, device="cuda")
            z = n - m
            # coarse: what is live is decided for a whole 128 x 128 tile, at its nearest cell
            tiles = n // 128 - m // 128
            far = torch.where(tiles > 0, tiles * 128 - 127, 0) if coarse else z
            lo, hi = int(far.min()), int(far.max())
            every = [r for r in range(h) if W[r] >= hi]
            dims = every + [r + h for r in every]
            s = q[..., dims] @ K[m0:m1][:, dims].T if dims else torch.zeros((g, b - a, m1 - m0), dtype=torch.float64, device="cuda")
            for r in range(h):
                if lo <= W[r] < hi:
                    s += (q[..., [r, r + h]] @ K[m0:m1][:, [r, r + h]].T) * (far <= W[r])
            S[..., m0:m1] = torch.where((z >= 0) & (far <= max(W)), s, -math.inf)
        lse[:, a - n0:b - n0] = torch.logsumexp(S, -1)
        O[:, a - n0:b - n0] = torch.softmax(S, -1) @ V[:b]
        a = b
    return O, lse


def exact(case, seed):
    """What run() returns, in 64 bits; None where that would take too long (and for the cache, which is a copy)."""
    Hq, Hkv, d, _, _ = LAYERS[case["layer"]]
    B, N, g = case["B"], _length(case), Hq // Hkv
    Nq = 1 if case["op"] == "decode" else case.get("Nq", N)
    if B * Hq * (Nq * (N - Nq) + Nq * (Nq + 1) // 2) > 2e10:
        return None
    theta, W = _frequencies(case)
    Q, K, V = _inputs(case, seed)
    coarse = case["mode"] == "coarse"
    if case["op"] == "decode":
        Q = Q[:, :, None]
        if case["cache"] == "unrotated":
            K = _rotated(K, theta, 0)
    else:
        Q, K = _rotated(Q, theta, N - Nq), _rotated(K, theta, 0)

    def attention(q, n0, tiles):
        O = torch.empty(q.shape, dtype=torch.float64, device="cuda")
        lse = torch.empty(q.shape[:3], dtype=torch.float64, device="cuda")
        for b in range(B):
            for k in range(Hkv):
                O[b, k * g:(k + 1) * g], lse[b, k * g:(k + 1) * g] = _attend(q[b, k * g:(k + 1) * g], K[b, k], V[b, k], W, n0, tiles)
        return O, lse

    if case["op"] == "decode":
        O, lse = attention(Q, N - 1, False)
        return O[:, :, 0] if case["cache"] == "rows" else (O[:, :, 0], lse[:, :, 0])
    O, lse = attention(Q, N - Nq, coarse)
    if case["op"] == "layer":
        return O, lse, attention(Q[:, :, -1:], N - 1, False)[0][:, :, 0], None
    return O, lse
