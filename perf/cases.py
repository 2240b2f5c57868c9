"""The work that is timed: what a mask-learning run has this library do, through its public calls.

A run trains one logit per weight of every linear layer of a model (the layer sets of
workloads.py are the models' shapes).  Each training step masks all layers (forward),
turns the gradients of the masked weights into logit gradients (backward, often fused
with the logits' AdamW step), and anneals the relaxation temperature tau from 1 to 0.05
and the sampling temperature lambda from 1 to 0.002 over 1500 of 2000 steps.  Finished
masks are exported; a layer's product with its masked weights may be formed directly.

Kinds of case:
  step    all tensors of `layers` transformer blocks (q, k, v, o, gate, up, down) in one
          batched forward and one batched backward call.  variant "soft": logit gradients;
          "adamw": the backward updates logits and moments; "st": straight-through, which
          also returns the gradient of the weights.
  call    one layer through the single-tensor calls, soft mask and weight gradient included.
  export  the deployment masks of one block's layers, with the pruned weights, and for 2:4
          the compressed form as well.
  linear  Y = X (W * S)^T for each layer of one block and T tokens.
"""
import math

import torch

import paper_2608_23048_gb300 as roi
import workloads as WL

T_ANNEAL = 1500
ADAMW = dict(lr=1e-3, beta1=0.9, beta2=0.95, eps=1e-8, weight_decay=0.05, t=40)


def _step(name, shape, layers, N, M, tau, lam=1.0, logits="normal", variant="soft"):
    s = WL.LAYER_SETS[shape]
    return dict(name=name, kind="step", hidden=s.hidden, kv=s.kv, inter=s.inter, layers=layers, N=N, M=M, tau=tau,
                lam=lam, logits=logits, variant=variant)


def listed():
    s = WL.LAYER_SETS["qwen2.5-7b"]
    block = dict(hidden=s.hidden, kv=s.kv, inter=s.inter, layers=1)
    return [
        # one small layer: a unit test, a toy model, a first call; latency counts
        dict(name="layer_2of4", kind="call", rows=128, cols=256, N=2, M=4, tau=1.0, lam=1.0, logits="logw"),
        # a pattern without a specialised kernel on one ordinary layer (75 % sparsity)
        dict(name="layer_1of4", kind="call", rows=896, cols=4864, N=1, M=4, tau=0.5, lam=1.0, logits="normal"),
        # a whole small model per step: 168 tensors, most of them small
        _step("set_0.5b_2of4", "qwen2.5-0.5b", 24, 2, 4, 0.1, logits="logw"),
        # blocks of the mid-sized models at their patterns and temperatures
        _step("set_1.5b_4of8", "qwen2.5-1.5b", 4, 4, 8, 0.5),
        _step("set_3b_8of16", "qwen2.5-3b", 2, 8, 16, 0.2, logits="logw"),
        _step("set_3b_16of32", "qwen2.5-3b", 1, 16, 32, 0.2, logits="logw"),
        # the largest layers at the start of the schedule, plain and with the fused optimizer
        _step("set_7b_2of4", "qwen2.5-7b", 2, 2, 4, 1.0),
        _step("adamw_7b_4of8", "qwen2.5-7b", 1, 4, 8, 1.0, variant="adamw"),
        # the last quarter of the schedule (both temperatures at their end values)
        _step("late_1.5b_2of4", "qwen2.5-1.5b", 4, 2, 4, 0.05, 0.002, variant="adamw"),
        # half-way through the annealing, the straight-through variant, the 2:8 pattern
        _step("mid_1.5b_2of8_st", "qwen2.5-1.5b", 4, 2, 8, *_temperatures(750), variant="st"),
        # deployment masks of a block, and its layers' products for a batch of tokens
        dict(name="export_7b", kind="export", N=2, M=4, logits="normal", **block),
        dict(name="linear_7b", kind="linear", N=2, M=4, tau=1.0, lam=1.0, logits="normal", T=256, **block),
    ]


def _temperatures(t):
    """tau and lambda at step t of the schedule."""
    f = min(1.0, t / T_ANNEAL)
    return round(0.05 ** f, 6), round(0.002 ** f, 6)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("step", "step", "step", "step", "call", "call", "export", "linear"))
    logits = rng.choice(("normal", "logw"))
    if kind == "call":
        N, M = rng.choice(((2, 4), (2, 4), (4, 8), (2, 8), (8, 16), (16, 32), (1, 4), (3, 4), (1, 8), (1, 2)))
        cols = M * log_int(max(1, 64 // M), 8192 // M)
        rows = log_int(1, min(4096, (1 << 22) // cols))
        # a few hundred groups without a near tie have no gradients to compare later on
        tau, lam = _temperatures(rng.randrange(0, min(_last_step(N, M), 400 if rows * cols < 65536 else 900)))
        return dict(kind=kind, rows=rows, cols=cols, N=N, M=M, tau=tau, lam=lam, logits=logits)
    if kind == "step":
        N, M = rng.choice(((2, 4), (2, 4), (4, 8), (2, 8), (8, 16), (16, 32)))
        variant = rng.choice(("soft", "soft", "adamw", "st"))
        tau, lam = _temperatures(rng.randrange(0, _last_step(N, M, variant)))
        hidden, kv, inter = _widths(rng, max(8, M), log_int(64, 2048))
        block = 2 * hidden * (hidden + kv) + 3 * hidden * inter
        layers = log_int(1, max(1, min(28, (60_000_000 if M <= 8 else 30_000_000) // block)))
        return dict(kind=kind, hidden=hidden, kv=kv, inter=inter, layers=layers, N=N, M=M, tau=tau, lam=lam,
                    logits=logits, variant=variant)
    N, M = rng.choice(((2, 4), (2, 4), (4, 8), (2, 8), (8, 16)))
    # the compressed form packs 32 elements a word
    hidden, kv, inter = _widths(rng, 32 if kind == "export" else 8, log_int(64, 3584))
    block = dict(hidden=hidden, kv=kv, inter=inter, layers=1)
    if kind == "export":
        return dict(kind=kind, N=N, M=M, logits=logits, **block)
    N, M = rng.choice(((2, 4), (2, 4), (4, 8), (2, 8)))
    tau, lam = _temperatures(rng.randrange(0, 2000))
    return dict(kind=kind, N=N, M=M, tau=tau, lam=lam, logits=logits, T=log_int(1, 256), **block)


def _widths(rng, unit, hidden):
    """Hidden, key/value and inner width of a block: multiples of `unit`, the ratios those of real models."""
    return [max(unit, int(x) // unit * unit) for x in
            (hidden, hidden / rng.choice((1, 2, 4, 6, 7, 8)), hidden * rng.uniform(2.0, 5.5))]


def _last_step(N, M, variant="soft"):
    """Steps of the schedule that are drawn.  A key's rounding grows with 1 / (tau lambda), and each of the N - 1
    corrections amplifies it: late gradients are zero but for a few near-tied groups, whose values 32-bit keys
    hardly determine, so that cases which return them alone stop earlier, the wide patterns' first of all.  The
    optimizer's state after one correction is well determined throughout."""
    return 300 if M > 8 else 2000 if variant == "adamw" and N == 2 else 900


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shapes(case):
    if case["kind"] == "call":
        return [(case["rows"], case["cols"])]
    h, kv, i = case["hidden"], case["kv"], case["inter"]
    return [(h, h), (kv, h), (kv, h), (h, h), (i, h), (i, h), (h, i)] * case["layers"]


def _offsets(case):
    """Start of every tensor in the flat buffers (each padded to 128 elements, 16 bytes of mask bits), and their length."""
    at, out = 0, []
    for r, c in _shapes(case):
        out.append(at)
        at += (r * c + 127) // 128 * 128
    return out, at


def _seeds(seed):
    return 0x9E3779B97F4A7C15 * (int(seed) + 1) & 0xFFFFFFFFFFFFFFFF, int(seed) % 1000


def _inputs(case, seed):
    """The flat inputs of all tensors: W ~ N(0, 0.02), logits, dWm ~ N(0, 1e-3) (as workloads.make_inputs)."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    _, E = _offsets(case)
    d = {"W": (torch.randn(E, generator=g, device="cuda") * 0.02).to(torch.bfloat16)}
    noise = torch.randn(E, generator=g, device="cuda")
    if case["logits"] == "logw":
        noise = torch.log(d["W"].float().abs().clamp_min(2.0 ** -126)) + 0.1 * noise
    d["phi"] = noise
    if case["kind"] in ("call", "step"):
        d["dWm"] = (torch.randn(E, generator=g, device="cuda") * 1e-3).to(torch.bfloat16)
    if case.get("variant") == "adamw":
        # moments after some steps, at the size of this case's logit gradients
        size = 2e-5 / (case["tau"] * case["lam"])
        d["m"] = 0.3 * size * torch.randn(E, generator=g, device="cuda")
        d["v"] = (size * (0.1 + torch.rand(E, generator=g, device="cuda"))) ** 2
    if case["kind"] == "linear":
        d["X"] = [torch.randn(case["T"], c, generator=g, device="cuda").to(torch.bfloat16) for _, c in _shapes(case)]
    return d


def _views(case, flat):
    offsets, _ = _offsets(case)
    return [flat[o:o + r * c].view(r, c) for o, (r, c) in zip(offsets, _shapes(case))]


def _states(case, seed):
    key, step = _seeds(seed)
    return [roi.NoiseState(key, step, i, case["lam"], 0) for i in range(len(_shapes(case)))]


def prepare(case, seed):
    d = _inputs(case, seed)
    offsets, E = _offsets(case)
    N, M = case["N"], case["M"]
    new = lambda dtype, n=E: torch.zeros(n, dtype=dtype, device="cuda")  # noqa: E731
    phi, W = _views(case, d["phi"]), _views(case, d["W"])
    hard = new(torch.int32, E // 32)
    words = [hard[o // 32:o // 32 + roi.hard_words(r, c)] for o, (r, c) in zip(offsets, _shapes(case))]
    s = dict(case=case, N=N, M=M, keep=d)
    if case["kind"] == "export":
        pruned = new(torch.bfloat16)
        s["out"] = {"hard": hard, "pruned": pruned}
        s["hard"] = list(zip(phi, words, W, _views(case, pruned)))
        s["compressed"] = []
        if (N, M) == (2, 4):
            values, codes = new(torch.bfloat16, E // 2), new(torch.int32, E // 32)
            s["out"].update(values=values, codes=codes)
            s["compressed"] = [(p, w, values[o // 2:o // 2 + r * c // 2].view(r, c // 2), codes[o // 32:o // 32 + r * c // 32])
                               for p, w, o, (r, c) in zip(phi, W, offsets, _shapes(case))]
        return s
    st = _states(case, seed)
    s["tau"] = case["tau"]
    if case["kind"] == "linear":
        s["Y"] = [torch.zeros(case["T"], r, device="cuda") for r, _ in _shapes(case)]
        need = max(roi.roi_masked_linear_workspace_size(case["T"], r, c) for r, c in _shapes(case))
        s["workspace"] = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
        s["layers"] = list(zip(d["X"], phi, W, st, s["Y"]))
        s["out"] = s["Y"]
        return s
    Wm = new(torch.bfloat16)
    s["out"] = {"Wm": Wm, "hard": hard}
    dWm, Wms = _views(case, d["dWm"]), _views(case, Wm)
    if case["kind"] == "call":
        s["out"].update(soft=new(torch.float32), dphi=new(torch.float32), dW=new(torch.bfloat16))
        soft, dphi, dW = (_views(case, s["out"][k])[0] for k in ("soft", "dphi", "dW"))
        s["fwd"] = (phi[0], W[0], N, M, case["tau"], st[0], Wms[0], soft, words[0])
        s["bwd"] = (phi[0], W[0], st[0], N, M, dWm[0], case["tau"], dphi, dW)
        return s
    s["fwd"] = roi.make_fwd_items([(p, w, t, o, None, b) for p, w, t, o, b in zip(phi, W, st, Wms, words)])
    if case["variant"] == "adamw":
        s["opt"] = roi.AdamW(*ADAMW.values())
        s["bwd"] = roi.make_adamw_items([(p, w, t, g, m, v, None, None) for p, w, t, g, m, v in
                                         zip(phi, W, st, dWm, _views(case, d["m"]), _views(case, d["v"]))])
        s["out"].update(phi=d["phi"], m=d["m"], v=d["v"])
    else:
        s["out"]["dphi"] = new(torch.float32)
        dphi = _views(case, s["out"]["dphi"])
        if case["variant"] == "st":
            s["out"]["dW"] = new(torch.bfloat16)
            s["bwd"] = roi.make_bwd_st_items(list(zip(phi, W, st, dWm, words, dphi, _views(case, s["out"]["dW"]))))
        else:
            s["bwd"] = roi.make_bwd_items([(p, w, t, g, o, None) for p, w, t, g, o in zip(phi, W, st, dWm, dphi)])
    return s


def run(s):
    kind, N, M = s["case"]["kind"], s["N"], s["M"]
    if kind == "export":
        for phi, bits, W, pruned in s["hard"]:
            roi.roi_hard_mask_export(phi, N, M, bits, W, pruned)
        for phi, W, values, codes in s["compressed"]:
            roi.roi_export_compressed_2of4(phi, W, values, codes)
    elif kind == "linear":
        for X, phi, W, st, Y in s["layers"]:
            roi.roi_masked_linear_fwd(X, phi, W, N, M, s["tau"], st, Y, s["workspace"])
    elif kind == "call":
        roi.roi_mask_fwd_ex(*s["fwd"])
        roi.roi_mask_bwd(*s["bwd"])
    elif s["case"]["variant"] == "adamw":
        roi.roi_mask_fwd_batch(s["fwd"], N, M, s["tau"])
        roi.roi_mask_bwd_adamw_batch(s["bwd"], N, M, s["tau"], s["opt"])
    elif s["case"]["variant"] == "st":
        roi.roi_mask_fwd_st_batch(s["fwd"], N, M, s["tau"])
        roi.roi_mask_bwd_st_batch(s["bwd"], N, M, s["tau"])
    else:
        roi.roi_mask_fwd_batch(s["fwd"], N, M, s["tau"])
        roi.roi_mask_bwd_batch(s["bwd"], N, M, s["tau"])
    return s["out"]


def work(case):
    E = sum(r * c for r, c in _shapes(case))
    bits = E / 8
    if case["kind"] == "linear":
        T = case["T"]
        return {"bytes": 6 * E + sum(2 * T * c + 4 * T * r for r, c in _shapes(case)), "flops": 2 * T * E}
    if case["kind"] == "export":
        # logits and weights in; bits and pruned weights out, and for 2:4 the same inputs again in
        # the second call, kept weights and codes out
        return {"bytes": 8 * E + bits + (7 * E + bits if (case["N"], case["M"]) == (2, 4) else 0), "flops": 0}
    fwd = 8 * E + bits + (4 * E if case["kind"] == "call" else 0)
    variant = case.get("variant", "call")
    bwd = {"soft": 12 * E, "adamw": 28 * E, "st": 14 * E + bits, "call": 14 * E}[variant]
    return {"bytes": fwd + bwd, "flops": 0}


def tolerance(case):
    """About four times the distance from exact() where a case's 32-bit outputs are the worst (relative / largest):
    1e-7 / 7e-6 at tau = 1, 6e-6 / 3e-4 for 2:4 at tau = 0.1, 4e-4 / 0.035 for 4:8 at tau = 0.2, lambda = 0.04,
    2e-4 to 6e-3 for the wide patterns at tau = 0.2 (a few near-tied groups hold it), 6e-5 / 0.04 at the end of the schedule: a key's rounding counts
    1 / (tau lambda) times in the relaxation.  Below that lie the roundings to bf16 that fall to the other side:
    1e-4, and one step of bf16 at the most."""
    if case["kind"] == "export":
        return "exact"
    # each of the N - 1 corrections amplifies a key's rounding again
    sharp = (case["N"] / 2) ** 2 / (case["tau"] * case["lam"])
    if case["M"] > 8:
        return {"rel": 0.024, "max": 0.99, "differ": 2e-5}
    return {"rel": min(0.01, 2e-4 + 4e-6 * sharp), "max": min(0.25, 0.01 + 2e-4 * sharp), "differ": 2e-5}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _philox(q, step, tensor_id, key):
    """Philox-4x32-10 of the counters (q low, q high, step, tensor_id): the words of elements 4q .. 4q + 3."""
    mask = 0xFFFFFFFF

    def mul(a, x):  # high and low word of the 32 x 32 bit product, in 64-bit signed arithmetic
        low = a * (x & 0xFFFF)
        high = a * (x >> 16) + (low >> 16)
        return high >> 16, (high & 0xFFFF) << 16 | low & 0xFFFF

    c = [q & mask, q >> 32, torch.full_like(q, step), torch.full_like(q, tensor_id)]
    k0, k1 = key & mask, key >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return torch.stack(c, -1).reshape(-1)


def _others(z):
    """log-sum-exp over the other members of each group, for every member ([members, groups])."""
    M = len(z)
    before, after = [z[0]], [z[M - 1]]
    for i in range(1, M - 1):
        before.append(torch.logaddexp(before[-1], z[i]))
        after.append(torch.logaddexp(after[-1], z[M - 1 - i]))
    inner = [torch.logaddexp(before[i - 1], after[M - 2 - i]) for i in range(1, M - 1)]
    return torch.stack([after[-1]] + inner + [before[-1]])


def _relax(kappa, N, tau, c=None):
    """Soft mask of the keys' groups ([members, groups]) and, with c = dL/dS, dL/dkappa."""
    alpha, S, steps = kappa, torch.zeros_like(kappa), []
    for k in range(N):
        z = alpha / tau
        total = torch.logsumexp(z, 0)
        mu, others = torch.exp(z - total), _others(z)
        S = S + mu
        alpha = alpha + others - total
        if c is not None:
            steps.append((z, mu, others))
    if c is None:
        return S, None
    b = torch.zeros_like(c)
    for k in reversed(range(N)):
        z, mu, others = steps.pop()
        grad = mu * (c - (c * mu).sum(0) - b.sum(0))
        for i in range(len(z) if k < N - 1 else 0):
            without = torch.exp(z - others[i])  # the softmax of the members but i
            without[i] = 0
            grad += b[i] * without
        b = b + grad / tau
    return S, b


def exact(case, seed):
    d = _inputs(case, seed)
    offsets, E = _offsets(case)
    N, M = case["N"], case["M"]
    if case["kind"] == "export":
        return None
    f64 = dict(dtype=torch.float64, device="cuda")
    variant = case.get("variant", "call")
    S, dphi = torch.zeros(E, **f64), torch.zeros(E, **f64)
    hard = torch.zeros(E, dtype=torch.bool, device="cuda")
    key, step = _seeds(seed)
    lam = float(torch.tensor(case["lam"], dtype=torch.float32))
    tau = float(torch.tensor(case["tau"], dtype=torch.float32))
    chunk = (1 << 22) // (4 * M) * 4 * M  # whole groups and whole noise blocks
    for i, (o, (r, c)) in enumerate(zip(offsets, _shapes(case))):
        for e in range(0, r * c, chunk):
            n = min(chunk, r * c - e)
            at = slice(o + e, o + e + n)
            words = _philox(torch.arange(e // 4, (e + n + 3) // 4, device="cuda"), step, i, key)[:n]
            u = ((words >> 9).double() + 0.5) * 2.0 ** -23
            kappa = (d["phi"][at].double() / lam - torch.log(-torch.log(u))).view(-1, M).T.contiguous()
            g = (d["dWm"][at].double() * d["W"][at].double()).view(-1, M).T.contiguous() if "dWm" in d else None
            soft, dk = _relax(kappa, N, tau, g)
            S[at] = soft.T.reshape(-1)
            if dk is not None:
                dphi[at] = dk.T.reshape(-1) / lam
            if variant == "st":
                hard[at] = (kappa >= kappa.sort(0).values[M - N]).T.reshape(-1)
    W = d["W"].double()
    if case["kind"] == "linear":
        Wm = (W * S).float().to(torch.bfloat16).double()
        return [X.double() @ w.T for X, w in zip(d["X"], _views(case, Wm))]
    out = {"Wm": W * S, "hard": None}
    if case["kind"] == "call":
        out.update(soft=S, dphi=dphi, dW=d["dWm"].double() * S)
    elif variant == "soft":
        out["dphi"] = dphi
    elif variant == "st":
        out.update(Wm=W * hard, dphi=dphi, dW=d["dWm"].double() * hard)
    else:
        o = ADAMW
        # the settings as the call receives them, in 32 bits
        lr, b1, b2, eps, wd = (float(torch.tensor(o[k], dtype=torch.float32)) for k in
                               ("lr", "beta1", "beta2", "eps", "weight_decay"))
        m = b1 * d["m"].double() + (1 - b1) * dphi
        v = b2 * d["v"].double() + (1 - b2) * dphi * dphi
        phi = d["phi"].double() * (1 - lr * wd)
        phi = phi - lr * (m / (1 - b1 ** o["t"])) / (torch.sqrt(v / (1 - b2 ** o["t"])) + eps)
        # the padding between tensors belongs to none of them
        belongs = torch.zeros(E, dtype=torch.bool, device="cuda")
        for a, (r, c) in zip(offsets, _shapes(case)):
            belongs[a:a + r * c] = True
        out.update({k: torch.where(belongs, x, d[k].double()) for k, x in (("phi", phi), ("m", m), ("v", v))})
    return out
