"""What is timed of the SwitchHead layer: the passes a user's program makes through the public binding.

A case is one layer, configured and loaded, and one pass over a batch that is on the GPU: the forward
pass in either storage type, or - `train` - the forward and the backward pass of the fp32 configuration,
which is the one that has a backward pass.  Sizes are those of the repository's own workloads
(`paper_2312_07987_b200.inputs.CONFIGS`) and of the paper's models (2 or 4 heads; d_head 76, 100, 112 or
132; 4, 5 or 8 experts; sequences of 256 and 512 tokens, a cache of one chunk with Transformer-XL's
relative positions, or rotary positions without a cache).
"""
import math

import torch

from paper_2312_07987_b200 import binding

DEFAULTS = dict(dtype="bf16", train=False, batch=1, seq=64, cache=0, d_model=128, heads=2, d_head=32, experts=4, k=2,
                causal=True, rope=False, positions=False, shared=False, out_f16=False, zipf=0.0)


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest layer: exact fp32 arithmetic on one short sequence (unit-test sized models, debugging);
        # launches and their latency are all there is
        _case("tiny_f32", dtype="f32", batch=1, seq=64, d_model=128, heads=2, d_head=32, experts=4, k=2),
        # fp32 evaluation of a 47M-parameter model's layer on a few sequences of a length that fits no tile;
        # d_model is the nearest the layer takes to the model's 412
        _case("eval_f32_ragged", dtype="f32", batch=4, seq=300, d_model=448, heads=2, d_head=76, experts=5, k=3),
        # a training step (output and all gradients) of the same model's layer on a slice of its batch
        _case("train_f32_47m", dtype="f32", train=True, batch=8, seq=256, d_model=448, heads=2, d_head=76, experts=5, k=3),
        # ... and of a 262M-parameter model's layer: two sequences per GPU and step
        _case("train_f32_262m", dtype="f32", train=True, batch=2, seq=512, d_model=1024, heads=4, d_head=112, experts=4, k=2),
        # serving: the prompt of one user through a 262M-parameter model's layer
        _case("prompt_bf16", batch=1, seq=200, d_model=1024, heads=4, d_head=112, experts=4, k=2),
        # a batch of a 47M-parameter model (three selected experts of five, narrow heads)
        _case("small_bf16", batch=32, seq=256, d_model=512, heads=2, d_head=64, experts=5, k=3),
        # a batch of the 262M-parameter model: the benchmark's default workload
        _case("c4_262m_bf16", batch=16, seq=512, d_model=1024, heads=4, d_head=128, experts=4, k=2),
        # long sequences: attention holds most of the work
        _case("long_ctx_bf16", batch=4, seq=4096, d_model=1024, heads=4, d_head=128, experts=8, k=2),
        # many experts, four selected, unevenly routed (a few experts take most tokens)
        _case("wide_skew_bf16", batch=8, seq=2048, d_model=2048, heads=8, d_head=128, experts=16, k=4, zipf=1.2),
        # a batch of the 262M-parameter Wikitext-103 model: two heads, four of eight experts, d_head 132
        _case("wt103_262m_bf16", batch=16, seq=512, d_model=1024, heads=2, d_head=132, experts=8, k=4),
        # the 262M-parameter model as the paper trains it: one cached chunk and Transformer-XL's positions
        _case("xl_262m_bf16", batch=16, seq=512, cache=512, d_model=1024, heads=4, d_head=112, experts=4, k=2, positions=True),
        # a model with rotary positions on a few sequences of an odd length, result handed on in fp16
        _case("rope_ragged_bf16", batch=5, seq=777, d_model=1024, heads=4, d_head=100, experts=4, k=2, rope=True, out_f16=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind of pass, then sizes over that kind's range; the batch shrinks (then the
    sequence) until it costs no more than the kind's largest listed case."""
    kind = rng.choice(["f32", "train", "bf16", "bf16", "bf16", "wide_head", "xl"])
    c = _case()
    c["experts"] = rng.choice([2, 3, 4, 4, 5, 8, 8, 16])
    c["k"] = rng.randint(1, min(4, c["experts"]))
    c["heads"] = rng.choice([1, 2, 2, 3, 4, 4, 8])
    c["causal"] = rng.random() < 0.85
    if kind in ("f32", "train"):
        limit = "train_f32_262m" if kind == "train" else "eval_f32_ragged"
        c.update(dtype="f32", train=kind == "train", seq=_log_int(rng, 16, 600), d_model=64 * rng.randint(1, 16),
                 d_head=rng.choice([32, 64, 76, 100, 112, 128, rng.randint(16, 168)]), batch=_log_int(rng, 1, 16))
        if kind == "f32":
            c["shared"] = rng.random() < 0.2
    elif kind == "bf16":
        limit = "wide_skew_bf16"
        c.update(seq=_log_int(rng, 32, 4096), d_model=128 * _log_int(rng, 2, 16), d_head=rng.choice([64, 76, 100, 112, 128, 128, rng.randint(24, 128)]),
                 batch=_log_int(rng, 1, 32), shared=rng.random() < 0.2, out_f16=rng.random() < 0.3, zipf=rng.choice([0.0, 0.0, 1.2]))
        c["rope"] = rng.random() < 0.25 and c["d_head"] % 2 == 0
    elif kind == "wide_head":
        limit = "wt103_262m_bf16"
        c.update(seq=_log_int(rng, 64, 1024), d_model=128 * rng.randint(4, 12), d_head=rng.choice([132, 168, rng.randint(130, 256)]),
                 heads=rng.choice([1, 2, 2, 4]), batch=_log_int(rng, 1, 16))
        c["rope"] = rng.random() < 0.25 and c["d_head"] % 2 == 0
    else:
        limit = "xl_262m_bf16"
        c.update(seq=128 * rng.randint(1, 6), cache=128 * rng.randint(1, 6), d_model=128 * rng.randint(2, 12),
                 d_head=rng.choice([64, 76, 112, 128]), heads=rng.choice([2, 4]), causal=True, positions=rng.random() < 0.7, batch=_log_int(rng, 1, 16))
    top = work(next(x for x in listed() if x["name"] == limit))
    while True:
        w = work(c)
        if w["flops"] <= top["flops"] and w["bytes"] <= top["bytes"]:
            return c
        if c["batch"] > 1:
            c["batch"] -= 1
        elif c["cache"]:
            c["heads"], c["d_model"] = max(1, c["heads"] // 2), max(128, c["d_model"] - 128)
        elif c["seq"] > 32:
            c["seq"] = c["seq"] * 3 // 4
        else:
            c["d_model"] = max(128, c["d_model"] - 128)


def _zipf_bias(c, g):
    """Per head a drawn permutation of the experts; their share falls off as rank^-zipf."""
    rows = []
    for _ in range(c["heads"]):
        rank = torch.randperm(c["experts"], generator=g, device="cuda").double() + 1
        lp = -c["zipf"] * torch.log(rank)
        rows.append((lp - lp.mean()).float())
    return torch.stack(rows).contiguous()


def _near_ties(x, gates, k, gap=1e-3):
    """Rows of x whose k-th and (k+1)-th gate logit of some head lie closer than gap."""
    bad = torch.zeros(x.shape[0], dtype=torch.bool, device=x.device)
    for W, bias in gates:
        z = torch.einsum("nm,hme->nhe", x.double(), W.double())
        if bias is not None:
            z = z + bias.double()
        if k < z.shape[2]:
            top = z.topk(k + 1, dim=2).values
            bad |= (top[..., k - 1] - top[..., k] < gap).any(dim=1)
    return bad.nonzero()[:, 0]


def _inputs(c, seed):
    """Weights, biases and batch of one case, in storage type, from the seed alone."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    store = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    H, E, M, D, k = c["heads"], c["experts"], c["d_model"], c["d_head"], c["k"]

    def normal(*shape, fan_in=1):
        return (torch.randn(*shape, generator=g, device="cuda") / math.sqrt(fan_in)).to(store)

    w = dict(Wq=normal(H, M, D, fan_in=M), Wk=normal(H, M, D, fan_in=M), Wv=normal(H, E, M, D, fan_in=M), Wo=normal(H, E, D, M, fan_in=D),
             Ws=normal(H, M, E, fan_in=M), Wd=None if c["shared"] else normal(H, M, E, fan_in=M))
    w["bias_s"] = _zipf_bias(c, g) if c["zipf"] else None
    w["bias_d"] = _zipf_bias(c, g) if c["zipf"] and not c["shared"] else None
    gates = [(w["Ws"], w["bias_s"])] + ([] if c["shared"] else [(w["Wd"], w["bias_d"])])
    n = c["batch"] * (c["cache"] + c["seq"])
    x = normal(n, M)
    # a token whose selection hangs on the last bits of a sum has two right answers: such rows are drawn again
    rows = _near_ties(x, gates, k)
    for _ in range(64):
        if rows.numel() == 0:
            break
        x[rows] = normal(rows.numel(), M)
        rows = rows[_near_ties(x[rows], gates, k)]
    x = x.view(c["batch"], c["cache"] + c["seq"], M)
    xl = None
    if c["positions"]:
        f32 = lambda *shape, fan_in=1: torch.randn(*shape, generator=g, device="cuda") / math.sqrt(fan_in)
        xl = (f32(H, M, D, fan_in=M), 0.5 * f32(H, D), 0.5 * f32(H, D))
    dout = torch.randn(c["batch"], c["seq"], M, generator=g, device="cuda") if c["train"] else None
    return w, x, xl, dout


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    w, x, xl, dout = _inputs(c, seed)
    layer = binding.Layer(c["d_model"], c["heads"], c["d_head"], c["experts"], c["k"], shared_selection=c["shared"])
    layer.sh_configure(binding.SH_F32 if c["dtype"] == "f32" else binding.SH_BF16, c["batch"], c["seq"], cache_len=c["cache"])
    layer.sh_set_weights(*[w[n] for n in ("Wq", "Wk", "Wv", "Wo", "Ws", "Wd", "bias_s", "bias_d")])
    layer.sh_set_causal(c["causal"])
    if c["rope"]:
        layer.sh_set_rope(10000.0)
    if c["out_f16"]:
        layer.sh_set_output_f16(True)
    if c["positions"]:
        layer.sh_set_xl_positions(*xl)
    state = dict(layer=layer, x=x)
    if c["train"]:
        state["dout"] = dout
    return state


def _select(x, W, bias, k):
    """Per head the gate values of the k largest logits, zero elsewhere: [n, H, E] (a lower index wins ties)."""
    z = torch.einsum("nm,hme->nhe", x, W)
    if bias is not None:
        z = z + bias
    order = torch.argsort(z.detach(), dim=2, descending=True, stable=True)[..., :k]
    return torch.sigmoid(z) * torch.zeros_like(z).scatter(2, order, 1.0)


def _layer64(c, w, x, xl):
    """The layer's equations in the precision of its arguments, plain torch."""
    B, T, C, M, H, D, E, k = (c[n] for n in ("batch", "seq", "cache", "d_model", "heads", "d_head", "experts", "k"))
    S = C + T
    flat = x.reshape(B * S, M)
    gs = _select(flat, w["Ws"], w["bias_s"], k)
    gd = gs if c["shared"] else _select(flat, w["Wd"], w["bias_d"], k)
    rows = torch.arange(B * S, device=x.device).view(B, S)[:, C:].reshape(-1)
    t = torch.arange(S, device=x.device)
    seen = t[None, :] <= t[C:, None] if c["causal"] else None
    y = torch.zeros(B * T, M, dtype=x.dtype, device=x.device)
    if c["rope"]:
        ang = t[:, None].double() * 10000.0 ** (-2.0 * torch.arange(D // 2, device=x.device).double() / D)
        cos, sin = torch.cos(ang), torch.sin(ang)
    if xl is not None:
        freq = 10000.0 ** (-2.0 * torch.arange(M // 2, device=x.device).double() / M)
        emb = torch.cat([torch.sin(t[:, None] * freq), torch.cos(t[:, None] * freq)], dim=1)
    for h in range(H):
        q, key = (flat[rows] @ w["Wq"][h]).view(B, T, D), (flat @ w["Wk"][h]).view(B, S, D)
        if c["rope"]:
            turn = lambda a: torch.stack([a[..., 0::2] * cos - a[..., 1::2] * sin, a[..., 0::2] * sin + a[..., 1::2] * cos], dim=-1).flatten(-2)
            q, key = turn(q), turn(key)
        v = sum(gs[:, h, e, None] * (flat @ w["Wv"][h, e]) for e in range(E)).view(B, S, D)
        read = []
        for b in range(B):
            s = q[b] @ key[b].T
            if xl is not None:
                s = (q[b] + xl[1][h]) @ key[b].T
                r = (q[b] + xl[2][h]) @ (emb @ xl[0][h]).T
                s = s + r.gather(1, (t[C:, None] - t[None, :]).clamp(min=0))
            s = s / math.sqrt(D)
            if seen is not None:
                s = s.masked_fill(~seen, -math.inf)
            read.append(torch.softmax(s, dim=1) @ v[b])
        read = torch.cat(read)
        for e in range(E):
            y = y + gd[rows][:, h, e, None] * (read @ w["Wo"][h, e])
    return y.view(B, T, M)


def exact(case, seed):
    c = dict(DEFAULTS, **case)
    w, x, xl, dout = _inputs(c, seed)
    d64 = lambda a: None if a is None else a.double()
    w, x, xl = {n: d64(a) for n, a in w.items()}, d64(x), None if xl is None else [d64(a) for a in xl]
    if not c["train"]:
        with torch.no_grad():
            return _layer64(c, w, x, xl)
    names = ("Wq", "Wk", "Wv", "Wo", "Ws", "Wd")
    wrt = [x] + [w[n] for n in names]
    for a in wrt:
        a.requires_grad_(True)
    out = _layer64(c, w, x, xl)
    grads = torch.autograd.grad(out, wrt, d64(dout))
    return dict(zip(["dx"] + ["d" + n for n in names], grads), out=out.detach())


def run(state):
    out = state["layer"].sh_forward(state["x"])
    if "dout" not in state:
        return out
    return dict(state["layer"].sh_backward(state["x"], state["dout"]), out=out)


def work(case):
    """Useful work: dense Q/K, the k selected V and O experts, both gates, the visible (query, key) pairs;
    every weight and input read once, every result written once.  The backward pass costs each
    projection twice (input and weight gradient) and attention five products where forward has two."""
    c = dict(DEFAULTS, **case)
    B, T, C, M, H, D, E, k = (c[n] for n in ("batch", "seq", "cache", "d_model", "heads", "d_head", "experts", "k"))
    nk, nq = B * (C + T), B * T
    sides = 1 if c["shared"] else 2
    proj = 2.0 * M * H * D * (nk + nq) + 2.0 * M * H * D * k * (nk + nq) + 2.0 * M * H * E * (nk + (sides - 1) * nq)
    pairs = B * H * (T * C + (T * (T + 1) / 2 if c["causal"] else T * T))
    attn = 2.0 * 2.0 * D * pairs
    flops = proj + attn + (2.0 * D * pairs if c["positions"] else 0.0)
    wide = 4 if c["dtype"] == "f32" else 2
    weights = wide * (2 * H * M * D + 2 * H * E * M * D + sides * H * M * E)
    nbytes = wide * nk * M + weights + (2 if c["out_f16"] else 4) * nq * M
    if c["train"]:
        flops += 2.0 * proj + 2.5 * attn
        nbytes += 4 * nq * M + weights + 4 * nk * M       # dout in; the weights' gradients and dx out
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error measured against a double-precision evaluation of the same inputs over
    the listed and drawn cases: fp32 passes up to 1.0e-6 (forward) and 1.5e-6 (gradients) relative, single
    values up to 2.7e-5 of the result's RMS; bf16 storage (fp16 intermediates) up to 6.5e-4 and 2.2e-2."""
    c = dict(DEFAULTS, **case)
    if c["dtype"] == "f32":
        return {"rel": 6e-6, "max": 1e-4}
    return {"rel": 2.6e-3, "max": 8e-2}
