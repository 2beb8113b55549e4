"""The work this library is used for, as cases that can be timed and compared: whole generations (prompt in, a run
of decode steps with trimming), the prompt side of a model layer by layer, and the two context-free attention calls.

A case is a dict of plain values; `kind` says which path it takes:
  decode   prefill_select, then `steps` decode steps, then the kept sets of the pruning layers are read.  `layers_per_call`
           is all layers (a replayed or batched step) or 1 (a decoder that calls once per layer); `overlap` is
           st3_set_overlap, for callers whose inputs are complete ahead of time.
  prompt   for every layer the causal attention of the prompt and then prefill_select of that layer.
  chain    the same with pruning as the paper words it: the scores of layer l's prompt attention prune layer l+1
           before it attends, and later layers run on the kept tokens only.
  attend   the causal prompt attention alone.
  noalloc  one query per head over dense K/V without a workspace.
Q/K/V are N(0,1) with a share of attentive visual tokens (keys shifted by +2 along the head's mean query direction),
the distribution the synthetic workloads of this repository use.
"""
import math

import torch

from paper_2412_20105_b200 import binding as B

_TORCH = {"bf16": torch.bfloat16, "f32": torch.float32}


def _decode(name, **kw):
    c = dict(name=name, kind="decode", dtype="bf16", layers=32, heads=32, dim=128, batch=1, sys=35, visual=576,
             text_min=64, text_max=64, steps=32, tau=50.0, first=3, stride=7, first_bp=5000, step_bp=1225,
             layers_per_call=32, overlap=False, shared=False, lazy=0)
    c.update(kw)
    return c


def _prompt(name, kind, **kw):
    c = dict(name=name, kind=kind, dtype="bf16", layers=32, heads=32, dim=128, batch=1, sys=35, visual=576, text=64,
             first=3, stride=7, first_bp=5000, step_bp=1225)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest calls: one fp32 layer of eight 64-wide heads (a small or debugging model); latency is all there is.
        _decode("decode_f32_small", dtype="f32", layers=1, heads=8, dim=64, sys=32, text_min=32, text_max=32, steps=16,
                first=0, stride=1, step_bp=0, layers_per_call=1),
        # One user in front of a 7B-shaped model, a whole answer, one call per token with the steps overlapping.
        _decode("decode_7b_b1", steps=256, tau=256.0, overlap=True),
        # The same model driven the way a decoder does it: a call per layer, in plain stream order.
        _decode("decode_7b_b1_layers", steps=24, layers_per_call=1),
        # A 13B-shaped model serving sixteen users, a call per layer.
        _decode("decode_13b_b16_layers", layers=40, heads=40, batch=16, stride=4, step_bp=500, steps=20, layers_per_call=1),
        # A full server: 32 users with prompts of different lengths, one call per token.
        _decode("decode_7b_b32", batch=32, text_min=16, text_max=128, overlap=True),
        # High-resolution images: five tiles of visual tokens, where trimming matters most.
        _decode("decode_next_b8", batch=8, visual=2880, text_min=128, text_max=128, overlap=True),
        # A few users, tokens shared inside a stage and layers that inherit attention (QK heredity), ragged prompts.
        _decode("decode_7b_b4_heredity", batch=4, text_min=16, text_max=128, steps=48, shared=True, lazy=0x370),
        # The prompt of one user through all layers: attention of the layer, then its cache is filled and trimmed.
        _prompt("prompt_7b_b1", "prompt"),
        # A batch of high-resolution prompts through four layers (the others are like them).
        _prompt("prompt_next_b8", "prompt", batch=8, visual=2880, text=128, layers=4),
        # Pruning between the layers of a prompt: two users, ragged lengths after every pruning layer.
        _prompt("chain_7b_b2", "chain", batch=2, text=41, layers=11, first=1, stride=3),
        # The prompt attention of a full batch in one call.
        _prompt("attend_7b_b32", "attend", batch=32, layers=1),
        # A plugin that may not allocate: one decode attention over a full 7B prompt.
        dict(name="noalloc_7b", kind="noalloc", dtype="bf16", heads=32, dim=128, rows=675),
    ]


# ---------------------------------------------------------------------------------------------- more of the same
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _seconds(case):
    w = work(case)
    return w["bytes"] / 6e12 + w["flops"] / 1e15


def draw(rng):
    most = max(_seconds(c) for c in listed())
    while True:
        c = _draw(rng)
        c.pop("name", None)
        if c["kind"] == "noalloc" and c["heads"] * -(-c["rows"] // 128) > 8192:
            continue
        if _seconds(c) <= most and _state_bytes(c) <= 30e9:
            return c


def _draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "prompt", "chain", "attend", "noalloc"])
    visual = rng.choice([144, 576, 576, 729, 1152, 2880]) if rng.random() < 0.7 else _log(rng, 100, 2880)
    sys_len = rng.randint(1, 64)
    if kind == "noalloc":
        return dict(kind=kind, dtype=rng.choice(["bf16", "bf16", "f32"]), heads=rng.randint(4, 64),
                    dim=rng.choice([64, 128, 128]), rows=_log(rng, 20, 8000))
    sched = dict(first_bp=5000, stride=rng.choice([1, 2, 4, 7]), step_bp=rng.choice([175, 500, 1225]))
    if kind != "decode":
        layers = {"attend": 1, "prompt": _log(rng, 3, 32), "chain": rng.randint(3, 12)}[kind]
        return _prompt("", kind, heads=rng.choice([8, 16, 32, 32, 40]), batch=_log(rng, 1, 4 if kind == "chain" else 32),
                       sys=sys_len, visual=visual, text=_log(rng, 8, 160), layers=layers, first=rng.choice([1, 3]), **sched)
    layers = rng.choice([4, 12, 24, 32, 32, 40])
    text = _log(rng, 8, 160)
    small = rng.random() < 0.2
    shared = rng.random() < 0.25
    c = _decode("", layers=layers, heads=rng.choice([8, 16, 32, 32, 40]), batch=_log(rng, 1, 32), sys=sys_len,
                visual=visual, text_min=max(1, text // rng.choice([1, 4])), text_max=text, steps=_log(rng, 8, 128),
                tau=rng.choice([50.0, 128.0, 256.0]), layers_per_call=rng.choice([layers, 1]),
                overlap=rng.random() < 0.5, shared=shared, **sched)
    if small:
        c.update(dtype=rng.choice(["f32", "bf16"]), dim=rng.choice([64, 64, 128]), layers=rng.choice([1, 2]),
                 batch=rng.randint(1, 4), steps=rng.randint(8, 32), first=rng.choice([0, 1]), lazy=0)
        c["layers_per_call"] = c["layers"]
    if shared and c["layers"] >= 12 and c["stride"] >= 4:
        c.update(lazy=0x370 if c["stride"] == 7 else 0x30, layers_per_call=c["layers"])
    return c


# ---------------------------------------------------------------------------------------------- inputs and handles
def _config(c, steps, text_max, tau):
    return B.make_config(num_layers=c["layers"], num_heads=c["heads"], head_dim=c["dim"], dtype=c["dtype"], batch=c["batch"],
                         sys_len=c["sys"], num_visual=c["visual"], max_text_len=text_max, max_decode_steps=steps,
                         stride=c["stride"], step_ratio_bp=c["step_bp"], first_ratio_bp=c["first_bp"],
                         first_prune_layer=c["first"], tau=tau, stage_shared=int(c.get("shared", False)),
                         lazy_mask=c.get("lazy", 0))


def _normal(g, dtype, *shape):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)


def _directions(g, c):
    u = _normal(g, torch.float32, c["layers"], c["heads"], c["dim"])
    return u / u.norm(dim=-1, keepdim=True)


def _plant(g, c, K, u):
    """Shifts the keys [layers][batch][heads][rows][dim] of 5 % of the visual tokens, other ones in each layer."""
    n = max(1, c["visual"] // 20)
    for l in range(c["layers"]):
        at = torch.rand(c["batch"], c["visual"], generator=g, device="cuda").topk(n, dim=1).indices + c["sys"]
        at = at[:, None, :, None].expand(-1, c["heads"], -1, c["dim"])
        K[l].scatter_add_(2, at, (2.0 * u[l]).to(K.dtype)[None, :, None, :].expand(c["batch"], -1, n, -1))


def _shift(q, u, dim):
    """Adds sqrt(dim) times the heads' directions to queries [..., layers, batch, heads, dim]."""
    q += (math.sqrt(dim) * u).to(q.dtype)[:, None]


def _pruning_layers(c):
    return [l for l in range(c["first"], c["layers"], c["stride"])]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return {"decode": _prepare_decode, "prompt": _prepare_prompt, "chain": _prepare_chain, "attend": _prepare_attend,
            "noalloc": _prepare_noalloc}[case["kind"]](case, g)


def _prepare_decode(c, g):
    dt = _TORCH[c["dtype"]]
    L, nb, H, D, n = c["layers"], c["batch"], c["heads"], c["dim"], c["steps"]
    u = _directions(g, c)
    T0 = c["sys"] + c["visual"] + c["text_max"]
    K, V = _normal(g, dt, L, nb, H, T0, D), _normal(g, dt, L, nb, H, T0, D)
    _plant(g, c, K, u)
    q, k, v = (_normal(g, dt, n + 1, L, nb, H, D) for _ in range(3))
    _shift(q, u, D)
    out = torch.empty_like(q)
    text = torch.randint(c["text_min"], c["text_max"] + 1, (nb,), generator=g, device="cuda").tolist()
    ctx = B.Context(_config(c, n, c["text_max"], c["tau"]))
    B.st3_set_overlap(ctx.handle, c["overlap"])
    # every call's tensors, as a model has them in hand: [step][call]
    per = c["layers_per_call"]
    cut = lambda t: [list(s.split(per)) for s in t]
    s = dict(case=c, ctx=ctx, text=text, K=list(K.split(per)), V=list(V.split(per)), q=cut(q), k=cut(k), v=cut(v), out=cut(out),
             whole_out=out, **_kept_buffers(c))
    return s


def _prepare_prompt(c, g):
    s = _prepare_attend(c, g)
    L, nb, H, D = c["layers"], c["batch"], c["heads"], c["dim"]
    T = c["sys"] + c["visual"] + c["text"]
    s["ctx"] = B.Context(_config(c, 1, c["text"], 50.0))
    s.update(_kept_buffers(c))
    five = lambda t: [x.view(1, nb, H, T, D) for x in t]
    s.update(text=[c["text"]] * nb, q_last=[x[:, -1].reshape(1, nb, H, D).contiguous() for x in s["q"]],
             k5=five(s["k"]), v5=five(s["v"]), last=torch.empty(L, 1, nb, H, D, dtype=_TORCH[c["dtype"]], device="cuda"))
    return s


def _prepare_attend(c, g):
    """Prompts of c["layers"] layers: q, k, v [batch * heads][T][dim] each."""
    dt = _TORCH[c["dtype"]]
    L, nb, H, D = c["layers"], c["batch"], c["heads"], c["dim"]
    T = c["sys"] + c["visual"] + c["text"]
    u = _directions(g, c)
    q, k, v = (_normal(g, dt, L, nb, H, T, D) for _ in range(3))
    _plant(g, c, k, u)
    q += (math.sqrt(D) * u).to(dt)[:, None, :, None, :]
    flat = lambda t: list(t.view(L, nb * H, T, D))
    return dict(case=c, T=T, q=flat(q), k=flat(k), v=flat(v), out=flat(torch.empty_like(q)),
                probs=torch.empty(nb * H, c["visual"], device="cuda"),
                scores=torch.empty(L, nb, c["visual"], device="cuda"),
                status=torch.zeros(1, dtype=torch.int32, device="cuda"))


def _prepare_chain(c, g):
    s = _prepare_prompt(c, g)
    L, nb, H, D = c["layers"], c["batch"], c["heads"], c["dim"]
    cfg = s["ctx"].cfg
    held = [B.st3_schedule_count(cfg, l, 0) for l in range(L)]
    lens = [c["sys"] + n + c["text"] for n in held]
    # what the projections of layer l give for the tokens it holds
    dense = [[_normal(g, _TORCH[c["dtype"]], nb * H, t, D) for _ in range(3)] for t in lens]
    s.update(held=held, lens=lens, dense=dense, dense_out=[torch.empty_like(d[0]) for d in dense],
             scores=[torch.empty(1, nb, c["visual"], device="cuda") for _ in range(L)],
             all_ids=torch.arange(c["visual"], dtype=torch.int32, device="cuda").repeat(nb, 1))
    for key in ("q", "k", "v", "out"):
        del s[key]
    return s


def _prepare_noalloc(c, g):
    dt = _TORCH[c["dtype"]]
    q = _normal(g, dt, c["heads"], c["dim"]) * 2
    k, v = (_normal(g, dt, c["heads"], c["rows"], c["dim"]) for _ in range(2))
    return dict(case=c, q=q, k=k, v=v, out=torch.empty_like(q))


# ---------------------------------------------------------------------------------------------- one pass
def run(state):
    return {"decode": _run_decode, "prompt": _run_prompt, "chain": _run_chain, "attend": _run_attend,
            "noalloc": _run_noalloc}[state["case"]["kind"]](state)


def _run_decode(s):
    c, ctx, per = s["case"], s["ctx"], s["case"]["layers_per_call"]
    q, k, v, out = s["q"], s["k"], s["v"], s["out"]
    for i in range(len(s["K"])):
        ctx.prefill_select(q[0][i], s["K"][i], s["V"][i], s["text"], out[0][i], layer_begin=i * per)
    for t in range(1, c["steps"] + 1):
        for i, (qi, ki, vi, oi) in enumerate(zip(q[t], k[t], v[t], out[t])):
            ctx.decode_step(t, qi, ki, vi, oi, layer_begin=i * per)
    return {"out": s["whole_out"], **_read_kept(s)}


def _kept_buffers(c):
    n, nb = len(_pruning_layers(c)), c["batch"]
    ids, mass = (torch.zeros(n, nb, c["visual"], dtype=t, device="cuda") for t in (torch.int32, torch.float32))
    return dict(ids=ids, count=torch.zeros(n, nb, dtype=torch.int32, device="cuda"), mass=mass)


def _read_kept(s):
    """The pruning layers' kept sets.  The ids come in cache order, which is not specified: the counts and each token's
    last score (by original index) are what is compared."""
    st = torch.cuda.current_stream().cuda_stream
    for i, l in enumerate(_pruning_layers(s["case"])):
        B.st3_get_kept(s["ctx"].handle, l, s["ids"][i].data_ptr(), s["count"][i].data_ptr(), s["mass"][i].data_ptr(), st)
    return {"count": s["count"], "mass": s["mass"]}


def _attend(s, l):
    c = s["case"]
    B.st3_prefill_attend(s["q"][l].data_ptr(), s["k"][l].data_ptr(), s["v"][l].data_ptr(), s["out"][l].data_ptr(),
                         s["probs"].data_ptr(), s["scores"][l].data_ptr(), s["status"].data_ptr(), c["batch"] * c["heads"],
                         c["heads"], s["T"], c["dim"], c["dtype"], c["sys"], c["visual"],
                         torch.cuda.current_stream().cuda_stream)


def _run_attend(s):
    for l in range(s["case"]["layers"]):
        _attend(s, l)
    return {"out": s["out"], "scores": s["scores"]}


def _run_prompt(s):
    c, ctx = s["case"], s["ctx"]
    for l in range(c["layers"]):
        _attend(s, l)
        ctx.prefill_select(s["q_last"][l], s["k5"][l], s["v5"][l], s["text"], s["last"][l], layer_begin=l)
    return {"out": s["out"], "scores": s["scores"], "last": s["last"], **_read_kept(s)}


def _run_chain(s):
    c, ctx, stream = s["case"], s["ctx"], torch.cuda.current_stream().cuda_stream
    nb, H, D = c["batch"], c["heads"], c["dim"]
    ids, n, kept = s["all_ids"], c["visual"], []
    for l in range(c["layers"]):
        if l == 0:
            ctx.prefill_select(s["q_last"][0], s["k5"][0], s["v5"][0], s["text"], s["last"][0])
        else:
            ctx.prefill_select_scored(s["q_last"][l], s["k5"][l], s["v5"][l], s["text"], s["scores"][l - 1], s["last"][l],
                                      layer_begin=l)
        if s["held"][l] != n:  # the tokens that go on, in the order of the sequence
            n = s["held"][l]
            got, _, _ = ctx.get_kept(l, with_mass=False)
            ids = got[:, :n].sort(dim=1).values.contiguous()
            kept.append(ids)
        q, k, v = s["dense"][l]
        B.st3_prefill_attend_kept(q.data_ptr(), k.data_ptr(), v.data_ptr(), s["dense_out"][l].data_ptr(), s["probs"].data_ptr(),
                                  s["scores"][l].data_ptr(), s["status"].data_ptr(), nb * H, H, s["lens"][l], D, c["dtype"],
                                  c["sys"], n, ids.data_ptr(), c["visual"], stream)
    return {"out": s["dense_out"], "scores": s["scores"], "last": s["last"], "kept": kept}


def _run_noalloc(s):
    c = s["case"]
    B.st3_attend_noalloc(s["q"].data_ptr(), s["k"].data_ptr(), s["v"].data_ptr(), s["out"].data_ptr(), c["heads"], c["rows"],
                         c["dim"], c["dtype"], torch.cuda.current_stream().cuda_stream)
    return s["out"]


# ---------------------------------------------------------------------------------------------- what a pass cannot do without
def _elem(c):
    return 2 if c["dtype"] == "bf16" else 4


def _count(c, tau, l, t):
    """Visual rows layer l holds after step t (the library's schedule, cosine annealing)."""
    if l < c["first"]:
        return c["visual"]
    bp = max(0, 10000 - c["first_bp"] - (l - c["first"]) // c["stride"] * c["step_bp"])
    n0 = c["visual"] * bp // 10000
    if t == 0:
        return n0
    return math.floor(n0 * (0.0 if t >= tau else math.cos(t * math.pi / (2 * tau))) + 1e-9)


def work(case):
    c = case
    e, H, D = _elem(c), c["heads"], c["dim"]
    row = H * D * e  # one position's keys (or values, query, output) of one layer
    if c["kind"] == "noalloc":
        return {"bytes": 2 * row * c["rows"] + 2 * row, "flops": 4 * H * D * c["rows"]}
    nb, L = c["batch"], c["layers"]
    if c["kind"] == "decode":
        text = (c["text_min"] + c["text_max"]) / 2
        size = flops = 0
        for l in range(L):
            lazy = c["lazy"] >> l & 1  # its keys are never read, it has no query
            kv, q = (1, 0) if lazy else (2, 1)
            t0 = c["sys"] + c["visual"] + text
            size += nb * row * (kv * t0 + kv * (t0 - c["visual"] + _count(c, c["tau"], l, 0)) + q + 1)
            flops += nb * 4 * H * D * t0
            for t in range(1, c["steps"] + 1):
                rows = c["sys"] + text + t + _count(c, c["tau"], l, t - 1)
                size += nb * row * (kv * rows + kv + q + 1)  # rows (the new one from the inputs), its copy to the cache, query, output
                flops += nb * (2 * kv) * H * D * rows
        return {"bytes": size, "flops": flops}
    size = flops = 0
    for l in range(L):
        held = _count(c, 50.0, l, 0)
        full = c["sys"] + c["visual"] + c["text"]
        t = c["sys"] + held + c["text"] if c["kind"] == "chain" else full
        size += nb * row * 4 * t
        flops += nb * H * 4 * D * t * (t + 1) / 2
        if c["kind"] != "attend":  # the kept rows go to the cache; last query in, last output out
            size += nb * row * (2 * (c["sys"] + held + c["text"]) + 2)
            flops += nb * 4 * H * D * t
        if c["kind"] == "chain":   # the prompt rows of the kept tokens, read from the layer's full prompt
            size += nb * row * 2 * t
    return {"bytes": size, "flops": flops}


def _state_bytes(c):
    e, row = _elem(c), c["heads"] * c["dim"] * _elem(c)
    if c["kind"] == "noalloc":
        return 2 * row * c["rows"]
    nb, L = c["batch"], c["layers"]
    if c["kind"] == "decode":
        t0 = c["sys"] + c["visual"] + c["text_max"]
        return nb * L * row * (4 * t0 + 6 * c["steps"])
    return nb * L * row * (10 if c["kind"] == "chain" else 6) * (c["sys"] + c["visual"] + c["text"])


def tolerance(case):
    # Measured with the path's own sums in another order (other chunk sizes): fp32 2e-7, bf16 decode 3e-5.  Decode may also
    # keep a visual token in place of one whose score ties with it to the last digits, which changes one token of a few
    # hundred for some steps: 2e-3, and `max` allows for the score of that token.  The prompt's attention rounds its
    # probabilities to bf16 ahead of the second product: 2e-3 against 64-bit sums.
    if case["dtype"] == "f32":
        return {"rel": 4e-6, "max": 0.01, "differ": 0.0}
    if case["kind"] in ("decode", "noalloc"):
        return {"rel": 2e-3, "max": 0.5, "differ": 0.002}
    return {"rel": 8e-3, "max": 0.5 if case["kind"] == "chain" else 0.1, "differ": 0.002}
