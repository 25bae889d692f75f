"""Performance cases: what a program that uses this library has it do, through its public
entry points (paper_2609_37241_gb300.scm), over the whole range of sizes, types and layouts.

A case is one pass of one of these workloads (its "op"):
  layers       a decoder step or a prefill: the non-GEMM chain of each of `layers` layers
               (add+RMSNorm, [q/k norm,] RoPE + KV append, add+RMSNorm, SwiGLU), by `entry`:
                 seq   one layer-chain call per layer through Scm.invoke_seq, the residual
                       passed from layer to layer (the layers depend on one another)
                 step  the same calls through Scm.invoke_step, each layer with its own
                       residual (independent chains: several sequences, or layers at once)
                 ops   four single-op calls per layer through Scm.invoke_seq, as a model
                       whose hidden size has no fused chain runs its layers
  add_rmsnorm, rmsnorm, rope, swiglu, silu, add, neg, masked_fill
               `calls` calls of the single op, each on buffers of its own, in one pass
               (what a step's layers do; small calls come several to a pass), by `entry`:
                 seq     Scm.invoke_seq (one call: Scm.invoke)
                 tree    Scm.call on nested arguments, packed per call (the norms)
                 noalloc trident_rope_kv_noalloc (RoPE)
A step that an engine repeats keeps its buffers and its argument tuples, so those are made in
prepare(), with the handle and its version table; new data would be written into the buffers.

Inputs: activations N(0, 1) in the activation type, norm weights N(1, 0.1), as the library's
synthetic workloads draw them; the fused projections' outputs (q|k|v rows, gate|up rows) are
views of one buffer where "layout" is "fused". Caches start as zeros; a decode's positions are
distinct and scattered, a prefill's consecutive.
"""
import math

import torch

from paper_2609_37241_gb300 import scm as S

EPS = 1e-6
TORCH = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}
CODE = {"bf16": S.BF16, "fp16": S.FP16, "fp32": S.FP32}
SIZE = {"bf16": 2, "fp16": 2, "fp32": 4}
NORMS = ("add_rmsnorm", "rmsnorm")
OPS = {"add_rmsnorm": S.OP_ADD_RMSNORM, "rmsnorm": S.OP_RMSNORM, "swiglu": S.OP_SWIGLU, "silu": S.OP_SILU,
       "add": S.OP_ADD, "neg": S.OP_NEG, "masked_fill": S.OP_MASKED_FILL}
CHAINS = (S.OP_LAYER_CHAIN, S.OP_LAYER_CHAIN_QKNORM)
ANY_TOKENS = (1, 1 << 30)


# ---------------------------------------------------------------- the cases
def _layers(entry, layers, tokens, hidden, q_heads, kv_heads, head, slots, inter, qk_norm, dtype="bf16",
            layout="fused"):
    return dict(op="layers", entry=entry, layers=layers, tokens=tokens, hidden=hidden, q_heads=q_heads,
                kv_heads=kv_heads, head=head, slots=slots, inter=inter, qk_norm=qk_norm, dtype=dtype,
                layout=layout, theta=1e6 if qk_norm else 5e5)


def _rows(op, calls, rows, width, dtype, layout="dense", entry="seq", in_place=False):
    """layout: dense rows; padded rows (row stride > width, 16-byte aligned); halves (gate and
    up as the halves of one row: swiglu); offset: dense, one element past a 16-byte boundary."""
    return dict(op=op, entry=entry, calls=calls, rows=rows, width=width, dtype=dtype, layout=layout,
                in_place=in_place)


def _rope(calls, tokens, q_heads, kv_heads, head, slots, qk_norm, dtype, layout="fused", entry="seq"):
    return dict(op="rope", entry=entry, calls=calls, tokens=tokens, q_heads=q_heads, kv_heads=kv_heads,
                head=head, slots=slots, qk_norm=qk_norm, dtype=dtype, layout=layout,
                theta=1e6 if qk_norm else 5e5)


def listed():
    return [
        # one token of one sequence through 36 dependent layers: launches and latency only
        dict(_layers("seq", 36, 1, 4096, 32, 8, 128, 2048, 12288, True), name="decode_1tok_36layers"),
        # a batch of 64 sequences' tokens, layer after layer: the headline decode size
        dict(_layers("seq", 16, 64, 4096, 32, 8, 128, 2048, 14336, False), name="decode_64tok_16layers"),
        # a whole step's independent chains in one launch
        dict(_layers("step", 36, 8, 4096, 32, 8, 128, 2048, 12288, True), name="step_8tok_36layers"),
        # prefill of one long prompt: the largest call
        dict(_layers("seq", 1, 8192, 4096, 32, 8, 128, 8192, 14336, False), name="prefill_8192tok"),
        # a hidden size without a fused chain: four calls per layer, a mid-size decode batch
        dict(_layers("ops", 8, 24, 5120, 40, 8, 128, 2048, 13824, False, "fp16"), name="decode_24tok_ops_h5120"),
        # a prefill's residual norm at that hidden size, in place, a ragged token count
        dict(_rows("add_rmsnorm", 1, 3001, 5120, "bf16", in_place=True), name="add_rmsnorm_3001x5120"),
        # short rows through nested arguments packed per call: dispatch cost
        dict(_rows("rmsnorm", 8, 1024, 128, "bf16", entry="tree"), name="rmsnorm_1024x128_tree"),
        # fp32 rows (a final norm kept in fp32), a width that is no power of two
        dict(_rows("rmsnorm", 1, 2050, 3000, "fp32"), name="rmsnorm_fp32_2050x3000"),
        # q/k norm, RoPE and cache append of a ragged prefill
        dict(_rope(1, 3333, 32, 8, 128, 8192, True, "fp16"), name="rope_qk_3333tok"),
        # the MLP's activation of a prefill, gate and up as halves of one projection
        dict(_rows("swiglu", 1, 4096, 14336, "bf16", "halves"), name="swiglu_4096x14336_halves"),
        # masked logits: an odd vocabulary, -inf
        dict(_rows("masked_fill", 1, 256, 50257, "bf16"), name="masked_fill_256x50257"),
        # a pointwise op over many short rows
        dict(_rows("silu", 1, 16384, 1000, "bf16"), name="silu_16384x1000"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _pick(rng, weighted):
    return rng.choices([v for v, _ in weighted], [w for _, w in weighted])[0]


def _draw_layers(rng):
    entry = _pick(rng, [("seq", 5), ("step", 3), ("ops", 3), ("prefill", 3)])
    dtype = _pick(rng, [("bf16", 3), ("fp16", 1)])
    qk = rng.random() < 0.5
    layout = _pick(rng, [("fused", 3), ("dense", 1)])
    if entry == "ops":
        head = _pick(rng, [(64, 1), (128, 2)])
        hidden = 128 * rng.randint(8, 56)
        q_heads = hidden // head
        kv_heads = rng.choice([k for k in (1, 2, 4, 8, q_heads) if q_heads % k == 0])
        inter = 64 * rng.randint(hidden * 5 // 128, hidden // 16)
    else:
        head, hidden, kv_heads = 128, _pick(rng, [(4096, 3), (8192, 1)]), 8
        q_heads = hidden // head
        inter = rng.choice([12288, 14336]) if hidden == 4096 else rng.choice([22016, 28672])
    if entry == "prefill":
        return _layers("seq", 1, _log(rng, 512, 8192), hidden, q_heads, kv_heads, head, 8192, inter, qk, dtype, layout)
    tokens = _log(rng, 1, 256)
    return _layers(entry, rng.randint(4, 36), tokens, hidden, q_heads, kv_heads, head, 2048, inter, qk, dtype, layout)


def _draw_rows(rng):
    op = _pick(rng, [("add_rmsnorm", 4), ("rmsnorm", 3), ("swiglu", 3), ("silu", 1), ("add", 1), ("neg", 1),
                     ("masked_fill", 1)])
    dtype = _pick(rng, [("bf16", 4), ("fp16", 2), ("fp32", 2)])
    kind = _pick(rng, [("power", 3), ("multiple", 4), ("any", 2)])
    lo, hi = {"add_rmsnorm": (512, 16384), "rmsnorm": (64, 16384), "swiglu": (1024, 28672)}.get(op, (64, 131072))
    width = _log(rng, lo, hi)
    if kind == "power":
        width = max(lo, min(hi, 1 << round(math.log2(width))))
    elif kind == "multiple":
        width = max(lo, width // 64 * 64)
    aligned = width * SIZE[dtype] % 16 == 0
    layouts = [("dense", 5), ("offset", 1)]
    if aligned:
        layouts.append(("halves" if op == "swiglu" else "padded", 2))
    entry = _pick(rng, [("seq", 4), ("tree", 1)]) if op in NORMS else "seq"
    c = _rows(op, 1, _log(rng, 1, 32768), width, dtype, _pick(rng, layouts), entry, rng.random() < 0.25)
    while work(c)["bytes"] > work(listed()[3])["bytes"]:
        c["rows"] = c["rows"] * 2 // 3
    c["calls"] = max(1, min(16, (16 << 20) // work(c)["bytes"]))
    return c


def _draw_rope(rng):
    head = _pick(rng, [(64, 2), (128, 5), (256, 1), (96, 1)])
    kv_heads = rng.choice([1, 2, 4, 8])
    entry = "noalloc" if head != 96 and rng.random() < 0.2 else "seq"
    c = _rope(1, _log(rng, 1, 16384), kv_heads * rng.choice([1, 2, 4, 5, 8]), kv_heads, head, 16384,
              rng.random() < 0.5, _pick(rng, [("bf16", 3), ("fp16", 1)]), _pick(rng, [("fused", 3), ("dense", 1)]),
              entry)
    c["calls"] = max(1, min(16, (16 << 20) // work(c)["bytes"]))
    return c


def draw(rng):
    c = _pick(rng, [(_draw_layers, 5), (_draw_rows, 5), (_draw_rope, 2)])(rng)
    if c["op"] == "layers":
        while work(c)["bytes"] > work(listed()[3])["bytes"]:
            c["layers"], c["tokens"] = max(1, c["layers"] * 2 // 3), max(1, c["tokens"] * 9 // 10)
    return c


# ---------------------------------------------------------------- inputs
class _Draws:
    """Seeded normal draws on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def act(self, shape, dtype):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32).to(TORCH[dtype])

    def weight(self, shape):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32) * 0.1 + 1.0


def _positions(d, tokens, slots, scattered):
    if scattered:
        return torch.randperm(slots, generator=d.gen, device="cuda")[:tokens].to(torch.int32)
    first = int(torch.randint(0, slots - tokens + 1, (1,), generator=d.gen, device="cuda"))
    return torch.arange(first, first + tokens, device="cuda", dtype=torch.int32)


def _heads(c, d, n):
    """q, k, v [n, T, heads, D] (views of one [n, T, (Hq + 2 Hkv) D] buffer where fused)."""
    T, Hq, Hkv, D = c["tokens"], c["q_heads"], c["kv_heads"], c["head"]
    if c["layout"] == "fused":
        qkv = d.act((n, T, Hq + 2 * Hkv, D), c["dtype"])
        return qkv[:, :, :Hq], qkv[:, :, Hq:Hq + Hkv], qkv[:, :, Hq + Hkv:]
    return tuple(d.act((n, T, h, D), c["dtype"]) for h in (Hq, Hkv, Hkv))


def _rope_inputs(c, d, n):
    i = {}
    i["q"], i["k"], i["v"] = _heads(c, d, n)
    i["pos"] = _positions(d, c["tokens"], c["slots"], c["tokens"] <= 256)
    shape = (n, c["kv_heads"], c["slots"], c["head"])
    i["k_cache"], i["v_cache"] = (torch.zeros(shape, device="cuda", dtype=TORCH[c["dtype"]]) for _ in range(2))
    if c["qk_norm"]:
        i["gamma_q"], i["gamma_k"] = d.weight((n, c["head"])), d.weight((n, c["head"]))
    return i


def _layer_inputs(c, d):
    L, T, H, I, dt = c["layers"], c["tokens"], c["hidden"], c["inter"], c["dtype"]
    i = _rope_inputs(c, d, L)
    i["h"], i["attn"] = d.act((L, T, H), dt), d.act((L, T, H), dt)
    i["r0"] = d.act((L if c["entry"] == "step" else 1, T, H), dt)
    i["gamma_a"], i["gamma_m"] = d.weight((L, H)), d.weight((L, H))
    if c["layout"] == "fused":
        gu = d.act((L, T, 2 * I), dt)
        i["g"], i["u"] = gu[:, :, :I], gu[:, :, I:]
    else:
        i["g"], i["u"] = d.act((L, T, I), dt), d.act((L, T, I), dt)
    return i


def _place(x, layout):
    """x [calls, rows, width] in the case's row layout (same values)."""
    n, rows, width = x.shape
    if layout == "padded":
        buf = torch.zeros((n, rows, width + 64), device=x.device, dtype=x.dtype)
        view = buf[:, :, :width]
    elif layout == "offset":  # each call's rows dense, starting one element past an aligned address
        per = (rows * width + 1 + 127) // 128 * 128
        view = torch.zeros((n, per), device=x.device, dtype=x.dtype)[:, 1:1 + rows * width].unflatten(1, (rows, width))
    else:
        return x
    return view.copy_(x)


def _row_inputs(c, d):
    n, rows, width, dt = c["calls"], c["rows"], c["width"], c["dtype"]
    i = {}
    if c["op"] == "swiglu" and c["layout"] == "halves":
        gu = d.act((n, rows, 2 * width), dt)
        i["x"], i["b"] = gu[:, :, :width], gu[:, :, width:]
    else:
        i["x"] = _place(d.act((n, rows, width), dt), c["layout"])
        if c["op"] in ("add_rmsnorm", "swiglu", "add"):
            i["b"] = _place(d.act((n, rows, width), dt), c["layout"])
    if c["op"] in NORMS:
        i["gamma"] = d.weight((n, width))
    if c["op"] == "masked_fill":
        mask = torch.rand((n, rows, width), generator=d.gen, device="cuda") < 0.3
        i["mask"] = _place(mask.to(torch.uint8), c["layout"])
    return i


def _inputs(c, seed):
    d = _Draws(seed)
    if c["op"] == "layers":
        return _layer_inputs(c, d)
    return _rope_inputs(c, d, c["calls"]) if c["op"] == "rope" else _row_inputs(c, d)


def _out_like(x, c):
    return _place(torch.zeros(x.shape, device=x.device, dtype=x.dtype), "dense" if c["layout"] == "halves" else c["layout"])


# ---------------------------------------------------------------- state
def _has_vector(op, fixed, dtype):
    """Whether rows of this version can be 16-byte aligned."""
    return op in (*CHAINS, S.OP_ROPE_KV, S.OP_QKNORM_ROPE_KV) or fixed[0] * SIZE[dtype] % 16 == 0


def _register(scm, op, dtype, fixed, theta=0.0):
    """The version table of a program: aligned rows first, then any alignment (not for chains)."""
    aligns = ([16] if _has_vector(op, fixed, dtype) else []) + ([] if op in CHAINS else [SIZE[dtype]])
    for align in aligns:
        scm.register(S.make_spec(op, CODE[dtype], fixed, *ANY_TOKENS, layout=S.LAYOUT_ANY, align_bytes=align,
                                 rope_theta=theta))


def _prepare_layers(c, i, scm, st):
    L, dt, theta = c["layers"], c["dtype"], c["theta"]
    heads = [c["q_heads"], c["kv_heads"], c["head"], c["slots"]]
    out = {k: torch.zeros_like(i["h"]) for k in ("x1", "r1", "x2", "r2")}
    out["o"] = torch.zeros((L, c["tokens"], c["inter"]), device="cuda", dtype=TORCH[dt])
    gqk = [[i["gamma_q"][l], i["gamma_k"][l]] if c["qk_norm"] else [] for l in range(L)]
    args = []
    if c["entry"] == "ops":
        rope_op = S.OP_QKNORM_ROPE_KV if c["qk_norm"] else S.OP_ROPE_KV
        _register(scm, S.OP_ADD_RMSNORM, dt, [c["hidden"]])
        _register(scm, rope_op, dt, heads, theta)
        _register(scm, S.OP_SWIGLU, dt, [c["inter"]])
    else:
        chain_op = S.OP_LAYER_CHAIN_QKNORM if c["qk_norm"] else S.OP_LAYER_CHAIN
        _register(scm, chain_op, dt, [c["hidden"], *heads, c["inter"]], theta)
    for l in range(L):
        r0 = i["r0"][l] if c["entry"] == "step" else (i["r0"][0] if l == 0 else out["r2"][l - 1])
        norm1 = [i["h"][l], r0, i["gamma_a"][l], out["x1"][l], out["r1"][l]]
        rope = [i["q"][l], i["k"][l], i["v"][l], i["pos"], i["k_cache"][l], i["v_cache"][l]]
        mlp = [i["g"][l], i["u"][l], out["o"][l]]
        if c["entry"] == "ops":
            args += [S.make_args(S.OP_ADD_RMSNORM, norm1, eps=EPS),
                     S.make_args(rope_op, rope + gqk[l], eps=EPS, rope_theta=theta),
                     S.make_args(S.OP_ADD_RMSNORM, [i["attn"][l], out["r1"][l], i["gamma_m"][l], out["x2"][l],
                                                    out["r2"][l]], eps=EPS),
                     S.make_args(S.OP_SWIGLU, mlp)]
        else:
            ts = norm1 + rope + [i["attn"][l], i["gamma_m"][l], out["x2"][l], out["r2"][l]] + mlp + gqk[l]
            args.append(S.make_args(chain_op, ts, eps=EPS, rope_theta=theta))
    st["args"] = (S.trident_args * len(args))(*args)
    st["out"] = dict(out, q=i["q"], k_cache=i["k_cache"], v_cache=i["v_cache"])


def _prepare_rope(c, i, scm, st):
    op = S.OP_QKNORM_ROPE_KV if c["qk_norm"] else S.OP_ROPE_KV
    args = []
    for l in range(c["calls"]):
        ts = [i["q"][l], i["k"][l], i["v"][l], i["pos"], i["k_cache"][l], i["v_cache"][l]]
        ts += [i["gamma_q"][l], i["gamma_k"][l]] if c["qk_norm"] else []
        args.append(S.make_args(op, ts, eps=EPS, rope_theta=c["theta"]))
    if c["entry"] != "noalloc":
        _register(scm, op, c["dtype"], [c["q_heads"], c["kv_heads"], c["head"], c["slots"]], c["theta"])
    st["args"] = (S.trident_args * len(args))(*args)
    st["out"] = dict(q=i["q"], k_cache=i["k_cache"], v_cache=i["v_cache"])


def _prepare_rows(c, i, scm, st):
    op, n = OPS[c["op"]], c["calls"]
    y = i["x"] if c["in_place"] else _out_like(i["x"], c)
    st["out"] = dict(y=y)
    if c["op"] == "add_rmsnorm":
        st["out"]["r_out"] = i["b"] if c["in_place"] else _out_like(i["b"], c)
    if c["entry"] == "tree":  # fn(x, residual or None, gamma, y or (y, r_out), eps)
        desc = S.make_spec(op, CODE[c["dtype"]], [c["width"]], *ANY_TOKENS, layout=S.LAYOUT_ANY,
                           align_bytes=SIZE[c["dtype"]])
        aligned = S.make_spec(op, CODE[c["dtype"]], [c["width"]], *ANY_TOKENS, layout=S.LAYOUT_ANY, align_bytes=16)
        if c["op"] == "rmsnorm":
            recipe = S.Recipe(S.Slot(0), None, S.Slot(1), S.Slot(2), S.EPS)
            st["calls"] = [(i["x"][l], None, i["gamma"][l], y[l], EPS) for l in range(n)]
        else:
            recipe = S.Recipe(S.Slot(0), S.Slot(1), S.Slot(2), (S.Slot(3), S.Slot(4)), S.EPS)
            st["calls"] = [(i["x"][l], i["b"][l], i["gamma"][l], (y[l], st["out"]["r_out"][l]), EPS)
                           for l in range(n)]
        if _has_vector(op, [c["width"]], c["dtype"]):
            scm.register_tree(aligned, recipe)
        scm.register_tree(desc, recipe)
        return
    _register(scm, op, c["dtype"], [c["width"]])
    args = []
    for l in range(n):
        ts = {"add_rmsnorm": lambda: [i["x"][l], i["b"][l], i["gamma"][l], y[l], st["out"]["r_out"][l]],
              "rmsnorm": lambda: [i["x"][l], i["gamma"][l], y[l]],
              "swiglu": lambda: [i["x"][l], i["b"][l], y[l]], "add": lambda: [i["x"][l], i["b"][l], y[l]],
              "masked_fill": lambda: [i["x"][l], i["mask"][l], y[l]]}.get(c["op"], lambda: [i["x"][l], y[l]])()
        args.append(S.make_args(op, ts, eps=EPS, scalar=-math.inf))
    st["args"] = (S.trident_args * n)(*args)


def prepare(case, seed):
    c = case
    i = _inputs(c, seed)
    st = dict(entry=c["entry"], inputs=i)
    scm = st["scm"] = None if c["entry"] == "noalloc" else S.Scm(device=torch.cuda.current_device(), flags=S.OPT_PDL)
    {"layers": _prepare_layers, "rope": _prepare_rope}.get(c["op"], _prepare_rows)(c, i, scm, st)
    return st


def run(state):
    stream = torch.cuda.current_stream().cuda_stream
    entry, scm = state["entry"], state["scm"]
    if entry == "step":
        status = scm.invoke_step(state["args"], stream)[0]
    elif entry == "tree":
        status = max((scm.call(*a, stream=stream) for a in state["calls"]), key=abs)
    elif entry == "noalloc":
        status = max((S.trident_rope_kv_noalloc(a, stream) for a in state["args"]), key=abs)
    elif len(state["args"]) == 1:
        status = scm.invoke(state["args"][0], stream)[0]
    else:
        status = scm.invoke_seq(state["args"], stream)[0]
    if status != S.OK:
        raise RuntimeError(f"{entry}: status {status}: {S.trident_scm_last_error()}")
    return state["out"]


# ---------------------------------------------------------------- what a pass cannot do without
def _rope_work(c):
    T, Hq, Hkv, D, es = c["tokens"], c["q_heads"], c["kv_heads"], c["head"], SIZE[c["dtype"]]
    flops = T * (Hq + Hkv) * D * (3 + (5 if c["qk_norm"] else 0))
    return T * (2 * Hq + 4 * Hkv) * D * es + 4 * T + (8 * D if c["qk_norm"] else 0), flops


def work(case):
    c = case
    if c["op"] == "layers":
        T, H, I, es = c["tokens"], c["hidden"], c["inter"], SIZE[c["dtype"]]
        b, f = _rope_work(c)
        # h, r0, attn read; x1, r1, x2, r2 written; gate, up read and the product written
        b += T * (7 * H + 3 * I) * es + 8 * H
        f += T * (12 * H + 6 * I)
        return {"bytes": c["layers"] * b, "flops": c["layers"] * f}
    if c["op"] == "rope":
        b, f = _rope_work(c)
        return {"bytes": c["calls"] * b, "flops": c["calls"] * f}
    n, es = c["rows"] * c["width"], SIZE[c["dtype"]]
    per = {"add_rmsnorm": 4, "rmsnorm": 2, "swiglu": 3, "add": 3}.get(c["op"], 2) * es
    b = n * (per + (1 if c["op"] == "masked_fill" else 0)) + (4 * c["width"] if c["op"] in NORMS else 0)
    f = n * {"add_rmsnorm": 5, "rmsnorm": 4, "swiglu": 6, "silu": 5}.get(c["op"], 1)
    return {"bytes": c["calls"] * b, "flops": c["calls"] * f}


# ---------------------------------------------------------------- results in 64 bits
def _norm64(x, gamma):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + EPS) * gamma.double()


def _rotate64(x, pos, theta):
    """Rotate-half RoPE of x [T, heads, D]."""
    D = x.shape[-1]
    f = theta ** (-2.0 * torch.arange(D // 2, device=x.device, dtype=torch.float64) / D)
    a = (pos.double()[:, None] * f)[:, None, :]
    lo, hi = x[..., :D // 2], x[..., D // 2:]
    return torch.cat([lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()], -1)


def _rope64(c, i):
    n = i["q"].shape[0]
    out = dict(q=torch.empty(i["q"].shape, device="cuda", dtype=torch.float64),
               k_cache=i["k_cache"].double(), v_cache=i["v_cache"].double())
    for l in range(n):
        q, k = i["q"][l].double(), i["k"][l].double()
        if c["qk_norm"]:
            q, k = _norm64(q, i["gamma_q"][l]), _norm64(k, i["gamma_k"][l])
        out["q"][l] = _rotate64(q, i["pos"], c["theta"])
        out["k_cache"][l][:, i["pos"].long()] = _rotate64(k, i["pos"], c["theta"]).transpose(0, 1)
        out["v_cache"][l][:, i["pos"].long()] = i["v"][l].double().transpose(0, 1)
    return out


def _layers64(c, i):
    """The residual is rounded to the activation type between the norms, as the operation says."""
    out = _rope64(c, i)
    for k in ("x1", "r1", "x2", "r2"):
        out[k] = torch.empty(i["h"].shape, device="cuda", dtype=torch.float64)
    out["o"] = torch.empty(i["g"].shape, device="cuda", dtype=torch.float64)
    dt = TORCH[c["dtype"]]
    r = i["r0"][0]
    for l in range(c["layers"]):
        if c["entry"] == "step":
            r = i["r0"][l]
        for x, y, ro, gamma in (("h", "x1", "r1", "gamma_a"), ("attn", "x2", "r2", "gamma_m")):
            s = i[x][l].double() + r.double()
            out[y][l], out[ro][l] = _norm64(s, i[gamma][l]), s
            r = s.to(dt)
        g = i["g"][l].double()
        out["o"][l] = g / (1 + torch.exp(-g)) * i["u"][l].double()
    return out


def exact(case, seed):
    c = case
    i = _inputs(c, seed)
    if c["op"] == "layers":
        return _layers64(c, i)
    if c["op"] == "rope":
        return _rope64(c, i)
    x = i["x"].double()
    if c["op"] == "add_rmsnorm":
        s = x + i["b"].double()
        return dict(y=_norm64(s, i["gamma"][:, None]), r_out=s)
    if c["op"] == "rmsnorm":
        return dict(y=_norm64(x, i["gamma"][:, None]))
    if c["op"] == "masked_fill":
        return dict(y=x.masked_fill(i["mask"] != 0, -math.inf))
    return dict(y={"swiglu": lambda: x / (1 + torch.exp(-x)) * i["b"].double(),
                   "silu": lambda: x / (1 + torch.exp(-x)), "add": lambda: x + i["b"].double(),
                   "neg": lambda: -x}[c["op"]]())


def tolerance(case):
    # add, neg and masked_fill: one exactly rounded operation, or none. Elsewhere one rounding
    # to the activation type: against exact() the outputs are off by about 1.7e-3 (bf16),
    # 2.1e-4 (fp16), 6e-8 (fp32) in the 2-norm; four times that, and for fp32, where sums in another
    # order move a row's scale by about 1e-7, eight. One value may land one unit in the last
    # place of the largest values away (bf16: 2^-8 of itself).
    if case["op"] in ("add", "neg", "masked_fill"):
        return "exact"
    return {"bf16": {"rel": 7e-3, "max": 2e-2}, "fp16": {"rel": 9e-4, "max": 4e-3},
            "fp32": {"rel": 5e-7, "max": 3e-6}}[case["dtype"]]
