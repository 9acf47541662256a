"""What a serving program has this library do, as cases that can be timed: decode steps and prompt prefills of the
per-layer hybrid attention, over the sizes, layouts and options of the configurations in `paper_2607_24788_b200.configs`.

A case is a dict of plain values:
  kind     "decode": one token for every sequence;  "prefill": a prompt (or a further turn) and then the first token
  layers   n_layers; windows per layer come from `pattern` (see `windows_of`) with `w` where the pattern has a size
  batch, heads, kv_heads, dim, dtype
  context  tokens the sequences hold before the pass (prefill with context 0: a new sequence in a used context)
  tokens   prefill: tokens of the call
  by_layer one library call per layer, as inside a model whose layer l + 1 computes its inputs from layer l's output
  slots    decode: the sequences have different lengths, and this many slots of the batch are parked (-1: level batch)
  phi, merge, gated   options of the context
"""
import math

import torch

from paper_2607_24788_b200 import configs, glide

# Capacity far above what any pass reaches, so that a state can be stepped for as long as a measurement wants.  It costs
# no memory: a ring never holds more than its window.
MAX_TOKENS = 1 << 28
STEP_INPUTS = 16   # different tokens a decode state goes round

_LLAMA = dict(layers=32, heads=32, kv_heads=8, dim=128, dtype="bf16")
_TINY = dict(layers=1, heads=4, kv_heads=4, dim=64, dtype="f32", pattern="uniform", w=64)
_PLAIN = dict(by_layer=False, slots=-1, phi=0, merge=0, gated=False)


def _case(name, kind, shape, **kw):
    c = dict(_PLAIN, name=name, kind=kind, tokens=0, w=0)
    c.update(shape)
    c.update(kw)
    return c


def windows_of(case):
    n, w, pattern = case["layers"], case["w"], case["pattern"]
    if pattern == "uniform":
        return [w] * n
    if pattern == "depth":      # windows shrink with depth: 4096, 1024, 256, 64 on 4, 8, 12, 8 of 32 layers
        return [w] * (n // 8) + [w // 4] * (n // 4) + [w // 16] * (3 * n // 8) + [w // 64] * (n - n // 8 - n // 4 - 3 * n // 8)
    if pattern == "block":      # the block-wise allocation (0, w/2, w): the last block is purely linear
        return configs.blockwise_windows(w, (0, w // 2, w), configs.three_block_split(n))
    if pattern == "decay":      # w_l = 4096 2^(-l/4), multiples of 16, at least 32
        return configs.mistral_decay_windows(n)
    if pattern == "long":       # two layers with a very long window, six middling ones, the rest short
        return [w] * 2 + [2048] * 6 + [128] * (n - 8)
    raise ValueError(pattern)


def listed():
    return [
        # The smallest calls: one fp32 layer of 4 heads, 512-token prompt.  Latency, launches and host work.
        _case("decode_tiny_f32", "decode", _TINY, batch=1, context=512),
        _case("prefill_tiny_f32", "prefill", _TINY, batch=1, context=0, tokens=512),
        # Interactive decode of one 32K-token sequence, the whole stack in one call ...
        _case("decode_b1_32k", "decode", _LLAMA, pattern="depth", w=4096, batch=1, context=32768),
        # ... and layer by layer, as a model runs it.
        _case("decode_layers_b1_32k", "decode", _LLAMA, pattern="depth", w=4096, batch=1, context=32768, by_layer=True),
        # A serving batch.
        _case("decode_b16_16k", "decode", _LLAMA, pattern="depth", w=4096, batch=16, context=16384),
        # Long documents: 128K tokens, two layers that keep all of them.
        _case("decode_b4_128k", "decode", _LLAMA, pattern="long", w=131072, batch=4, context=131072),
        # The learned feature map.
        _case("decode_learned_b1_32k", "decode", _LLAMA, pattern="depth", w=4096, batch=1, context=32768, phi=1),
        # Continuous batching: slots of different lengths, two of them idle.
        _case("decode_slots_b7_8k", "decode", _LLAMA, pattern="decay", batch=7, context=8192, slots=2),
        # One long prompt, layer by layer, a length that is no multiple of any tile.
        _case("prefill_layers_b1_8k", "prefill", _LLAMA, pattern="depth", w=4096, batch=1, context=0, tokens=8001, by_layer=True),
        # A batch of prompts, the whole stack in one call.
        _case("prefill_b8_2k", "prefill", _LLAMA, pattern="decay", batch=8, context=0, tokens=2048),
        # A further turn of long conversations: 1000 tokens on top of 128K.
        _case("prefill_turn_b4_128k", "prefill", _LLAMA, pattern="long", w=131072, batch=4, context=131072, tokens=1000),
        # The gated recurrence: a prompt of 1000 tokens.
        _case("prefill_gated_b1_1k", "prefill", _LLAMA, pattern="depth", w=4096, batch=1, context=0, tokens=1000, gated=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: decode or prefill, fp32 or bf16, 1 to 16 sequences, windows from a few dozen tokens to all
    of them, whole-stack and layer-by-layer calls, every option."""
    if rng.random() < 0.2:   # small fp32 contexts
        w = _log_int(rng, 16, 300)
        c = _case("", "decode", dict(_TINY, w=w, layers=rng.randint(1, 4)), batch=rng.randint(1, 4), context=_log_int(rng, 65, 2100))
        if rng.random() < 0.5:
            c.update(kind="prefill", tokens=_log_int(rng, 17, 700), context=rng.choice([0, c["context"]]))
        del c["name"]
        return c
    pattern = rng.choice(["uniform", "depth", "block", "decay", "long"])
    w = {"uniform": _log_int(rng, 32, 4096), "depth": 64 * _log_int(rng, 8, 64), "block": 2 * _log_int(rng, 32, 1024), "decay": 0,
         "long": _log_int(rng, 4096, 65536)}[pattern]
    batch = _log_int(rng, 1, 16 if pattern != "long" else 4)
    context = _log_int(rng, 1000, 32768)
    option = rng.choice(["", "", "", "learned", "gated", "sum"])
    opts = dict(phi=int(option == "learned"), gated=option == "gated", merge=rng.choice([1, 2]) if option == "sum" else 0)
    c = _case("", "decode", _LLAMA, pattern=pattern, w=w, batch=batch, context=context, **opts)
    how = rng.random()
    if how < 0.45:   # prefill: a new prompt or a further turn
        c["kind"] = "prefill"
        c["by_layer"] = rng.random() < 0.5
        most = 700 if c["gated"] else 6000
        c["tokens"] = max(16, min(most, _log_int(rng, 16, 8000)) // c["batch"])
        if rng.random() < 0.5:
            c["context"] = 0
        if c["gated"]:
            c["context"] = min(c["context"], 2000)
    elif how < 0.65:
        c["by_layer"] = True
    elif how < 0.8 and batch > 1 and not c["gated"]:
        c["slots"] = rng.randint(0, batch - 1)
    del c["name"]
    return c


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


class _Inputs:
    """Seeded inputs on the GPU.  Queries and keys have unit variance (logits of unit variance at the default scale), values
    too; gates are close to 1, as a trained decay is."""

    def __init__(self, case, seed):
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        self.dtype = _dtype(case)

    def normal(self, *shape, scale=1.0):
        x = torch.randn(shape, generator=self.gen, device="cuda", dtype=self.dtype)
        return x if scale == 1.0 else x.mul_(scale)

    def gates(self, *shape):
        return 1.0 - 0.05 * torch.rand(shape, generator=self.gen, device="cuda", dtype=torch.float32)


def _fill(g, case, inp):
    """The context's tokens, state only: layer by layer, or slot by slot where the slots hold different lengths."""
    L, B, Hkv, d, n = case["layers"], case["batch"], case["kv_heads"], case["dim"], case["context"]
    if case["slots"] >= 0:
        for b in range(B):
            if b < case["slots"]:
                g.glide_park_seq(b)
                continue
            t = max(1, n * (b + 1) // B)
            k, v = inp.normal(L, t, Hkv, d), inp.normal(L, t, Hkv, d)
            g.glide_reset_seq(b)
            g.glide_prefill_seq(b, None, k, v)
        return
    for l in range(L if n else 0):
        k, v = inp.normal(1, B, n, Hkv, d), inp.normal(1, B, n, Hkv, d)
        if case["gated"]:
            g.glide_prefill_gated(None, k, v, inp.gates(1, B, n, Hkv), layer_begin=l, layer_count=1)
        else:
            g.glide_prefill(None, k, v, layer_begin=l, layer_count=1)


def prepare(case, seed):
    L, B, H, Hkv, d = case["layers"], case["batch"], case["heads"], case["kv_heads"], case["dim"]
    inp = _Inputs(case, seed)
    kw = {}
    if case["phi"]:
        kw = dict(phi=glide.GLIDE_PHI_PROJ_SOFTMAX2, phi_wq=inp.normal(L, H, d, d, scale=d ** -0.5),
                  phi_wk=inp.normal(L, Hkv, d, d, scale=d ** -0.5))
    g = glide.Glide(windows_of(case), B, H, Hkv, d, MAX_TOKENS, dtype=_dtype(case), merge=case["merge"], gated=case["gated"], **kw)
    _fill(g, case, inp)
    steps = []
    for _ in range(STEP_INPUTS if case["kind"] == "decode" else 1):
        q, k, v = inp.normal(L, B, H, d), inp.normal(L, B, Hkv, d), inp.normal(L, B, Hkv, d)
        steps.append((q, k, v, inp.gates(L, B, Hkv) if case["gated"] else None))
    state = dict(g=g, case=case, steps=steps, at=0, out=torch.zeros_like(steps[0][0]))
    if case["kind"] == "prefill":
        T = case["tokens"]
        state["prompt"] = (inp.normal(L, B, T, H, d), inp.normal(L, B, T, Hkv, d), inp.normal(L, B, T, Hkv, d),
                           inp.gates(L, B, T, Hkv) if case["gated"] else None)
        state["prompt_out"] = torch.zeros_like(state["prompt"][0])
    return state


def _step(state):
    """One token for every layer and sequence; the layer's attention output goes to the state's own buffer."""
    g, case, out = state["g"], state["case"], state["out"]
    q, k, v, gate = state["steps"][state["at"]]
    state["at"] = (state["at"] + 1) % len(state["steps"])
    if case["gated"]:
        g.glide_decode_step_gated(q, k, v, gate, out)
    elif case["by_layer"]:
        for l in range(case["layers"]):
            g.glide_decode_step_layers(q[l:l + 1], k[l:l + 1], v[l:l + 1], out[l:l + 1], l, 1)
    else:
        g.glide_decode_step(q, k, v, out)
    return out


def run(state):
    """One pass.  The library keeps rings and recurrent state in its own workspace, where no caller reads them; what a pass
    leaves there is seen in the outputs of the passes after it."""
    case, g = state["case"], state["g"]
    if case["kind"] == "decode":
        return _step(state)
    # A prompt, then the first generated token: its output is read from the state that the prompt has left (window rows
    # and recurrent state), so a wrong state shows in it.
    q, k, v, gate = state["prompt"]
    out = state["prompt_out"]
    if case["context"] == 0:
        g.glide_reset()
    ranges = [(l, 1) for l in range(case["layers"])] if case["by_layer"] else [(0, case["layers"])]
    for l, n in ranges:
        s = slice(l, l + n)
        if case["gated"]:
            g.glide_prefill_gated(q[s], k[s], v[s], gate[s], out[s], layer_begin=l, layer_count=n)
        else:
            g.glide_prefill(q[s], k[s], v[s], out[s], layer_begin=l, layer_count=n)
    return out, _step(state)


def _positions(case):
    """Tokens each live sequence holds before the pass."""
    n, B = case["context"], case["batch"]
    if case["slots"] < 0:
        return [n] * B
    return [max(1, n * (b + 1) // B) for b in range(case["slots"], B)]


def _step_work(case, positions):
    H, Hkv, d = case["heads"], case["kv_heads"], case["dim"]
    elem = 4 if case["dtype"] == "f32" else 2
    feat = (2 if case["phi"] else 1) * d
    byts = flops = 0
    for w in windows_of(case):
        for n in positions:
            seen = min(w, n + 1)
            byts += 2 * seen * Hkv * d * elem + (2 * H + 2 * Hkv) * d * elem + (2 * Hkv * d * elem if w else 0)
            flops += 4 * H * d * seen
            if n >= w or case["merge"] == 2:
                byts += 2 * Hkv * (feat * d + feat) * 4
                flops += 2 * (H + Hkv) * feat * d
        if case["phi"]:
            byts += (H + Hkv) * d * d * elem
            flops += 2 * (H + Hkv) * d * d * len(positions)
    return byts, flops


def work(case):
    """One pass: every input and every window row or state that the results depend on read once, every result written
    once.  Prefill: the call's own tensors, the rings' rows older than the call, the state read and written; multiply-adds
    of the causal window products, of the state's readout and of its update."""
    positions = _positions(case)
    if case["kind"] == "decode":
        byts, flops = _step_work(case, positions)
        return dict(bytes=byts, flops=flops)
    T = case["tokens"]
    byts, flops = _step_work(case, [n + T for n in positions])
    H, Hkv, d = case["heads"], case["kv_heads"], case["dim"]
    elem = 4 if case["dtype"] == "f32" else 2
    feat = (2 if case["phi"] else 1) * d
    for w in windows_of(case):
        for n in positions:
            byts += T * (2 * H + 2 * Hkv) * d * elem + 2 * min(w, n) * Hkv * d * elem + 2 * min(w, T) * Hkv * d * elem
            full = max(0, min(T, n + T - w + 1) if n < w else T)     # queries with a full window
            part = T - full                                          # the others see all tokens up to themselves
            pairs = full * w + part * n + part * (part + 1) // 2
            flops += 4 * H * d * pairs
            evicted = max(0, n + T - (0 if case["merge"] == 2 else w))
            if evicted:
                late = min(T, evicted)
                byts += 2 * Hkv * (feat * d + feat) * 4
                flops += 2 * (H + Hkv) * feat * d * late
                if case["phi"]:
                    flops += 2 * (H + Hkv) * d * d * late
        if case["phi"]:
            byts += (H + Hkv) * d * d * elem
    return dict(bytes=byts, flops=flops)


def tolerance(case):
    """bf16: the tensor-core kernels and the fp32 CUDA-core kernels differ by 1.9e-3 to 2.3e-3 (2-norm) and by up to 0.053 in
    one value on these inputs (window weights and outputs rounded to bf16): four times that.  fp32: the same formula in fp32
    against fp64 differs by 2.6e-7, two orders of the fp32 sums by 2.4e-7; twice as much for the longer sums of the larger
    contexts, times four."""
    return dict(rel=2e-6, max=1e-4) if case["dtype"] == "f32" else dict(rel=8.5e-3, max=0.2)
