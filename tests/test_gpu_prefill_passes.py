"""Prefill passes of the tensor-core pipeline: several chunks per pass (their sums go over consumed scratch rows and are added
up by a scan), passes of few layers, and the gated recurrence on the tcgen05 kernel with split operands; against the oracle."""
import pytest
import torch

from paper_2607_24788_b200 import glide
from tests.parity_util import run_case

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


# chunk 144: the smallest with room for a chunk's sums (129 rows) that is no multiple of 128; 64: passes of one chunk.
# Calls of 1 token, of a chunk and one token, and of more chunks than a pass holds for one layer (6 layers: 6 chunks).
@pytest.mark.parametrize("chunk,calls", [(144, [145, 1, 300]), (256, [1, 600, 257]), (144, [1000]), (64, [130, 65])])
@pytest.mark.parametrize("kw", [dict(), dict(merge=glide.GLIDE_MERGE_SUM_EVICTED), dict(phi=1), dict(gated=True)],
                         ids=["shared", "sum", "learned", "gated"])
def test_passes_of_several_chunks(chunk, calls, kw):
    run_case([0, 16, 100, 128, 304, 1 << 20], 1, 4, 2, 128, BF16, calls, 2, amp=128 ** -0.5 * 4, seed=41, prefill_chunk=chunk, **kw)


# one query head per KV head to eight (rows of a tile per token), two sequences, the call boundary inside a key tile
@pytest.mark.parametrize("G,chunk,calls", [(1, 0, [300, 131]), (2, 512, [40, 520]), (8, 0, [70, 33, 5])])
def test_gated_prefill_on_tcgen05(G, chunk, calls):
    run_case([0, 33, 129, 1 << 20], 2, 2 * G, 2, 128, BF16, calls, 2, amp=128 ** -0.5 * 4, seed=43 + G, gated=True, prefill_chunk=chunk)


# CUDA-core passes: chunk sums per unit from one (prefill_chunk 16) to four, calls of one token, of a chunk and one token, of
# several passes; row tiles of 16 to 2 tokens; every merge
@pytest.mark.parametrize("dtype,d,G,merge,chunk,calls", [
    (torch.float32, 64, 1, 0, 0, [1, 65, 512]), (torch.float32, 64, 4, 1, 0, [700, 3]), (torch.float32, 128, 2, 2, 0, [130, 257]),
    (torch.float32, 64, 8, 0, 16, [40, 300]), (torch.float32, 128, 1, 0, 512, [600]), (BF16, 64, 2, 0, 0, [65, 300])])
@pytest.mark.parametrize("gated", [False, True])
def test_cuda_core_passes(dtype, d, G, merge, chunk, calls, gated):
    amp = 4 * d ** -0.5
    run_case([0, 16, 100, 300, 1 << 20], 2, 2 * G, 2, d, dtype, calls, 2, amp=amp, seed=47 + G, merge=merge, gated=gated and merge == 0,
             prefill_chunk=chunk)


# one CTA per unit (decode on the CUDA cores): rings at and beside the length where the work list takes over, rows not
# filling a warp's batch, every merge, the learned map, gates
@pytest.mark.parametrize("dtype,d,G,windows,kw", [
    (torch.float32, 64, 1, [0, 1, 63, 512], dict()), (torch.float32, 64, 1, [513, 64], dict()), (torch.float32, 128, 8, [320, 7], dict()),
    (torch.float32, 128, 2, [321], dict(merge=1)), (BF16, 128, 4, [40, 0], dict(merge=2, decode_impl=glide.GLIDE_DECODE_FMA)),
    (torch.float32, 128, 4, [33, 0, 1 << 20], dict(phi=1)), (torch.float32, 64, 2, [31, 0], dict(gated=True))])
def test_decode_by_unit(dtype, d, G, windows, kw):
    run_case(windows, 2, 2 * G, 2, d, dtype, [70], 3, amp=4 * d ** -0.5, seed=53 + G, max_tokens=600, **kw)


# CUDA-core passes of so many chunks that their sums are scanned (more than 8 of d = 64, 4 of d = 128), with the first delayed
# token in the pass's first, a middle and its last chunk; gates
@pytest.mark.parametrize("dtype,d,G,chunk,calls,gated", [
    (torch.float32, 64, 1, 0, [700, 90], False), (torch.float32, 64, 4, 64, [640, 1], True), (torch.float32, 128, 2, 80, [500, 33], False),
    (BF16, 64, 2, 0, [650], True)])
def test_cuda_core_passes_with_a_scan(dtype, d, G, chunk, calls, gated):
    run_case([0, 64, 300, 630], 2, 2 * G, 2, d, dtype, calls, 2, amp=4 * d ** -0.5, seed=73 + G, gated=gated, prefill_chunk=chunk)


# The same prompt with outputs (many chunks of few layers, their sums scanned) and without (one chunk of all layers after the other,
# sums straight to S), in one call and in calls of two chunks: the same additions, so the same bits.  (Not so for the sum-of-terms
# merges in bf16, whose phi comes from another kernel when there are outputs.)
@pytest.mark.parametrize("dtype,d,kw", [
    (BF16, 128, dict(prefill_chunk=256)), (BF16, 128, dict(prefill_chunk=144, gated=True)),
    (torch.float32, 64, dict(prefill_chunk=32)), (torch.float32, 128, dict(prefill_chunk=16, merge=2))])
def test_passes_leave_the_same_state(dtype, d, kw):
    chunk, L = kw["prefill_chunk"], 5
    T = 4 * chunk + 9
    gen = torch.Generator(device="cuda").manual_seed(107)
    q, k, v = (torch.randn((L, 1, T, h, d), generator=gen, device="cuda").to(dtype) for h in (4, 2, 2))
    states = []
    for with_outputs, step in ((True, T), (False, T), (True, 2 * chunk)):
        g = glide.Glide([0, 16, 100, 300, 1 << 20], 1, 4, 2, d, 1 << 20, dtype=dtype, **kw)
        for c in range(0, T, step):
            part = [x[:, :, c:c + step].contiguous() for x in (q, k, v)]
            g.glide_prefill(part[0] if with_outputs else None, part[1], part[2], torch.empty_like(part[0]) if with_outputs else None)
        # (slots that no token has reached hold whatever the workspace held: a ring longer than the prompt is compared up to T)
        states.append([x[:, :, :T].clone() if i < 2 else x.clone() for l in range(4) for i, x in enumerate(g.glide_export_state(l))])
        assert g.glide_device_status() == 0
        g.glide_destroy()
    for other in states[1:]:
        for a, b in zip(states[0], other):
            assert torch.equal(a, b)


# Chunk sums on tcgen05: stages of 32 tokens with every kind of remainder, the first delayed token inside a stage, chunks from one
# stage to the largest (passes of one chunk update S in place), rings that wrap, no ring at all.  Against fp64; bound: the tensor core
# adds 3 chunk / 16 products to a running sum without rounding to nearest (2^-23 of it each at most), the scan one sum per chunk.
@pytest.mark.parametrize("chunk,w,calls", [(64, 16, [97]), (144, 0, [145, 31]), (160, 33, [481, 1]), (256, 300, [513, 40, 700]), (1024, 31, [1055]),
                                           (0, 100, [101, 1000])])
def test_chunk_sums_on_tcgen05(chunk, w, calls):
    T = sum(calls)
    gen = torch.Generator(device="cuda").manual_seed(chunk + w)
    q, k, v = (torch.randn((1, 2, T, h, 128), generator=gen, device="cuda").to(BF16) for h in (4, 2, 2))
    g = glide.Glide([w], 2, 4, 2, 128, 1 << 20, prefill_chunk=chunk)
    at = 0
    for n in calls:
        part = [x[:, :, at:at + n].contiguous() for x in (q, k, v)]
        g.glide_prefill(*part, torch.empty_like(part[0]))
        at += n
    S, z = g.glide_export_state(0)[2:]
    phi = torch.softmax(k[0].double(), -1)[:, :T - w].transpose(1, 2)
    for got, want in ((S, phi.transpose(-1, -2) @ v[0, :, :T - w].double().transpose(1, 2)), (z, phi.sum(2))):
        bound = (3 * (chunk or 256) / 16 + T / (chunk or 256) + 2) * 2.0 ** -23
        assert ((got - want).norm() / want.norm()).item() <= bound
    assert g.glide_device_status() == 0


# Launches that start while the one before them runs out (programmatic dependent launch): reset, prompt of several passes and decode
# steps issued back to back leave the bits that they leave with the device idle between any two calls.
@pytest.mark.parametrize("dtype,d,heads,windows,kw", [
    (torch.float32, 64, 2, [64], dict()), (torch.float32, 64, 2, [0, 16, 100], dict(gated=True)), (torch.float32, 128, 8, [40, 0], dict(prefill_chunk=16)),
    (BF16, 128, 8, [0, 16, 100, 300], dict(prefill_chunk=144)), (BF16, 128, 8, [16, 600, 100], dict(gated=True)), (BF16, 128, 4, [33, 0], dict(merge=1))])
def test_calls_back_to_back(dtype, d, heads, windows, kw):
    L, T, steps = len(windows), 700, 4
    gen = torch.Generator(device="cuda").manual_seed(109)
    q, k, v = (torch.randn((L, 2, T + steps, h, d), generator=gen, device="cuda").to(dtype) for h in (heads, 2, 2))
    prompt, tokens = [x[:, :, :T].contiguous() for x in (q, k, v)], [[x[:, :, T + i].contiguous() for x in (q, k, v)] for i in range(steps)]
    results = []
    for idle in (True, False, False):
        g = glide.Glide(windows, 2, heads, 2, d, 1 << 20, dtype=dtype, **kw)
        outs = [torch.empty_like(prompt[0])] + [torch.empty_like(t[0]) for t in tokens]
        torch.cuda.synchronize()
        for _ in range(2):   # (the second prompt begins in what the first has left)
            decode = [lambda t=t, o=o: g.glide_decode_step(*t, o) for t, o in zip(tokens, outs[1:])]
            for call in [g.glide_reset, lambda: g.glide_prefill(*prompt, outs[0])] + decode:
                call()
                if idle:
                    torch.cuda.synchronize()
        state = [x for l, w in enumerate(windows) for x in g.glide_export_state(l)[(0 if w else 2):]]
        assert g.glide_device_status() == 0
        results.append(outs + state)
        g.glide_destroy()
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert torch.equal(a, b)


def _time_ms(run, repeats=6):
    """The shortest of some runs (the first one left out), by events around it; all of a run is queued before the device begins it."""
    times = []
    for _ in range(repeats + 1):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(8_000_000)   # (4 ms and more)
        a.record()
        run()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return min(times[1:])


# The thread blocks of a launch that has started early keep their places while they wait, and what is launched behind them gets the
# places that are left.  Each case is one that this made slower than launches that do not overlap (thread blocks for less than half of
# the SMs, long chains of launches): back to back against the same tokens with an event, which nothing overlaps, between any two calls.
# The bounds lie between the ratios with the next launch let go as late as is useful (0.74, 0.40, 0.89) and at a kernel's beginning
# (0.82, 0.50, 1.03).
@pytest.mark.parametrize("what,bound", [("decode", 0.79), ("cuda-core prefill", 0.45), ("gated prefill", 0.96)])
def test_overlapping_launches_hold_nothing_up(what, bound):
    gen = torch.Generator(device="cuda").manual_seed(131)
    rows = lambda L, n, h, d, dtype: torch.randn((L, 1, n, h, d), generator=gen, device="cuda").to(dtype)
    if what == "decode":
        g = glide.Glide([512] * 8, 1, 8, 8, 64, 1 << 20, dtype=torch.float32)
        q, k, v, out = (rows(8, 600, 8, 64, torch.float32) for _ in range(4))
        g.glide_prefill(None, k, v, None)
        step = [x[:, :, 0].contiguous() for x in (q, k, v, out)]
        together = lambda: [g.glide_decode_step(*step) for _ in range(32)]
        calls = [lambda: g.glide_decode_step(*step)] * 32
    elif what == "cuda-core prefill":
        g = glide.Glide([64, 300], 1, 4, 4, 128, 1 << 20, dtype=torch.float32, prefill_chunk=256)
        k, v = (rows(2, 8192, 4, 128, torch.float32) for _ in range(2))
        together = lambda: g.glide_prefill(None, k, v, None)
        parts = [[x[:, :, c:c + 256].contiguous() for x in (k, v)] for c in range(0, 8192, 256)]
        calls = [lambda p=p: g.glide_prefill(None, *p, None) for p in parts]
    else:
        g = glide.Glide([4096, 1024, 256, 64], 1, 32, 8, 128, 1 << 20, dtype=BF16, gated=True)
        k, v = (rows(4, 4096, 8, 128, BF16) for _ in range(2))
        together = lambda: g.glide_prefill_gated(None, k, v, None, None)
        parts = [[x[:, :, c:c + 256].contiguous() for x in (k, v)] for c in range(0, 4096, 256)]
        calls = [lambda p=p: g.glide_prefill_gated(None, *p, None, None) for p in parts]
    between = torch.cuda.Event(enable_timing=True)

    def apart():
        for call in calls:
            call()
            between.record()

    t_together, t_apart = _time_ms(together), _time_ms(apart)
    assert g.glide_device_status() == 0
    g.glide_destroy()
    print(f"{what}: {t_together * 1e3:.1f} us, with events between {t_apart * 1e3:.1f}")
    assert t_together <= bound * t_apart


# A chunk's sum in passes of several chunks (their sums by row in the scratch, added up by the scan): six layers, a call with outputs of
# three chunks or more, so that a pass holds three at least.  The layer with w = T - 1 has one delayed token, of the pass's last chunk,
# w = T - 3 three.  Chunk 144: stages with a remainder.
def _states_after(windows, chunk, calls, B=2):
    T = sum(calls)
    gen = torch.Generator(device="cuda").manual_seed(chunk + T)
    q, k, v = (torch.randn((len(windows), B, T, h, 128), generator=gen, device="cuda").to(BF16) for h in (4, 2, 2))
    g = glide.Glide(windows, B, 4, 2, 128, 1 << 20, prefill_chunk=chunk)
    at = 0
    for n in calls:
        part = [x[:, :, at:at + n].contiguous() for x in (q, k, v)]
        g.glide_prefill(*part, torch.empty_like(part[0]))
        at += n
    states = [g.glide_export_state(l)[2:] for l in range(len(windows))]
    assert g.glide_device_status() == 0
    g.glide_destroy()
    return k, v, states


# Bound: the tensor core adds without rounding to nearest, so the error grows with the number of products added to a running sum, 3 of
# 16 tokens each; 8.2e-7 was measured with chunks of 256 tokens, random keys and values.  Not twice that, and in proportion for
# longer chunks.  (A phi of two terms instead of three is 2.3e-6 to 2.6e-6 off by itself.)
@pytest.mark.parametrize("chunk,calls", [(144, [1000]), (256, [700, 900]), (1024, [3100])])
def test_sums_of_several_chunks_against_fp64(chunk, calls):
    windows, T, bound = [0, 16, 100, 304, 31, 1 << 20], sum(calls), 1.5e-6 * max(1, chunk / 256)
    k, v, states = _states_after(windows, chunk, calls)
    for l, w in enumerate(windows[:-1]):
        S, z = states[l]
        phi = torch.softmax(k[l].double(), -1)[:, :T - w].transpose(1, 2)
        want = phi.transpose(-1, -2) @ v[l][:, :T - w].double().transpose(1, 2)
        err, errz = ((S - want).norm() / want.norm()).item(), ((z - phi.sum(2)).norm() / phi.sum(2).norm()).item()
        print(f"chunk {chunk}, w = {w}: S {err:.2e}, z {errz:.2e}")
        assert err <= bound and errz <= bound


# One delayed token: z is its phi(k) in fp32 and S the products of the three terms of that with V, exact but for two sums of the tensor
# core, each operand of which loses less than 2^-23 of the result.  (Without the third term 2^-18 at most, 2e-6 on average.)  A pass of
# one chunk and passes of several; three tokens: three such sums each.
@pytest.mark.parametrize("layers,chunk", [(1, 64), (1, 256), (6, 144), (6, 256)])
def test_terms_of_phi_in_the_carry(layers, chunk):
    T = 3 * chunk + 17
    k, v, states = _states_after([T - 1, T - 3, 16, 100, 304, 0][:layers], chunk, [T])
    S, z = (x.double() for x in states[0])
    exact = z[..., None] * v[0][:, 0].double()[:, :, None, :]
    assert ((S - exact).abs() <= 4 * 2.0 ** -23 * exact.abs()).all()
    if layers > 1:
        S, z = (x.double() for x in states[1])
        phi = torch.softmax(k[1].double(), -1)[:, :3].transpose(1, 2)
        want = phi.transpose(-1, -2) @ v[1][:, :3].double().transpose(1, 2)
        # (phi itself: the exponent is rounded at up to 2^3, the sum and the quotient: 8 2^-24 ln 2 and a few 2^-24)
        assert ((S - want).norm() / want.norm()).item() <= (8 + 8) * 2.0 ** -24


# As test_calls_back_to_back, for calls that it leaves out: slots of different lengths, reset, parked and filled again between steps (the
# streaming decode kernel reads their offsets before it waits for what is in front), and layer by layer, with the learned map (its
# feature kernel asks for its matrices before it waits) and without.
@pytest.mark.parametrize("kind,dtype,d,heads,kw", [
    ("slots", BF16, 128, 8, dict()), ("slots", torch.float32, 64, 4, dict()), ("slots", BF16, 128, 8, dict(gated=True)), ("layers", BF16, 128, 8, dict(phi=1)),
    ("layers", BF16, 128, 8, dict()), ("layers", torch.float32, 64, 2, dict()), ("layers", torch.float32, 128, 4, dict(phi=1))])
def test_slots_and_layers_back_to_back(kind, dtype, d, heads, kw):
    windows, B, T, steps = [0, 16, 300], 3, 400, 4
    L, kw = len(windows), dict(kw)
    gen = torch.Generator(device="cuda").manual_seed(137)
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda").to(dtype)
    if kw.get("phi"):
        kw.update(phi_wq=(rand(L, heads, d, d) * d ** -0.5).contiguous(), phi_wk=(rand(L, 2, d, d) * d ** -0.5).contiguous())
    prompts = [[rand(L, T - 90 * b, h, d) for h in (heads, 2, 2)] for b in range(B)]
    level = [rand(L, B, T, h, d) for h in (heads, 2, 2)]
    tokens = [[rand(L, B, h, d) for h in (heads, 2, 2)] for _ in range(steps)]
    results = []
    for idle in (True, False, False):
        g = glide.Glide(windows, B, heads, 2, d, 1 << 20, dtype=dtype, **kw)
        outs, calls = [], []

        def step(t, l=None):
            s = slice(0, L) if l is None else slice(l, l + 1)
            outs.append(torch.zeros_like(t[0][s]))
            calls.append(lambda o=outs[-1]: g.glide_decode_step(*t, o) if l is None else g.glide_decode_step_layers(*(x[s] for x in t), o, l, 1))

        def fill(b):
            outs.append(torch.zeros_like(prompts[b][0]))
            calls.extend([lambda: g.glide_reset_seq(b), lambda o=outs[-1]: g.glide_prefill_seq(b, *prompts[b], o)])

        for _ in range(2):
            if kind == "slots":
                for b in range(B):
                    fill(b)
                calls.append(lambda: g.glide_park_seq(1))
                step(tokens[0])
                step(tokens[1])
                fill(0)
                step(tokens[2])
                fill(1)
                step(tokens[3])
            else:
                calls.append(g.glide_reset)
                for l in range(L):
                    outs.append(torch.zeros_like(level[0][l:l + 1]))
                    calls.append(lambda o=outs[-1], l=l: g.glide_prefill(*(x[l:l + 1] for x in level), o, layer_begin=l, layer_count=1))
                for t in tokens[:3]:
                    for l in range(L):
                        step(t, l)
                step(tokens[3])
        torch.cuda.synchronize()
        for call in calls:
            call()
            if idle:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert g.glide_device_status() == 0
        results.append(outs + [x for l, w in enumerate(windows) for x in g.glide_export_state(l)[2:]])
        g.glide_destroy()
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert torch.equal(a, b)
