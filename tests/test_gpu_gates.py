"""The gated recurrence where its gates matter: a state that lasts over many chunks, gates of 0, gates that are not numbers, and
the precision of the tensor-core prefill against that of the CUDA-core one."""
import numpy as np
import pytest
import torch

from oracle import glide_oracle as orc
from paper_2607_24788_b200 import glide
from tests.parity_util import f32_scale, run_case, to_np

pytestmark = pytest.mark.gpu
BF16, F32 = torch.bfloat16, torch.float32


# Gates of 0.99 to 1: a chunk of 64 to 256 tokens leaves a quarter to three quarters of the state it started from.  The
# CUDA-core passes with the sums of the chunks before (four chunks) and with a scan (eleven, five), the tcgen05 kernel with
# passes of one chunk (prefill_chunk 64) and of several, the learned map, decode of a state that has lasted
@pytest.mark.parametrize("dtype,d,G,calls,kw", [
    (F32, 64, 1, [256, 30], dict(prefill_chunk=64)), (F32, 64, 2, [700], {}), (F32, 128, 4, [400, 99], dict(prefill_chunk=80)),
    (BF16, 64, 2, [500], {}), (BF16, 128, 4, [700, 40], {}), (BF16, 128, 2, [300], dict(prefill_chunk=64)), (BF16, 128, 8, [600], dict(prefill_chunk=144)),
    (BF16, 128, 1, [300, 1, 30], dict(phi=1)), (F32, 64, 1, [130], dict(phi=1, prefill_chunk=32))])
def test_states_that_last(dtype, d, G, calls, kw):
    run_case([0, 40, 200], 2, 2 * G, 2, d, dtype, calls, 6, amp=4 * d ** -0.5, seed=79 + G, gated=True, gate_lo=0.99, **kw)


# A gate of 0 empties the state.  (Every 200th token: the running sums of log-gates inside a chunk then stay below 210, where
# two of them differ by at most 2^-17 from what they should: 8e-6 of a weight.)
@pytest.mark.parametrize("dtype,d,G,calls,kw", [
    (F32, 64, 1, [450], {}), (F32, 128, 2, [300, 60], dict(prefill_chunk=64)), (BF16, 128, 4, [700, 20], {}),
    (BF16, 128, 2, [150, 150], dict(prefill_chunk=64)), (F32, 64, 2, [220], dict(phi=1, prefill_chunk=64))])
def test_a_gate_of_zero_empties_the_state(dtype, d, G, calls, kw):
    run_case([0, 40, 150], 2, 2 * G, 2, d, dtype, calls, 3, amp=4 * d ** -0.5, seed=83 + G, gated=True, gate_lo=0.95, zero_gate_every=200, **kw)


@pytest.mark.parametrize("dtype,d,kw", [(F32, 64, {}), (BF16, 128, {}), (BF16, 128, dict(prefill_impl=glide.GLIDE_PREFILL_FMA))])
def test_a_gate_that_is_no_number_shows(dtype, d, kw):
    """Token 150 enters the state of a window of 40 with token 190: outputs before it are untouched, all later ones are NaN."""
    T, H, Hkv, w = 300, 4, 2, 40
    gen = torch.Generator(device="cuda").manual_seed(89)
    q, k, v = (torch.randn((1, 1, T, h, d), generator=gen, device="cuda").to(dtype) for h in (H, Hkv, Hkv))
    gate = 0.95 + 0.05 * torch.rand((1, 1, T, Hkv), generator=gen, device="cuda")
    outs = []
    for bad in (False, True):
        if bad:
            gate[:, :, 150] = float("nan")
        g = glide.Glide([w], 1, H, Hkv, d, 1 << 20, dtype=dtype, gated=True, **kw)
        outs.append(torch.zeros_like(q))
        g.glide_prefill_gated(q, k, v, gate, outs[-1])
        assert g.glide_device_status() == 0
        g.glide_destroy()
    assert torch.equal(outs[1][:, :, :190], outs[0][:, :, :190])
    assert bool(torch.isnan(outs[1][:, :, 190:].float()).all())


@pytest.mark.parametrize("w,gate_lo", [(64, 0.95), (64, 0.99), (256, 0.999)])
def test_precision_of_the_tensor_core_prefill(w, gate_lo):
    """Outputs and state of 1000 tokens, bf16, against the fp64 oracle, by the tcgen05 kernel and by the CUDA cores.
    Outputs: what is rounded to bf16 differs from the exact value by the split operands' 2^-17 or so (1e-5), which adds
    (1e-5 / 1.6e-3)^2 / 2 = 2e-5 of it to the rounding's own 1.6e-3.  State: fp32 sums of up to 1000 terms of one sign, three-way
    splits of 2^-24; one rounding per 32 tokens and per chunk (measured 2e-7; summed up in the tensor core alone 7.6e-7)."""
    T, H, Hkv, d = 1000, 8, 2, 128
    gen = torch.Generator().manual_seed(97)
    q, k, v = (torch.randn((1, 1, T, h, d), generator=gen).to(BF16).cuda() for h in (H, Hkv, Hkv))
    gate = (gate_lo + (1 - gate_lo) * torch.rand((1, 1, T, Hkv), generator=gen)).cuda()
    stack = orc.Stack([w], 1, H, Hkv, d, f32_scale(d))
    ref = stack.prefill(to_np(q), to_np(k), to_np(v), gate=to_np(gate))
    oS = stack.cells[0][0].export()[2]
    err = {}
    for impl in (glide.GLIDE_PREFILL_AUTO, glide.GLIDE_PREFILL_FMA):
        g = glide.Glide([w], 1, H, Hkv, d, 1 << 20, dtype=BF16, softmax_scale=f32_scale(d), gated=True, prefill_impl=impl)
        out = torch.zeros_like(q)
        g.glide_prefill_gated(q, k, v, gate, out)
        S = to_np(g.glide_export_state(0)[2][0])
        err[impl] = (np.linalg.norm(to_np(out) - ref) / np.linalg.norm(ref), np.linalg.norm(S - oS) / np.linalg.norm(oS))
        g.glide_destroy()
    print(f"w={w} gates {gate_lo}..1: outputs, S: tcgen05 {err[0]}, CUDA cores {err[3]}")
    assert err[glide.GLIDE_PREFILL_AUTO][0] <= err[glide.GLIDE_PREFILL_FMA][0] * (1 + 2e-5)
    assert err[glide.GLIDE_PREFILL_AUTO][1] <= 3e-7


# phi(q) is made from the Q tile that TMA wrote (neighbouring heads of a group) or that its own threads copied (heads of a group
# apart): the same rows either way, so the same bits
@pytest.mark.parametrize("G,kw", [(2, {}), (4, dict(merge=1)), (4, dict(gated=True)), (8, {})])
def test_order_of_heads(G, kw):
    T, Hkv, d, H = 200, 2, 128, 2 * G
    gen = torch.Generator(device="cuda").manual_seed(101)
    q, k, v = (torch.randn((1, 1, T, h, d), generator=gen, device="cuda").to(BF16) for h in (H, Hkv, Hkv))
    apart = [h % Hkv for h in range(H)]                                   # query head h belongs to KV head h % 2
    order = sorted(range(H), key=lambda h: (apart[h], h))                 # its heads side by side
    outs = []
    for heads, q_to_kv in ((order, None), (list(range(H)), apart)):
        g = glide.Glide([16], 1, H, Hkv, d, 1 << 20, dtype=BF16, q_to_kv=q_to_kv, **kw)
        out = torch.zeros_like(q)
        g.glide_prefill(q[:, :, :, heads].contiguous(), k, v, out)
        outs.append(out)
        g.glide_destroy()
    assert torch.equal(outs[0], outs[1][:, :, :, order])


def _gated_outputs_f64(q, k, v, gate, w, n0):
    """Outputs of tokens n0 .. of one sequence, shared normaliser, in fp64: q [T][H][d] from token n0 on, k, v, gate of all tokens."""
    N, Hkv, d = k.shape
    G, j = q.shape[1] // Hkv, torch.arange(N, device=q.device)
    t = j[n0:, None]
    outs = []
    for h in range(q.shape[1]):
        qq, kk, vv, log_g = q[:, h].double(), k[:, h // G].double(), v[:, h // G].double(), gate[:, h // G].double().log().cumsum(0)
        s = torch.where((j <= t) & (j > t - w), qq @ kk.T * f32_scale(d), -torch.inf)
        m = s.amax(-1, keepdim=True)
        phi = torch.softmax(qq, -1) @ torch.softmax(kk, -1).T * (log_g[(t - w).clamp(min=0)] - log_g[None]).clamp(max=0).exp()
        p = (s - m).exp() + torch.where(j <= t - w, phi * (-m).exp(), 0.)
        outs.append(p @ vv / p.sum(-1, keepdim=True))
    return torch.stack(outs, 1)


# Key tiles without a masked key on the tcgen05 kernel: rows of every group size, a window whose first whole tile is also the row's
# first (a turn behind a long context), scores that grow from tile to tile, so that the reference moves in each, and scores that stay.
# Bound: an output is within 2^-9 of itself when it is rounded to bf16; two split terms of the weights and V in bf16 add 2^-17.
@pytest.mark.parametrize("G,w,n0,T,growing", [(1, 700, 900, 300, True), (2, 1 << 20, 0, 700, True), (4, 512, 1024, 200, False), (4, 385, 640, 129, True),
                                              (8, 300, 513, 97, False), (8, 1 << 20, 1000, 33, True)])
def test_gated_key_tiles_without_a_masked_key(G, w, n0, T, growing):
    N, Hkv, d = n0 + T, 2, 128
    gen = torch.Generator(device="cuda").manual_seed(113 + G)
    q, k, v = (torch.randn((1, 1, N, h, d), generator=gen, device="cuda") for h in (Hkv * G, Hkv, Hkv))
    if growing:   # (the largest of 128 scores grows by more than 2^8 per tile)
        k *= (1 + torch.arange(N, device="cuda") / 32).view(1, 1, N, 1, 1)
    q, k, v = (x.to(BF16) for x in (q, k, v))
    gate = 0.99 + 0.01 * torch.rand((1, 1, N, Hkv), generator=gen, device="cuda")
    g = glide.Glide([w], 1, Hkv * G, Hkv, d, 1 << 20, dtype=BF16, softmax_scale=f32_scale(d), gated=True)
    if n0:
        g.glide_prefill_gated(None, *(x[:, :, :n0].contiguous() for x in (k, v, gate)), None)
    new = [x[:, :, n0:].clone() for x in (q, k, v, gate)]   # (a slice of one sequence is contiguous, but not on a multiple of 16 bytes)
    out = torch.full_like(new[0], float("nan"))
    g.glide_prefill_gated(*new, out)
    assert g.glide_device_status() == 0
    want = _gated_outputs_f64(new[0][0, 0], k[0, 0], v[0, 0], gate[0, 0], w, n0)
    assert ((out[0, 0] - want).norm() / want.norm()).item() <= 2.0 ** -9 + 2.0 ** -17


def test_a_gated_long_window_takes_its_products_time():
    """A gated key tile has three products where one without gates has two (K, and V with the weights' two terms): on long windows
    the call takes no longer than that by more than a fifteenth (1.33 times as long; 1.68 when whole tiles went through the masked
    tiles' code)."""
    T, H, Hkv, d, w, n = 2048, 32, 8, 128, 16384, 3
    gen = torch.Generator(device="cuda").manual_seed(127)
    q, k, v = (torch.randn((2, 1, T, h, d), generator=gen, device="cuda").to(BF16) for h in (H, Hkv, Hkv))
    out, took = torch.empty_like(q), {}
    for gated in (False, True):
        g = glide.Glide([w, w], 1, H, Hkv, d, 1 << 20, dtype=BF16, gated=gated)
        for _ in range(w // T):
            g.glide_prefill(None, k, v, None)
        times = []
        for _ in range(1 + n):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.glide_prefill(q, k, v, out)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        took[gated] = min(times[1:])
        g.glide_destroy()
    print(f"without gates {took[False]:.3f} ms, gated {took[True]:.3f}")
    assert took[True] <= 1.6 * took[False]
