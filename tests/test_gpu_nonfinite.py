"""A value that is not finite reaches the outputs of the tokens that see its row, and no others: a query's window and state hold
tokens up to itself alone, so what stands in V behind it (a padded tail, memory never written) must not matter.  Each case
runs the same prompt twice, with and without the bad rows: outputs of tokens before them are the same but for the order of their
sums, the others are what the sums give (every weight of a finite prompt is positive)."""
import math

import pytest
import torch

from paper_2607_24788_b200 import glide

pytestmark = pytest.mark.gpu
BF16, F32 = torch.bfloat16, torch.float32


def _prompt(dtype, d, G, w, gated, calls, bad, value, **kw):
    """Outputs [T][H][d], S [Hkv][d][d]; V rows `bad` hold `value`."""
    T, Hkv = sum(calls), 2
    gen = torch.Generator(device="cuda").manual_seed(61 + d + G)
    q, k, v = (torch.randn((1, 1, T, h, d), generator=gen, device="cuda").to(dtype) for h in (G * Hkv, Hkv, Hkv))
    gate = 0.95 + 0.05 * torch.rand((1, 1, T, Hkv), generator=gen, device="cuda")
    for j in bad:
        v[0, 0, j] = value
    g = glide.Glide([w], 1, G * Hkv, Hkv, d, 1 << 20, dtype=dtype, gated=gated, **kw)
    out = torch.zeros_like(q)
    at = 0
    for n in calls:
        s = slice(at, at + n)
        part = [x[:, :, s].contiguous() for x in (q, k, v, out)]
        if gated:
            g.glide_prefill_gated(*part[:3], gate[:, :, s].contiguous(), part[3])
        else:
            g.glide_prefill(*part)
        out[:, :, s] = part[3]
        at += n
    S = g.glide_export_state(0)[2][0].clone()
    assert g.glide_device_status() == 0
    g.glide_destroy()
    return out[0, 0].float(), S


def _check(dtype, d, G, w, gated, calls, bad, value, **kw):
    clean, _ = _prompt(dtype, d, G, w, gated, calls, (), 0.0, **kw)
    got, S = _prompt(dtype, d, G, w, gated, calls, bad, value, **kw)
    first = min(bad)
    # fp32: two orders of sums of up to 300 weights of sum 1 times values below 5; bf16: neighbouring roundings
    tol = 1e-5 if dtype == F32 else 2 ** -7
    torch.testing.assert_close(got[:first], clean[:first], rtol=tol, atol=tol)
    seen = got[first:] if first < got.shape[0] else got[:0]
    assert bool((torch.isnan(seen) if math.isnan(value) else seen == value).all())
    if w <= sum(calls) - 1 - first:   # the row has entered the state
        assert bool((torch.isnan(S) if math.isnan(value) else S == value).all())
    else:
        assert bool(torch.isfinite(S).all())


# windows shorter and longer than a tile and none; a call boundary before and behind the bad row; the padded tail of a call
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("dtype,d,G,w,gated,calls,bad", [
    (F32, 64, 1, 40, False, [300], (150,)), (F32, 64, 4, 16, True, [100, 200], (150, 151)), (F32, 128, 2, 0, False, [130, 40], (60,)),
    (F32, 128, 8, 200, True, [300], (150, 280)), (BF16, 64, 2, 64, False, [257], (256,)), (F32, 64, 8, 90, False, [64, 100], tuple(range(120, 164)))])
def test_cuda_core_prefill(dtype, d, G, w, gated, calls, bad, value):
    _check(dtype, d, G, w, gated, calls, bad, value)


# gated bf16 states of d = 128 are carried by the tensor cores: chunks on their own and in a pass, phi made there and in front
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("w,calls,kw", [(40, [300], {}), (0, [100, 60], dict(prefill_chunk=64)), (100, [700], dict(prefill_chunk=144))])
def test_gated_state(w, calls, kw, value):
    _, S = _prompt(BF16, 128, 4, w, True, calls, (50,), value, **kw)
    assert bool((torch.isnan(S) if math.isnan(value) else S == value).all())


# bf16, d = 128 with gates runs on the tcgen05 kernel, whose tiles are 128 rows of keys by 128 of queries: windows inside a tile,
# over several, longer than a chunk and none; window rows from the ring; a chunk that is carried on its own and in a pass
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("G,w,calls,bad,kw", [
    (4, 40, [300], (150,), {}), (1, 16, [100, 200], (150, 299), {}), (8, 0, [300], (60,), {}), (2, 600, [700], (300, 690), {}),
    (4, 64, [257], (256,), {}), (2, 120, [160, 60], (170,), dict(prefill_chunk=64)), (4, 300, [700], (200,), dict(prefill_chunk=144))])
def test_gated_prefill_on_tcgen05(G, w, calls, bad, kw, value):
    _check(BF16, 128, G, w, True, calls, bad, value, **kw)
