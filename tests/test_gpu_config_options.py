"""Options of a context that choose how its work is cut: an explicit value is what the kernels use, also where the library
would choose another way by itself."""
import pytest
import torch

from paper_2607_24788_b200 import glide
from tests.parity_util import run_case

pytestmark = pytest.mark.gpu
BF16, F32 = torch.bfloat16, torch.float32


@pytest.mark.parametrize("kw,items", [
    (dict(), 1),                                              # one item per unit where the rings are short
    (dict(decode_chunk=16), 4 + 2), (dict(decode_chunk=8), 8 + 2),   # ring of 64 slots; the state in two row blocks by default
    (dict(decode_state_splits=4), 1 + 4), (dict(decode_chunk=32, decode_state_splits=1), 2 + 1)])
def test_decode_items_per_unit(kw, items):
    g = glide.Glide([64], 2, 4, 2, 64, 1000, dtype=F32, **kw)
    assert g.glide_decode_launch_info()["work_items"] == 2 * 2 * items
    g.glide_destroy()


# the work list with units cut in many records (18 to 38 of them), every merge, the learned map, gates; more records than
# one ring of short windows has, so that the merge takes several batches
@pytest.mark.parametrize("dtype,d,G,kw", [
    (F32, 64, 1, dict(merge=1)), (F32, 128, 4, dict(merge=2)), (F32, 64, 2, dict(phi=1)), (F32, 128, 8, dict(gated=True)),
    (BF16, 128, 2, dict(phi=1, gated=True, decode_impl=glide.GLIDE_DECODE_FMA)), (BF16, 64, 8, dict(merge=2, gated=True))])
def test_decode_work_list_with_many_records(dtype, d, G, kw):
    run_case([0, 5, 150, 1 << 20], 2, 2 * G, 2, d, dtype, [260], 4, amp=4 * d ** -0.5, seed=59 + G, max_tokens=300, decode_chunk=8,
             **kw)


# prefill_chunk is the chunk of the scan: a call of eight chunks, eight calls of one, and one slot after the other give the
# same bits (the same sums in the same order); 16: less than a chunk sum's rows, 272: more than the kernels choose themselves
@pytest.mark.parametrize("d,gated,chunk", [(64, False, 16), (64, True, 80), (128, False, 48), (128, True, 272)])
def test_prefill_chunk_cuts_the_scan(d, gated, chunk):
    L, B, H, Hkv, T = 2, 2, 4, 2, 8 * chunk
    gen = torch.Generator(device="cuda").manual_seed(67)
    q, k, v = (torch.randn((L, B, T, h, d), generator=gen, device="cuda") for h in (H, Hkv, Hkv))
    gate = 0.99 + 0.01 * torch.rand((L, B, T, Hkv), generator=gen, device="cuda")

    def prefill(cuts, by_slot):
        g = glide.Glide([100, 0], B, H, Hkv, d, 1 << 20, dtype=F32, gated=gated, prefill_chunk=chunk)
        out = torch.zeros_like(q)
        for s in ([slice(b, b + 1) for b in range(B)] if by_slot else [slice(0, B)]):
            for c in range(0, T, T // cuts):
                part = [x[:, s, c:c + T // cuts].contiguous() for x in (q, k, v, out, gate)]
                if by_slot:
                    g.glide_prefill_seq(s.start, *(x[:, 0] for x in part[:4]))
                elif gated:
                    g.glide_prefill_gated(*part[:3], part[4], part[3])
                else:
                    g.glide_prefill(*part[:4])
                out[:, s, c:c + T // cuts] = part[3]
        states = [x.clone() for l in range(L) for x in g.glide_export_state(l)[2:]]
        assert g.glide_device_status() == 0
        g.glide_destroy()
        return [out, *states]

    one = prefill(1, False)
    for other in [prefill(8, False)] + ([] if gated else [prefill(2, True)]):   # (a slot's call takes no gates)
        for a, b in zip(one, other):
            assert torch.equal(a, b)


# one CTA per unit or the work list: the longest ring of the launch, head_dim, group size, type and map, and whether the units
# are more than the chip has SMs (148 here): (L, B, H_kv, G, d, window) with one item per unit, and the same with one slot more
@pytest.mark.parametrize("dtype,L,B,Hkv,G,d,w,kw", [
    (F32, 1, 1, 4, 1, 64, 512, {}), (F32, 8, 8, 4, 1, 64, 512, {}), (F32, 1, 2, 4, 8, 128, 64, {}), (BF16, 8, 8, 4, 8, 128, 16, dict(decode_impl=2)),
    (F32, 1, 2, 4, 4, 64, 192, {}), (F32, 8, 8, 4, 4, 128, 320, {}), (F32, 8, 8, 4, 2, 128, 320, dict(phi=1))])
def test_decode_by_unit_or_by_list(dtype, L, B, Hkv, G, d, w, kw):
    units = L * B * Hkv
    if kw.get("phi"):
        kw = dict(kw, phi_wq=torch.zeros((L, G * Hkv, d, d), device="cuda", dtype=dtype),
                  phi_wk=torch.zeros((L, Hkv, d, d), device="cuda", dtype=dtype))
    for longer in (0, 1):
        g = glide.Glide([w + longer] + [w] * (L - 1), B, G * Hkv, Hkv, d, 1 << 20, dtype=dtype, **kw)
        assert (g.glide_decode_launch_info()["work_items"] == units) == (longer == 0)
        g.glide_destroy()


@pytest.mark.parametrize("G,d,kw", [(4, 64, {}), (2, 64, dict(phi=1)), (8, 64, dict(merge=1))])
def test_decode_many_small_units_take_the_work_list(G, d, kw):
    """More units than SMs with several heads of 64: the list, against the oracle; a range of few of its layers: by unit."""
    run_case([16] * 5, 16, 2 * G, 2, d, F32, [20], 2, amp=4 * d ** -0.5, seed=71 + G, max_tokens=40, **kw)


# one CTA per unit, for sure: every merge, the learned map, gates, rings of no, one and a few slots and of the longest there
@pytest.mark.parametrize("dtype,d,G,windows,kw", [
    (F32, 128, 2, [320, 7], dict(merge=1)), (F32, 64, 4, [192, 0, 1], dict(merge=2)), (F32, 128, 4, [256, 0, 33], dict(phi=1)),
    (F32, 64, 8, [128, 5], dict(phi=1, merge=1)), (F32, 64, 2, [384, 0], dict(gated=True)), (F32, 128, 8, [64, 0], dict(phi=1, gated=True)),
    (BF16, 64, 1, [512, 3], dict(merge=1)), (BF16, 128, 4, [40, 0], dict(phi=1, decode_impl=glide.GLIDE_DECODE_FMA))])
def test_decode_by_unit_every_kind(dtype, d, G, windows, kw):
    weights = {}
    if kw.get("phi"):
        weights = dict(phi_wq=torch.zeros((len(windows), 2 * G, d, d), device="cuda", dtype=dtype),
                       phi_wk=torch.zeros((len(windows), 2, d, d), device="cuda", dtype=dtype))
    g = glide.Glide(windows, 2, 2 * G, 2, d, 600, dtype=dtype, **kw, **weights)
    assert g.glide_decode_launch_info()["work_items"] == len(windows) * 2 * 2
    g.glide_destroy()
    run_case(windows, 2, 2 * G, 2, d, dtype, [70], 3, amp=4 * d ** -0.5, seed=103 + G, max_tokens=600, **kw)
