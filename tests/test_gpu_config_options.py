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
