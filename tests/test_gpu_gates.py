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
