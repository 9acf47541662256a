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
