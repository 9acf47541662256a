"""What the options of a context do to the workspace it asks for (host only)."""
import pytest
import torch

from paper_2607_24788_b200 import build, glide

BF16, F32 = torch.bfloat16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()
    glide.load_library()


def _bytes(dtype, d, **kw):
    cfg, keep = glide.make_config(**dict(dict(windows=[64] * 16, batch=4, n_q_heads=8, n_kv_heads=8, head_dim=d, max_tokens=4096,
                                              dtype=dtype), **kw))
    return glide.glide_workspace_bytes(cfg)


UNITS = 16 * 4 * 8
SLACK = 3 << 20   # alignment of the streamed arrays, small tables


# the prefill scratch holds prefill_chunk rows of fp32 per unit (or one chunk sum for every unit of one layer, which is less here)
@pytest.mark.parametrize("dtype,d,kw", [(F32, 64, {}), (F32, 128, {}), (F32, 128, dict(gated=True)), (BF16, 64, {}),
                                        (BF16, 128, dict(prefill_impl=glide.GLIDE_PREFILL_FMA))])
def test_prefill_chunk_bounds_the_scratch(dtype, d, kw):
    rows = (256 - 16) * UNITS
    assert abs(_bytes(dtype, d, prefill_chunk=256, **kw) - _bytes(dtype, d, prefill_chunk=16, **kw) - rows * d * 4) < rows * 8 + SLACK


# the bf16 copies that the tcgen05 prefill kernel reads (phi(K') rows and S; two of each with gates) are laid out only where
# the context can run that kernel
@pytest.mark.parametrize("gated,halves", [(False, 1), (True, 2)])
@pytest.mark.parametrize("kw", [dict(prefill_impl=glide.GLIDE_PREFILL_FMA), dict(decode_impl=glide.GLIDE_DECODE_FMA)])
def test_no_scratch_for_a_kernel_that_is_ruled_out(gated, halves, kw):
    copies = halves * UNITS * (64 + 128) * 128 * 2
    more = _bytes(BF16, 128, gated=gated, prefill_chunk=64) - _bytes(BF16, 128, gated=gated, prefill_chunk=64, **kw)
    assert abs(more - copies) < UNITS * 1024 + SLACK
