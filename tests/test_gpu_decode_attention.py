"""The decode kernel's attention phase: 8 (bf16, head size 64) to 1 (float32, 128) positions side by side in a warp, four of
each group in flight, so rounds of 64 to 512 positions of a block, over up to 8 splits of the positions per head."""
import numpy as np
import pytest

import spd_inputs as si
from tests.gpu_common import compare_first_step, compare_step, make_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shapes():
    out = {}
    for hd in (64, 128):
        shape = si.ModelShape("attn%d" % hd, 2, 2 * hd, 2, 256, 600)
        out[hd] = shape, si.make_weights(shape, seed=101), si.make_ngram_tables(shape.vocab, 1.1, 20_000, (2, 3), 2000, seed=102)
    return out


@pytest.mark.parametrize("images", [True, False])
@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("m", [1, 2, 31, 62, 127, 520])   # 62, 127: the steps cross to two and to three splits; 520: eight, more than a round each (float32)
def test_decode_behind_m_positions(shapes, m, hd, kv_dtype, images):
    shape, weights, tables = shapes[hd]
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), [0.3, 0.2] + [0.0] * 6, 0.4, 0.2, 0.05, 640, kv_dtype, images=images)
    compare_first_step(ctx, orc, si.make_prefix("zipf", m, shape.vocab, 1.1, seed=103 + m))
    for _ in range(4):
        compare_step(ctx, orc)
    ctx.close()


def test_nan_in_the_cache_reaches_the_logits(shapes):
    """A NaN key of one head makes that head's output NaN, as a softmax does, wherever the position lies in a round."""
    shape, weights, tables = shapes[128]
    for at in (0, 3, 17, 39):
        ctx, _ = make_pair(shape, weights, tables, 3, (2, 3), [0.3, 0.2] + [0.0] * 6, 0.4, 0.2, 0.05, 256, "bf16")
        ctx.spd_prefill(si.make_prefix("zipf", 40, shape.vocab, 1.1, seed=104))
        keys = ctx.workspace[: 256 * 256 * 2].view(__import__("torch").bfloat16).view(256, 256)   # first layer [max_pos][d_model]
        keys[at, 5] = float("nan")
        ctx.spd_step()
        assert np.isnan(ctx.spd_debug_read("LOGITS")).all()
        ctx.close()


@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("hd", [32, 64, 128])
def test_positions_that_score_minus_infinity_have_no_weight(hd, kv_dtype):
    """The first 40 of 41 keys of a head infinite in one dimension: with the sign that makes their scores -inf they drop out of
    the softmax, to the bit as with a score of -1e27 or so; with the other, scores of +inf, the head's output is NaN.  Most
    groups of lanes meet nothing but -inf."""
    import paper_2405_18400_b200 as P
    import torch
    shape = si.ModelShape("inf%d" % hd, 2, 2 * hd, 2, 256, 600)
    packed = P.pack_weights(si.make_weights(shape, seed=105), "cuda:0")
    ctx = P.SpdContext(shape, packed, [], 3, (2, 3), [0.0] * 8, 0.4, 0.2, 0.05, 64, kv_dtype)
    prefix = si.make_prefix("zipf", 41, shape.vocab, 1.1, seed=106)
    dtype, size = (torch.bfloat16, 2) if kv_dtype == "bf16" else (torch.float32, 4)

    def step(value):
        ctx.spd_prefill(prefix)
        keys = ctx.workspace[: 64 * 2 * hd * size].view(dtype).view(64, 2 * hd)   # first layer [max_pos][d_model]
        keys[:40, hd + 5] = value
        ctx.spd_step()
        return ctx.spd_debug_read("LOGITS")

    large = {s: step(s * 1e30) for s in (1.0, -1.0)}
    infinite = {s: step(s * float("inf")) for s in (1.0, -1.0)}
    assert all(np.isfinite(z).all() for z in large.values())
    sign = 1.0 if np.isnan(infinite[-1.0]).all() else -1.0
    assert np.isnan(infinite[-sign]).all()
    assert np.array_equal(infinite[sign], large[sign])
    ctx.close()
