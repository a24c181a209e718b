"""Attention of a job of prefix tokens: up to 128 tokens over a bf16 cache the warps of a block share 16 of them (64 positions a
round), over a float32 cache a round is 32 positions of 16 tokens."""
import pytest

import spd_inputs as si
from tests.gpu_common import compare_first_step, compare_step, make_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shapes():
    """16 MB of matrices and more per layer, so prefixes of any length run as jobs."""
    out = {}
    for hd in (64, 128):
        shape = si.ModelShape("jobattn%d" % hd, 2, 1024, 1024 // hd, 2048, 800)
        out[hd] = shape, si.make_weights(shape, seed=131), si.make_ngram_tables(shape.vocab, 1.1, 20_000, (2, 3), 2000, seed=132)
    return out


# Positions on both sides of the ends of rounds and of a block's 16 tokens; 194 positions make jobs of 128 tokens, so the longer
# prefixes leave a job of 1, 15, 17 and 64 tokens behind 128 cached positions.  The restart's job stands behind any position.
@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("m", [1, 15, 16, 17, 31, 33, 63, 64, 65, 96, 112, 127, 128, 129, 143, 145, 192])
def test_job_attention(shapes, m, hd, kv_dtype):
    shape, weights, tables = shapes[hd]
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), [0.3, 0.2] + [0.0] * 6, 0.4, 0.2, 0.05, 194 if m > 128 else 200, kv_dtype)
    compare_first_step(ctx, orc, si.make_prefix("zipf", m, shape.vocab, 1.1, seed=133 + m))
    if m < 192:
        compare_step(ctx, orc)
    if m < 190:
        compare_first_step(ctx, orc, None, reset_draft=1)
    ctx.close()
