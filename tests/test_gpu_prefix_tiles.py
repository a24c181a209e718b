"""Tiles of token rows in steps of 16, and the tokens that a context's jobs take."""
import numpy as np
import pytest

import spd_inputs as si
from tests.gpu_common import compare_first_step, compare_step, make_pair

pytestmark = pytest.mark.gpu

LAM = [0.3, 0.2] + [0.0] * 6


@pytest.fixture(scope="module")
def wide():
    """25 MB of matrices per layer, so prefixes of any length run as jobs; d_ffn leaves a ragged last row tile."""
    shape = si.ModelShape("wide", 2, 1024, 16, 2712, 1504)
    return shape, si.make_weights(shape, seed=111), si.make_ngram_tables(shape.vocab, 1.1, 50_000, (2, 3), 5000, seed=112)


# One tile of 80, 96, 112, 144, 208, 240 rows and one row more; three of 96 and of 112, four of 112 and of 128 rows.  Halves of 40,
# 56, 72 and 104 rows are no multiple of the 16 columns of a tensor-memory load.
@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("m", [80, 81, 97, 112, 113, 144, 145, 208, 209, 240, 241, 272, 300, 385, 448, 449])
def test_tiles_in_steps_of_16_rows(wide, m, kv_dtype):
    shape, weights, tables = wide
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), LAM, 0.4, 0.2, 0.05, 600, kv_dtype)
    compare_first_step(ctx, orc, si.make_prefix("zipf", m, shape.vocab, 1.1, seed=113 + m))
    assert ctx.spd_launch_count() == 9 * shape.n_layers + 1
    compare_step(ctx, orc)
    ctx.close()


@pytest.mark.parametrize("max_pos,m,jobs", [(194, 193, 2), (193, 192, 2), (259, 256, 1), (322, 321, 2), (386, 385, 2), (465, 400, 2), (449, 448, 2), (514, 512, 1), (600, 599, 2)])
def test_tokens_of_a_job(wide, max_pos, m, jobs):
    """The longest prefix of the context rounded down to a multiple of 128, 512 at most."""
    shape, weights, tables = wide
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), LAM, 0.4, 0.2, 0.05, max_pos, "f32")
    compare_first_step(ctx, orc, si.make_prefix("zipf", m, shape.vocab, 1.1, seed=114 + m))
    assert ctx.spd_launch_count() == 9 * shape.n_layers * jobs + 1
    ctx.close()


@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("m,least,most", [(200, 202, 257), (300, 302, 385), (400, 402, 513)])
def test_room_in_the_context_does_not_change_a_prefix(wide, m, least, most, kv_dtype):
    """From the first to the last context whose jobs take as many tokens, a prefix has the same bits."""
    import paper_2405_18400_b200 as P
    shape, weights, tables = wide
    packed, dtabs = P.pack_weights(weights, "cuda:0"), P.build_ngram_tables(tables, "cuda:0")
    prefix = si.make_prefix("zipf", m, shape.vocab, 1.1, seed=115 + m)
    z = []
    for max_pos in (least, most):
        ctx = P.SpdContext(shape, packed, dtabs, 3, (2, 3), LAM, 0.4, 0.2, 0.05, max_pos, kv_dtype)
        ctx.spd_prefill(prefix)
        z.append(ctx.spd_debug_read("LOGITS"))
        ctx.close()
    assert np.isfinite(z[0]).all() and np.array_equal(z[0], z[1])
