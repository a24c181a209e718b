"""Tiles of token rows in steps of 16, and the tokens that a context's jobs take."""
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


@pytest.mark.parametrize("max_pos,m,jobs", [(194, 193, 1), (193, 192, 2), (322, 321, 1), (465, 400, 1), (450, 449, 1), (449, 448, 2), (600, 599, 2)])
def test_tokens_of_a_job(wide, max_pos, m, jobs):
    """The longest prefix of the context to the nearest multiple of 128, 512 at most: at 193, 321 and 449 tokens it is rounded up,
    at one less down."""
    shape, weights, tables = wide
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), LAM, 0.4, 0.2, 0.05, max_pos, "f32")
    compare_first_step(ctx, orc, si.make_prefix("zipf", m, shape.vocab, 1.1, seed=114 + m))
    assert ctx.spd_launch_count() == 9 * shape.n_layers * jobs + 1
    ctx.close()


@pytest.mark.parametrize("m", [129, 200, 257, 300, 400])
def test_a_job_that_stands_for_two_is_as_exact(wide, m):
    """In a context of m + 65 positions these prefixes are one job, longer than the positions rounded down to a multiple of 128:
    chains of 24 additions, the small terms first.  The logits are below 8, a rounding of float32 there is 2.4e-7 at most;
    twenty of them are the bound (chains of 96 additions: 1.6e-5 and more at 7B width)."""
    import numpy as np
    shape, weights, tables = wide
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), LAM, 0.4, 0.2, 0.05, m + 65, "f32")
    worst = []
    for seed in range(3):
        prefix = si.make_prefix("zipf", m, shape.vocab, 1.1, seed=115 + seed)
        before = ctx.spd_launch_count()
        ctx.spd_prefill(prefix)
        assert ctx.spd_launch_count() - before == 9 * shape.n_layers + 1
        orc.prefill(prefix)
        worst.append(float(np.abs(ctx.spd_debug_read("LOGITS").astype(np.float64) - orc.logits()).max()))
        assert np.abs(orc.logits()).max() < 8
    assert np.mean(worst) < 4.8e-6, worst
    ctx.close()
