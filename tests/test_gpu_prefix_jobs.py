"""Prefixes that run wholly as jobs of the long-prefix path: the last job carries the last token's row through the last
layer alone and ends with the launch that multiplies the LM head and takes the first timestep (Eq. 1).  Models whose
layers hold 16 MB of matrices and more send runs of any length there, smaller ones runs of more than 16 tokens."""
import numpy as np
import pytest

import spd_inputs as si
from tests.gpu_common import compare_first_step, compare_step, make_pair, make_tiny_pair

pytestmark = pytest.mark.gpu

LAM = [0.3, 0.2] + [0.0] * 6


@pytest.fixture(scope="module")
def wide():
    """25 MB of matrices per layer; a vocabulary that does not divide among the blocks or by the rows a warp takes."""
    shape = si.ModelShape("wide", 2, 1024, 16, 2752, 1501)
    return shape, si.make_weights(shape, seed=61), si.make_ngram_tables(shape.vocab, 1.1, 50_000, (2, 3), 5000, seed=62)


def _pair(wide, max_pos, kv_dtype, k=3):
    shape, weights, tables = wide
    return make_pair(shape, weights, tables, k, (2, 3), LAM, 0.4, 0.2, 0.05, max_pos, kv_dtype)


# One token; the products' instances for up to 16, 32, 64, 128 and 256 token rows at both ends of their ranges (96 and 97, 160
# and 161: a step in the rows of a tile).  Up to 256 rows a tile may be cut: a layer's products have 192, 64, 352 and 172 stages
# there, cut into 48, 16, 74 and 43 runs, so tiles of two to four parts (129 rows on: two segments of a run at least).  More
# rows make uncut tiles of up to 128 rows, all alike: three of 96 (257, 288), three of 128 (289, 384), four of 128 (385, 512).
# 513 = a job of 512 and one of one token.
@pytest.mark.parametrize("m,jobs", [(1, 1), (2, 1), (16, 1), (17, 1), (32, 1), (33, 1), (64, 1), (65, 1), (96, 1), (97, 1), (128, 1), (129, 1),
                                    (160, 1), (161, 1), (256, 1), (257, 1), (288, 1), (289, 1), (320, 1), (321, 1), (384, 1), (385, 1), (512, 1),
                                    (513, 2)])
def test_whole_prefix_as_jobs(wide, m, jobs):
    ctx, orc = _pair(wide, 768, "bf16" if m % 2 else "f32", k=5)
    prefix = si.make_prefix("zipf", m, wide[0].vocab, 1.1, seed=800 + m)
    compare_first_step(ctx, orc, prefix)
    assert ctx.spd_launch_count() == 9 * wide[0].n_layers * jobs + 1
    for _ in range(2):
        compare_step(ctx, orc)
    # a restart (Section 5.3) runs the three generated tokens as a job behind the cached positions
    compare_first_step(ctx, orc, None, reset_draft=2)
    compare_step(ctx, orc)
    ctx.close()


def test_end_of_a_job_leaves_what_the_prefill_kernel_leaves(wide):
    """Residual row and logits of the last token, drafts and weights: a context of 128 positions has no long-prefix
    buffers and sends the same prefix through the 16-token kernel; so does a traced call."""
    a, _ = _pair(wide, 128, "f32")
    b, _ = _pair(wide, 256, "f32")
    c, _ = _pair(wide, 256, "f32")
    c.spd_debug_trace(True)
    prefix = si.make_prefix("zipf", 30, wide[0].vocab, 1.1, seed=5)
    got = [x.spd_prefill(prefix) for x in (a, b, c)]
    # (traced: a job of 16 tokens without an end, then the 16-token kernel)
    assert [x.spd_launch_count() for x in (a, b, c)] == [2, 9 * wide[0].n_layers + 1, 9 * wide[0].n_layers + 1]
    for x, (ids, g) in zip((b, c), got[1:]):
        assert ids.tolist() == got[0][0].tolist() and np.abs(g - got[0][1]).max() < 1e-3
        for what in ("LOGITS", "HIDDEN"):
            assert np.abs(x.spd_debug_read(what) - a.spd_debug_read(what)).max() < 1e-4
    assert np.abs(c.spd_debug_read("TRACE")[-1, 1] - b.spd_debug_read("HIDDEN")).max() < 1e-4
    for x in (a, b, c):
        x.close()


@pytest.mark.parametrize("m,launches", [(16, 1), (17, 19), (32, 19), (513, 9 * 2 + 1)])
def test_small_model(tiny_inputs, m, launches):
    """The tiny model's jobs begin at 17 tokens; the one token that a job of 512 leaves over goes through the 16-token kernel."""
    wl, _, _, _ = tiny_inputs
    ctx, orc = make_tiny_pair(tiny_inputs, max_pos=1024)
    compare_first_step(ctx, orc, si.make_prefix("zipf", m, wl.shape.vocab, 1.1, seed=820 + m))
    assert ctx.spd_launch_count() == launches
    compare_step(ctx, orc)
    ctx.close()


@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("d,heads", [(256, 4), (256, 2)])
def test_batched_attention_rounds(d, heads, kv_dtype):
    """A batch's attention takes 32 (float32, head size 128) to 128 positions (bf16, 64) per round of a block: contexts of
    one position, around one and two rounds, and their growth across a round's end, all in one batch."""
    import paper_2405_18400_b200 as P
    from oracle import spd_oracle as so

    shape = si.ModelShape("hd%d" % (d // heads), 2, d, heads, 512, 1000)
    weights = si.make_weights(shape, seed=71)
    tables = sorted(si.make_ngram_tables(shape.vocab, 1.1, 50_000, (2, 3), 5000, seed=72), key=lambda t: int(t["n"]))
    packed, dtabs = P.pack_weights(weights, "cuda:0"), P.build_ngram_tables(tables, "cuda:0")
    reqs = []
    for r, m in enumerate((1, 30, 31, 62, 63, 64, 126, 127, 128, 255, 257)):
        ctx = P.SpdContext(shape, packed, dtabs, 3, (2, 3), LAM, 0.4, 0.2, 0.05, 300, kv_dtype)
        orc = so.Oracle(so.make_config(shape, 3, (2, 3), LAM, 0.4, 0.2, 0.05, 300, kv_dtype), weights, tables)
        compare_first_step(ctx, orc, si.make_prefix("zipf", m, shape.vocab, 1.1, seed=840 + r))
        reqs.append((ctx, orc))
    for _ in range(3):
        for (ctx, orc), got in zip(reqs, P.spd_batch_step([c for c, _ in reqs])):
            compare_step(ctx, orc, None, stepped=got, path="prefill")
    for ctx, orc in reqs:
        ctx.close()
        orc.close()


@pytest.mark.parametrize("m", [17, 64, 80, 128, 200, 300])
def test_first_timestep_is_as_exact_as_float32_sums(tiny_inputs, m):
    """The products' accumulators add with truncation; short chains between two moves to registers keep the logits within a
    few roundings of 64 bits, whatever the number of token rows.  The logits here are below 2, so a rounding is 2^-24 of that at
    most: 1.2e-7; ten of them are the bound (measured 4e-7 to 9e-7; with a row's 48 additions in one chain 1.6e-6 to 3e-6)."""
    wl, _, _, _ = tiny_inputs
    ctx, orc = make_tiny_pair(tiny_inputs, kv_dtype="f32", max_pos=512)
    worst = []
    for seed in range(4):
        prefix = si.make_prefix("zipf", m, wl.shape.vocab, 1.1, seed=860 + seed)
        ctx.spd_prefill(prefix)
        orc.prefill(prefix)
        worst.append(float(np.abs(ctx.spd_debug_read("LOGITS").astype(np.float64) - orc.logits()).max()))
        assert np.abs(orc.logits()).max() < 2
    assert np.mean(worst) < 1.2e-6, worst
    ctx.close()
