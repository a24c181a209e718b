"""The decode kernel's ring with weights in fragment order: where units do not fill their stages, a stage may hold the
end of a unit, several units or a part of one, and a tile of 128 rows may end inside a stage."""
import numpy as np
import pytest

import spd_inputs as si
from tests.gpu_common import compare_first_step, compare_step, make_pair

pytestmark = pytest.mark.gpu


# d_model, heads, d_ffn, vocabulary, rings (stage bytes, stages): a unit of 8 rows has d_model / 32 pairs of column blocks of 512
# bytes.  33 pairs in stages of 4, 16 and 67; 3 pairs in stages of one, of several units and of more than a block has; 8 pairs
# and up to 17 units a block of gate / up, so a second tile of rows.
@pytest.mark.parametrize("d,heads,f,vocab,rings", [
    (1056, 33, 512, 1200, [(2176, 2), (2176, 9), (8192, 3), (34304, 5)]),
    (96, 3, 160, 200, [(512, 16), (640, 2), (2048, 4), (65536, 2)]),
    (256, 4, 9600, 9728, [(19200, 2), (19200, 9), (38400, 4)]),
])
def test_results_do_not_depend_on_the_ring(d, heads, f, vocab, rings):
    shape = si.ModelShape("ring", 2, d, heads, f, vocab)
    weights = si.make_weights(shape, seed=121)
    tables = si.make_ngram_tables(vocab, 1.1, 20_000, (2, 3), 2000, seed=122)
    ctx, orc = make_pair(shape, weights, tables, 3, (2, 3), [0.3, 0.2] + [0.0] * 6, 0.4, 0.2, 0.05, 64, "f32")
    prefix = si.make_prefix("zipf", 7, vocab, 1.1, seed=123)
    compare_first_step(ctx, orc, prefix)
    want = []
    for _ in range(3):
        compare_step(ctx, orc)
        want.append(ctx.spd_debug_read("LOGITS"))
    for stage_bytes, stages in rings:
        ctx.spd_set_ring(stage_bytes, stages)
        ctx.spd_prefill(prefix)
        for z in want:   # a unit's pairs go to the same warps in the same order whatever the stages
            ctx.spd_step()
            assert np.array_equal(ctx.spd_debug_read("LOGITS"), z), (stage_bytes, stages)
    ctx.close()


def test_stage_smaller_than_a_pair_of_column_blocks_is_refused():
    import paper_2405_18400_b200 as P
    shape = si.ModelShape("ring", 1, 96, 3, 160, 200)
    weights = si.make_weights(shape, seed=121)
    tables = si.make_ngram_tables(200, 1.1, 20_000, (2, 3), 2000, seed=122)
    for images in (True, False):
        ctx, _ = make_pair(shape, weights, tables, 3, (2, 3), [0.3, 0.2] + [0.0] * 6, 0.4, 0.2, 0.05, 64, "f32", images=images)
        if images:
            with pytest.raises(P.SpdError) as e:
                ctx.spd_set_ring(384, 4)
            assert e.value.status == -1
        else:
            ctx.spd_set_ring(384, 4)
        ctx.spd_prefill(si.make_prefix("zipf", 7, 200, 1.1, seed=123))
        ctx.spd_step()
        ctx.close()
