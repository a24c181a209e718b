"""The serial end of a timestep: per-block lists of the best logits (a lane keeps up to eight rows of its block in registers,
more are read again each round) and their merge (a lane walks the heads of its lists)."""
import pytest

import spd_inputs as si
from tests.gpu_common import compare_first_step, compare_step, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,k,hot", [
    (96, 16, None),        # fewer rows than blocks: empty lists and lists of one, all shorter than k
    (1504, 16, (40, 56)),  # the k best rows in two or three neighbouring blocks: a list is used up
    (37888, 8, (4, 8)),    # 256 rows a block: the most that stay in registers; some of the best in one lane's stride
    (40000, 5, None),      # more than that
])
def test_keep_topk_lists(vocab, k, hot):
    shape = si.ModelShape("tail", 1, 128, 2, 128, vocab)
    weights = si.make_weights(shape, seed=91)
    if hot:
        weights["lm_head"][hot[0]:hot[1]] *= 8   # exact in bf16; these rows' logits are the largest and the smallest
    tables = si.make_ngram_tables(vocab, 1.1, 20_000, (2, 3), 2000, seed=92)
    ctx, orc = make_pair(shape, weights, tables, k, (2, 3), [0.3, 0.2] + [0.0] * 6, 0.4, 0.2, 0.05, 256, "f32")
    compare_first_step(ctx, orc, si.make_prefix("zipf", 9, vocab, 1.1, seed=93))   # the 16-token kernel's end
    for _ in range(2):
        compare_step(ctx, orc)
    compare_first_step(ctx, orc, si.make_prefix("zipf", 20, vocab, 1.1, seed=94))  # the end of a job
    compare_step(ctx, orc)
    ctx.close()


@pytest.mark.parametrize("vocab,k", [(96, 16), (1504, 3), (1504, 16), (37888, 8), (40000, 16)])
def test_equal_logits_are_kept_by_id(vocab, k):
    """The kept tokens are the largest of the device's own logits, equal ones by ascending id: a row and its negative, eight times as
    large as the others, in twelve places each make ties at the top, between lanes, between blocks and (k = 3, 8) between the last kept
    and the first left out; rows of zeros make logits of zero."""
    import numpy as np
    import paper_2405_18400_b200 as P
    shape = si.ModelShape("ties", 1, 128, 2, 128, vocab)
    weights = si.make_weights(shape, seed=95)
    head = weights["lm_head"]
    step = vocab // 12
    for r in range(12):
        head[r * step + 1] = head[step + 3] * 8      # exact in bf16
        head[r * step + 2] = head[step + 3] * -8
        head[r * step] = 0
    ctx = P.SpdContext(shape, P.pack_weights(weights, "cuda:0"), [], k, (2, 3), [0.0] * 8, 0.4, 0.2, 0.05, 192, "f32")
    prefixes = [si.make_prefix("zipf", 20, vocab, 1.1, seed=s) for s in (96, 97, 98, 99)]
    tied = 0
    for prefix in prefixes:
        ctx.spd_prefill(prefix)
        for _ in range(3):
            z = ctx.spd_debug_read("LOGITS")
            order = np.lexsort((np.arange(vocab), -z.astype(np.float64)))
            assert ctx.spd_debug_read("CAND_TOK").tolist() == order[:k].tolist()
            tied += int(len(np.unique(z[order[:k + 1]])) < k + 1)
            ctx.spd_step()
    assert tied                                      # (a step whose hidden row is nearly at right angles to that row has none)
    ctx.close()


@pytest.mark.parametrize("vocab", [20000, 37888, 40000])     # 136 rows a block, 256 (the most that stay in registers), 272
def test_nan_logits_are_passed_over(vocab):
    """Logits that are NaN are left out of the kept tokens, wherever they lie beside them."""
    import numpy as np
    import paper_2405_18400_b200 as P
    shape = si.ModelShape("nan", 1, 128, 2, 128, vocab)
    weights = si.make_weights(shape, seed=109)
    make = lambda: P.SpdContext(shape, P.pack_weights(weights, "cuda:0"), [], 8, (2, 3), [0.0] * 8, 0.4, 0.2, 0.05, 192, "f32")
    prefixes = [si.make_prefix("zipf", m, vocab, 1.1, seed=110 + m) for m in (9, 40)]      # the 16-token kernel's end, a job's
    sound = make()
    top = set()
    for prefix in prefixes:
        top |= set(sound.spd_prefill(prefix)[0].tolist())
    # rows of the kept tokens' lanes (a lane has every 32nd row of its block), none of the kept ones
    bad = [r for r in sorted({t + o for t in top for o in (-96, -64, -32, 32)} - top) if 0 <= r < vocab]
    weights["lm_head"][bad] = float("nan")
    damaged = make()
    for prefix in prefixes:
        want = sound.spd_prefill(prefix)[0]
        z = sound.spd_debug_read("LOGITS")
        z[bad] = np.nan
        got = damaged.spd_prefill(prefix)[0]
        assert np.array_equal(damaged.spd_debug_read("LOGITS"), z, equal_nan=True)
        assert got.tolist() == want.tolist()
    # and with all but three rows lost, those three, then the lost ones by their ids
    keep = sound.spd_debug_read("CAND_TOK")[:3].tolist()
    weights["lm_head"][[r for r in range(vocab) if r not in keep]] = float("nan")
    lost = make()
    for prefix in prefixes:
        lost.spd_prefill(prefix)
        z = lost.spd_debug_read("LOGITS")
        best = sorted(keep, key=lambda t: (-float(z[t]), t))
        first = [r for r in range(11) if r not in keep][:5]
        assert lost.spd_debug_read("CAND_TOK").tolist() == best + first
    for c in (sound, damaged, lost):
        c.close()


@pytest.mark.parametrize("k", [3, 6, 8, 16])                  # 9 to 256 options: one to eight of a lane
def test_nan_scores_rank_last(k):
    """Options whose score is NaN (a draft's or a kept token's log-probability is) are chosen when nothing else is left, by index."""
    import numpy as np
    import paper_2405_18400_b200 as P
    shape = si.ModelShape("nan", 1, 128, 2, 128, 800)
    ctx = P.SpdContext(shape, P.pack_weights(si.make_weights(shape, seed=114), "cuda:0"), [], k, (2, 3), [0.0] * 8, 0.4, 0.2, 0.05, 64, "f32")
    rng = np.random.default_rng(k)
    for lost_drafts, lost_tokens in ([0], []), ([], [0]), (list(range(k - 1)), []), (list(range(k - 1)), [0, k - 1]), (list(range(1, k)), [1]), ([], []):
        logp, cand_lp = rng.normal(-8, 2, k).astype(np.float32), rng.normal(-3, 1, k).astype(np.float32)
        logp[k // 2] = -1.0                                   # the best draft's options lie beside the first draft's in their lanes (k = 8)
        logp[lost_drafts] = np.nan
        cand_lp[lost_tokens] = np.nan
        ctx.spd_debug_score(rng.integers(0, 800, (k, 2)), logp, rng.permutation(800)[:k].astype(np.int32), cand_lp)
        score = ctx.spd_debug_read("SCORE").astype(np.float64).reshape(-1)
        assert np.isnan(score).sum() == k * k - (k - len(lost_drafts)) * (k - len(lost_tokens))
        order = np.lexsort((np.arange(k * k), -np.where(np.isnan(score), -np.inf, score), np.isnan(score)))
        assert ctx.spd_debug_read("SEL").tolist() == order[:k].tolist(), (lost_drafts, lost_tokens)
    ctx.close()
