"""Batched timesteps: B requests, each a context of its own over shared weights, stepped together with one pass over
the weights per timestep, every request compared element by element with its own CPU oracle (B independent
oracles: a request's step does not depend on the batch it runs in)."""
import numpy as np
import pytest
import torch

import spd_inputs as si
from oracle import spd_oracle as so
from tests.gpu_common import compare_first_step, compare_step

pytestmark = pytest.mark.gpu


def _requests(P, shape, packed, dtabs, host, tables, n, k, orders, lam, alpha, tau, delta, max_pos, kv_dtype, prefix_len, zipf_s):
    out = []
    otabs = sorted(tables, key=lambda t: int(t["n"]))
    for r in range(n):
        ctx = P.SpdContext(shape, packed, dtabs, k, orders, lam, alpha, tau, delta, max_pos, kv_dtype)
        cfg = so.make_config(shape, k, orders, lam, alpha, tau, delta, max_pos, kv_dtype)
        orc = so.Oracle(cfg, host, otabs)
        prefix = si.make_prefix("zipf", prefix_len + (r % 5), shape.vocab, zipf_s, seed=700 + r)   # own prefix, own length
        out.append((ctx, orc, prefix))
    return out


# the products' instances for up to 16, 32, 64 and 128 token rows
@pytest.mark.parametrize("n,kv_dtype", [(2, "bf16"), (8, "f32"), (32, "bf16"), (48, "bf16"), (70, "f32")])
def test_batched_steps_tiny(tiny_inputs, n, kv_dtype):
    import paper_2405_18400_b200 as P

    wl, weights, tables, _ = tiny_inputs
    packed = P.pack_weights(weights, "cuda:0")
    dtabs = P.build_ngram_tables(tables, "cuda:0")
    reqs = _requests(P, wl.shape, packed, dtabs, weights, tables, n, wl.k, wl.orders, wl.lambdas(), wl.alpha, wl.tau, wl.delta,
                     256, kv_dtype, 12, wl.zipf_s)
    for ctx, orc, prefix in reqs:
        compare_first_step(ctx, orc, prefix)
    ctxs = [r[0] for r in reqs]
    before = ctxs[0].spd_launch_count()
    for step in range(3):
        res = P.spd_batch_step(ctxs)
        for (ctx, orc, _), got in zip(reqs, res):
            ids, par, g = compare_step(ctx, orc, None, stepped=got, path="prefill")
            assert abs(float(g.sum()) - 1.0) < 1e-5 and np.all(np.diff(g) <= 0)
    # a timestep of the batch is 9 launches per layer and three around them, whatever the number of requests
    assert ctxs[0].spd_launch_count() - before == 3 * (9 * wl.shape.n_layers + 3)
    # requests leave the batch and carry on alone, or in another batch, from where they are
    compare_step(reqs[0][0], reqs[0][1])
    if n > 2:
        sub = reqs[1: n // 2 + 1]
        res = P.spd_batch_step([r[0] for r in sub])
        for (ctx, orc, _), got in zip(sub, res):
            compare_step(ctx, orc, None, stepped=got, path="prefill")
    # several timesteps in one call equal the same number of single calls
    a = reqs[-1][0]
    b_ctx = P.SpdContext(wl.shape, packed, dtabs, wl.k, wl.orders, wl.lambdas(), wl.alpha, wl.tau, wl.delta, 256, kv_dtype)
    pf = reqs[-1][2]
    b_ctx.spd_prefill(pf)
    P.spd_batch_generate([b_ctx], 3)
    c_ctx = P.SpdContext(wl.shape, packed, dtabs, wl.k, wl.orders, wl.lambdas(), wl.alpha, wl.tau, wl.delta, 256, kv_dtype)
    c_ctx.spd_prefill(pf)
    for _ in range(3):
        P.spd_batch_step([c_ctx])
    assert np.array_equal(b_ctx.spd_debug_read("LOGITS"), c_ctx.spd_debug_read("LOGITS"))
    assert np.array_equal(b_ctx.spd_debug_read("LOGP"), c_ctx.spd_debug_read("LOGP"))
    for ctx, orc, _ in reqs:
        ctx.close(); orc.close()
    b_ctx.close(); c_ctx.close()


def test_batched_steps_7b_width():
    """Eight requests at the 7B shape's width (two layers): rows of 4096 and 11008 columns through the batched
    products, head size 128, five n-gram orders."""
    import paper_2405_18400_b200 as P

    shape = si.ModelShape("w7b", 2, 4096, 32, 11008, 2000)
    dev = torch.device("cuda:0")
    weights = si.make_weights(shape, seed=51, device=dev)
    host = {n: ([t.cpu() for t in v] if isinstance(v, list) else v.cpu()) for n, v in weights.items()}
    tables = si.make_ngram_tables(shape.vocab, 1.1, 100_000, (2, 3, 4, 5, 6), 5000, seed=52)
    lam = [0.01, 0.04, 0.15, 0.18, 0.12, 0.0, 0.0, 0.0]
    packed = P.pack_weights(weights, dev, consume=True)
    del weights
    dtabs = P.build_ngram_tables(tables, dev)
    reqs = _requests(P, shape, packed, dtabs, host, tables, 8, 3, (2, 3, 4, 5, 6), lam, 0.54, 0.06, 0.01, 192, "bf16", 15, 1.1)
    stats = []
    for ctx, orc, prefix in reqs:
        compare_first_step(ctx, orc, prefix, stats)
    ctxs = [r[0] for r in reqs]
    for step in range(2):
        res = P.spd_batch_step(ctxs)
        for (ctx, orc, _), got in zip(reqs, res):
            compare_step(ctx, orc, stats, stepped=got, path="prefill")
    assert max(s["eps_z"] for s in stats if "eps_z" in s) < 2e-3
    for ctx, orc, _ in reqs:
        ctx.close(); orc.close()


def test_batch_argument_checks(tiny_inputs):
    import paper_2405_18400_b200 as P

    wl, weights, tables, prefix = tiny_inputs
    packed = P.pack_weights(weights, "cuda:0")
    dtabs = P.build_ngram_tables(tables, "cuda:0")
    mk = lambda max_pos=256, **kw: P.SpdContext(wl.shape, packed, dtabs, wl.k, wl.orders, wl.lambdas(), wl.alpha, wl.tau, wl.delta,
                                                max_pos, "bf16", **kw)
    a, b, small, stopper = mk(), mk(), mk(64), mk(eos_id=5)
    for c in (a, small, stopper):
        c.spd_prefill(prefix)

    def status(ctxs, steps=1):
        with pytest.raises(P.SpdError) as e:
            P.spd_batch_generate(ctxs, steps)
        return e.value.status

    assert status([a, b]) == -2                 # b was not prefilled
    b.spd_prefill(prefix)
    assert status([a, a]) == -1                 # a request twice
    assert status([small, a]) == -3             # the leading context has no long-prefix buffers to lend
    assert status([a, stopper]) == -1           # stop tokens are a single-request feature
    assert status([a, b], 0) == -3 and status([a, b], 1000) == -3
    P.spd_batch_generate([a, small], 2)         # only the leading context needs the buffers
    assert a.spd_debug_read("CAND_TOK").tolist() == small.spd_debug_read("CAND_TOK").tolist()
    for c in (a, b, small, stopper):
        c.close()


@pytest.mark.parametrize("kv_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("heads,k", [(4, 3), (2, 16)])
def test_a_nan_in_the_cache_reaches_the_logits(heads, k, kv_dtype):
    """A damaged cache row is not left out of the softmax: behind a NaN key, at whichever position and so in whichever group
    of lanes, a request's logits are NaN, and only that request's.  (19 positions: most groups hold one.)"""
    import paper_2405_18400_b200 as P

    shape = si.ModelShape("hd%d" % (256 // heads), 2, 256, heads, 512, 1000)
    packed = P.pack_weights(si.make_weights(shape, seed=73), "cuda:0")
    args = (k, (2, 3), [0.0] * 8, 0.4, 0.2, 0.05, 256, kv_dtype)
    ctxs = [P.SpdContext(shape, packed, [], *args) for _ in range(2)]
    prefixes = [si.make_prefix("zipf", 18, shape.vocab, 1.1, seed=74 + r) for r in range(2)]
    dtype, size = (torch.bfloat16, 2) if kv_dtype == "bf16" else (torch.float32, 4)
    sound = None
    for position in (None, 0, 1, 9, 17):
        for ctx, prefix in zip(ctxs, prefixes):
            ctx.spd_prefill(prefix)
        if position is not None:
            # keys of the first layer, the workspace's first bytes: [max_pos][d_model]; the last head's first dimension
            keys = ctxs[1].workspace[: 256 * 256 * size].view(dtype).view(256, 256)
            keys[position, 256 - 256 // heads] = float("nan")
        P.spd_batch_step(ctxs)
        z = [ctx.spd_debug_read("LOGITS") for ctx in ctxs]
        if position is None:
            sound = z[0]
            assert np.isfinite(z[1]).all()
        else:
            assert np.isnan(z[1]).all(), position
        assert np.array_equal(z[0], sound)
        for ids, par, _ in P.spd_batch_step(ctxs):     # and the drafts stay ones that can be carried on
            assert ids.min() >= 0 and ids.max() < shape.vocab and par.min() >= 0 and par.max() < k
    for ctx in ctxs:
        ctx.close()


def test_a_malformed_table_of_one_request_stops_only_that_request(tiny_inputs):
    """A table image without an empty slot makes one request's probes run to their bound in the first of three timesteps: the
    call reports it, that request has no drafts to go on from, the others are where a batch without it has them."""
    import paper_2405_18400_b200 as P

    wl, weights, tables, prefix = tiny_inputs
    packed = P.pack_weights(weights, "cuda:0")
    good = P.build_ngram_tables(tables, "cuda:0")
    slots = 1 << 15
    img = np.zeros((slots, 4), np.uint32)
    img[:, 0] = np.arange(slots, dtype=np.uint32) | 0xfff00000          # keys no lookup asks for
    img[:, 3] = 1
    full = torch.from_numpy(img.view(np.uint8).reshape(-1)).to("cuda:0")
    bad = [dict(t) for t in good]
    bad[0] = {"n": 2, "ngram_slots": slots, "ctx_slots": slots, "ngram": full, "ctx": full}
    mk = lambda tabs: P.SpdContext(wl.shape, packed, tabs, wl.k, wl.orders, wl.lambdas(), wl.alpha, wl.tau, wl.delta, 256, "f32")
    for at in (0, 1, 2):                        # the leading context, whose workspace the batch borrows, among them
        ctxs, sound = [mk(bad if r == at else good) for r in range(3)], [mk(good) for _ in range(3)]
        for r in range(3):
            for c in (ctxs[r], sound[r]):
                c.spd_prefill(np.roll(prefix, r))
        with pytest.raises(P.SpdError) as e:
            P.spd_batch_generate(ctxs, 3)
        assert e.value.status == -6
        P.spd_batch_generate(sound, 3)
        with pytest.raises(P.SpdError) as e:
            ctxs[at].spd_step()
        assert e.value.status == -2
        others = [r for r in range(3) if r != at]
        for _ in range(2):
            for r in others:
                for what in ("LOGITS", "LOGP", "SEL"):
                    assert np.array_equal(ctxs[r].spd_debug_read(what), sound[r].spd_debug_read(what)), (at, r, what)
            P.spd_batch_step([ctxs[r] for r in others])
            P.spd_batch_step([sound[r] for r in others])
        ctxs[at].spd_prefill(prefix)            # and the request itself can be taken up again, up to its table
        for c in ctxs + sound:
            c.close()


@pytest.mark.parametrize("heads", [16, 8])
def test_batches_behind_long_prefixes(heads):
    """24 requests behind 2 to 900 positions, float32 and bf16 caches among them: the attention asks for the first rows of a cache ahead,
    as many as a block's share of L2 (341 float32, 682 bf16 here), so for all rows of some requests and a part of others'."""
    import paper_2405_18400_b200 as P

    shape = si.ModelShape("long%d" % heads, 1, 1024, heads, 512, 600)
    weights = si.make_weights(shape, seed=121)
    packed = P.pack_weights(weights, "cuda:0")
    tables = si.make_ngram_tables(shape.vocab, 1.1, 20_000, (2, 3), 2000, seed=122)
    dtabs = P.build_ngram_tables(tables, "cuda:0")
    otabs = sorted(tables, key=lambda t: int(t["n"]))
    lam = [0.3, 0.2] + [0.0] * 6
    lengths = [2, 341, 342, 343, 682, 683, 900, 100] + [40 * (r + 1) for r in range(16)]
    ctxs, orcs = [], {}
    for r, m in enumerate(lengths):
        kv_dtype = "bf16" if r % 2 else "f32"
        ctx = P.SpdContext(shape, packed, dtabs, 3, (2, 3), lam, 0.4, 0.2, 0.05, 920, kv_dtype)
        prefix = si.make_prefix("zipf", m, shape.vocab, 1.1, seed=123 + r)
        if r in (0, 2, 4, 5, 6):
            orcs[r] = so.Oracle(so.make_config(shape, 3, (2, 3), lam, 0.4, 0.2, 0.05, 920, kv_dtype), weights, otabs)
            compare_first_step(ctx, orcs[r], prefix)
        else:
            ctx.spd_prefill(prefix)
        ctxs.append(ctx)
    for _ in range(2):
        res = P.spd_batch_step(ctxs)
        for r, orc in orcs.items():
            compare_step(ctxs[r], orc, None, stepped=res[r], path="prefill")
    for c in ctxs + list(orcs.values()):
        c.close()
