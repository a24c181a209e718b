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


@pytest.fixture(scope="module")
def kernels(tmp_path_factory):
    import ctypes as C
    import os
    import shutil
    import subprocess
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = str(tmp_path_factory.mktemp("attn") / "libattn.so")
    subprocess.check_call([shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-I", os.path.join(root, "include"), "-I", os.path.join(root, "paper_2405_18400_b200", "csrc"), "-o", out,
                           os.path.join(root, "tests", "attn_kernels.cu")])
    lib = C.CDLL(out)
    lib.attn_run.argtypes = [C.c_int, C.c_int] + [C.c_void_p] * 4 + [C.c_int] * 6
    return lib


# A prefix's tokens keep their bits whichever job they fall into, so the kernel of up to 128 tokens and those of longer jobs have to agree.
@pytest.mark.parametrize("pos0", [0, 1, 47, 48, 63, 64, 384, 1900])
@pytest.mark.parametrize("hd", [64, 128])
def test_short_and_long_jobs_kernels_agree_to_the_bit(kernels, hd, pos0):
    import torch
    heads, rows, max_pos = 3, 130, 2048
    g = torch.Generator(device="cuda:0").manual_seed(hd + pos0)
    torch.cuda.synchronize()
    assert kernels.attn_prepare() == 0
    q = torch.randn(rows, heads * hd, generator=g, device="cuda:0") * 3
    k, v = (torch.randn(2, max_pos, heads * hd, generator=g, device="cuda:0").to(torch.bfloat16) for _ in range(2))
    for n_tok in (1, 2, 15, 16, 17, 64, 65, 100, 128):
        out = {}
        for which in (0, 4, 8):
            x = torch.full((3, rows, heads * hd), -1, dtype=torch.int16, device="cuda:0")
            torch.cuda.synchronize()
            assert kernels.attn_run(which, hd, q.data_ptr(), k.data_ptr(), v.data_ptr(), x.data_ptr(), heads, rows, max_pos, 1, pos0, n_tok) == 0
            out[which] = x
        assert torch.equal(out[0], out[4]) and torch.equal(out[0], out[8]), n_tok
        assert (out[0][:, n_tok:] == -1).all()
        # and the terms are a softmax's output
        o = (out[0][:, :n_tok].to(torch.int32) << 16).view(torch.float32).double().sum(0).view(n_tok, heads, hd)
        T = pos0 + n_tok
        s = torch.einsum("thc,phc->htp", q[:n_tok].view(n_tok, heads, hd).double(), k[1, :T].view(T, heads, hd).double()) / hd ** 0.5
        s.masked_fill_(torch.arange(T, device="cuda:0")[None, None] > pos0 + torch.arange(n_tok, device="cuda:0")[None, :, None], float("-inf"))
        want = torch.einsum("htp,phc->thc", s.softmax(-1), v[1, :T].view(T, heads, hd).double())
        # (a score of up to 16 is a float32, so is __expf's argument: 1e-6 of a weight each, and half of that for the sums; 1e-5 is four times it)
        assert float((o - want).abs().max()) <= 1e-5 * float(want.abs().max())
