"""The host side of the library on a runtime without a device (tests/fake_cuda.cpp): what a call that fails leaves behind."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
L = 2     # layers
ESTATE, ECUDA = -2, -5


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2405_18400_b200.binding import SpdConfig, _Weights
    src = os.path.join(ROOT, "paper_2405_18400_b200", "csrc")
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.check_call(["g++", "-x", "c++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                           "-I", os.path.join(ROOT, "include"), "-I", src, "-o", out, os.path.join(src, "spd_api.cu"),
                           os.path.join(ROOT, "tests", "fake_cuda.cpp")])
    lib = C.CDLL(out)
    lib.spd_create.argtypes = [C.POINTER(SpdConfig), C.POINTER(_Weights), C.c_void_p, C.c_int32, C.c_void_p, C.c_size_t, C.POINTER(C.c_void_p)]
    lib.spd_prefill.argtypes = [C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p]
    lib.spd_step.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.spd_generate.argtypes = [C.c_void_p, C.c_int32] + [C.c_void_p] * 4
    lib.spd_sample.argtypes = [C.c_void_p, C.c_int32, C.c_float, C.c_float] + [C.c_void_p] * 4
    lib.spd_batch_generate.argtypes = [C.c_void_p, C.c_int32, C.c_int32]
    lib.spd_batch_step.argtypes = [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.spd_destroy.argtypes = [C.c_void_p]
    return lib


PREFIX = np.arange(5, dtype=np.int32)


class Context:
    def __init__(self, lib):
        from paper_2405_18400_b200.binding import SpdConfig, _Weights, _PP
        cfg = SpdConfig()
        cfg.n_layers, cfg.d_model, cfg.n_heads, cfg.d_ffn, cfg.vocab, cfg.max_pos = L, 128, 2, 128, 512, 192
        cfg.rms_eps, cfg.rope_theta, cfg.k, cfg.n_min, cfg.n_max = 1e-5, 10000.0, 2, 2, 3
        cfg.alpha, cfg.tau, cfg.delta, cfg.eos_id, cfg.kv_dtype = 0.5, 0.1, 0.01, -1, 1
        w = _Weights()
        place = 1 << 20                       # no kernel runs: an aligned address is all that is wanted
        w.tok_emb = w.final_norm = w.lm_head = place
        layers = (C.c_void_p * L)(*[place] * L)
        for name in ("attn_norm", "wqkv", "wo", "ffn_norm", "wgate_up", "wdown"):
            setattr(w, name, C.cast(layers, _PP))
        n = C.c_size_t()
        assert lib.spd_workspace_bytes(C.byref(cfg), C.byref(n)) == 0
        self.lib, self.buf, self.h = lib, np.zeros(n.value + 256, np.uint8), C.c_void_p()
        at = self.buf.ctypes.data
        assert lib.spd_create(C.byref(cfg), C.byref(w), None, 0, at + -at % 256, n.value, C.byref(self.h)) == 0

    def prefill(self):
        return self.lib.spd_prefill(self.h, PREFIX.ctypes.data, 5, None, None)

    def step(self):
        return self.lib.spd_step(self.h, None, None, None)

    def generate(self):
        return self.lib.spd_generate(self.h, 2, None, None, None, None)

    def sample(self):
        u = np.zeros(2, np.float32)
        return self.lib.spd_sample(self.h, 2, 0.9, 1.0, u.ctypes.data, None, None, None)


@pytest.fixture
def pair(lib):
    ctxs = [Context(lib) for _ in range(2)]
    for c in ctxs:
        assert c.prefill() == 0
    yield ctxs, (C.c_void_p * 2)(*[c.h for c in ctxs])
    lib.fake_fail(-1, -1)
    for c in ctxs:
        lib.spd_destroy(c.h)


# the first copy of a batch brings the requests' parameters to the device, the second their results back
@pytest.mark.parametrize("call", ["generate", "step"])
@pytest.mark.parametrize("copies,waits", [(1, -1), (-1, 0)])
def test_a_batch_that_fails_leaves_no_request_to_go_on_from(lib, pair, copies, waits, call):
    ctxs, handles = pair
    lib.fake_fail(copies, waits)
    rc = lib.spd_batch_generate(handles, 2, 3) if call == "generate" else lib.spd_batch_step(handles, 2, None, None, None)
    assert rc == ECUDA
    lib.fake_fail(-1, -1)
    assert [c.step() for c in ctxs] == [ESTATE] * 2 and lib.spd_batch_generate(handles, 2, 1) == ESTATE
    assert [c.prefill() for c in ctxs] == [0, 0] and lib.spd_batch_generate(handles, 2, 3) == 0 and [c.step() for c in ctxs] == [0, 0]


@pytest.mark.parametrize("call", [Context.step, Context.generate])
@pytest.mark.parametrize("copies,waits", [(0, -1), (-1, 0)])      # the copy of the result, the wait for it
def test_steps_that_fail_leave_no_drafts_to_go_on_from(lib, pair, copies, waits, call):
    ctx = pair[0][0]
    lib.fake_fail(copies, waits)
    assert call(ctx) == ECUDA
    lib.fake_fail(-1, -1)
    assert ctx.step() == ESTATE
    assert ctx.prefill() == 0 and call(ctx) == 0 and ctx.step() == 0


@pytest.mark.parametrize("call", ["prefill", "sample", "batch"])
def test_calls_that_wait_are_refused_under_capture(lib, pair, call):
    """Before anything has changed: nothing is enqueued, and the contexts go on from where they were."""
    ctxs, handles = pair
    calls = {"prefill": ctxs[0].prefill, "sample": ctxs[0].sample, "batch": lambda: lib.spd_batch_generate(handles, 2, 3)}
    before = lib.fake_enqueued()
    lib.fake_capture(1)
    assert calls[call]() == ECUDA
    lib.fake_capture(0)
    assert lib.fake_enqueued() == before
    assert calls["sample"]() == 0 and calls["batch"]() == 0       # sampling continues a prefix behind which no step was taken yet
    assert ctxs[0].step() == 0
