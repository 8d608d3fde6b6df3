"""Host code of the runtime without a GPU: the library's own sources, linked with a stand-in for the CUDA runtime that runs
every queued copy as late as it may (tests/fake_cudart.cpp)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2305_13144_b200 import api, build, synth

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    lib = str(tmp_path_factory.mktemp("fake") / "libseqsched_fake.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-shared", "-cudart", "none", "-Xcompiler", "-fPIC",
                    "-Xlinker", "-Bsymbolic", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    *(os.path.join(build.CSRC, s) for s in build.SOURCES), os.path.join(HERE, "fake_cudart.cpp"), "-o", lib],
                   check=True, capture_output=True)
    with pytest.MonkeyPatch.context() as mp:
        mp.setattr(api, "LIB_PATH", lib)
        mp.setattr(api, "_lib_handle", None)
        L = api.lib()
        L.fake_changed_sources.restype = L.fake_pending.restype = C.c_int64
        L.fake_pending.argtypes = [C.c_char_p]
        L.fake_loaded.restype, L.fake_loaded.argtypes = C.c_int64, [C.c_char_p]
        L.fake_wait_limit.restype, L.fake_wait_limit.argtypes = C.c_int64, [C.c_char_p]
        L.fake_fail_wait_behind.argtypes = [C.c_char_p, C.c_int]
        yield L


def _engine(L, max_prefill=32, max_new=8, max_batch=16):
    """An engine over host memory; its weights are loaded (and read as zeros by nobody)."""
    shape = synth.ModelShape(n_layers=1, d_model=64, n_heads=1, head_dim=64, d_ffn=64, vocab=64)
    m, rt = api.model_cfg(shape), api.runtime_cfg(max_batch, 64, max_prefill, max_new, 2048)
    arena = np.empty(api.ss_arena_bytes(m, rt) + 1024, dtype=np.uint8)
    base = arena.ctypes.data + (-arena.ctypes.data) % 1024
    h = C.c_void_p()
    assert L.ss_create(C.byref(m), C.byref(rt), C.c_void_p(base), arena.size - 1024, None, C.byref(h)) == api.SS_OK
    eng = api.Ctx(h, arena, None, m, rt)
    api.ss_load_weights(eng, {k: synth.to_bf16_bits(v) for k, v in synth.make_weights(shape, seed=1).items()})
    return eng


def _batch(seed, lens):
    rng = np.random.default_rng(seed)
    cu = np.zeros(len(lens) + 1, dtype=np.int32)
    cu[1:] = np.cumsum(lens)
    return rng.integers(3, 64, size=int(cu[-1])).astype(np.int32), cu


def test_staging_is_not_refilled_before_its_copies_have_run(fake):
    """Prompt chunks and batches one behind the other, nothing waited for by the caller: what a copy reads is what it was given."""
    eng = _engine(fake)
    before = fake.fake_changed_sources()
    for seed in range(3):
        toks, cu = _batch(seed, [20, 17, 30, 5, 9])        # 32 tokens a chunk: four chunks
        api.ss_prefill(eng, toks, cu, None, 4)
        api.ss_keep_prompts(eng, np.arange(5) + 5 * (seed % 2), cu[1:] - cu[:-1])
        api.ss_decode_steps(eng, 2)
        api.ss_release_batch(eng)
        for ids in ([0, 3], [2]):
            api.ss_resume(eng, ids, None, 4)
            api.ss_decode_steps(eng, 1)
            api.ss_release_batch(eng)
    api.ss_last_device_status(eng)                         # everything that is queued runs
    assert fake.fake_changed_sources() == before
    api.ss_destroy(eng)


def test_prompt_pass_returns_behind_its_layers(fake):
    """When ss_prefill returns, the hidden states that it hands out are there and an error of the layers has been reported."""
    eng = _engine(fake)
    toks, cu = _batch(1, [20, 17, 30])
    api.ss_prefill(eng, toks, cu, None, 4)
    assert fake.fake_pending(b"gather_last_rmsnorm") == 0
    assert fake.fake_pending(b"lmhead_tile_argmax") == 1   # nothing is gained by waiting for these
    api.ss_release_batch(eng)
    api.ss_last_device_status(eng)
    fake.fake_fail_wait_behind(b"gather_last_rmsnorm", 719)       # cudaErrorLaunchFailure
    with pytest.raises(api.SSError) as e:
        api.ss_prefill(eng, toks, cu, None, 4)
    assert e.value.code == api.SS_ERR_CUDA and api.ss_last_cuda_error(eng) == 719
    api.ss_prefill(eng, toks, cu, None, 4)                 # the failed batch was released
    api.ss_release_batch(eng)
    api.ss_destroy(eng)


def test_the_wait_limit_reaches_the_prompt_pass(fake):
    """Both GEMMs (chunks of up to 256 tokens and longer ones) and the attention."""
    eng = _engine(fake, max_prefill=512)
    for ms in (7, 50):
        api.ss_set_wait_limit_ms(eng, ms)
        for lens in ([20, 30], [60] * 6):
            toks, cu = _batch(4, lens)
            api.ss_prefill(eng, toks, cu, None, 4)
            api.ss_release_batch(eng)
        for kernel in (b"gemm_wx_kernel", b"gemm_wx_pair_kernel", b"attn_prefill"):
            assert fake.fake_wait_limit(kernel) == ms * 1965000, kernel
    api.ss_last_device_status(eng)
    api.ss_destroy(eng)


def test_a_context_loads_the_kernels_that_it_can_launch(fake):
    """Four instantiations of the decode step (up to 16, 64, 128 and 256 rows of its head size), the traced ones when asked for."""
    fake.fake_loaded(b"")
    eng = _engine(fake)
    assert fake.fake_loaded(b"decode_step_mega") == 4
    api.ss_set_trace(eng, False)
    assert fake.fake_loaded(b"decode_step_mega") == 0
    api.ss_set_trace(eng, True)
    assert fake.fake_loaded(b"decode_step_mega") == 4
    api.ss_destroy(eng)


def _resident():
    return int(open("/proc/self/statm").read().split()[1]) * os.sysconf("SC_PAGE_SIZE")


def test_host_memory_follows_the_batch_and_not_the_limits(fake):
    """A context for 256 rows of up to a million tokens: its host memory grows with what a batch brings back."""
    before = _resident()
    eng = _engine(fake, max_batch=256, max_new=1 << 20)
    assert _resident() - before < 64 << 20
    toks, cu = _batch(3, [20, 17, 30])
    api.ss_prefill(eng, toks, cu, None, 30)
    out, lens, _ = api.ss_read_batch(eng, 3, 30)           # no kernel ran, so no token was generated
    assert lens.tolist() == [0, 0, 0]
    assert _resident() - before < 64 << 20
    api.ss_destroy(eng)
