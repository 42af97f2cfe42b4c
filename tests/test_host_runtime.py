"""CPU tests of the runtime's host code on a CUDA runtime that needs no GPU (fake_cuda.cpp): what a context does with
its memory, and with calls that CUDA refuses."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2609_15160_gb300 import build, synth, tlf

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    """The library's objects linked against the fake runtime; the binding uses it while this module runs."""
    build.build()
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    out = str(tmp_path_factory.mktemp("fake") / "libtlf_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cuda.cpp"), *[os.path.join(build.BUILD, x.replace(".cu", ".o")) for x in build.SOURCES],
                    "-Wl,-Bsymbolic", "-o", out], check=True)
    fake = tlf.load_library(out)
    for name in ("fake_live", "fake_syncs", "fake_launches", "fake_graph_launches"):
        getattr(fake, name).restype = C.c_long
    fake.fake_launches.argtypes = [C.c_char_p]
    fake.fake_refuse_copy.argtypes = [C.c_void_p]
    fake.fake_device_buffer.restype, fake.fake_device_buffer.argtypes = C.c_void_p, [C.c_size_t]
    fake.fake_free.argtypes = [C.c_void_p]
    real, tlf._LIB = tlf._LIB, fake
    yield fake
    tlf._LIB = real


def _model(dtype="bf16", **kw):
    return synth.tiny_config(**{**dict(vocab=96, d_model=128, n_heads=2, n_kv_heads=2, head_dim=64, n_layers=2,
                                       ffn_hidden=96, max_loops=3, dtype=dtype), **kw})


def _context(m, **kw):
    return tlf.Context(m, synth.make_weights(m), **{**dict(max_seqs=4, max_batch=4, max_seq_len=200, prefill_chunk=64), **kw})


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_a_context_gives_back_all_its_device_memory(lib, dtype):
    before = lib.fake_live()
    with _context(_model(dtype, conditioning=True, router_hidden=16)) as ctx:
        ctx.prefill([1, 2], [np.arange(70, dtype=np.int32), np.arange(5, dtype=np.int32)])
        ctx.decode_step([1, 2], [3, 4])
    assert lib.fake_live() == before


class _DeviceBuffer:
    """A buffer that the fake runtime takes for device memory."""

    def __init__(self, lib, nbytes):
        self.lib, self.ptr = lib, lib.fake_device_buffer(nbytes)

    def data_ptr(self):
        return self.ptr

    def free(self):
        self.lib.fake_free(self.ptr)


@pytest.fixture
def loops(lib):
    """loops(batch, n): from now on every step's results say n loops for each row (nothing computes them here)."""
    hooks = []

    def set_loops(batch, n):
        size = 2 * batch * 4 + 4  # loop counts, margins, error word

        def fill(dst, src, nbytes):
            if nbytes == size:
                C.memmove(dst, (C.c_int32 * batch)(*[n] * batch), 4 * batch)
        hooks.append(C.CFUNCTYPE(None, C.c_void_p, C.c_void_p, C.c_size_t)(fill))
        lib.fake_on_copy(hooks[-1])
    yield set_loops
    lib.fake_on_copy(None)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_a_refused_logits_copy_leaves_host_and_device_at_the_same_lengths(lib, loops, dtype):
    """The step has run by then: the call waits for it and advances the lengths, as the device has, before it fails."""
    m = _model(dtype)
    with _context(m) as ctx:
        loops(4, 2)
        ctx.load_cache(1, synth.make_cache_positions(m, 10, 3))
        want = [ctx.cache_len(1, r) for r in (1, 2, 3)]
        out = _DeviceBuffer(lib, 4 * m.vocab)
        lib.fake_refuse_copy(out.ptr)
        for step in range(3):  # directly, captured, replayed
            syncs = lib.fake_syncs()
            with pytest.raises(tlf.TlfError) as e:
                ctx.decode_step([1], [5], logits=out)
            assert e.value.name == "CUDA" and "logits copy" in str(e.value)
            assert lib.fake_syncs() > syncs
            want = [want[0] + 1, want[1] + 1, want[2]]
            assert [ctx.cache_len(1, r) for r in (1, 2, 3)] == want
        lib.fake_refuse_copy(None)
        ctx.decode_step([1], [5], logits=out)
        out.free()


@pytest.mark.parametrize("refused", ["first launch", "capture", "replay"])
def test_a_refused_cooperative_launch_falls_back_to_a_launch_per_stage(lib, loops, refused):
    """Steps of up to 16 rows want every SM at once; where CUDA says no, the step and all later ones run as kernels of
    their own, and are still captured and replayed."""
    m = _model()
    with _context(m) as ctx:
        loops(4, 1)
        ctx.load_cache(1, synth.make_cache_positions(m, 10, 3))

        def step():
            """(persistent kernels, projections, replayed graphs) of one step, and the launches it reports"""
            names = (b"k_step_small", b"k_gemm_tc")
            before = [lib.fake_launches(n) for n in names] + [lib.fake_graph_launches()]
            ctx.decode_step([1], [5], logits=False)
            after = [lib.fake_launches(n) for n in names] + [lib.fake_graph_launches()]
            return [b - a for a, b in zip(before, after)], ctx.last_step_profile()[2]

        stages = 4 * m.n_layers * m.max_loops
        try:
            good = {"first launch": 0, "capture": 1, "replay": 2}[refused]
            for i in range(good):
                assert step()[0] == [1, 0, i]  # a capture counts as a launch, and its graph is replayed
            lib.fake_refuse_cooperative(1)
            lib.fake_refuse_graph(int(refused == "replay"))
            got, reported = step()
            assert got[:2] == [0, stages] and reported > stages
            lib.fake_refuse_graph(0)
            for i in range(4):
                got, reported = step()
                assert got[0] == 0 and reported > stages
            assert got == [0, 0, 1]  # replayed
        finally:
            lib.fake_refuse_cooperative(0)
            lib.fake_refuse_graph(0)
        assert ctx.cache_len(1, 1) == 10 + good + 5


def _kernel_of_step(lib, ctx, ids):
    """Which kernel ran the block of a (directly launched) step."""
    names = (b"k_step_small", b"k_step_row", b"k_attn_decode")
    before = [lib.fake_launches(n) for n in names]
    ctx.decode_step(ids, [5] * len(ids), logits=False)
    ran = [n for n, b in zip(names, before) if lib.fake_launches(n) > b]
    assert len(ran) == 1
    return ran[0].decode()


@pytest.mark.parametrize("rows,pages_a_group,want", [(1, 100, "k_step_small"), (1, 125, "k_attn_decode"),
                                                     (8, 100, "k_step_small"), (16, 50, "k_step_small"),
                                                     (16, 65, "k_attn_decode")])
def test_the_persistent_step_leaves_long_caches_to_the_launches(lib, monkeypatch, rows, pages_a_group, want):
    """The rule counts the pages of the first loop that each of the kernel's 2 x 152 groups of warps gets."""
    monkeypatch.setenv("TLF_NO_GRAPH", "1")
    m = _model(n_heads=8, n_kv_heads=8, head_dim=32, n_layers=1, max_loops=2)
    keys = pages_a_group * 304 * 64 // (8 * rows)
    with _context(m, max_seqs=rows, max_batch=rows, max_seq_len=keys + 10, kv_pool_pages=rows * 2 * (keys // 64 + 2)) as ctx:
        for i in range(rows):
            ctx.load_cache(i, {"positions": [np.arange(keys, dtype=np.int32), np.arange(0, dtype=np.int32)]})
        assert _kernel_of_step(lib, ctx, list(range(rows))) == want


# layers of 996, 393 and 200 KB; the last is staged in shared memory
ROW_MODELS = {"wide": dict(d_model=192, n_heads=3, n_kv_heads=3, head_dim=64, ffn_hidden=176),
              "narrow": dict(d_model=128, n_heads=4, n_kv_heads=2, head_dim=32, n_layers=1, ffn_hidden=128),
              "tiny": dict(d_model=64, n_heads=4, n_kv_heads=4, head_dim=16, n_layers=1, ffn_hidden=176)}


@pytest.mark.parametrize("model,rows,keys,want", [
    ("wide", 1, 15, "k_step_row"), ("wide", 1, 40, "k_attn_decode"), ("wide", 64, 200, "k_step_row"),
    ("wide", 64, 300, "k_attn_decode"), ("wide", 256, 550, "k_step_row"), ("wide", 256, 650, "k_attn_decode"), ("narrow", 1, 600, "k_step_row"),
    ("narrow", 1, 700, "k_attn_decode"), ("tiny", 1, 1000, "k_step_row"), ("tiny", 256, 1000, "k_step_row"),
    ("tiny", 1, 1024, "k_attn_decode")])
def test_the_row_kernel_takes_what_one_sm_can_read(lib, monkeypatch, model, rows, keys, want):
    """The rule counts a layer's weights, unless they are staged, and the K and V of the longest row's heads."""
    monkeypatch.setenv("TLF_NO_GRAPH", "1")
    m = _model("f32", **ROW_MODELS[model])
    with _context(m, max_seqs=rows, max_batch=rows, max_seq_len=1100, kv_pool_pages=rows * 3 + 60) as ctx:
        for i in range(rows):
            n = keys if i == 0 else 3
            ctx.load_cache(i, {"positions": [np.arange(n, dtype=np.int32)] + [np.arange(0, dtype=np.int32)] * 2})
        assert _kernel_of_step(lib, ctx, list(range(rows))) == want
