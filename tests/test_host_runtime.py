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
