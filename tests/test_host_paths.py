"""The host code of the C ABI on a fake runtime and fake launchers (no GPU): what a call that fails half-way leaves behind."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run([NVCC, "-O1", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-shared",
                    "--cudart", "none", "-o", out, os.path.join(HERE, "fake_launches.cu")], check=True)
    return ctypes.CDLL(out)


def _verify(lib, words):
    """A verify call on the library's own scratch whose streaming launch uses `words` hand-over words."""
    buf = ctypes.create_string_buffer(4096 + 16)
    p = ctypes.c_void_p((ctypes.addressof(buf) + 15) & ~15)   # (never read or written: the launchers are fakes)
    return lib.sgbv_verify(p, p, p, p, words, 1, 1, 64, ctypes.c_float(1.0), p, p, p, None)


def test_a_call_that_failed_half_way_leaves_no_published_words_behind(lib):
    """The finishing launch is refused after the streaming kernel has published 148 words; a small call (10 words) and then
    a large one follow.  Neither may find a word published before its own streaming kernel runs."""
    lib.fake_set(0, 0, 0)
    assert _verify(lib, 148) == 0 and lib.fake_stale() == 0
    lib.fake_set(1, 0, 0)
    assert _verify(lib, 148) < 0
    lib.fake_set(0, 0, 0)
    for words in (10, 148, 256):
        assert _verify(lib, words) == 0 and lib.fake_stale() == 0, words


def test_words_in_doubt_stay_so_until_they_have_been_cleared(lib):
    """Neither a call that is only captured nor one whose own clearing fails ends the doubt."""
    lib.fake_set(1, 0, 1)
    assert _verify(lib, 148) < 0
    lib.fake_set(0, 1, 0)
    assert _verify(lib, 148) == 0
    lib.fake_set(0, 0, 1)
    streamed = lib.fake_streamed()
    assert _verify(lib, 10) < 0 and lib.fake_streamed() == streamed
    lib.fake_set(0, 0, 0)
    for words in (10, 148):
        assert _verify(lib, words) == 0 and lib.fake_stale() == 0, words
