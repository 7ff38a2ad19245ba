"""CPU: which launches a resolve makes, and what it does when the cooperative
one is refused: csrc/host.cu linked against a runtime that launches nothing and
notes what it was asked for (fake_runtime.cpp, fake_kernels.cu)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2606_05613_gb300 import build as nb
from paper_2606_05613_gb300 import native as bk

HERE = os.path.dirname(os.path.abspath(__file__))
TOO_LARGE, NOT_SUPPORTED = 720, 801      # cudaErrorCooperativeLaunchTooLarge, ...NotSupported
F32, BF16 = bk.BKMOO_F32, bk.BKMOO_BF16


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    d = tmp_path_factory.mktemp("fake")
    inc = ["-I", nb.INCLUDE, "-I", nb.CSRC, "-std=c++17", "-Xcompiler", "-fPIC"]
    objs = []
    for src in (os.path.join(nb.CSRC, "host.cu"), os.path.join(HERE, "fake_kernels.cu"),
                os.path.join(HERE, "fake_runtime.cpp")):
        objs.append(str(d / (os.path.basename(src) + ".o")))
        subprocess.run([nb.nvcc()] + nb.ARCH + inc + ["-c", src, "-o", objs[-1]], check=True)
    so = str(d / "libfake.so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so] + objs + ["-lpthread"], check=True)
    lib = ctypes.CDLL(so)
    lib.fake_notes.restype = ctypes.c_char_p
    return lib


def _resolve(lib, K, dt, off, flags=0, rng=None, error=0, events=False):
    """(return code, launches) of a call on made-up, never touched addresses."""
    off = np.asarray(off, dtype=np.int64)
    p = bk.bkmoo_default_params()
    p.flags |= flags
    if events:
        arr = (ctypes.c_void_p * 4)(1, 2, 3, 4)
        p.events = ctypes.addressof(arr)
    grads = (ctypes.c_void_p * K)(*[(k + 1) << 40 for k in range(K)])
    B = ctypes.c_int64(len(off) - 1)
    lib.fake_reset(error)
    args = [grads, K, dt, off.ctypes.data_as(ctypes.c_void_p), B]
    tail = [bk.RULES["mgda"], ctypes.byref(p), ctypes.c_void_p(1 << 60), dt, None, None,
            ctypes.c_void_p(1 << 59), ctypes.c_size_t(1 << 40), None]
    if rng is None:
        code = lib.bkmoo_resolve(*args, *tail)
    else:
        code = lib.bkmoo_resolve_buckets(*args, ctypes.c_int64(rng[0]), ctypes.c_int64(rng[1]),
                                         *tail)
    return code, lib.fake_notes().decode().split()


PLAN = np.arange(0, 21, dtype=np.int64) * 10 * 16384      # 20 buckets of 10 chunks


def test_cooperative_launch_that_does_not_fit_falls_back(fake):
    three = ["gram", "solve", "combine-last-first"]
    assert _resolve(fake, 4, F32, PLAN) == (bk.BKMOO_OK, ["stream"])
    assert _resolve(fake, 4, F32, PLAN, error=TOO_LARGE) == (
        bk.BKMOO_OK, ["stream", "cleared"] + three)
    assert _resolve(fake, 4, F32, PLAN, rng=(3, 20), error=TOO_LARGE) == (
        bk.BKMOO_OK, ["stream", "cleared"] + three)
    # any other refusal is the caller's: nothing else is launched
    for r in (None, (0, 20)):
        assert _resolve(fake, 4, F32, PLAN, rng=r, error=NOT_SUPPORTED) == (
            bk.BKMOO_ERR_CUDA, ["stream"])
    # the events of a call that falls back lie between the passes
    assert _resolve(fake, 4, F32, PLAN, error=TOO_LARGE, events=True) == (
        bk.BKMOO_OK, ["event", "stream", "cleared", "gram", "event", "solve", "event",
                      "combine-last-first", "event"])
    assert _resolve(fake, 4, F32, PLAN, events=True) == (
        bk.BKMOO_OK, ["event", "stream", "event", "event", "event"])


@pytest.mark.parametrize("K,dt,off,kernels", [
    (4, F32, PLAN, ["gram", "solve", "combine-last-first"]),
    (4, BF16, PLAN * 2, ["gram", "solve", "combine-prefetch"]),
    (3, BF16, PLAN * 2, ["gram", "solve", "combine-last-first"]),
    (8, F32, PLAN, ["gram", "solve", "combine-prefetch"]),
    (6, F32, PLAN, ["gram-bulk", "solve", "combine-prefetch"]),
    (6, F32, [0, 5, 90], ["gram", "solve", "combine-prefetch"]),
    (6, F32, [0, 5, 90, 91], ["gram-bulk", "solve", "combine-prefetch"]),
    (8, F32, [0, 2 * 16384], ["gram", "solve", "combine-prefetch"]),
    (8, F32, [0, 2 * 16384 + 1], ["gram-bulk", "solve", "combine-prefetch"]),
    (12, F32, PLAN, ["gram-prefetch", "solve", "combine-prefetch"]),
    (4, F32, [0, 152 * 16384], ["gram-bulk", "solve", "combine-prefetch"]),
    (4, F32, [0, 153 * 16384], ["gram", "solve", "combine-last-first"]),
    (4, F32, [0, 768 * 16384], ["gram", "solve", "combine-last-first"]),      # 192 MiB
    (4, F32, [0, 768 * 16384 + 1], ["gram", "solve", "combine-prefetch"]),
    # 200 chunks, nine sixteenths full and a little more
    (8, F32, np.arange(0, 201) * 9216, ["gram", "solve", "combine-last-first"]),
    (8, F32, np.arange(0, 201) * 9217, ["gram", "solve", "combine-prefetch"]),
    (8, F32, np.arange(0, 153) * 9216, ["gram-bulk", "solve", "combine-prefetch"]),
    # 1 GiB of half-full chunks
    (8, F32, np.arange(0, 4097) * 8192, ["gram", "solve", "combine-last-first"]),
    (8, F32, np.arange(0, 4098) * 8192, ["gram", "solve", "combine-prefetch"]),
    # 1001 chunks of a quarter of their length: 66 MB
    (4, F32, np.arange(0, 1002) * 4097, ["gram", "solve", "combine-last-first"]),
    (12, BF16, [0, 152 * 32768], ["gram-prefetch", "solve", "combine-prefetch"]),
    (12, BF16, [0, 153 * 32768], ["gram-prefetch", "solve", "combine-last-first"]),
    (16, BF16, [0, 768 * 32768], ["gram-prefetch", "solve", "combine-last-first"]),   # 768 MiB
    (16, BF16, [0, 768 * 32768 + 1], ["gram-prefetch", "solve", "combine-prefetch"]),
    (11, BF16, [0, 153 * 32768], ["gram", "solve", "combine-prefetch"]),
    (16, F32, [0, 153 * 16384], ["gram-prefetch", "solve", "combine-prefetch"]),
    (4, F32, [0, 1025 * 16384], ["gram", "groups", "solve", "combine-prefetch"]),
])
def test_kernels_of_the_three_launches(fake, K, dt, off, kernels):
    assert _resolve(fake, K, dt, off, bk.BKMOO_FLAG_THREE_PASS) == (bk.BKMOO_OK, kernels)


def test_ranges_stream_above_two_buckets(fake):
    for flags in (0, bk.BKMOO_FLAG_FUSED):
        for n in (1, 2):
            assert "stream" not in _resolve(fake, 4, F32, PLAN, flags, rng=(5, 5 + n))[1]
        assert _resolve(fake, 4, F32, PLAN, flags, rng=(5, 8))[1] == ["stream"]
    assert "stream" not in _resolve(fake, 4, F32, PLAN, bk.BKMOO_FLAG_THREE_PASS, rng=(5, 8))[1]
    assert _resolve(fake, 4, F32, PLAN, rng=(5, 5)) == (bk.BKMOO_OK, [])
