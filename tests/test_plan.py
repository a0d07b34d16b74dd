"""The planner of the tensor-core kernel, compiled for the host: every shape the path takes can be planned, fits shared and
tensor memory, and keeps the kernel's reads inside what is staged."""
import ctypes
import random
import subprocess
from pathlib import Path

import numpy as np
import pytest

ROOT = Path(__file__).resolve().parent.parent
WORDS, CHAIN, SIGNS = 0, 1, 2
SMS = 148


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = tmp_path_factory.mktemp("plan") / "plan.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", f"-I{ROOT}/include", f"-I{ROOT}/paper_2110_09195_b200/csrc",
                    "-I/usr/local/cuda/include", "-o", str(so), str(ROOT / "tests/plan_harness.cpp")], check=True)
    lib = ctypes.CDLL(str(so))
    lib.plan_make.restype = ctypes.c_char_p
    return lib


def _array(shapes):
    return np.array(shapes, np.int32).ctypes.data_as(ctypes.POINTER(ctypes.c_int))


def takes(lib, shape, f16):
    return bool(lib.plan_takes(_array(shape), int(f16)))


def make(lib, shapes, f16=False, kind=WORDS):
    """[(lg, Np, tma, tiles)] of the problems (N, H, W, C, K, stride, pad, ksize)."""
    out = np.zeros((len(shapes), 4), np.int32)
    err = lib.plan_make(_array(shapes), len(shapes), int(f16), kind, SMS, out.ctypes.data_as(ctypes.POINTER(ctypes.c_int)))
    assert err is None, (err, shapes, f16, kind)
    return out.tolist()


def draw(rng):
    log = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    ksize = rng.choice((3, 3, 3, 1))
    return (log(1, 300), log(3, 700), log(3, 700), log(1, 1200), log(1, 1200), rng.choice((1, 2)),
            0 if ksize == 1 else rng.choice((0, 1)), ksize)


@pytest.mark.parametrize("f16", [False, True])
def test_every_shape_the_path_takes_can_be_planned(lib, f16):
    rng = random.Random(5)
    taken = 0
    for _ in range(4000):
        shape = draw(rng)
        if not takes(lib, shape, f16):
            continue
        taken += 1
        for kind in (WORDS,) if f16 else (WORDS, SIGNS, CHAIN):
            make(lib, [shape], f16, kind)
    assert taken > 500


@pytest.mark.parametrize("f16", [False, True])
def test_every_group_of_such_shapes_can_be_planned(lib, f16):
    rng = random.Random(6)
    for _ in range(60):
        shapes = [s for s in (draw(rng) for _ in range(80)) if takes(lib, s, f16)][:rng.randint(2, 32)]
        for kind in (WORDS,) if f16 else (WORDS, SIGNS):
            make(lib, shapes, f16, kind)
