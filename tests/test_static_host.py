"""The no-allocation entry point's host code on a fake CUDA runtime: a status page that cannot be pinned at one call is tried
again by the next (never under capture), a wait that gave up is reported once, and plans are a device's own."""
import ctypes
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
SNN_OK, SNN_ERR_TIMEOUT = 0, 5


@pytest.fixture
def call(tmp_path):
    # one library, and one set of its globals, per test; -Bsymbolic: its calls stay inside, whatever runtime the process has loaded
    so = tmp_path / "static.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-I{ROOT}/include", f"-I{ROOT}/paper_2110_09195_b200/csrc",
                    "-I/usr/local/cuda/include", "-o", str(so), str(ROOT / "tests/static_harness.cpp")], check=True)
    lib = ctypes.CDLL(str(so))

    def one(register_fails=-1, capturing=0, device=0):
        out = (ctypes.c_int * 3)()
        return lib.static_call(register_fails, capturing, out, device), *out

    def planned():
        out = (ctypes.c_int * 3)()
        lib.static_planned(out)
        return tuple(out)
    one.report, one.planned = lib.static_report, planned
    return one


def test_each_device_has_plans_for_its_own_sms(call):
    """SMs planned for, plans made, questions asked: a plan is kept for the shape on that device, and so is the number of SMs."""
    for device, want in ((0, (148, 1, 1)), (0, (148, 1, 1)), (1, (132, 2, 2)), (0, (148, 2, 2)), (1, (132, 2, 2))):
        assert call(device=device)[0] == SNN_OK
        assert call.planned() == want


def test_pinning_that_failed_is_tried_again(call):
    assert call(register_fails=2) == (SNN_OK, 1, 0, 1)
    assert call() == (SNN_OK, 2, 0, 2)
    assert call() == (SNN_OK, 3, 1, 2)
    assert call() == (SNN_OK, 3, 2, 2)


def test_nothing_is_pinned_under_capture(call):
    assert call(capturing=1) == (SNN_OK, 0, 0, 1)
    assert call() == (SNN_OK, 1, 1, 1)
    assert call(capturing=1) == (SNN_OK, 1, 2, 1)


def test_a_wait_that_gave_up_is_reported_once(call):
    assert call() == (SNN_OK, 1, 1, 0)
    call.report(3)
    assert call() == (SNN_ERR_TIMEOUT, 1, 1, 0)
    assert call() == (SNN_OK, 1, 2, 0)
