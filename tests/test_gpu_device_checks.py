"""Device functions on their own: the track model's shortcuts (reciprocals,
quantiser, conversions) against the operations that they stand for, bit for
bit over every operand."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SWEEP = ("frcp2, first operand", "frcp2, second operand", "quant to the pad limit",
         "quant to the time limit", "time_to_t", "pad_to_y")


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_02206_gb300 import build
    so = str(tmp_path_factory.mktemp("checks") / "device_checks.so")
    r = subprocess.run([build.nvcc(), *build.FLAGS, *build.ARCH, "-shared", "-o", so,
                        os.path.join(HERE, "device_checks.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    torch.zeros(1, device="cuda:0")
    return ctypes.CDLL(so)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def test_model_shortcuts_over_all_operands(checks):
    import torch
    bad = torch.zeros(len(SWEEP), dtype=torch.int64, device="cuda:0")
    torch.cuda.synchronize()
    assert checks.check_sweep(_ptr(bad)) == 0
    assert {k: int(v) for k, v in zip(SWEEP, bad.cpu())} == dict.fromkeys(SWEEP, 0)
