"""Device functions on their own: the track model's shortcuts (reciprocals,
quantiser, conversions) against the operations that they stand for, bit for
bit over every operand, and the bounded wait of the grid barrier."""
import ctypes
import os
import subprocess
import time

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


@pytest.mark.parametrize("blocks, extra", [(1, 0), (5, 0), (152, 0), (1, 1), (5, 1)])
def test_grid_barrier_passes_or_gives_up(checks, blocks, extra):
    """All arrivals: every block passes.  One that never comes: every block
    gives up by itself, and the device is usable afterwards."""
    import torch
    arrivals = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    out = torch.zeros(blocks, dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    assert checks.check_barrier(blocks, extra, _ptr(arrivals), _ptr(out)) == 0
    assert time.perf_counter() - t0 < 30.0
    assert out.tolist() == [2 if extra else 1] * blocks
    assert int(arrivals.item()) == blocks
