"""What the bounded device waits do when they run out: on a barrier at which nobody arrives, with nothing in flight."""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_2504_08966_b200 import build

pytestmark = pytest.mark.gpu

WARPS = 4


@pytest.fixture(scope="module")
def waits(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("waits") / "waits.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "waits.cu")
    subprocess.check_call([build._nvcc(), "-shared", "-o", lib, src, "-I", build.CSRC] + build.FLAGS)
    return C.CDLL(lib)


def _stream():
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("late", [-1, 0, 1, WARPS - 1])
def test_any_warp_reports_a_wait_that_ran_out(waits, late):
    status, ok = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((WARPS,), 7, dtype=torch.int32, device="cuda")
    assert waits.late_warp(late, WARPS, C.c_void_p(status.data_ptr()), C.c_void_p(ok.data_ptr()), _stream()) == 0
    torch.cuda.synchronize()
    assert ok.tolist() == [int(w != late) for w in range(WARPS)]
    assert status.tolist() == [-5 if late >= 0 else 0]


def test_a_cta_that_has_given_up_does_not_wait_again(waits):
    """Twenty waits after one another take the second of the first one, not twenty."""
    failed = torch.zeros(WARPS, dtype=torch.int32, device="cuda")
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    begin.record()
    assert waits.many_waits(20, WARPS, C.c_void_p(failed.data_ptr()), _stream()) == 0
    end.record()
    torch.cuda.synchronize()
    assert failed.tolist() == [20] * WARPS
    assert begin.elapsed_time(end) < 3000
