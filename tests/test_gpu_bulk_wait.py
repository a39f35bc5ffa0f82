"""The wait for a block's bulk copies: one answer for all threads, whoever of them gave up, and an end where nothing arrives."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2405_17517_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("probe") / "bulk_wait_probe.so")
    source = os.path.join(os.path.dirname(os.path.abspath(__file__)), "bulk_wait_probe.cu")
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-shared", source, "-o", lib], check=True)
    call = ctypes.CDLL(lib).bulk_wait_probe
    call.argtypes = [ctypes.c_int, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    return call


@pytest.mark.parametrize("threads", [64, 128])
@pytest.mark.parametrize("arrive,first_warp,others,want", [(1, 64, 64, 1),    # all see the copies
                                                           (1, 0, 64, 0),     # one warp gives up, the others see them
                                                           (1, 64, 0, 0),
                                                           (1, 0, 0, 0),      # all give up
                                                           (0, 8, 8, 0)])     # nothing arrives: the wait ends
def test_every_thread_gets_one_answer(probe, threads, arrive, first_warp, others, want):
    torch.cuda.init()
    answer = torch.full((threads,), 7, dtype=torch.int32, device="cuda")
    clocks = torch.zeros(threads, dtype=torch.int64, device="cuda")
    assert probe(arrive, first_warp, others, threads, answer.data_ptr(), clocks.data_ptr()) == 0
    assert answer.tolist() == [want] * threads
