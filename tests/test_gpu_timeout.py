"""The device-side timeout status, exercised without hanging or faulting anything.

Every barrier wait in the library's kernels is bounded: after its limit it records
SPARKATTN_E_DEVICE_TIMEOUT plus an id of the wait in the workspace's status words and the kernel
winds down.  The product kernels never meet that case on valid input, so this test builds tiny
kernels of its own (tests/cuda/timeout_probe.cu) that call the same helpers, `mbar_wait` (d = 64 forward,
compensation) and `pipe_wait` with `report_abort` (pipelined forward), on a barrier nothing arrives at, with
a limit of one millisecond, and reads the status back through the library's sparkattn_read_status."""
import ctypes
import os
import subprocess
import time

import pytest
import torch

import paper_2609_23153_b200 as sa

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libtimeout_probe.so")
    src = os.path.join(HERE, "cuda", "timeout_probe.cu")
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-gencode", "arch=compute_100a,code=sm_100a", "-shared",
                    "-Xcompiler", "-fPIC", "-o", out, src], check=True)
    lib = ctypes.CDLL(out)
    lib.timeout_probe.restype = ctypes.c_int
    lib.timeout_probe.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    return lib


@pytest.mark.parametrize("pipelined,threads", [(0, 32), (1, 64)])
def test_expired_wait_sets_timeout_status_and_returns(probe, pipelined, threads):
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda:0")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    t0 = time.perf_counter()
    assert probe.timeout_probe(ctypes.c_void_p(ws.data_ptr()), 1_000_000, 77, pipelined, stream) == 0
    assert sa.read_status(ws) == sa.E_DEVICE_TIMEOUT          # synchronises: the kernel has returned
    elapsed = time.perf_counter() - t0
    words = ws.view(torch.int32).cpu()
    assert int(words[1]) == 77                                 # the id of the first wait that gave up
    assert int(words[2]) == threads and int(words[3]) == 0          # every thread left its wait unsuccessfully
    assert elapsed < 1.0, f"a 1 ms wait limit took {elapsed:.3f} s"
    # the context is still usable and a later library call on the same workspace starts clean
    x = torch.ones(1024, device="cuda:0")
    assert float(x.sum()) == 1024.0


@pytest.mark.parametrize("overlap", [0, 1])
def test_failed_launch_is_reported_once(probe, overlap):
    """A launch that the runtime refuses on the host: the library's launch helper reports it and takes the runtime's
    last error with it, so that the check after a later, unrelated launch does not find it again."""
    assert probe.launch_probe(overlap) == 0


@pytest.mark.parametrize("early", [0, 1])
@pytest.mark.parametrize("words", [(0, 0), (0, 5), (0x5A5A5A5A, 1), (-1515870811, -1515870811), (-1, -1), (sa.E_BAD_INDEX, 3), (sa.E_DEVICE_TIMEOUT, 9), (-9, 0)])
def test_bad_index_is_reported_in_any_order(probe, early, words):
    """A kernel that clears the status itself: a report made milliseconds before the first CTA begins is kept, whatever the
    memory held (nothing, anything, an earlier call's code), and what an earlier call left is gone."""
    probe.header_probe.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    nb, kmax = 7, 40
    good = torch.arange(2 * kmax, dtype=torch.int32, device="cuda:0") % nb
    bad = good.clone()
    bad[2 * kmax - 3] = nb + 4
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for lists, status, detail in ((good, sa.OK, 0), (bad, sa.E_BAD_INDEX, nb + 4)):
        ws = torch.zeros(64, dtype=torch.int32)
        ws[0], ws[1] = words
        ws = ws.cuda()
        assert probe.header_probe(ctypes.c_void_p(ws.data_ptr()), ctypes.c_void_p(lists.data_ptr()), nb, kmax, early, stream) == 0
        assert ws[:2].tolist() == [status, detail]
