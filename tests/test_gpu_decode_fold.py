"""The fold of the decode kernel's clusters where a block hands its share in late or not at all: a result that is not complete is not a
number and reported, and the block that gave up leaves after the others."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2603_14303_b200 import binding, build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HERE = os.path.dirname(os.path.abspath(__file__))
MS = 1_000_000


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("fold") / "probe.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, *build.NVCC_FLAGS, "-Xcompiler", "-fvisibility=default", "-shared", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    os.path.join(HERE, "decode_fold_probe.cu"), "-o", lib], check=True)
    run = ctypes.CDLL(lib).run_probe
    run.argtypes = [ctypes.c_longlong, ctypes.c_ulonglong] + [ctypes.c_void_p] * 4

    def call(delay_ms, limit_ms):
        out, status = torch.full((17,), -1.0, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        left = torch.zeros(2, dtype=torch.int64, device=DEV)
        assert run(int(delay_ms * MS), int(limit_ms * MS), out.data_ptr(), status.data_ptr(), left.data_ptr(),
                   torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        return out.cpu(), int(status), left.cpu().tolist()
    return call


@pytest.mark.parametrize("delay_ms,limit_ms", [(0, 500), (75, 50)])   # in time; later than the limit, within the second one
def test_slices_that_arrive(probe, delay_ms, limit_ms):
    out, status, _ = probe(delay_ms, limit_ms)
    assert status == binding.SC_OK and bool((out[:16] == 2.0).all()) and float(out[16]) == 0.0


@pytest.mark.parametrize("delay_ms", [-1, 250])   # never; later than both limits
def test_slices_that_do_not(probe, delay_ms):
    out, status, (left, other_left) = probe(delay_ms, 50)
    assert status == binding.SC_ERR_TIMEOUT
    assert bool(out[:16].isnan().all()) and float(out[16]) == 0.0   # a merge with other partials takes it in
    if delay_ms > 0:
        assert left >= other_left - 5 * MS   # (each block's clock is read a little before it has left)
