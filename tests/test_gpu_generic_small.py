"""The generic clustering and merge kernels over short inputs, whose launches are as large as the input can need: texts of delimiters only (more
segments than warps), of none and mixed ones, against the oracle; and the time of a very short one."""
import pytest
import torch

from helpers import compare_compressed, oracle_compress
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _inputs(B, H, n, d, dtype, ends):
    g = torch.Generator().manual_seed(n * 7 + d)
    ids = torch.full((B, n), 7, dtype=torch.int32)
    if ends == "all":
        ids[:] = 13
    elif ends == "some":
        ids[torch.rand((B, n), generator=g) < 0.4] = 13
    centre = torch.randn((3, d), generator=g)
    near = torch.randint(0, 3, (B, H, n), generator=g)
    K = (centre[near] + 0.1 * torch.randn((B, H, n, d), generator=g)).to(dtype)
    return ids, K, torch.randn((B, H, n, d), generator=g).to(dtype)


@pytest.mark.parametrize("dtype,d", [(torch.float32, 128), (torch.float32, 160), (torch.bfloat16, 64), (torch.bfloat16, 256)])
@pytest.mark.parametrize("ends", ["all", "none", "some"])
@pytest.mark.parametrize("B,H,n", [(1, 1, 1), (1, 1, 2), (1, 2, 3), (1, 1, 31), (2, 3, 50), (1, 8, 200)])
def test_short_inputs(B, H, n, ends, dtype, d):
    ids, K, V = _inputs(B, H, n, d, dtype, ends)
    plan = binding.chunk(ids.to(DEV), (13,))
    got = binding.compress(K.to(DEV), V.to(DEV), plan, 0.8, want_assign=True)
    binding.check_status(plan.status)
    compare_compressed(got, oracle_compress(ids, K, V, (13,), 0.8), dtype)


def _us(n):
    ids, K, V = _inputs(1, 8, n, 128, torch.float32, "some")
    K, V, plan, ws = K.to(DEV), V.to(DEV), binding.chunk(ids.to(DEV), (13,)), binding.compress_workspace(1, 8, n, DEV)
    out = binding.compress(K, V, plan, 0.8, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(10):
            binding.compress(K, V, plan, 0.8, workspace=ws, out=out)
    best = float("inf")
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        graph.replay()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 100)
    return best


def test_a_short_input_is_a_small_launch():
    # 0.4 of the time of 2048 tokens; 0.8 with launches of 64 blocks per SM
    assert _us(64) < 0.6 * _us(2048)
