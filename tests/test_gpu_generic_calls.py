"""The generic calls: a decode workspace that starts on any float and is shared with the tensor-core kernel, and a launch that
the runtime refuses, which is an error of its own call only."""
import ctypes

import pytest
import torch

from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(cap=1500, H=2, d=40):
    g = torch.Generator().manual_seed(cap)
    k, v = torch.randn((1, H, cap, d), generator=g), torch.randn((1, H, cap, d), generator=g)
    y = binding.CompressedLayer(k.to(DEV), v.to(DEV), torch.ones((1, H, cap), dtype=torch.int32, device=DEV),
                                torch.full((1, H), cap, dtype=torch.int32, device=DEV))
    q = torch.randn((1, 2 * H, d), generator=g)
    x = torch.einsum("hgd,htd->hgt", q.view(H, 2, d).double(), k[0].double()) / d ** 0.5
    return q.to(DEV), y, torch.einsum("hgt,htd->hgd", torch.softmax(x, -1), v[0].double()).reshape(1, 2 * H, d).numpy()


@pytest.mark.parametrize("shift", [0, 4, 8, 12])
def test_decode_workspace_on_any_float(shift):
    q, y, ref = _layer()
    need = binding.lib().sc_decode_workspace_bytes(1, 4, 2, 40, 1500)
    whole = torch.zeros(need + 64, dtype=torch.uint8, device=DEV)
    whole[shift + need:] = 77
    got = binding.decode_attn(q, y, workspace=whole[shift:shift + need])
    assert_close_vectors(to_f64(got), ref, TOL[torch.float32], f"workspace shifted by {shift}")
    assert bool((whole[shift + need:] == 77).all()) and bool((whole[:shift] == 0).all())


def test_a_refused_launch_is_not_an_error_of_the_next_call():
    q, y, ref = _layer()
    none = ctypes.c_void_p(q.data_ptr())
    # 2^33 queries are 2^31 blocks of four, one more than a grid can have: the runtime refuses the launch, nothing runs
    code = binding.lib().sc_prefill_attn(none, binding.SC_F32, 1 << 20, 1 << 13, 1 << 13, 1, 40, none, none, None, 8, none, 0.0, 0, none, None, None)
    assert code == binding.SC_ERR_CUDA
    assert_close_vectors(to_f64(binding.decode_attn(q, y)), ref, TOL[torch.float32], "decode")


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_one_workspace_for_both_kinds_of_kernel(dtype):
    # the batch's long heads meet through counters in front of the workspace, which the generic kernels have to leave alone
    B, H, cap, d = 4, 2, 9000, 128
    g = torch.Generator(device=DEV).manual_seed(3)
    rand = lambda *shape: torch.randn(shape, generator=g, device=DEV)
    k, v = rand(B, H, cap, d), rand(B, H, cap, d)
    count = torch.randint(1, 9, (B, H, cap), generator=g, device=DEV, dtype=torch.int32)
    lens = torch.tensor([[9000], [300], [20], [0]], dtype=torch.int32, device=DEV).expand(B, H).contiguous()
    y = binding.CompressedLayer(k.bfloat16(), v.bfloat16(), count, lens)
    z = binding.CompressedLayer(k.to(dtype), v.to(dtype), count, lens)
    q = rand(B, 4 * H, d)
    ws = binding.decode_workspace(B, 4 * H, H, d, cap, DEV)
    want = binding.decode_attn(q.bfloat16(), y)
    for _ in range(2):
        binding.decode_attn(q.to(dtype), z, workspace=ws, flags=binding.SC_FLAG_GENERIC)
        assert torch.equal(binding.decode_attn(q.bfloat16(), y, workspace=ws), want)
