"""The generic decode kernels with fewer and with more blocks than the GPU has SMs (blocks of eight and of four warps), against attention in
64 bits; and a batch's time, which follows the number of rows."""
import pytest
import torch

from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(B, H, cap, d, dtype, lens):
    g = torch.Generator(device=DEV).manual_seed(B + cap + d)
    k = torch.randn((B, H, cap, d), generator=g, device=DEV)
    v = torch.randn((B, H, cap, d), generator=g, device=DEV)
    count = torch.randint(1, 9, (B, H, cap), generator=g, device=DEV, dtype=torch.int32)
    ln = torch.tensor([lens[i % len(lens)] for i in range(B * H)], dtype=torch.int32, device=DEV).view(B, H)
    return binding.CompressedLayer(k.to(dtype), v.to(dtype), count, ln)


@pytest.mark.parametrize("dtype,d", [(torch.float32, 128), (torch.float32, 40), (torch.float32, 256), (torch.bfloat16, 64), (torch.bfloat16, 200)])
@pytest.mark.parametrize("B,H,cap", [(1, 2, 31), (1, 4, 1500), (4, 4, 4608), (37, 4, 512), (37, 4, 513), (149, 1, 300)])   # 2, 12, 144, 148, 296, 149 splits
def test_blocks_on_either_side_of_the_sms(B, H, cap, dtype, d):
    G = 3
    y = _layer(B, H, cap, d, dtype, [cap, cap - 1, cap // 2 + 1, 1, 0, 33 % cap])
    q = torch.randn((B, H * G, d), generator=torch.Generator(device=DEV).manual_seed(d), device=DEV).to(dtype)
    got = binding.decode_attn(q, y)
    x = torch.einsum("bhgd,bhtd->bhgt", q.double().view(B, H, G, d), y.core_k.double()) / d ** 0.5 + torch.log(y.count.double()).unsqueeze(2)
    x = x.masked_fill(torch.arange(cap, device=DEV) >= y.core_len.view(B, H, 1, 1), -torch.inf)
    want = torch.einsum("bhgt,bhtd->bhgd", torch.softmax(x, -1).nan_to_num(0.0), y.core_v.double()).reshape(B, H * G, d)   # (no row: zeros)
    assert_close_vectors(to_f64(got), to_f64(want), TOL[dtype], f"{B} x {H} x {cap}, d {d}")
    assert torch.equal(binding.decode_attn(q, y), got)


def _us(B, dtype, d):
    H, G, cap = 8, 4, 8192
    y = _layer(B, H, cap, d, dtype, [4096])
    q = torch.randn((B, H * G, d), device=DEV).to(dtype)
    out, ws = torch.empty_like(q), binding.decode_workspace(B, H * G, H, d, cap, DEV)
    best = float("inf")
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(20):
            binding.decode_attn(q, y, out=out, workspace=ws)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 50)
    return best


@pytest.mark.parametrize("dtype,d,most", [(torch.float32, 128, 10.5), (torch.bfloat16, 64, 10.5)])
def test_a_batch_uses_the_whole_of_every_sm(dtype, d, most):
    # sixteen sequences of 2048 blocks against one of 128, one per SM: 8.4 and 6.6 times the time with three to five blocks to an
    # SM; 13.1 and 16.6 when an SM held one
    assert _us(16, dtype, d) < most * _us(1, dtype, d)
