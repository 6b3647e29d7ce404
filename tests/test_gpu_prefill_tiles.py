"""sc_prefill_attn where a CTA walks a whole head (as many CTAs as fill the GPU, so that keys are not split): heads of one to nine key tiles,
so that either softmax group has the last tile and each place of the rings is the last one, against attention in 64 bits."""
import pytest
import torch

from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("slope", [6.0, -6.0, 0.0])   # scores (natural units) grow, fall or stay from tile to tile
def test_heads_of_one_to_nine_tiles(slope, causal):
    B, H, G, m, d, cap = 4, 9, 4, 150, 128, 1152   # 600 rows: five query tiles of 36 heads are 180 CTAs
    g = torch.Generator(device=DEV).manual_seed(int(slope) + causal)
    lens = torch.tensor([[128 * t - cut for t in range(1, 10)] for cut in (0, 1, 64, 127)], dtype=torch.int32, device=DEV).clamp(min=1)
    q = torch.randn((B, H * G, m, d), generator=g, device=DEV)
    q[..., 0] = 8.0
    q[:, :, ::3, 0] = 5.0
    k = torch.randn((B, H, cap, d), generator=g, device=DEV)
    k[..., 0] = slope * (torch.arange(cap, device=DEV) // 128) * d ** 0.5 / 8.0
    v = torch.randn((B, H, cap, d), generator=g, device=DEV)
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    count = torch.randint(1, 9, (B, H, cap), generator=g, device=DEV, dtype=torch.int32)
    layer = binding.CompressedLayer(k, v, count, lens)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = binding.prefill_attn(q, layer, status=status, causal=causal)
    binding.check_status(status)
    # a row i of m sees the keys before len - (m - 1 - i), or all of them
    see = lens.view(B, H, 1, 1, 1) - (torch.arange(m - 1, -1, -1, device=DEV).view(1, 1, 1, m, 1) if causal else 0)
    x = torch.einsum("bhgid,bhtd->bhgit", q.double().view(B, H, G, m, d), k.double()) / d ** 0.5 + torch.log(count.double()).view(B, H, 1, 1, cap)
    x = x.masked_fill(torch.arange(cap, device=DEV) >= see, -torch.inf)
    want = torch.einsum("bhgit,bhtd->bhgid", torch.softmax(x, -1).nan_to_num(0.0), v.double()).reshape(B, H * G, m, d)   # (no key: zeros)
    assert_close_vectors(to_f64(got), to_f64(want), TOL[torch.bfloat16], f"slope {slope}")
    for _ in range(5):
        assert torch.equal(binding.prefill_attn(q, layer, causal=causal), got)
