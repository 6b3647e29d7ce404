"""sc_prefill_attn on either side of the choice between one and two groups of softmax warps (few key tiles and many, split over a cluster and
not, rows that stand in the tile once, twice and four times), heads from empty to full, against attention in 64 bits."""
import pytest
import torch

from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("m", [1, 8, 9, 16, 17, 70])
@pytest.mark.parametrize("cap,causal", [(100, False), (128, False), (204, False), (205, False), (206, True), (300, True), (512, False), (900, True), (1500, False)])
def test_one_group_and_two(cap, causal, m):
    B, H, G, d = 2, 3, 4, 128
    if cap < m:
        pytest.skip("a causal block is part of the cache")
    g = torch.Generator(device=DEV).manual_seed(cap + m)
    lens = torch.tensor([[cap, cap // 2, 1], [0, min(cap, 129), 5 * cap // 8]], dtype=torch.int32, device=DEV)
    q, k, v = (torch.randn(s, generator=g, device=DEV).bfloat16() for s in ((B, H * G, m, d), (B, H, cap, d), (B, H, cap, d)))
    count = torch.randint(1, 9, (B, H, cap), generator=g, device=DEV, dtype=torch.int32)
    layer = binding.CompressedLayer(k, v, count, lens)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = binding.prefill_attn(q, layer, status=status, causal=causal)
    binding.check_status(status)
    see = lens.view(B, H, 1, 1, 1) - (torch.arange(m - 1, -1, -1, device=DEV).view(1, 1, 1, m, 1) if causal else 0)
    x = torch.einsum("bhgid,bhtd->bhgit", q.double().view(B, H, G, m, d), k.double()) / d ** 0.5 + torch.log(count.double()).view(B, H, 1, 1, cap)
    x = x.masked_fill(torch.arange(cap, device=DEV) >= see, -torch.inf)
    want = torch.einsum("bhgit,bhtd->bhgid", torch.softmax(x, -1).nan_to_num(0.0), v.double()).reshape(B, H * G, m, d)   # (no key: zeros)
    assert_close_vectors(to_f64(got), to_f64(want), TOL[torch.bfloat16], f"capacity {cap}, m = {m}")
    assert torch.equal(binding.prefill_attn(q, layer, causal=causal), got)
