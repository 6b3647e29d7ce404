"""sc_decode_attn at the head counts and capacities where the split plan changes -- clusters of 16 down to 2, several per
head, none, short capacities, raw caches -- with heads from empty to full, against the oracle's Eq. 4; twice on one
workspace."""
import pytest
import torch

import oracle
from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,Hkv,G,cap,raw", [
    (1, 1, 4, 50000, False), (1, 4, 7, 24001, False), (1, 8, 4, 8200, False), (1, 8, 4, 63, False), (1, 8, 4, 1024, False), (1, 8, 2, 4096, False),
    (2, 7, 4, 8193, False), (2, 8, 4, 8193, False), (3, 6, 1, 3000, False), (5, 4, 4, 5000, False), (7, 4, 7, 2000, False), (7, 8, 4, 2100, False),
    (19, 4, 4, 1200, False), (16, 8, 4, 1100, False), (19, 8, 3, 900, False), (1, 2, 4, 9000, True), (2, 8, 4, 8192, True), (9, 8, 1, 8200, True),
    (1, 8, 4, 700, True)])
def test_decode_split_plans(B, Hkv, G, cap, raw):
    d = 128
    g = torch.Generator().manual_seed(B * 1000 + Hkv * 10 + G)
    lens = torch.randint(0, cap + 1, (B, Hkv), generator=g, dtype=torch.int32)
    lens.view(-1)[0] = cap
    if B * Hkv > 2:
        lens.view(-1)[1], lens.view(-1)[2] = 0, 1
    k = torch.randn((B, Hkv, cap, d), generator=g)
    k = (k / k.norm(dim=3, keepdim=True)).bfloat16()
    v = torch.randn((B, Hkv, cap, d), generator=g).bfloat16()
    count = torch.randint(1, 9, (B, Hkv, cap), generator=g, dtype=torch.int32)
    layer = binding.CompressedLayer(k.to(DEV), v.to(DEV), count.to(DEV), lens.to(DEV))
    ws = binding.decode_workspace(B, Hkv * G, Hkv, d, cap, DEV)
    for step in range(2):
        q = torch.randn((B, Hkv * G, d), generator=g).bfloat16()
        got = binding.decode_attn(q.to(DEV), layer, workspace=ws, use_count=not raw)
        ref = oracle.attn(synth.to_numpy_bits(q), synth.to_numpy_bits(k), synth.to_numpy_bits(v), None if raw else count.numpy(), lens.numpy())
        assert_close_vectors(to_f64(got), ref, TOL[torch.bfloat16], f"{B} x {Hkv} x {G}, capacity {cap}, step {step}")
