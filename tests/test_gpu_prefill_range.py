"""sc_prefill_attn with raw products of tens of thousands and scale 1, of both signs, against the oracle's Eq. 4: the softmax
reference of a row has to be its own largest score, not one that is larger by a share of it (2^-7 of 32 K would put every
weight below the smallest float)."""
import pytest
import torch

import oracle
from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("m,cap", [(3, 300), (13, 129), (40, 900), (8, 3000)])   # the rows stand in a tile four times, twice, once; a key split
@pytest.mark.parametrize("base", [32512, -32512, 16384])
def test_prefill_large_scores(m, cap, base):
    # All entries are integers that bf16 holds exactly: q.k = base + delta, |delta| <= 8, without rounding in fp32.  A score in
    # base-2 units is below 2^16, where fp32 has steps of 2^-8: weights are off by at most 2 ln 2 * 2^-9 = 0.27 %, inside the tolerance.
    B, H, G, d = 1, 2, 4, 128
    g = torch.Generator().manual_seed(m)
    k = torch.zeros((B, H, cap, d))
    k[..., 1:127] = 16.0
    k[..., 0] = torch.randint(-8, 9, (B, H, cap), generator=g).float()
    q = torch.zeros((B, H * G, m, d))
    q[..., 0] = 1.0
    rest = base // 16
    q[..., 1:127] = float(int(rest / 126))
    q[..., 127] = 1.0
    k[..., 127] = base - 16.0 * 126 * int(rest / 126)
    assert float((k.bfloat16().float() - k).abs().max()) == 0.0
    v = torch.randn((B, H, cap, d), generator=g).bfloat16()
    q, k = q.bfloat16(), k.bfloat16()
    prod = torch.einsum("bgmd,btd->bgmt", q[:, :1].double(), k[:, 0].double())
    assert float(prod.min()) >= base - 8 and float(prod.max()) <= base + 8
    count = torch.randint(1, 9, (B, H, cap), generator=g, dtype=torch.int32)
    lens = torch.tensor([[cap, cap - 37]], dtype=torch.int32)
    layer = binding.CompressedLayer(k.to(DEV), v.to(DEV), count.to(DEV), lens.to(DEV))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = binding.prefill_attn(q.to(DEV), layer, scale=1.0, status=status)
    binding.check_status(status)
    ref = oracle.attn_multi(synth.to_numpy_bits(q), synth.to_numpy_bits(k), synth.to_numpy_bits(v), count.numpy(), lens.numpy(), scale=1.0)
    assert_close_vectors(to_f64(got), ref, TOL[torch.bfloat16], f"m = {m}, products around {base}")
