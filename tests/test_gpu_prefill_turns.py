"""sc_prefill_attn where the row's softmax reference moves from key tile to key tile (the two softmax groups settle it in turn and
rescale one accumulator): scores that grow, fall or jump along the cache, heads of one to eight tiles, against the oracle."""
import pytest
import torch

import oracle
from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("m", [3, 13, 40])   # the rows stand in a tile four times, twice, once
@pytest.mark.parametrize("slope", [6.0, -6.0, 0.0])
def test_prefill_reference_moves_from_tile_to_tile(m, slope):
    B, H, G, d, cap = 2, 4, 4, 128, 1024
    g = torch.Generator().manual_seed(m)
    lens = torch.tensor([[128, 129, 256, 300], [385, 640, 1000, 1024]], dtype=torch.int32)
    # Scores (natural units) slope * tile + N(0, 1), every third row 3 lower: a step of 6 is 8.7 in base 2, just above what the
    # reference lets pass, so it moves in every tile or, falling, only once.  All entries are bf16 before either side reads them.
    t = torch.arange(cap) // 128
    q = torch.randn((B, H * G, m, d), generator=g)
    q[..., 0] = 8.0
    q[:, :, ::3, 0] = 5.0
    k = torch.randn((B, H, cap, d), generator=g)
    k[..., 0] = slope * t * d ** 0.5 / 8.0
    v = torch.randn((B, H, cap, d), generator=g).bfloat16()
    q, k = q.bfloat16(), k.bfloat16()
    count = torch.randint(1, 9, (B, H, cap), generator=g, dtype=torch.int32)
    layer = binding.CompressedLayer(k.to(DEV), v.to(DEV), count.to(DEV), lens.to(DEV))
    for causal in (False, True):
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        got = binding.prefill_attn(q.to(DEV), layer, status=status, causal=causal)
        binding.check_status(status)
        ref = oracle.attn_multi(synth.to_numpy_bits(q), synth.to_numpy_bits(k), synth.to_numpy_bits(v), count.numpy(), lens.numpy(), causal=causal)
        assert_close_vectors(to_f64(got), ref, TOL[torch.bfloat16], f"m = {m}, slope {slope}, causal {causal}")
