"""sc_prefill_attn at the query counts and batch sizes where the width of the key split changes (clusters of 10, 9, 7, 5, 3
and 2 CTAs, odd widths among them, none at last), against the oracle's Eq. 4 with a block of queries."""
import pytest
import torch

import oracle
from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,Hkv,G,m", [(1, 8, 4, 3), (1, 8, 4, 33), (2, 8, 4, 5), (3, 8, 4, 8), (5, 8, 4, 2), (9, 8, 4, 1), (1, 4, 7, 19),
                                       (1, 3, 4, 40), (1, 1, 4, 7)])
@pytest.mark.parametrize("causal", [False, True])
def test_prefill_split_widths(B, Hkv, G, m, causal):
    cap, d = 6000, 128
    g = torch.Generator().manual_seed(B * 100 + m)
    lens = torch.randint(m, cap + 1, (B, Hkv), generator=g, dtype=torch.int32)
    lens[0, 0] = cap
    k = torch.randn((B, Hkv, cap, d), generator=g)
    k = (k / k.norm(dim=3, keepdim=True)).bfloat16()
    v = torch.randn((B, Hkv, cap, d), generator=g).bfloat16()
    count = torch.randint(1, 9, (B, Hkv, cap), generator=g, dtype=torch.int32)
    q = torch.randn((B, Hkv * G, m, d), generator=g).bfloat16()
    layer = binding.CompressedLayer(k.to(DEV), v.to(DEV), count.to(DEV), lens.to(DEV))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = binding.prefill_attn(q.to(DEV), layer, status=status, causal=causal)
    binding.check_status(status)
    ref = oracle.attn_multi(synth.to_numpy_bits(q), synth.to_numpy_bits(k), synth.to_numpy_bits(v), count.numpy(), lens.numpy(), causal=causal)
    assert_close_vectors(to_f64(got), ref, TOL[torch.bfloat16], f"{B} x {Hkv} x {G} x {m}")


@pytest.mark.parametrize("B,Hkv,G,m,cap", [(1, 8, 4, 8, 6000), (1, 8, 4, 9, 6000), (1, 4, 7, 9, 3000), (2, 4, 4, 16, 700), (1, 2, 1, 1, 40), (2, 3, 7, 4, 700), (20, 8, 4, 2, 300), (1, 4, 8, 4, 129)])
@pytest.mark.parametrize("causal", [False, True])
def test_prefill_few_rows(B, Hkv, G, m, cap, causal):
    """Up to 32 and up to 64 query rows per KV head: heads of every length around a key tile, its halves and its quarters."""
    d = 128
    g = torch.Generator().manual_seed(B * 100 + m)
    lens = torch.randint(m, cap + 1, (B, Hkv), generator=g, dtype=torch.int32)
    some = [n for n in (cap, m, 31, 32, 33, 65, 97, 128, 129) if m <= n <= cap][:B * Hkv]
    lens.view(-1)[:len(some)] = torch.tensor(some, dtype=torch.int32)
    k = torch.randn((B, Hkv, cap, d), generator=g)
    k = (k / k.norm(dim=3, keepdim=True)).bfloat16()
    v = torch.randn((B, Hkv, cap, d), generator=g).bfloat16()
    for b in range(B):
        for h in range(Hkv):
            k[b, h, int(lens[b, h]):] = float("nan")
            v[b, h, int(lens[b, h]):] = float("nan")
    count = torch.randint(1, 9, (B, Hkv, cap), generator=g, dtype=torch.int32)
    q = (3 * torch.randn((B, Hkv * G, m, d), generator=g)).bfloat16()
    layer = binding.CompressedLayer(k.to(DEV), v.to(DEV), count.to(DEV), lens.to(DEV))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = binding.prefill_attn(q.to(DEV), layer, status=status, causal=causal)
    binding.check_status(status)
    ref = oracle.attn_multi(synth.to_numpy_bits(q), synth.to_numpy_bits(k), synth.to_numpy_bits(v), count.numpy(), lens.numpy(), causal=causal)
    assert_close_vectors(to_f64(got), ref, TOL[torch.bfloat16], f"{B} x {Hkv} x {G} x {m}, capacity {cap}")
