"""A threshold of zero, of either sign: Sim > 0 is false for orthogonal keys and for keys without length, so none of them merge."""
import numpy as np
import pytest
import torch

from helpers import compare_compressed, oracle_compress
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("tau", [0.0, -0.0])
@pytest.mark.parametrize("run", [20, 200])   # a tile of several segments, a tile of one
@pytest.mark.parametrize("flags", [0, binding.SC_FLAG_TWO_PASS, binding.SC_FLAG_GENERIC])
def test_orthogonal_and_zero_keys_stay_apart(tau, run, flags):
    n, d = 3 * run, 128
    ids = torch.full((1, n), 7, dtype=torch.int32)
    ids[0, run - 1::run] = 13
    K = torch.zeros((1, 2, n, d))
    K[0, 0, torch.arange(n), torch.arange(n) % 100] = 1.0      # equal or exactly orthogonal
    K[0, 1, ::3, 5] = 2.0                                      # two of three keys have no length
    K, V = K.bfloat16(), torch.randn((1, 2, n, d), generator=torch.Generator().manual_seed(run)).bfloat16()
    plan = binding.chunk(ids.to(DEV), (13,))
    got = binding.compress(K.to(DEV), V.to(DEV), plan, tau, want_assign=True, flags=flags)
    binding.check_status(plan.status)
    compare_compressed(got, oracle_compress(ids, K, V, (13,), 0.0), torch.bfloat16)


@pytest.mark.parametrize("tau", [0.0, -0.0])
def test_layers_at_once(tau):
    n, d = 40, 128
    ids = torch.full((1, n), 7, dtype=torch.int32, device=DEV)
    K = torch.zeros((1, 1, n, d), dtype=torch.bfloat16, device=DEV)
    K[0, 0, torch.arange(n), torch.arange(n)] = 1.0
    plan = binding.chunk(ids, (13,))
    outs = [binding.CompressedLayer(torch.zeros_like(K), torch.zeros_like(K), torch.zeros((1, 1, n), dtype=torch.int32, device=DEV),
                                    torch.zeros((1, 1), dtype=torch.int32, device=DEV)) for _ in range(2)]
    binding.sc_compress_layers([K, K], [K, K], plan, tau, outs, binding.compress_layers_workspace(2, 1, 1, n, DEV), plan.status)
    binding.check_status(plan.status)
    for o in outs:
        assert int(o.core_len) == n and np.array_equal(o.count.cpu().numpy().ravel(), np.ones(n, dtype=np.int32))
