"""Keys that are infinite or not a number are similar to nothing and merge with nothing; keys without length neither."""
import numpy as np
import pytest
import torch

from helpers import oracle_compress
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("tau", [0.0, 0.6])
@pytest.mark.parametrize("run", [8, 128, 129, 256])   # tiles of several segments, of one, of one longer than 128 tokens
@pytest.mark.parametrize("bad", [float("nan"), -float("nan"), float("inf"), -float("inf"), 0.0, -0.0])
def test_partition_matches_oracle(bad, run, tau):
    n, d = 3 * run, 128
    ids = torch.full((1, n), 7, dtype=torch.int32)
    ids[0, run - 1::run] = 13
    g = torch.Generator().manual_seed(run)
    # Rows of +-1 around two centres: products are whole numbers, exact in fp32, and far from either threshold.
    centre = torch.randint(0, 2, (2, d), generator=g) * 2.0 - 1.0
    K = centre[torch.randint(0, 2, (2 * n,), generator=g)].view(1, 2, n, d).clone()
    K[0, :, 1::5, 3] = bad
    if bad == 0.0:
        K[0, :, 1::5, :] = bad
    K, V = K.bfloat16(), torch.randn((1, 2, n, d), generator=g).bfloat16()
    plan = binding.chunk(ids.to(DEV), (13,))
    got = binding.compress(K.to(DEV), V.to(DEV), plan, tau, want_assign=True)
    binding.check_status(plan.status)
    ref = oracle_compress(ids, K, V, (13,), tau)
    assert np.array_equal(got.assign.cpu().numpy(), ref["assign"])
    assert np.array_equal(got.core_len.cpu().numpy(), ref["core_len"])
    for h in range(2):
        L = int(ref["core_len"][0, h])
        assert np.array_equal(got.count[0, h, :L].cpu().numpy(), ref["count"][0, h, :L])
