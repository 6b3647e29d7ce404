"""The fused compress kernel where its tiles and its pooling product can go wrong: values that are not finite (a product
with a 0/1 matrix must not carry them into other clusters), beside clusters that share sixteen rows or columns with
them, in tiles of up to 128 tokens and in longer ones."""
import numpy as np
import pytest
import torch

from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("gap,n", [(20, 128), (31, 500), (64, 777), (130, 524), (200, 603)])
@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
def test_values_that_are_not_finite_stay_in_their_cluster(gap, n, bad):
    w = synth.config(0).replace(n=n, Hkv=2, Hq=8, gap=("fixed", gap), seed=gap)
    ids, run_id, run_lens = synth.token_ids(w)
    K, V = synth.layer_kv(w, 0, run_id, run_lens)
    rng = np.random.default_rng(n)
    for t in rng.choice(n, size=4, replace=False):
        V[0, :, int(t), int(rng.integers(128))] = bad
    plan = binding.chunk(ids.to(DEV), w.delims)
    got = binding.compress(K.to(DEV), V.to(DEV), plan, w.tau, want_assign=True)
    ref = binding.compress(K.to(DEV), V.to(DEV), plan, w.tau, want_assign=True, flags=binding.SC_FLAG_GENERIC)
    binding.check_status(plan.status)
    assert torch.equal(got.core_len, ref.core_len) and torch.equal(got.assign, ref.assign)
    for h in range(w.Hkv):
        m = int(ref.core_len[0, h])
        assert torch.equal(got.count[0, h, :m], ref.count[0, h, :m])
        for a, b in ((got.core_k, ref.core_k), (got.core_v, ref.core_v)):
            a, b = to_f64(a[0, h, :m]), to_f64(b[0, h, :m])
            odd = ~np.isfinite(b)
            assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[np.isinf(b)], b[np.isinf(b)])
            # both sides add bf16 values in float32 and round once to bf16: the repository's bf16 tolerance
            assert_close_vectors(np.where(odd, 0, a), np.where(odd, 0, b), TOL[torch.bfloat16], f"head {h}")
