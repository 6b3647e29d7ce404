"""float32 clustering and merge of segments longer than 32 tokens (taken 32 rows at a time, 16 where a row has more than 128 columns) and
cluster order in short ones, against the oracle."""
import pytest
import torch

import oracle
from helpers import TOL, assert_close_vectors, compare_compressed, oracle_compress, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [128, 160])
@pytest.mark.parametrize("length,centroids", [(31, 9), (47, 5), (48, 6), (63, 8), (64, 40), (65, 3), (96, 12), (97, 97), (255, 17)])
def test_generic_long_segments(length, centroids, d):
    w = synth.config(0, n=900, Hkv=2, Hq=4, d=d, dtype="f32", gap=("fixed", length), centroids=("uniform", centroids), seed=length)
    ids, run_id, run_lens = synth.token_ids(w)
    K, V = synth.layer_kv(w, 0, run_id, run_lens)
    tau = 0.8
    ref = oracle_compress(ids, K, V, w.delims, tau, w.max_chunk_len)
    assert ref["margin"] > 1e-5   # every comparison is clear of the threshold by more than float32 can move it
    plan = binding.chunk(ids.to(DEV), w.delims, w.max_chunk_len)
    got = binding.compress(K.to(DEV), V.to(DEV), plan, tau, want_assign=True)
    binding.check_status(plan.status)
    compare_compressed(got, ref, torch.float32)
    q = torch.randn((1, 4, d), generator=torch.Generator().manual_seed(length))
    want = oracle.attn(q.numpy(), ref["core_k"], ref["core_v"], ref["count"], ref["core_len"])
    assert_close_vectors(to_f64(binding.decode_attn(q.to(DEV), got)), want, TOL[torch.float32], f"{length} tokens, d {d}")
