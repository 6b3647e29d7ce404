"""The generic (float32, other head sizes) kernels where they change their way: segments around 8, 16 and 32 tokens, more than
sixteen clusters in a segment, head sizes that leave lanes idle; then one decode step over the cores.  Against the oracle."""
import pytest
import torch

import oracle
from helpers import TOL, assert_close_vectors, compare_compressed, oracle_compress, to_f64
from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [128, 40])
@pytest.mark.parametrize("length,centroids", [(1, 1), (2, 2), (7, 3), (8, 8), (9, 4), (16, 5), (17, 6), (25, 24), (32, 16), (32, 32), (33, 8)])
def test_generic_segments_and_decode(length, centroids, d):
    w = synth.config(0, n=611, Hkv=3, Hq=9, d=d, dtype="f32", gap=("fixed", length), centroids=("uniform", centroids), seed=length)
    ids, run_id, run_lens = synth.token_ids(w)
    K, V = synth.layer_kv(w, 0, run_id, run_lens)
    tau = 0.8
    ref = oracle_compress(ids, K, V, w.delims, tau, w.max_chunk_len)
    assert ref["margin"] > 1e-5   # every comparison is clear of the threshold by more than float32 can move it
    plan = binding.chunk(ids.to(DEV), w.delims, w.max_chunk_len)
    got = binding.compress(K.to(DEV), V.to(DEV), plan, tau, want_assign=True)
    binding.check_status(plan.status)
    compare_compressed(got, ref, torch.float32)
    q = torch.randn((1, 9, d), generator=torch.Generator().manual_seed(length))
    out = binding.decode_attn(q.to(DEV), got)
    want = oracle.attn(q.numpy(), ref["core_k"], ref["core_v"], ref["count"], ref["core_len"])
    assert_close_vectors(to_f64(out), want, TOL[torch.float32], f"{length} tokens, d {d}")
