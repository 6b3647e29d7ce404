"""Calls in one stream without a synchronisation between them, each of which needs what the one before wrote: kernels are set up
beside their predecessors, some with tensor memory of their own, and have to give what they give one at a time."""
import pytest
import torch

from paper_2603_14303_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,n,m", [(1, 200, 4), (2, 3000, 40), (5, 700, 9)])
def test_compress_and_attention_by_turns(B, n, m):
    w = synth.Workload("order", B=B, n=n, L=1, Hkv=4, Hq=16, d=128, gap=("poisson", 20.0), centroids=("uniform", 4), seed=n)
    ids, run_id, run_lens = synth.token_ids(w)
    K0, V0 = (t.to(DEV) for t in synth.layer_kv(w, 0, run_id, run_lens))
    ids = ids.to(DEV)
    q = torch.randn((B, 16, m, 128), generator=torch.Generator(device=DEV).manual_seed(1), device=DEV).bfloat16()
    ws, dws = binding.compress_workspace(B, 4, n, DEV), binding.decode_workspace(B, 16, 4, 128, n, DEV)

    def steps(sync):
        done = torch.cuda.synchronize if sync else lambda: None
        K, V, x, seen = K0.clone(), V0.clone(), q, []
        out = None
        for i in range(12):
            plan = binding.chunk(ids, w.delims)
            done()
            out = binding.compress(K, V, plan, w.tau, workspace=ws, flags=binding.SC_FLAG_TWO_PASS if i % 3 == 2 else 0)
            done()
            x = binding.prefill_attn(x, out)
            done()
            o = binding.decode_attn(x[:, :, 0].contiguous(), out, workspace=dws)
            done()
            V = V + o[:, ::4].unsqueeze(2)      # the next compression pools what this step gave
            done()
            seen.append((x, o, out.core_len))
        torch.cuda.synchronize()
        binding.check_status(plan.status)
        return seen

    for got, want in zip(steps(False), steps(True)):
        assert all(torch.equal(a, b) for a, b in zip(got, want))
