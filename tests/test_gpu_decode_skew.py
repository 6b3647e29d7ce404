"""sc_decode_attn over batches of very different lengths: heads that take part of the work from spare blocks beside heads that
have none to give, against plain attention in 64 bits; one workspace for batches of different sizes in turn; and the time, which
follows the number of rows and not the longest sequence."""
import pytest
import torch

from helpers import TOL, assert_close_vectors, to_f64
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(lens, cap, H, seed, equal_heads=True):
    B, d = len(lens), 128
    g = torch.Generator(device=DEV).manual_seed(seed)
    ln = torch.tensor(lens, dtype=torch.int32, device=DEV).view(B, 1).expand(B, H).contiguous()
    if not equal_heads:
        ln = (ln * (0.5 + 0.5 * torch.rand((B, H), generator=g, device=DEV))).int()
    k = torch.randn((B, H, cap, d), generator=g, device=DEV)
    k = (k / k.norm(dim=3, keepdim=True)).bfloat16()
    v = torch.randn((B, H, cap, d), generator=g, device=DEV).bfloat16()
    count = torch.randint(1, 9, (B, H, cap), generator=g, device=DEV, dtype=torch.int32)
    return binding.CompressedLayer(k, v, count, ln)


def _reference(q, y, raw):
    B, Hq, d = q.shape
    H = y.core_k.shape[1]
    out = torch.zeros((B, Hq, d), dtype=torch.float64, device=DEV)
    for b in range(B):
        for h in range(H):
            n = int(y.core_len[b, h])
            rows = slice(h * (Hq // H), (h + 1) * (Hq // H))
            if n == 0:
                continue
            x = q[b, rows].double() @ y.core_k[b, h, :n].double().T / d ** 0.5
            if not raw:
                x = x + torch.log(y.count[b, h, :n].double())
            out[b, rows] = torch.softmax(x, -1) @ y.core_v[b, h, :n].double()
    return out.cpu().numpy()


@pytest.mark.parametrize("lens,cap,H,G,raw,equal", [
    ([16000] + [500] * 15, 16384, 8, 4, False, True),       # one long sequence: twelve units each for its heads
    ([500] * 15 + [16000], 16384, 8, 4, False, True),       # the same, last
    ([0] * 7 + [9000], 9000, 4, 7, False, True),            # all rows in one sequence
    ([0, 0, 0, 0], 40000, 8, 4, False, True),               # none at all
    ([4095, 12300, 1, 8191, 0, 16, 17, 7000], 12300, 8, 4, False, False),
    ([30000, 2000], 32768, 4, 4, False, True),              # wide clusters
    ([20000, 900, 900], 20000, 11, 2, False, False),        # 33 heads: the pool's units start in the middle of 32
    ([3000] * 40 + [9000] * 3, 9000, 8, 1, False, False),   # more heads than clusters of two: one block each
    ([9000, 9000, 9000, 9001], 9001, 8, 4, True, True),     # raw caches: equal, and not
    ([30000, 1000, 1000, 1000], 30000, 8, 4, True, True),
    ([12000] + [800] * 9, 12000, 8, 4, True, False),        # 80 raw heads
    ([12000] + [300] * 40, 12000, 4, 4, True, True),        # 164 raw heads
    # more blocks of clusters than counters, several clusters per long head: a head's blocks share one
    ([9000, 4000] + [300] * 38, 9000, 8, 4, False, True),   # 320 heads, clusters of three
    ([200] * 20 + [9000] + [0] * 17, 9000, 8, 7, False, False),   # 304
    ([8200] + [100] * 20 + [5000], 8200, 8, 1, True, True),       # 176 raw heads, clusters of three
    ([100] * 39 + [8200], 8200, 8, 4, True, False)])              # 320, of two
def test_lengths_far_apart(lens, cap, H, G, raw, equal):
    y = _layer(lens, cap, H, len(lens), equal)
    ws = binding.decode_workspace(len(lens), H * G, H, 128, cap, DEV)
    outs = []
    for step in range(2):
        q = torch.randn((len(lens), H * G, 128), generator=torch.Generator(device=DEV).manual_seed(step), device=DEV).bfloat16()
        got = binding.decode_attn(q, y, workspace=ws, use_count=not raw)
        assert_close_vectors(to_f64(got), _reference(q, y, raw), TOL[torch.bfloat16], f"lengths {lens[:4]}..., step {step}")
        outs.append((q, got))
    q, first = outs[0]
    assert torch.equal(binding.decode_attn(q, y, workspace=ws, use_count=not raw), first)


def test_one_workspace_for_batches_of_different_sizes():
    H, G, cap = 8, 4, 40000
    big = _layer([8000] + [300] * 15, 8192, H, 1)
    small = _layer([40000], cap, 4, 2)             # several clusters per head
    pair = _layer([30000, 500], 32768, H, 3)
    need = [binding.lib().sc_decode_workspace_bytes(*s) for s in ((16, 32, 8, 128, 8192), (1, 16, 4, 128, cap), (2, 32, 8, 128, 32768))]
    ws = torch.zeros(max(need), dtype=torch.uint8, device=DEV)
    want = {}
    for turn in range(3):
        for name, y, h in (("big", big, H), ("small", small, 4), ("pair", pair, H)):
            q = torch.randn((y.core_k.shape[0], h * G, 128), generator=torch.Generator(device=DEV).manual_seed(5), device=DEV).bfloat16()
            got = binding.decode_attn(q, y, workspace=ws)
            want.setdefault(name, binding.decode_attn(q, y))   # a workspace of its own
            assert torch.equal(got, want[name]), (turn, name)


def _us(y, H, G):
    q = torch.randn((y.core_k.shape[0], H * G, 128), device=DEV).bfloat16()
    out, ws = torch.empty_like(q), binding.decode_workspace(y.core_k.shape[0], H * G, H, 128, y.core_k.shape[2], DEV)
    best = float("inf")
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(20):
            binding.decode_attn(q, y, out=out, workspace=ws)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 50)
    return best


def test_a_long_sequence_does_not_hold_up_the_batch():
    # the same number of rows, in one long and fifteen short sequences and in sixteen equal ones; with equal shares for all
    # heads the first took three and a half times as long
    H, G = 8, 4
    skewed, even = _us(_layer([32768] + [1024] * 15, 32768, H, 1), H, G), _us(_layer([3008] * 16, 32768, H, 1), H, G)
    assert skewed < 2 * even, (skewed, even)


@pytest.mark.parametrize("B,H,G,cap,raw", [(19, 4, 2, 8192, True), (11, 8, 1, 8200, True), (22, 8, 1, 8192, True), (38, 8, 1, 8192, True),
                                           (38, 8, 4, 8200, False), (42, 8, 1, 8192, False), (2, 8, 4, 7300, False), (1, 8, 4, 5300, False)])
def test_more_heads_than_seats(B, H, G, cap, raw):
    """Where a block per head would leave SMs idle in the last round: clusters of two and three; and widths that are passed over."""
    lens = [cap - 37 * b for b in range(B)]
    y = _layer(lens, cap, H, B)
    q = torch.randn((B, H * G, 128), generator=torch.Generator(device=DEV).manual_seed(B), device=DEV).bfloat16()
    got = binding.decode_attn(q, y, use_count=not raw)
    assert_close_vectors(to_f64(got), _reference(q, y, raw), TOL[torch.bfloat16], f"{B} x {H} x {G}, capacity {cap}")


@pytest.mark.parametrize("flag", [binding.SC_FLAG_OVERLAP_PREV, binding.SC_FLAG_OVERLAP_CHAIN])
def test_overlapped_launches_with_spare_units(flag):
    """Layers of one skewed batch, eager and from a graph, with one workspace: the same bits as launches in plain stream order."""
    H, G, B = 8, 4, 4
    ys = [_layer([30000, 900, 40, 2500], 32768, H, i, False) for i in range(5)]
    q = torch.randn((B, H * G, 128), generator=torch.Generator(device=DEV).manual_seed(1), device=DEV).bfloat16()
    ws = binding.decode_workspace(B, H * G, H, 128, 32768, DEV)

    def layers(flags, outs):
        x = q
        for y, o in zip(ys, outs):
            r = binding.decode_attn(x, y, out=o, workspace=ws, flags=flags)
            x = r if flag == binding.SC_FLAG_OVERLAP_CHAIN else q
        return outs

    want = layers(0, [torch.empty_like(q) for _ in ys])
    torch.cuda.synchronize()
    outs = [torch.empty_like(q) for _ in ys]
    for _ in range(3):
        layers(flag, outs)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        layers(flag, outs)
    for o in outs:
        o.zero_()
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(outs, want))
