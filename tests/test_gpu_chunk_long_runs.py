"""sc_chunk on text whose delimiters are rare or absent: the run a tile starts in may begin anywhere before it.  Lengths
around the 2048-token tiles, the 16 K-token looks back and the 262144 tokens from which a block takes several tiles."""
import numpy as np
import pytest
import torch

import oracle
from helpers import compare_plan
from paper_2603_14303_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
DELIMS = (13, 29889, 29892)


def _run(ids, max_len):
    plan = binding.chunk(torch.from_numpy(ids).to(DEV), DELIMS, max_len)
    seg_off, seq_seg_off = oracle.chunk(ids, DELIMS, max_len)[:2]
    compare_plan(plan, seg_off, seq_seg_off)


@pytest.mark.parametrize("n", [2047, 2049, 4096 + 257, 18432, 18433, 2048 * 17 + 255, 262144, 262145, 2048 * 259 + 77])
@pytest.mark.parametrize("max_len", [256, 37])
def test_rare_delimiters(n, max_len):
    rng = np.random.default_rng(n)
    ids = rng.integers(100, 1000, size=(2, n), dtype=np.int32)
    # a few delimiters at places where a look back ends or a tile begins; the second sequence has one, near its start
    for p in (0, 2047, 2048, 4095, 18431, 18432 - 256, 2048 * 130 - 1, 2048 * 131 + 5):
        if p < n and rng.random() < 0.6:
            ids[0, p] = DELIMS[int(rng.integers(3))]
    ids[1, min(3, n - 1)] = DELIMS[0]
    _run(ids, max_len)


@pytest.mark.parametrize("n", [2048 * 9 + 1, 2048 * 141])
def test_no_delimiters(n):
    _run(np.full((1, n), 7, dtype=np.int32), 100)


def test_text_without_delimiters_takes_no_multiple_of_text_with_them():
    n = 1 << 20
    g = torch.Generator(device=DEV).manual_seed(1)
    ids = torch.randint(100, 1000, (1, n), generator=g, device=DEV, dtype=torch.int32)
    text = ids.clone()
    text[torch.rand((1, n), generator=g, device=DEV) < 0.05] = DELIMS[0]

    def us(x):
        p = binding.chunk(x, DELIMS)
        ws = torch.empty(binding.lib().sc_chunk_workspace_bytes(1, n), dtype=torch.uint8, device=DEV)
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(5):
                binding.sc_chunk(x, DELIMS, 256, p.seg_off, p.seq_seg_off, p.n_seg, p.tile_seg, p.seq_tile_cnt, ws, p.status)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1) * 200)
        return best

    # 196 us against 226: there are 21 times fewer segments to write and pack.  A look back whose work grows with the square of the
    # length took 8.5 times as long as text with delimiters; twice leaves room for a busy machine.
    assert us(ids) < 2 * us(text)
