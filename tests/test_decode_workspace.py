"""Sizes of the decode workspace (host side only): one that was sized for the largest batch and capacity serves every smaller
call, and the fixed scratch of sc_decode_attn_static is not what limits a batch."""
import pytest

from paper_2603_14303_b200 import binding, build


@pytest.fixture(scope="module")
def size():
    build.build()
    f = binding.lib().sc_decode_workspace_bytes
    return lambda B, Hq, Hkv, cap: f(B, Hq, Hkv, 128, cap)


@pytest.mark.parametrize("Hkv,G", [(8, 4), (4, 7), (1, 8), (16, 1)])
def test_the_largest_batch_covers_the_smaller_ones(size, Hkv, G):
    caps = [1, 63, 64, 65, 512, 1024, 1280, 4096, 8192, 32768, 131072]
    for cap, wider in zip(caps, caps[1:] + caps[-1:]):
        for B in list(range(1, 70)) + [127, 128, 500]:
            assert size(B, Hkv * G, Hkv, cap) <= size(B + 1, Hkv * G, Hkv, cap)
            assert size(B, Hkv * G, Hkv, cap) <= size(B, Hkv * G, Hkv, wider)


@pytest.mark.parametrize("B,Hq,Hkv,cap", [(1, 32, 8, 131072), (16, 32, 8, 8192), (500, 32, 8, 512), (2000, 8, 1, 500), (60, 16, 16, 8192)])
def test_shapes_the_fixed_scratch_holds(size, B, Hq, Hkv, cap):
    splits = min(64, -(-cap // 512))
    assert 4 * B * Hq * splits * 130 + 256 <= binding.SC_STATIC_SCRATCH_BYTES
    assert size(B, Hq, Hkv, cap) <= binding.SC_STATIC_SCRATCH_BYTES
