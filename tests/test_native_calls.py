"""The extension entry points take and refuse the argument values that ctypes takes and refuses for the same prototypes; no
call here gets as far as a CUDA call (its pointers are null)."""
import numpy as np
import pytest

from paper_2603_14303_b200 import binding, build


@pytest.fixture(scope="module")
def native():
    build.build()
    return binding._native()


def _chunk(native, delims, max_len=256, B=1, n=8):
    return native.chunk(None, B, n, delims, max_len, None, 8, None, None, None, 3, None, None, 0, None, None)


@pytest.mark.parametrize("delims", [(), [13], (13, 29889), {13}, {13: 0}, np.array([13, 14]), [np.int64(13)], ["13"], [13.7], [-1],
                                    [1 << 40, -(1 << 63)], [1 << 63, 1 << 200]])
def test_delimiters_accepted(native, delims):
    assert _chunk(native, delims) == binding.SC_ERR_INVALID_ARG   # converted; then refused for its null pointers


@pytest.mark.parametrize("delims", [(i for i in (13,)), iter([13]), 13, None, ["x"], [None], [13, object()]])
def test_delimiters_refused(native, delims):
    with pytest.raises((TypeError, ValueError)):
        _chunk(native, delims)


def test_integers(native):
    # more than 32 bits are cut, as by c_int32: a negative length is what the library then sees
    assert _chunk(native, (), max_len=(1 << 32) + 256) == binding.SC_ERR_INVALID_ARG
    assert _chunk(native, (), max_len=True) == binding.SC_ERR_INVALID_ARG
    assert _chunk(native, (), max_len=np.int64(256)) == binding.SC_ERR_INVALID_ARG
    assert native.chunk_sizes(1 << 31, 1)[0] == binding.SC_ERR_INVALID_ARG
    for bad in (256.0, "256", None):
        with pytest.raises(TypeError):
            _chunk(native, (), max_len=bad)


def test_flags_are_taken_modulo_two_to_the_32(native):
    call = lambda flags: native.prefill_attn(None, binding.SC_BF16, 0, 8, 8, 1, 128, None, None, None, 0, None, 0.0, flags, None, None, None)
    assert call(0) == binding.SC_OK                                  # no sequences: nothing to do
    assert call(1 << 32) == binding.SC_OK
    assert call(-1) == binding.SC_ERR_INVALID_ARG                    # unknown flags
