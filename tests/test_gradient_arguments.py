"""Argument checks of the emulator network's gradients: operands that the
kernels could not read (16-byte pieces) are refused before any launch, so no
GPU is needed here and none is touched."""
import ctypes

import pytest

SG_ERR_ARG = -1


@pytest.fixture(scope="module")
def lib():
    from paper_1605_01421_gb300 import binding
    try:
        binding.build()
    except FileNotFoundError:
        pytest.skip("nvcc not available")
    return binding.lib()


def _call(lib, feat=4096, W=(8192, 16384, 32768, 65536)):
    nb = ctypes.c_int64()
    assert lib.sg_mlp_gradients_scratch(8, ctypes.byref(nb)) == 0
    ptrs = lambda ps: (ctypes.c_void_p * 4)(*ps)  # noqa: E731
    v = ctypes.c_void_p
    return lib.sg_mlp_gradients(v(feat), v(4096), 8, ptrs(W), ptrs([4096] * 4), ptrs([4096] * 4),
                                ptrs([4096] * 4), v(4096), v(4096), nb.value, None)


@pytest.mark.parametrize("off", [2, 4, 8])
def test_misaligned_operands_are_refused(lib, off):
    assert _call(lib, feat=4096 + off) == SG_ERR_ARG
    for layer in range(4):
        W = [8192, 16384, 32768, 65536]
        W[layer] += off
        assert _call(lib, W=W) == SG_ERR_ARG
