"""The mixed-radix passes with compile-time radices vs the FP64 oracle: every multiple of
16 that tests/test_gpu_fft_mixed.py does not hold, once along each axis."""

import pytest

import test_gpu_fft_mixed as mixed

pytestmark = pytest.mark.gpu

LENGTHS = [48, 80, 96, 112, 144, 160, 176, 208, 224, 240]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", LENGTHS)
def test_length_along_every_axis(n, axis):
    shape = [10, 8, 6]
    shape[axis] = n
    mixed.test_operator_and_warp_match_oracle(tuple(shape), 2, 4)
