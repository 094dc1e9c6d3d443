"""The wavelet shrinkage scales exactly: with threshold zero it is the identity, bit for
bit on whole numbers (whose sums over a cube are exact), so a solve's iterations do not
shrink the image by rounding."""

import numpy as np
import pytest

from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("shape", [(16, 32, 48), (48, 16, 16), (16, 16, 80)])
@pytest.mark.parametrize("levels", [0, 1, 2, 3, 4])
def test_zero_threshold_is_the_identity(shape, levels):
    from paper_2501_16713_gb300 import wavelet_shrink
    rng = np.random.default_rng(181)
    v = (rng.integers(-500, 500, shape) + 1j * rng.integers(-500, 500, shape)).astype(np.complex64)
    assert np.array_equal(wavelet_shrink(to_dev(v), 0.0, levels).cpu().numpy(), v)
