"""Device sort of the displaced voxels: plans whose points are spread over blocks,
crowded into a few (rank over large groups) or crowded beyond the device sort's limit
(host fallback) give the oracle's T^H, the same values on every build, and the same
values whether an order is built with the plan or when a tuning choice asks for it."""

import ctypes

import numpy as np
import pytest

import synth
from helpers import TOL_FP32, crandn, rel_l2, to_dev
from oracle import operators as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("shape,phases,kind", [((14, 10, 18), 1, "smooth"), ((14, 10, 18), 3, "smooth"),
                                               ((16, 16, 16), 1, "crowd"), ((16, 16, 16), 4, "crowd"),
                                               ((24, 24, 24), 1, "crowd"), ((24, 24, 24), 3, "crowd")])
def test_orders_match_oracle(shape, phases, kind):
    import torch
    from paper_2501_16713_gb300 import Plan
    from paper_2501_16713_gb300.nrsense import Tuning
    rng = np.random.default_rng(111)
    d = np.stack([synth.bump_displacement(shape, 112 + j, 1.4, width_range=(1.0, 3.0))
                  for j in range(phases)])
    if kind == "crowd":  # all voxels into one cell: up to 13824 points per group and phase
        n = np.stack(np.meshgrid(*[np.arange(s, dtype=np.float32) for s in shape], indexing="ij"))
        d = np.stack([3.0 + 0.4 * rng.random((3,) + shape) - n for _ in range(phases)])
    d = to_dev(np.ascontiguousarray(d, dtype=np.float32))
    w = crandn(rng, (phases,) + shape)
    wt = to_dev(w)
    geo = O.Geometry(shape)
    dh = d.cpu().numpy().astype(np.float64)
    ref = sum(O.warp_adjoint(geo, w[j].astype(np.complex128), dh[j]) for j in range(phases))
    plan = Plan(shape, disp=d, n_phases=phases)
    x = plan.warp_adjoint(wt)
    assert rel_l2(x.cpu().numpy(), ref) < TOL_FP32
    again = Plan(shape, disp=d, n_phases=phases)
    assert torch.equal(again.warp_adjoint(wt), x)
    # the other orders, built on demand; then back to the first
    m0 = plan.warp_forward(x)
    for image, home in ((0, 1), (1, 0), (2, 0)):
        t = Tuning()
        t.spread_variant, t.interp_coils, t.spread_image_warp = 3, 8, image
        t.interp_image_home, t.image_fft_pruned = home, int(shape == (16, 16, 16))
        assert plan.lib.nrsense_plan_set_tuning(plan._h, ctypes.byref(t)) == 0
        assert rel_l2(plan.warp_adjoint(wt).cpu().numpy(), ref) < TOL_FP32
        assert torch.equal(plan.warp_forward(x), m0)
    assert torch.equal(plan.warp_adjoint(wt), x)
    plan.close()
    again.close()


def test_bad_displacements_are_refused():
    import torch
    from paper_2501_16713_gb300 import NrsenseError, Plan
    for v in (float("nan"), float("inf"), 2e6):
        d = torch.zeros((1, 3, 8, 8, 8), device="cuda")
        d[0, 1, 3, 4, 5] = v
        with pytest.raises(NrsenseError):
            Plan((8, 8, 8), disp=d, n_phases=1)
