"""Sub-block k-space spreads with FP32-accurate sums (1 to 4 coils by FMAs, more by
tensor cores; W = 4 and 6) and the one-coil interpolation vs the FP64 oracle.

Ragged grids (the last tiles 2, 4 or 6 wide), partial coil chunks, odd coil counts
(8-byte aligned rows), few samples (most sub-blocks empty), dense samples (split
work items) and samples on the periodic edge.
"""

import numpy as np
import pytest

import synth
from helpers import TOL_FP32, crandn, make_plan, rel_l2, to_dev
from oracle import operators as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


CASES = [  # shape, sigma, W, coils, samples
    ((10, 12, 14), 2, 4, 1, 40), ((10, 12, 14), 2, 4, 2, 3000), ((10, 14, 22), 2, 4, 3, 700),
    ((12, 10, 18), 2, 4, 5, 900), ((16, 16, 16), 2, 4, 8, 40000), ((10, 12, 14), 2, 4, 13, 1500),
    ((10, 12, 14), 2, 6, 1, 900), ((12, 14, 10), 2, 6, 2, 20000), ((20, 12, 16), 1.5, 6, 4, 700),
    ((18, 12, 22), 1.5, 6, 7, 1200), ((16, 16, 16), 1.25, 6, 8, 30000), ((10, 12, 14), 2, 6, 9, 20),
]


@pytest.mark.parametrize("shape,osf,width,coils,samples", CASES)
def test_adjoint_matches_oracle(shape, osf, width, coils, samples):
    import torch
    c = synth.small_case(shape, coils, 2, [samples, max(1, samples // 3)], seed=101, uniform_coords=True)
    # some samples exactly on the periodic edge and on grid points
    edge = np.array([[-np.pi, 0.0, np.pi / 2], [0.0, -np.pi, -np.pi]], np.float32)
    c["coords"][0][:min(2, samples)] = edge[:min(2, samples)]
    plan = make_plan(c, shape, identity_warp=True, osf=osf, width=width)
    geo = O.Geometry(shape, osf=osf, width=width)
    rng = np.random.default_rng(102)
    y = crandn(rng, (sum(plan.counts), coils))
    ys = np.split(y.astype(np.complex128), [plan.counts[0]])
    ref = O.stacked_adjoint(geo, ys, [None, None], c["smaps"], c["coords"])
    yt = to_dev(y)
    x = plan.adjoint(yt)
    err = rel_l2(x.cpu().numpy(), ref)
    print(shape, osf, width, coils, samples, "adjoint rel L2 %.2e" % err)
    # sigma 1.25: the band edge divides FP32 rounding by the kernel transform's 1/15
    assert err < (5e-5 if osf == 1.25 else TOL_FP32)
    assert torch.equal(plan.adjoint(yt), x)
    fwd = plan.forward(to_dev(c["x"])).cpu().numpy()
    f_ref = np.concatenate(O.stacked_forward(geo, c["x"].astype(np.complex128), [None, None],
                                             c["smaps"], c["coords"]))
    assert rel_l2(fwd, f_ref) < (5e-5 if osf == 1.25 else TOL_FP32)
    plan.close()


@pytest.mark.parametrize("shape,width,samples", [((10, 12, 14), 4, 60), ((16, 16, 16), 4, 30000),
                                                 ((12, 10, 14), 6, 2000)])
def test_density_compensation_matches_oracle(shape, width, samples):
    from oracle import motion as OM
    c = synth.small_case(shape, 5, 1, samples, seed=103)
    plan = make_plan(c, shape, identity_warp=True, width=width)
    w = plan.dcf(0, iters=4).cpu().numpy()
    ref, _ = OM.dcf_pipe_menon(O.Geometry(shape, width=width), c["coords"][0], 4)
    assert rel_l2(w, ref) < TOL_FP32
    plan.close()


@pytest.mark.parametrize("wpc,coils", [(1, 8), (2, 6), (4, 11)])
def test_tuned_sub_blocks_sum_in_fp32(wpc, coils):
    """Positive data, where a truncated running sum drifts one way.  Weights, sums, transform
    and coil combination are FP32 steps of at most some 2.5e-7 each: 1e-6 together."""
    import ctypes
    from paper_2501_16713_gb300.nrsense import Tuning
    shape = (16, 14, 18)
    c = synth.small_case(shape, coils, 1, [40000], seed=104)
    plan = make_plan(c, shape, identity_warp=True)
    t = Tuning()
    t.spread_variant, t.interp_coils, t.interp_tma = 4, 8, 0
    t.spread_mma_wpc, t.spread_mma_cube = wpc, 1
    assert plan.lib.nrsense_plan_set_tuning(plan._h, ctypes.byref(t)) == 0
    y = (1.0 + 0.1 * crandn(np.random.default_rng(105), (40000, coils))).astype(np.complex64)
    ref = O.stacked_adjoint(O.Geometry(shape), [y.astype(np.complex128)], [None], c["smaps"], c["coords"])
    err = rel_l2(plan.adjoint(to_dev(y)).cpu().numpy(), ref)
    print(wpc, coils, "adjoint rel L2 %.2e" % err)
    assert err < 1e-6
    plan.close()
