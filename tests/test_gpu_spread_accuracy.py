"""An untuned plan spreads more than four coils on the tensor cores no less accurately than
by the FP32 register kernel.

Data that belong to an image (coherent, the centre of k space large), where the tensor
core's truncated sums add up.  Both spreads of the same data on the same plan against the
FP64 oracle; the mean error over the inputs may exceed the register kernel's by 3 %, the
scatter of such a mean.
"""

import ctypes

import numpy as np
import pytest

import synth
from helpers import c64, make_plan, rel_l2, to_dev
from oracle import operators as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("shape,coils,samples", [((32, 32, 32), 6, 3000), ((24, 30, 28), 12, 6000)])
def test_untuned_spread_is_as_accurate_as_the_register_kernel(shape, coils, samples):
    from paper_2501_16713_gb300.nrsense import Tuning
    geo = O.Geometry(shape)
    errs = []
    for seed in range(191, 196):
        c = synth.small_case(shape, coils, 1, [samples], seed=seed)
        y = c64(O.stacked_forward(geo, c["x"].astype(np.complex128), [None], c["smaps"], c["coords"])[0])
        ref = O.stacked_adjoint(geo, [y.astype(np.complex128)], [None], c["smaps"], c["coords"])
        plan = make_plan(c, shape, identity_warp=True)
        e = [rel_l2(plan.adjoint(to_dev(y)).cpu().numpy(), ref)]
        t = Tuning()
        t.spread_variant, t.interp_coils, t.interp_tma = 1, 4, 1
        t.fft_pruned = int(shape == (32, 32, 32))  # the transforms of the plan as created
        assert plan.lib.nrsense_plan_set_tuning(plan._h, ctypes.byref(t)) == 0
        e.append(rel_l2(plan.adjoint(to_dev(y)).cpu().numpy(), ref))
        errs.append(e)
        plan.close()
    mine, register = np.mean(errs, axis=0)
    print(shape, coils, "as created %.3e, register %.3e, ratio %.3f" % (mine, register, mine / register))
    assert mine < 1.03 * register
