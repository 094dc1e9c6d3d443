"""Tuning choices that need another point order or work-item split, with their
memory refused.

The library's host fault injection (NRSENSE_FAULT=alloc:N refuses allocations of a plan
that holds N already, so a growing N stops the call at each of its allocations in turn;
upload refuses the first copy).  A refused call gives back what it allocated and leaves
the plan as it was; the same call with memory again builds everything, and the results
are the oracle's.
"""

import ctypes

import numpy as np
import pytest

import synth
from helpers import TOL_FP32, crandn, make_plan, rel_l2, to_dev
from oracle import operators as O

pytestmark = pytest.mark.gpu

SHAPE = (16, 14, 18)  # grid 32 x 28 x 36: ragged tiles, whole 4^3 blocks


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def _setup(phases, samples=6000):
    """Plan with its data, the present adjoint and the oracle's."""
    c = synth.small_case(SHAPE, 2, phases, [samples] * phases, seed=151)
    plan = make_plan(c, SHAPE)
    y = crandn(np.random.default_rng(152), (samples * phases, 2))
    ref = O.stacked_adjoint(O.Geometry(SHAPE), np.split(y.astype(np.complex128), phases),
                            [d.astype(np.float64) for d in c["disp"]], c["smaps"], c["coords"])
    yt = to_dev(y)
    return plan, yt, plan.adjoint(yt), ref


def _set(plan, **kw):
    from paper_2501_16713_gb300.nrsense import Tuning
    t = Tuning()
    t.spread_variant, t.interp_coils, t.interp_tma, t.spread_image_warp = 4, 2, 1, 2
    for k, v in kw.items():
        setattr(t, k, v)
    return plan.lib.nrsense_plan_set_tuning(plan._h, ctypes.byref(t))


# one phase: the plan starts with block rows, four: with home tiles
@pytest.mark.parametrize("phases,choice", [
    (1, {"spread_image_warp": 0}), (1, {"spread_image_warp": 1}), (1, {"interp_image_home": 1}),
    (4, {"spread_image_warp": 0}), (4, {"spread_image_warp": 1})])
def test_refused_point_order_is_built_by_the_next_call(monkeypatch, phases, choice):
    import torch
    plan, y, x0, ref = _setup(phases)
    held = plan.info()["device_bytes"]
    monkeypatch.setenv("NRSENSE_FAULT", "upload")
    assert _set(plan, **choice) == -4
    assert plan.info()["device_bytes"] == held
    refused = 0
    for n in range(1, 200):
        monkeypatch.setenv("NRSENSE_FAULT", "alloc:%d" % n)
        st = _set(plan, **choice)
        if st == 0:
            break
        assert st == -2
        assert plan.info()["device_bytes"] == held
        assert torch.equal(plan.adjoint(y), x0)
        refused += 1
    monkeypatch.delenv("NRSENSE_FAULT")
    assert st == 0 and refused > 5
    assert plan.info()["device_bytes"] > held
    x = plan.adjoint(y)
    assert rel_l2(x.cpu().numpy(), ref) < TOL_FP32
    assert torch.equal(plan.adjoint(y), x)
    assert plan.device_status() == 0
    plan.close()


def test_refused_work_item_split_leaves_a_plan_that_runs(monkeypatch):
    """Three phases re-split one after the other, stopped at every allocation: the adjoint
    and a captured CG solve stay right in between.  Phases already re-split sum their tiles
    in another order, so results agree to rounding, which three iterations on a system of
    condition 2 or so carry on without growth."""
    plan, y, x0, ref = _setup(3, samples=40000)
    lam = 1e6
    cg = lambda: plan.solve_cg(y, lam, tol=0.0, maxit=3, graph=True)[0].cpu().numpy()  # noqa: E731
    cg0 = cg()
    split = plan.info()["split_tiles"]
    refused = 0
    for n in range(1, 300):
        monkeypatch.setenv("NRSENSE_FAULT", "alloc:%d" % n)
        st = _set(plan, spread_max_item=512)
        monkeypatch.delenv("NRSENSE_FAULT")
        if st == 0:
            break
        assert st == -2
        refused += 1
        assert rel_l2(plan.adjoint(y).cpu().numpy(), ref) < TOL_FP32
        assert rel_l2(cg(), cg0) < TOL_FP32
    assert st == 0 and refused > 5
    assert plan.info()["split_tiles"] > split
    assert rel_l2(plan.adjoint(y).cpu().numpy(), ref) < TOL_FP32
    assert rel_l2(cg(), cg0) < TOL_FP32
    plan.close()
