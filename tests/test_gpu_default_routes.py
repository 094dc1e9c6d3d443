"""The kernels an untuned plan takes, against the ones it could take: a default rule
picks the faster side of its line.

Times are the library's own stage times, medians over several runs; the sides measured
here differ by 1.2 and more, the default may lose a tenth.
"""

import ctypes

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


def _contraction(shape, phases, factor):
    n = np.stack(np.meshgrid(*[np.arange(s, dtype=np.float32) for s in shape], indexing="ij"))
    c = np.array([(s - 1) / 2 for s in shape], np.float32)[:, None, None, None]
    return np.stack([(factor - 1.0) * (n - c) + 0.1 * (j + 1) for j in range(phases)]).astype(np.float32)


def _stage(plan, name, run, repeat=7):
    """Median time of a stage, ms."""
    import torch
    for _ in range(3):
        run()
    ts = []
    for _ in range(repeat):
        plan.profile_start(200)
        for _ in range(4):
            run()
        torch.cuda.synchronize()
        ts.append(plan.profile_stop()[0][name][0] / 4)
    return sorted(ts)[repeat // 2]


def _set(plan, **kw):
    from paper_2501_16713_gb300.nrsense import Tuning
    t = Tuning()
    t.spread_variant, t.interp_coils, t.interp_tma, t.spread_image_warp = 1, 8, 0, 0
    for k, v in kw.items():
        setattr(t, k, v)
    assert plan.lib.nrsense_plan_set_tuning(plan._h, ctypes.byref(t)) == 0


@pytest.mark.parametrize("shape,osf,phases", [((64, 64, 64), 1.5, 1), ((128, 128, 128), 1.5, 1),
                                              ((96, 80, 104), 1.25, 2), ((128, 128, 128), 2, 8),
                                              ((64, 64, 64), 2.5, 1), ((32, 32, 32), 2, 8),
                                              ((96, 96, 96), 2, 1)])
def test_image_interpolation(shape, osf, phases):
    import torch
    from paper_2501_16713_gb300 import Plan
    size = max(shape)  # motion as in the benchmark: bumps of up to 6 % of the image
    d = np.stack([synth.bump_displacement(shape, 169 + j, 0.06 * size, width_range=(0.05 * size, 0.1 * size))
                  for j in range(phases)])
    plan = Plan(shape, disp=to_dev(d), n_phases=phases, osf=osf)
    x = to_dev(crandn(np.random.default_rng(161), shape))
    out = plan.warp_forward(x)
    run = lambda: plan.warp_forward(x, out=out)  # noqa: E731
    ms, first = _stage(plan, "interp_image", run), out.clone()
    other = []
    dt = to_dev(d)
    edge = ((dt < 0) & (dt > -1e-7)).any(1)
    own = int(osf == 2 and set(shape) <= {16, 32, 64, 128})  # power-of-two transforms, as created
    for home in (0, 1):
        _set(plan, interp_image_home=home, spread_image_warp=2, image_fft_pruned=own)
        other.append(_stage(plan, "interp_image", run))
        # the same values, bit for bit but where a displacement component is negative and
        # below 1e-7: the sorted positions (FP64) round up to the grid point, whose taps
        # start one later with the fraction 0 instead of 1
        same = (out == first) | edge
        assert bool(same.all()) and float((out - first).abs().max()) < 1e-6 * float(first.abs().max())
    print(shape, osf, phases, "default %.4f, per voxel %.4f, super-tiles %.4f ms" % (ms, *other))
    assert ms < 1.1 * min(other)
    plan.close()


@pytest.mark.parametrize("width,factor,rows", [(4, 1.0, True), (4, 0.8, True), (4, 0.5, False),
                                               (4, 0.15, False), (6, 1.0, True), (6, 0.5, True),
                                               (6, 0.15, False), (6, 0.05, False)])
def test_image_spread_of_crowded_points(width, factor, rows):
    """Images contracted about their centre: block rows (one kernel) until the crowd is one
    warp's, then home tiles or split halo lists (two)."""
    import torch
    from paper_2501_16713_gb300 import Plan
    shape = (128, 128, 128)
    w = to_dev(crandn(np.random.default_rng(162), (1,) + shape))

    def kernels(factor):
        plan = Plan(shape, disp=to_dev(_contraction(shape, 1, factor)), n_phases=1, width=width)
        out = plan.warp_adjoint(w)
        plan.profile_start(100)
        plan.warp_adjoint(w, out=out)
        torch.cuda.synchronize()
        st, own = plan.profile_stop()
        print(width, factor, "%.4f ms, %d kernels" % (st["spread_image"][0], own))
        plan.close()
        return own

    assert kernels(factor) - kernels(1.0) == (0 if rows else 1)


@pytest.mark.parametrize("n,samples", [(64, 40000), (128, 20000), (192, 100000), (64, 2000000)])
def test_two_coil_spread(n, samples):
    """The sub-block kernel only where items hold enough points: against it and the register
    kernel."""
    import torch
    from paper_2501_16713_gb300 import Plan
    gen = torch.Generator(device="cuda").manual_seed(163)
    k = (torch.rand((samples, 3), device="cuda", generator=gen) * 2 - 1) * 3.1
    maps = torch.ones((2, n, n, n), dtype=torch.complex64, device="cuda")
    plan = Plan((n, n, n), coords=[k], smaps=maps, identity_warp=True)
    y = torch.randn((samples, 2), dtype=torch.complex64, device="cuda", generator=gen)
    out = plan.adjoint(y)
    run = lambda: plan.adjoint(y, out=out)  # noqa: E731
    ms, other = _stage(plan, "spread_kspace", run), []
    for variant in (1, 4):
        _set(plan, spread_variant=variant)
        other.append(_stage(plan, "spread_kspace", run))
    print(n, samples, "default %.4f, register %.4f, sub-blocks %.4f ms" % (ms, *other))
    assert ms < 1.1 * min(other)
    plan.close()


@pytest.mark.parametrize("shape,width,coils,samples", [
    ((24, 20, 28), 4, 2, 120), ((24, 20, 28), 4, 2, 900), ((24, 20, 28), 6, 3, 60),
    ((24, 20, 28), 6, 4, 60), ((24, 20, 28), 6, 3, 900), ((18, 22, 20), 6, 3, 30)])
def test_few_coils_on_both_sides_of_the_line(shape, width, coils, samples):
    c = synth.small_case(shape, coils, 2, [samples, samples // 2], seed=164, uniform_coords=True)
    plan = make_plan(c, shape, identity_warp=True, width=width)
    y = crandn(np.random.default_rng(165), (samples + samples // 2, coils))
    ref = O.stacked_adjoint(O.Geometry(shape, width=width), np.split(y.astype(np.complex128), [samples]),
                            [None, None], c["smaps"], c["coords"])
    assert rel_l2(plan.adjoint(to_dev(y)).cpu().numpy(), ref) < TOL_FP32
    plan.close()


@pytest.mark.parametrize("shape,osf,own", [((256, 256, 12), 4, False), ((256, 32, 224), 4, False),
                                           ((256, 32, 32), 4, True), ((32, 256, 224), 4, True)])
def test_coil_transforms_at_1024_points(shape, osf, own):
    """cuFFT along z of 1024 points and another long axis, own passes else; either way the
    adjoint of the forward operator (whose parts are held against the oracle at small sizes)."""
    import torch
    from paper_2501_16713_gb300 import Plan
    gen = torch.Generator(device="cuda").manual_seed(166)
    k = (torch.rand((5000, 3), device="cuda", generator=gen) * 2 - 1) * 3.1
    maps = torch.randn((1,) + shape, dtype=torch.complex64, device="cuda", generator=gen)
    plan = Plan(shape, coords=[k], smaps=maps, identity_warp=True, osf=osf)
    x = torch.randn(shape, dtype=torch.complex64, device="cuda", generator=gen)
    y = torch.randn((5000, 1), dtype=torch.complex64, device="cuda", generator=gen)
    plan.forward(x)
    plan.profile_start(100)
    ax, ahy = plan.forward(x), plan.adjoint(y)
    torch.cuda.synchronize()
    st = plan.profile_stop()[0]
    assert (st["fft_pruned"][1] > 0, st["fft_gc"][1] > 0) == (own, not own)
    a = (ax.conj().to(torch.complex128) * y).sum()
    b = (x.conj().to(torch.complex128) * ahy).sum()
    scale = ax.to(torch.complex128).norm() * y.to(torch.complex128).norm()
    assert abs(a - b) < 1e-6 * scale
    plan.close()


@pytest.mark.parametrize("coils", [2, 3, 4])
@pytest.mark.parametrize("samples", [50, 40000])
def test_tuned_sub_blocks_of_few_coils(coils, samples):
    """The tuner's sub-block choice with two to four coils (partial chunk with three, ragged
    tiles, split items) against the oracle.  Positive data, FP32 steps of at most some 2.5e-7
    each: 1e-6 together."""
    shape = (16, 14, 18)
    c = synth.small_case(shape, coils, 1, [samples], seed=167)
    plan = make_plan(c, shape, identity_warp=True)
    _set(plan, spread_variant=4)
    y = (1.0 + 0.1 * crandn(np.random.default_rng(168), (samples, coils))).astype(np.complex64)
    ref = O.stacked_adjoint(O.Geometry(shape), [y.astype(np.complex128)], [None], c["smaps"], c["coords"])
    yt = to_dev(y)
    x = plan.adjoint(yt)
    err = rel_l2(x.cpu().numpy(), ref)
    print(coils, samples, "adjoint rel L2 %.2e" % err)
    assert err < 1e-6
    plan.close()
