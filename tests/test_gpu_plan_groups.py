"""Plans whose phases are too many samples to list at once: the host builds them in
groups, and every phase comes out as in a plan of its own."""

import pytest

from helpers import TOL_FP32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def test_phases_listed_in_groups():
    import torch
    from paper_2501_16713_gb300 import Plan
    shape, counts = (24, 20, 28), [4000000, 4000000, 700000, 5]  # groups {0, 1} and {2, 3}
    gen = torch.Generator(device="cuda").manual_seed(171)
    coords = [(torch.rand((m, 3), device="cuda", generator=gen) * 2 - 1) * 3.1 for m in counts]
    maps = torch.randn((1,) + shape, dtype=torch.complex64, device="cuda", generator=gen)
    x = torch.randn(shape, dtype=torch.complex64, device="cuda", generator=gen)
    plan = Plan(shape, coords=coords, smaps=maps, identity_warp=True)
    y = plan.forward(x)
    w = torch.randn(y.shape, dtype=torch.complex64, device="cuda", generator=gen)
    total = 0
    for j in range(len(counts)):
        one = Plan(shape, coords=[coords[j]], smaps=maps, identity_warp=True)
        assert torch.equal(one.forward(x), plan.phase_slice(y, j))
        total = total + one.adjoint(plan.phase_slice(w, j).contiguous()).to(torch.complex128)
        one.close()
    err = (plan.adjoint(w).to(torch.complex128) - total).norm() / total.norm()
    assert float(err) < TOL_FP32
    plan.close()
