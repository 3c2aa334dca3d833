"""Map counts that are not a group width: the maps past the eights run as one
padded group, and q^t holds a group's maps in packs of two (QtView).  A map's
result does not depend on its group, so every comparison is for equality."""
import pytest

from paper_1110_4874_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402


# max_depth 0: residual blocks write q^t themselves; residual_recurrence: regenerated ones do
@pytest.mark.parametrize("nside,lmax,opts", [
    (16, 33, {}), (33, 70, {"max_depth": 0}), (32, 64, {"residual_recurrence": True}),
    (16, 40, {"max_depth": 0, "residual_recurrence": True})])
@pytest.mark.parametrize("nmaps", [2, 3, 6, 7, 9, 12])
def test_grouped_maps_equal_single_maps(nside, lmax, opts, nmaps):
    plan = sh.Plan(nside, lmax, 1e-10, **opts)
    a = torch.from_numpy(synthetic.gaussian_alm(lmax, nmaps, seed=nmaps)).cuda()
    maps = plan.synthesize(a)
    back = plan.adjoint(maps)
    q = torch.empty(nmaps, 2, 2 * nside, lmax + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_butterfly(plan.handle, a, q, nmaps)
    host = torch.empty(nmaps, plan.npix, dtype=torch.float64)
    sh.shtb_synthesize_host(plan.handle, a.cpu(), host, nmaps)
    torch.cuda.synchronize()
    assert torch.equal(host, maps.cpu())
    for b in range(nmaps):
        assert torch.equal(plan.synthesize(a[b]), maps[b])
        assert torch.equal(plan.adjoint(maps[b]), back[b])
        one = torch.empty_like(q[:1])
        sh.shtb_test_butterfly(plan.handle, a[b:b + 1].contiguous(), one, 1)
        assert torch.equal(one[0], q[b])


@pytest.mark.parametrize("npairs", [2, 3, 5])
def test_grouped_pairs_equal_single_pairs(npairs):
    plan = sh.Plan(24, 50, 1e-10, spin=2)
    a = torch.from_numpy(synthetic.gaussian_alm(50, 2 * npairs, seed=4)).cuda().reshape(npairs, 2, -1)
    maps = plan.synthesize_spin(a)
    back = plan.adjoint_spin(maps)
    for p in range(npairs):
        assert torch.equal(plan.synthesize_spin(a[p]), maps[p])
        assert torch.equal(plan.adjoint_spin(maps[p]), back[p])
