"""The uncompressed Legendre stage, whose sums over the maps are integer
(shtb_legendre.cu), where that can go wrong: last chunks of a few rings, chains
around the step and tile sizes, map counts of every width, scales at the ends
of the range, zero maps, infinities and NaN.

Tolerance against the oracle: both sides run the recurrence in FP64, whose
rounding grows by about 2^-53 a step, so 4 (lmax + 16) 2^-53 of the norm
allows each side twice that."""
import numpy as np
import pytest

import oracle as orc
from paper_1110_4874_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402


def alm_of(lmax, nmaps, seed):
    return torch.from_numpy(synthetic.gaussian_alm(lmax, nmaps, seed=seed)).cuda()


# half-rings 2 nside: 2, 16, 32, 34, 64, 66, 40; chains of 1 to 101 steps
@pytest.mark.parametrize("nside,lmax", [(1, 2), (8, 7), (16, 9), (17, 64), (32, 67), (33, 131), (20, 201)])
@pytest.mark.parametrize("nmaps", [1, 2, 3, 4, 8])
def test_sums_match_the_oracle(nside, lmax, nmaps):
    plan, rings = sh.Plan(nside, lmax, 0.0), orc.healpix_rings(nside)
    tol = 4 * (lmax + 16) * 2.0 ** -53
    a = alm_of(lmax, nmaps, 3)
    maps = plan.synthesize(a)
    back = plan.adjoint(maps)
    for b in {0, nmaps - 1}:
        want = orc.synthesize(rings, lmax, a[b].cpu().numpy())
        got = maps[b].cpu().numpy()
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
        want = orc.adjoint(rings, lmax, got)
        assert np.linalg.norm(back[b].cpu().numpy() - want) <= tol * np.linalg.norm(want)
        assert torch.equal(plan.synthesize(a[b:b + 1])[0], maps[b])
        assert torch.equal(plan.adjoint(maps[b:b + 1])[0], back[b])


@pytest.mark.parametrize("nmaps", [1, 2, 4, 8])
def test_scales_and_zero_maps(nmaps):
    plan = sh.Plan(32, 80, 0.0)
    a = alm_of(80, nmaps, 6)
    base, back = plan.synthesize(a), plan.adjoint(plan.synthesize(a))
    for p in (2.0 ** -500, 2.0 ** 500):        # exact: powers of two in the sums' range
        assert torch.equal(plan.synthesize(a * p), base * p)
        assert torch.equal(plan.adjoint(base * p), back * p)
    for p in (2.0 ** -960, 2.0 ** 990):        # FP64 sums of 41 terms (synthesis), 64 (adjoint), and ring sums
        s, t = plan.synthesize(a * p), plan.adjoint(base * p)
        assert float(((s / p) - base).norm() / base.norm()) <= 80 * 2.0 ** -53
        assert float(((t / p) - back).norm() / back.norm()) <= 80 * 2.0 ** -53
    assert torch.count_nonzero(plan.synthesize(torch.zeros_like(a))) == 0
    z = a.clone()
    z[0] = 0                                    # a zero map among others
    got = plan.synthesize(z)
    assert torch.count_nonzero(got[0]) == 0
    assert torch.equal(got[1:], base[1:])


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_maps_stay_apart(bad):
    plan = sh.Plan(32, 80, 0.0)
    a = alm_of(80, 8, 7)
    base, f = plan.synthesize(a), plan.synthesize(a)
    b = a.clone()
    b[3, int(synthetic.alm_index(80, 40, 2))] = complex(bad, 0.0)
    got = plan.synthesize(b)
    keep = [i for i in range(8) if i != 3]
    assert torch.equal(got[keep], base[keep])
    assert not torch.isfinite(got[3]).any()     # order 2 reaches every ring
    f[5, 1000] = bad
    back, want = plan.adjoint(f), plan.adjoint(base)
    keep = [i for i in range(8) if i != 5]
    assert torch.equal(back[keep], want[keep])
    assert not torch.isfinite(back[5]).all()


# 4, 5, 8 and 9 chunks of 32 half-rings: 8 and 16 warps an order
@pytest.mark.parametrize("nside", [64, 65, 128, 129])
@pytest.mark.parametrize("nmaps", [1, 2, 4, 8])
def test_adjoint_at_the_lines_between_block_sizes(nside, nmaps):
    lmax = 40
    plan, rings = sh.Plan(nside, lmax, 0.0), orc.healpix_rings(nside)
    f = torch.from_numpy(synthetic.gaussian_map(plan.npix, nmaps, seed=9)).cuda()
    back = plan.adjoint(f)
    want = orc.adjoint(rings, lmax, f[nmaps - 1].cpu().numpy())
    got = back[nmaps - 1].cpu().numpy()
    assert np.linalg.norm(got - want) <= 4 * (lmax + 16) * 2.0 ** -53 * np.linalg.norm(want)
    assert torch.equal(plan.adjoint(f[nmaps - 1]), back[nmaps - 1])
