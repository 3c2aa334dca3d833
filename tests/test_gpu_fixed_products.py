"""The butterfly's block products in fixed-point digits (shtb_bf_fix.cuh) at
the places where they can go wrong: block shapes around the tile and chunk
sizes, map counts of every width, zero maps, scales at the ends of the range,
infinities and NaN, and plan files, which hold doubles."""
import pytest

from paper_1110_4874_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402


def alm_of(lmax, nmaps, seed):
    return torch.from_numpy(synthetic.gaussian_alm(lmax, nmaps, seed=seed)).cuda()


# chain lengths and ranks from below 8 to several chunks of 32, by way of the
# leaf width and the depth limit
@pytest.mark.parametrize("nside,lmax,opts", [
    (4, 5, {}), (8, 16, {"max_depth": 0}), (16, 70, {"max_depth": 0}), (33, 61, {"leaf_cols": 7}),
    (64, 128, {"leaf_cols": 64}), (48, 200, {"leaf_cols": 17}), (100, 255, {"leaf_cols": 100}),
])
@pytest.mark.parametrize("nmaps", [1, 3, 8])
def test_products_match_the_uncompressed_operator(nside, lmax, opts, nmaps):
    """At eps = 1e-13 the compression error is below 5e-13 (0.4-3 eps, Table
    accuracy, and the recurrence's own rounding below 2e-13 at these sizes),
    so the fixed-point products have to be good to that."""
    ref, plan = sh.Plan(nside, lmax, 0.0), sh.Plan(nside, lmax, 1e-13, **opts)
    a = alm_of(lmax, nmaps, 5)
    want, got = ref.synthesize(a), plan.synthesize(a)
    assert float((want - got).norm() / want.norm()) <= 5e-13
    want_a, got_a = ref.adjoint(want), plan.adjoint(want)
    assert float((want_a - got_a).norm() / want_a.norm()) <= 5e-13


@pytest.mark.parametrize("nmaps", [1, 2, 4, 8])
def test_scale_invariance_zero_maps_and_extremes(nmaps):
    plan = sh.Plan(32, 80, 1e-10)
    a = alm_of(80, nmaps, 6)
    base, back = plan.synthesize(a), plan.adjoint(plan.synthesize(a))
    for p in (2.0 ** -500, 2.0 ** 500):        # exact: powers of two in the digits' range
        assert torch.equal(plan.synthesize(a * p), base * p)
        assert torch.equal(plan.adjoint(base * p), back * p)
    for p in (2.0 ** -960, 2.0 ** 990):        # the FP64 loop takes over: a rounding of 50 terms at most
        s = plan.synthesize(a * p)
        assert float(((s / p) - base).norm() / base.norm()) <= 50 * 2.0 ** -53
    assert torch.count_nonzero(plan.synthesize(torch.zeros_like(a))) == 0
    z = a.clone()
    z[0] = 0                                    # a zero map among others
    got = plan.synthesize(z)
    assert torch.count_nonzero(got[0]) == 0
    assert torch.equal(got[1:], base[1:])


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_maps_stay_apart(bad):
    plan = sh.Plan(32, 80, 1e-10)
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


def test_plan_file_holds_the_same_operator(tmp_path):
    plan = sh.Plan(64, 130, 1e-10)
    one, two = str(tmp_path / "a.bin"), str(tmp_path / "b.bin")
    plan.save(one)
    back = sh.Plan.load(one)
    back.save(two)                              # doubles of words made from doubles
    again = sh.Plan.load(two)
    a = alm_of(130, 3, 8)
    want = plan.synthesize(a)
    for p in (back, again):
        assert torch.equal(p.synthesize(a), want)
        assert torch.equal(p.adjoint(want), plan.adjoint(want))
