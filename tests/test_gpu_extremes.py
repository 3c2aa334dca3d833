"""Maps and coefficients of extreme magnitude, and maps with infinities or NaN
(masked pixels): powers of two pass through the transforms exactly, a value
that is not finite stays in its ring, and neither costs more than a small
multiple of an ordinary call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402

BAD = [float("nan"), float("inf"), -float("inf")]


def ms(fn):
    """best of seven"""
    fn()
    best = 1e30
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


class Rings:
    """The ring stage alone."""
    def __init__(self, nside, lmax, nmaps):
        self.plan, self.n = sh.Plan(nside, lmax, 0.0), nmaps
        g = torch.Generator(device="cuda").manual_seed(3)
        self.f = torch.randn(nmaps, self.plan.npix, dtype=torch.float64, device="cuda", generator=g)
        q = torch.randn(nmaps, self.plan.nrings, lmax + 1, 2, dtype=torch.float64, device="cuda", generator=g)
        q[:, :, 0, 1] = 0
        self.q = torch.view_as_complex(q)

    def synth(self, q):
        out = torch.empty_like(self.f)
        sh.shtb_test_phi(self.plan.handle, q, out, self.n)
        return out

    def adjoint(self, f):
        out = torch.empty_like(self.q)
        sh.shtb_test_phi_adjoint(self.plan.handle, f, out, self.n)
        return out


# rings of every transform kind
@pytest.mark.parametrize("nside", [1, 21, 47, 64])
@pytest.mark.parametrize("power", [-980, -900, -800, 750, 900, 1000])
def test_rings_scale_exactly_by_powers_of_two(nside, power):
    """No result is subnormal: |q| and |f| are above 2^-30, 2^-1010 in all."""
    r, p = Rings(nside, 60, 2), 2.0 ** power
    assert torch.equal(r.synth(r.q * p), r.synth(r.q) * p)
    assert torch.equal(r.adjoint(r.f * p), r.adjoint(r.f) * p)


def test_rings_of_subnormal_values():
    """Whole multiples of 2^-1074 up to 2^20 of them: exact inputs, results off by
    the rounding of the results to that unit and of the transforms."""
    r = Rings(47, 60, 1)
    k = torch.round(r.f * 2.0 ** 18)
    want, got = r.adjoint(k), r.adjoint(k * 2.0 ** -1074)
    back = torch.view_as_real(got) * 2.0 ** 1000 * 2.0 ** 74
    assert float((back - torch.view_as_real(want)).abs().max()) <= 0.5 + 1e-6


@pytest.mark.parametrize("bad", BAD)
def test_a_value_that_is_not_finite_fills_its_ring(bad):
    r = Rings(47, 60, 2)
    maps, back = r.synth(r.q), r.adjoint(r.f)
    J = 4 * np.minimum(np.minimum(np.arange(1, 188), 47), 188 - np.arange(1, 188))
    start = np.concatenate([[0], np.cumsum(J)])
    for ring in (0, 3, 22, 46, 47, 120, 186):
        q, f = r.q.clone(), r.f.clone()
        q[1, ring, 7] = complex(0.0, bad)
        f[0, start[ring] + J[ring] // 2] = bad
        m, b = r.synth(q), r.adjoint(f)
        inside = torch.zeros_like(maps, dtype=torch.bool)
        inside[1, start[ring]:start[ring + 1]] = True
        assert torch.isnan(m[inside]).all() and torch.equal(m[~inside], maps[~inside])
        rest = torch.ones(2, r.plan.nrings, dtype=torch.bool, device="cuda")
        rest[0, ring] = False
        assert torch.isnan(torch.view_as_real(b[0, ring])).all() and torch.equal(b[rest], back[rest])


def test_extreme_rings_cost_little():
    r = Rings(256, 512, 4)
    t_s, t_a = ms(lambda: r.synth(r.q)), ms(lambda: r.adjoint(r.f))
    for p in BAD + [2.0 ** -900, 2.0 ** 900]:
        q, f = r.q * p, r.f * p
        assert ms(lambda: r.synth(q)) <= 2 * t_s + 0.05, p
        assert ms(lambda: r.adjoint(f)) <= 2 * t_a + 0.05, p


def coefficients(plan, nmaps):
    g = torch.Generator(device="cuda").manual_seed(5)
    a = torch.randn(nmaps, plan.nalm, 2, dtype=torch.float64, device="cuda", generator=g)
    a[:, :plan.lmax + 1, 1] = 0
    return torch.view_as_complex(a)


# compressed plans, several chunks of 32 (max_depth 0) and many levels
@pytest.mark.parametrize("nside,lmax,opts", [(32, 80, {}), (16, 70, {"max_depth": 0}), (64, 200, {"leaf_cols": 17})])
@pytest.mark.parametrize("nmaps", [1, 2, 4, 8])
def test_compressed_plans_scale_exactly_by_powers_of_two(nside, lmax, opts, nmaps):
    """Nothing is subnormal: the operator's elements and their products are zero
    or above 2^-120."""
    plan = sh.Plan(nside, lmax, 1e-10, **opts)
    a = coefficients(plan, nmaps)
    maps = plan.synthesize(a)
    back = plan.adjoint(maps)
    for power in (-850, -700, 700, 850, 980):
        p = 2.0 ** power
        assert torch.equal(plan.synthesize(a * p), maps * p), power
        assert torch.equal(plan.adjoint(maps * p), back * p), power
    # one map of another scale, or not finite, leaves the rest alone
    for x in BAD + [2.0 ** -850, 2.0 ** 900]:
        b, f = a.clone(), maps.clone()
        b[0] *= x
        f[0] *= x
        assert torch.equal(plan.synthesize(b)[1:], maps[1:])
        assert torch.equal(plan.adjoint(f)[1:], back[1:])
        if x in BAD or x != x:
            assert not torch.isfinite(plan.synthesize(b)[0]).any()
            assert not torch.isfinite(torch.view_as_real(plan.adjoint(f)[0])[lmax + 1:]).any()


@pytest.mark.parametrize("eps,most", [(1e-10, 2), (0.0, 4)])       # uncompressed sums take FP64 there
@pytest.mark.parametrize("nmaps", [1, 8])
def test_extreme_maps_cost_little(eps, most, nmaps):
    plan = sh.Plan(256, 512, eps)
    a = coefficients(plan, nmaps)
    maps = plan.synthesize(a)
    t_s, t_a = ms(lambda: plan.synthesize(a)), ms(lambda: plan.adjoint(maps))
    for x in BAD + [2.0 ** -850, 2.0 ** 900]:
        b, f = a * x, maps * x
        assert ms(lambda: plan.synthesize(b)) <= most * t_s + 0.05, x
        assert ms(lambda: plan.adjoint(f)) <= most * t_a + 0.05, x
