"""The ring stage in 64-bit fixed point (shtb_phi_items.cuh): every transform
kind and radix, flat and peaked spectra, the ends of the exponent range, zero
rings, infinities and NaN."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402


def spectrum(plan, kind, seed):
    rng = np.random.default_rng(seed)
    L = plan.lmax
    q = rng.standard_normal((2, plan.nrings, L + 1)) + 1j * rng.standard_normal((2, plan.nrings, L + 1))
    if kind == "steep":
        q *= 10.0 ** (-12.0 * np.arange(L + 1) / max(L, 1))
    elif kind == "peak":
        q *= 1e-9
        q[..., min(3, L)] = 1.0
    q[..., 0].imag = 0
    return q


# L = 2 Nside gives ring lengths J = 4i: halves 2i over every radix (2 .. 13),
# Rader primes, Bluestein lengths; 1 and 2 are the shortest transforms
@pytest.mark.parametrize("nside,lmax", [(1, 2), (2, 9), (13, 26), (30, 200), (47, 94), (64, 40), (105, 230)])
@pytest.mark.parametrize("kind", ["flat", "steep", "peak"])
def test_ring_transforms_match_the_oracle(nside, lmax, kind):
    """Relative rms below 1e-15: the tables and the fold's FP64 sums are
    rounded to 2^-53 and each fixed-point pass adds a few 2^-58 of the ring's
    largest point, so a few 1e-16 are expected."""
    plan = sh.Plan(nside, lmax, 0.0)
    rings = oracle.healpix_rings(nside)
    q = spectrum(plan, kind, 3)
    want = oracle.phi_synth(rings, lmax, q)
    maps = torch.empty(2, plan.npix, dtype=torch.float64, device="cuda")
    sh.shtb_test_phi(plan.handle, torch.from_numpy(q).cuda(), maps, 2)
    assert np.linalg.norm(maps.cpu().numpy() - want) <= 1e-15 * np.linalg.norm(want)
    want_q = oracle.phi_adjoint(rings, lmax, want)
    back = torch.empty(2, plan.nrings, lmax + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_phi_adjoint(plan.handle, torch.from_numpy(want).cuda(), back, 2)
    assert np.linalg.norm(back.cpu().numpy() - want_q) <= 1e-15 * np.linalg.norm(want_q)


def test_scales_zero_rings_and_non_finite_values():
    nside, lmax = 21, 50
    plan = sh.Plan(nside, lmax, 0.0)
    q = torch.from_numpy(spectrum(plan, "steep", 4)).cuda()
    maps = torch.empty(2, plan.npix, dtype=torch.float64, device="cuda")

    def synth(x):
        out = torch.empty_like(maps)
        sh.shtb_test_phi(plan.handle, x.contiguous(), out, 2)
        return out

    def adjoint(f):
        out = torch.empty_like(q)
        sh.shtb_test_phi_adjoint(plan.handle, f.contiguous(), out, 2)
        return out

    base = synth(q)
    back = adjoint(base)
    for p in (2.0 ** -600, 2.0 ** 600):                  # powers of two only move the exponent
        assert torch.equal(synth(q * p), base * p)
        assert torch.equal(adjoint(base * p), back * p)
    for p in (2.0 ** -950, 2.0 ** 1000):                 # the direct FP64 sum: 2 (L + 1) roundings at most
        assert float((synth(q * p) / p - base).norm() / base.norm()) <= 2 * (lmax + 1) * 2.0 ** -53
    z = q.clone()
    z[0, 5] = 0                                          # one ring of zeros
    got = synth(z)
    start = sum(4 * min(i, nside) for i in range(1, 6))
    ring = slice(start, start + 4 * 6)
    assert torch.count_nonzero(got[0, ring]) == 0
    keep = torch.ones(plan.npix, dtype=torch.bool)
    keep[ring] = False
    assert torch.equal(got[0, keep], base[0, keep]) and torch.equal(got[1], base[1])
    for bad in (float("nan"), float("inf")):
        z = q.clone()
        z[0, 5, 2] = complex(bad, 0.0)                   # only its own ring
        got = synth(z)
        assert not torch.isfinite(got[0, ring]).any()
        assert torch.equal(got[0, keep], base[0, keep]) and torch.equal(got[1], base[1])
        f = base.clone()
        f[1, start] = bad
        ab = adjoint(f)
        assert not torch.isfinite(torch.view_as_real(ab[1, 5])).all()
        rest = [i for i in range(plan.nrings) if i != 5]
        assert torch.equal(ab[1, rest], back[1, rest]) and torch.equal(ab[0], back[0])


@pytest.mark.parametrize("nside", [768, 769])
def test_rings_at_the_line_between_block_sizes(nside):
    """Longest rings of 4 x 768 pixels run 128 threads a block, longer ones
    256; the bound is that of the transforms above."""
    lmax = 24
    plan = sh.Plan(nside, lmax, 0.0)
    rings = oracle.healpix_rings(nside)
    q = spectrum(plan, "flat", 5)
    want = oracle.phi_synth(rings, lmax, q)
    maps = torch.empty(2, plan.npix, dtype=torch.float64, device="cuda")
    sh.shtb_test_phi(plan.handle, torch.from_numpy(q).cuda(), maps, 2)
    assert np.linalg.norm(maps.cpu().numpy() - want) <= 1e-15 * np.linalg.norm(want)
    want_q = oracle.phi_adjoint(rings, lmax, want)
    back = torch.empty(2, plan.nrings, lmax + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_phi_adjoint(plan.handle, torch.from_numpy(want).cuda(), back, 2)
    assert np.linalg.norm(back.cpu().numpy() - want_q) <= 1e-15 * np.linalg.norm(want_q)
