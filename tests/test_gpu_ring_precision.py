"""The ring transforms keep FP64's precision ring by ring, also where one value
is far above the others: a bright pixel (adjoint), a strong low order
(synthesis).

Tolerance: an FP64 transform adds about 2^-53 of its points' rms a pass (its
products, sums and rounded roots); up to 9 passes, the fold or unwrap, the
packing and the last rounding are sqrt(12) 2^-53, so 2^-51 as the rms over
many rings.  Rader and Bluestein rings run three transforms: sqrt(3) 2^-51.  A
single ring, of which the shortest have 4 pixels, may reach twice that."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402

NSIDE, LMAX = 256, 520


def prime_factors(n):
    out, p = [], 2
    while n > 1:
        while n % p == 0:
            out.append(p)
            n //= p
        p += 1
    return out


def kind(k):
    """power of two, largest odd radix, or 'long' (Rader and Bluestein)"""
    top = max(prime_factors(k), default=2)
    return "long" if top > 13 else top


@pytest.fixture(scope="module")
def setting():
    n = [min(i, NSIDE, 4 * NSIDE - i) for i in range(1, 4 * NSIDE)]
    return sh.Plan(NSIDE, LMAX, 0.0), oracle.healpix_rings(NSIDE), 4 * np.array(n), np.array(
        [str(kind(2 * i)) for i in n])


def check(err, kinds):
    for k in sorted(set(kinds)):
        e = err[kinds == k]
        tol = 2.0 ** -51 * (3.0 ** 0.5 if k == "long" else 1.0)
        assert np.sqrt(np.mean(e ** 2)) <= tol, k
        assert e.max() <= 2 * tol, k


@pytest.mark.parametrize("contrast", [1.0, 1e3, 1e5, 1e8])
def test_adjoint_of_a_bright_pixel_in_every_ring(setting, contrast):
    plan, rings, J, kinds = setting
    rng = np.random.default_rng(11)
    f = rng.standard_normal(plan.npix)
    starts = np.concatenate([[0], np.cumsum(J)[:-1]])
    f[starts + rng.integers(J)] *= contrast
    want = oracle.phi_adjoint(rings, LMAX, f[None])[0]
    q = torch.empty(1, plan.nrings, LMAX + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_phi_adjoint(plan.handle, torch.from_numpy(f[None]).cuda(), q, 1)
    got = q.cpu().numpy()[0]
    check(np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1), kinds)


@pytest.mark.parametrize("contrast", [1.0, 1e3, 1e5, 1e8])
def test_synthesis_of_a_strong_order(setting, contrast):
    plan, rings, J, kinds = setting
    rng = np.random.default_rng(12)
    q = rng.standard_normal((plan.nrings, LMAX + 1)) + 1j * rng.standard_normal((plan.nrings, LMAX + 1))
    q[:, 1] *= contrast
    q[:, 0].imag = 0
    want = oracle.phi_synth(rings, LMAX, q[None])[0]
    maps = torch.empty(1, plan.npix, dtype=torch.float64, device="cuda")
    sh.shtb_test_phi(plan.handle, torch.from_numpy(q[None]).cuda(), maps, 1)
    got = maps.cpu().numpy()[0]
    ends = np.cumsum(J)
    err = np.array([np.linalg.norm(got[e - j:e] - want[e - j:e]) / np.linalg.norm(want[e - j:e])
                    for e, j in zip(ends, J)])
    check(err, kinds)
