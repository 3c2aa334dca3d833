"""The uncompressed Legendre sums keep FP64's precision for each coefficient and
each ring, whatever the others' sizes: a run of 32 a or g whose sizes differ
much is summed in FP64, others in integers (shtb_legendre.cu).

The reference sums, in extended precision, the values of the same recurrence
that the kernels run (shtb_test_host_recurrence), so that only the sums differ.

Tolerance, against the sum of a result's terms' magnitudes: an FP64 sum of n
products rounds each term by at most n 2^-53, and the factors (sigma, the
halves' sum, the last scaling) by a few 2^-53 more: (n + 8) 2^-53.  The integer
sums cut a or g at 2^-51 of their run's largest or less."""
import numpy as np
import pytest

from paper_1110_4874_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402

NSIDE, LMAX = 150, 260
Z = 2 * NSIDE
ORDERS = [0, 1, 2, 9, 17, 23, 29, 40, 77, 131, 200, 260]
KINDS = ["flat", "polar", "steep", "stairs", "spread", "holes", "ends", "single", "subnormal"]
ULP = 2.0 ** -53


def weights(kind, n, rng):
    """Sizes of n values along a chain (l upwards) or over half-rings (from the pole)"""
    i = np.arange(n)
    if kind == "polar":
        return np.where(i < 3, 1e12, 1.0)
    if kind == "steep":
        return 10.0 ** (-40.0 * (i / n) ** 2)
    if kind == "stairs":                     # runs in integers, in FP64 and in integers again
        lo, hi = (40, 200) if n == Z else (72, 120)
        return 10.0 ** (-14.0 * np.clip((i - lo) / (hi - lo), 0, 1))
    if kind == "ends":                       # ... and in nothing between
        return np.where((i > 40) & (i < n - 20), 0.0, 1.0)
    if kind == "spread":
        return 2.0 ** rng.integers(-60, 61, n)
    if kind == "holes":
        return np.where(i // 7 % 3 == 1, 0.0, 1.0)
    if kind == "single":
        return np.where(i == n // 2, 1.0, 0.0)
    if kind == "subnormal":
        return np.where(i % 2, 1e-310, 1.0) if n % 2 else np.full(n, 1e-310)
    return np.ones(n)


@pytest.fixture(scope="module")
def setting():
    P = {m: np.array([sh.shtb_test_host_recurrence(NSIDE, LMAX, m, r) for r in range(Z)]) for m in ORDERS}
    return sh.Plan(NSIDE, LMAX, 0.0), P                                  # P[m][half-ring][l - m]


def chain(m):
    return slice(int(synthetic.alm_index(LMAX, m, m)), int(synthetic.alm_index(LMAX, LMAX, m)) + 1)


def exact(A, x):
    """A x of a real matrix and a complex vector, in extended precision"""
    A = A.astype(np.longdouble)
    return A @ x.real.astype(np.longdouble) + 1j * (A @ x.imag.astype(np.longdouble))


@pytest.mark.parametrize("kind", KINDS)
def test_each_ring_of_a_synthesis(setting, kind):
    plan, P = setting
    rng = np.random.default_rng(21)
    a = rng.standard_normal((8, plan.nalm)) + 1j * rng.standard_normal((8, plan.nalm))
    for m in range(LMAX + 1):
        a[:, chain(m)] *= weights(kind, LMAX - m + 1, rng)
    a[1:4] = rng.standard_normal((3, plan.nalm)) + 1j * rng.standard_normal((3, plan.nalm))
    a[:, :LMAX + 1].imag = 0
    at = torch.from_numpy(a).cuda()
    q = torch.empty(8, plan.nrings, LMAX + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_legendre(plan.handle, at, q, 8)
    for b in (0, 7):
        got = q[b].cpu().numpy()
        for m in ORDERS:
            c = a[b, chain(m)]
            even, odd = exact(P[m][:, 0::2], c[0::2]), exact(P[m][:, 1::2], c[1::2])
            size, n = np.abs(P[m]) @ np.abs(c), (len(c) + 1) // 2
            tol = (n + 8) * ULP * size + n * 1e-321
            assert np.all(np.abs(got[:Z, m] - (even + odd)) <= tol), m
            assert np.all((np.abs(got[:Z - 1:-1, m] - (even - odd)[:-1]) <= tol[:-1])), m
    for n in (1, 2, 4):                                                  # the same bits at every width
        one = torch.empty_like(q[:n])
        sh.shtb_test_legendre(plan.handle, at[:n].contiguous(), one, n)
        assert torch.equal(one, q[:n])


@pytest.mark.parametrize("kind", KINDS)
def test_each_coefficient_of_an_adjoint(setting, kind):
    plan, P = setting
    rng = np.random.default_rng(22)
    F = rng.standard_normal((8, plan.nrings, LMAX + 1)) + 1j * rng.standard_normal((8, plan.nrings, LMAX + 1))
    w = weights(kind, Z, rng)
    F *= np.concatenate([w, w[-2::-1]])[:, None]
    F[1:4] = rng.standard_normal((3, plan.nrings, LMAX + 1))
    F[..., 0].imag = 0
    Ft = torch.from_numpy(F).cuda()
    out = torch.empty(8, plan.nalm, dtype=torch.complex128, device="cuda")
    sh.shtb_test_legendre_adjoint(plan.handle, Ft, out, 8)
    for b in (0, 7):
        got = out[b].cpu().numpy()
        south = np.zeros((Z, LMAX + 1), dtype=complex)
        south[:-1] = F[b, :Z - 1:-1]
        for m in ORDERS:
            for t, g in enumerate((F[b, :Z, m] + south[:, m], F[b, :Z, m] - south[:, m])):
                cm, R = (1 if m == 0 else 2), P[m][:, t::2].T
                size = cm * (np.abs(R) @ np.abs(g))
                err = np.abs(got[chain(m)][t::2] - cm * exact(R, g))
                assert np.all(err <= (Z + 8) * ULP * size + Z * 1e-321), (m, t)
    for n in (1, 2, 4):
        one = torch.empty_like(out[:n])
        sh.shtb_test_legendre_adjoint(plan.handle, Ft[:n].contiguous(), one, n)
        assert torch.equal(one, out[:n])


@pytest.mark.parametrize("nside", [129, 130, 131, 144])                  # last runs of 2, 4, 6 and 32 rings
def test_adjoint_beside_a_bright_equator(nside):
    """The equator adds nothing to the odd chains: their coefficients stay exact
    beside it.  The even functions have their extremum there."""
    lmax, half = 150, 2 * nside
    plan = sh.Plan(nside, lmax, 0.0)
    rng = np.random.default_rng(23)
    F = rng.standard_normal((2, plan.nrings, lmax + 1)) + 1j * rng.standard_normal((2, plan.nrings, lmax + 1))
    F[0, half - 1] *= 1e12
    F[..., 0].imag = 0
    out = torch.empty(2, plan.nalm, dtype=torch.complex128, device="cuda")
    sh.shtb_test_legendre_adjoint(plan.handle, torch.from_numpy(F).cuda(), out, 2)
    for b in (0, 1):
        got = out[b].cpu().numpy()
        south = np.zeros((half, lmax + 1), dtype=complex)
        south[:-1] = F[b, :half - 1:-1]
        for m in (0, 1, 5, 40, 100, 150):
            P = np.array([sh.shtb_test_host_recurrence(nside, lmax, m, r) for r in range(half)])
            at = int(synthetic.alm_index(lmax, m, m))
            for t, g in enumerate((F[b, :half, m] + south[:, m], F[b, :half, m] - south[:, m])):
                cm, R = (1 if m == 0 else 2), P[:, t::2].T
                size = cm * (np.abs(R) @ np.abs(g))
                err = np.abs(got[at:at + lmax - m + 1][t::2] - cm * exact(R, g))
                assert np.all(err <= (half + 8) * ULP * size), (b, m, t)
