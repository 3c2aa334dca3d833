"""The butterfly's block products (shtb_bf_fix.cuh) against sums of the same
elements in extended precision.  Plans of depth 0 apply their residual blocks
and nothing else, and unit inputs show the blocks' elements themselves.

Tolerance: 2^-52 max|T| max|v| sqrt(k) for a chunk of k entries.  Per product the
vector's cut (2^-56 of max|v| at most), the digit diagonals left out (2^-57 of
max|T| max|v| rms) and, once, the last rounding make about 2^-55 sqrt(k) rms; the
lowest diagonal that is kept is worth 2^-47 or more, so losing it fails."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_4874_gb300 as sh  # noqa: E402
from paper_1110_4874_gb300 import synthetic  # noqa: E402

L, CHUNK, ULP2 = 70, 32, 2.0 ** -52


def chain(m):
    return slice(int(synthetic.alm_index(L, m, m)), int(synthetic.alm_index(L, L, m)) + 1)


def legendre(plan, a):
    q = torch.empty(a.shape[0], 2, 2 * plan.nside, L + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_butterfly(plan.handle, torch.from_numpy(a).cuda(), q, a.shape[0])
    return q.cpu().numpy()


class Operator:
    """R[m][t]: [half-ring][chain row] as the plan holds it"""
    def __init__(self, nside, leaf):
        self.plan = sh.Plan(nside, L, 1e-10, max_depth=0, leaf_cols=leaf)
        unit = np.zeros((L + 1, self.plan.nalm), dtype=complex)
        for m in range(L + 1):
            unit[np.arange(L + 1 - m), np.arange(chain(m).start, chain(m).stop)] = 1.0
        q = legendre(self.plan, unit).real
        self.R = [[q[t:L + 1 - m:2, t, :, m].T.copy() for t in (0, 1)] for m in range(L + 1)]


@pytest.fixture(scope="module")
def operators():
    made = {}

    def get(nside, leaf):
        if (nside, leaf) not in made:
            made[nside, leaf] = Operator(nside, leaf)
        return made[nside, leaf]
    return get


def vector(kind, shape, rng):
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    if kind == "spread":
        x *= 2.0 ** rng.integers(-40, 41, shape)
    elif kind == "peak":
        x[..., ::11] *= 1e8
    return x


def exact(R, x):
    R = R.astype(np.longdouble)
    return R @ x.real.astype(np.longdouble), R @ x.imag.astype(np.longdouble)


# chains of 1 to 36 rows against blocks of 7 to 33 columns
@pytest.mark.parametrize("nside,leaf", [(16, 7), (16, 8), (16, 16), (16, 17), (16, 32), (33, 33)])
@pytest.mark.parametrize("kind", ["flat", "spread", "peak"])
@pytest.mark.parametrize("nmaps", [1, 2, 4, 8])
def test_synthesis_blocks(operators, nside, leaf, kind, nmaps):
    op = operators(nside, leaf)
    a = vector(kind, (nmaps, op.plan.nalm), np.random.default_rng(31))
    a[:, :L + 1].imag = 0
    got = legendre(op.plan, a)
    for b in {0, nmaps - 1}:
        for m in range(L + 1):
            for t in (0, 1):
                R, x = op.R[m][t], a[b, chain(m)][t::2]
                if R.shape[1] == 0:
                    continue
                tol = np.zeros(len(R))
                for k0 in range(0, len(x), CHUNK):
                    c, v = R[:, k0:k0 + CHUNK], x[k0:k0 + CHUNK]
                    big = max(np.abs(v.real).max(), np.abs(v.imag).max())
                    tol += ULP2 * np.sqrt(len(v)) * np.abs(R).max(1) * big
                re, im = exact(R, x)
                assert np.all(np.abs(got[b, t, :, m].real - re) <= tol), (m, t)
                assert np.all(np.abs(got[b, t, :, m].imag - im) <= tol), (m, t)


@pytest.mark.parametrize("nside,leaf", [(16, 7), (16, 8), (16, 16), (16, 17), (16, 32), (33, 33)])
@pytest.mark.parametrize("nmaps", [1, 2, 4, 8])
def test_adjoint_blocks(operators, nside, leaf, nmaps):
    op = operators(nside, leaf)
    plan, Z = op.plan, 2 * nside
    f = torch.from_numpy(np.random.default_rng(32).standard_normal((nmaps, plan.npix))).cuda()
    F = torch.empty(nmaps, plan.nrings, L + 1, dtype=torch.complex128, device="cuda")
    sh.shtb_test_phi_adjoint(plan.handle, f, F, nmaps)
    F, got = F.cpu().numpy(), plan.adjoint(f).cpu().numpy()
    chunks = sum(-(-min(leaf, Z - s) // CHUNK) for s in range(0, Z, leaf))
    for b in {0, nmaps - 1}:
        south = np.zeros((Z, L + 1), dtype=complex)
        south[:-1] = F[b, :Z - 1:-1]
        for m in range(L + 1):
            for t, g in enumerate((F[b, :Z, m] + south[:, m], F[b, :Z, m] - south[:, m])):
                R, cm = op.R[m][t], (1 if m == 0 else 2)
                if R.shape[1] == 0:
                    continue
                big = (np.abs(R).max(1) * np.maximum(np.abs(g.real), np.abs(g.imag))).max()
                tol = cm * ULP2 * chunks * np.sqrt(min(leaf, CHUNK)) * big
                re, im = exact(R.T, g)
                out = got[b, chain(m)][t::2]
                assert np.all(np.abs(out.real - cm * re) <= tol), (m, t)
                if m:
                    assert np.all(np.abs(out.imag - cm * im) <= tol), (m, t)
