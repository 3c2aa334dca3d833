"""Workloads of the spherical-harmonic transforms, for timing and comparing builds.

Each case is one call (or one differentiation step, or one run of a prepared
batch) through the package's public entry points, at the sizes its
configurations, tests and benchmark use: HEALPix grids with L about 2 Nside,
compressed plans at eps = 1e-10 and 1e-12 and uncompressed ones, one map per
call and many.  `exact` evaluates the definition (Sec. 2.1: one-step Legendre
recurrence, a direct sum over l and a Fourier sum per ring) in 64 bits with
plain torch.
"""
import collections
import math

import torch

import paper_1110_4874_gb300 as sh

# Plans are what a user's program builds once and keeps: the ones used last
# stay here, so that new inputs meet the plan they would meet in earnest.
_MAX_PLANS = 3
_plans = collections.OrderedDict()


def _plan(nside, lmax, eps, spin=0):
    key = (nside, lmax, eps, spin)
    if key not in _plans:
        while len(_plans) >= _MAX_PLANS:
            _plans.popitem(last=False)
        _plans[key] = sh.Plan(nside, lmax, eps, spin=spin, gpu_build=eps > 0)
    _plans.move_to_end(key)
    return _plans[key]


def _case(op, nside, lmax, eps, nmaps, **more):
    return {"op": op, "nside": nside, "lmax": lmax, "eps": eps, "nmaps": nmaps, **more}


def listed():
    return [
        # a quick look at one low-resolution map: launches and latency count
        {"name": "synth_64_1", **_case("synth", 64, 128, 1e-10, 1)},
        # one sky per call at the middle resolution (a sampler's inner step)
        {"name": "synth_512_1", **_case("synth", 512, 1024, 1e-10, 1)},
        # simulations by the batch at the middle resolution
        {"name": "synth_512_8", **_case("synth", 512, 1024, 1e-10, 8)},
        # a grid that is no power of two, tighter tolerance, an odd map count
        {"name": "synth_300_3", **_case("synth", 300, 701, 1e-12, 3)},
        # simulations by the batch at high resolution: the largest
        {"name": "synth_1024_8", **_case("synth", 1024, 2048, 1e-10, 8)},
        # map-making: the transpose of a batch of maps
        {"name": "adjoint_512_8", **_case("adjoint", 512, 1024, 1e-10, 8)},
        # gradient of a pixel-space misfit through the autograd function
        {"name": "grad_1024_4", **_case("grad", 1024, 2048, 1e-10, 4)},
        # uncompressed reference transforms (accuracy checks, small grids)
        {"name": "synth_exact_256_4", **_case("synth", 256, 512, 0.0, 4)},
        {"name": "adjoint_exact_100_1", **_case("adjoint", 100, 255, 0.0, 1)},
        # polarised skies
        {"name": "spin_256_2", **_case("spin", 256, 512, 1e-10, 2)},
        # map analysis with Jacobi refinement
        {"name": "analyze_128_3", **_case("analyze", 128, 256, 1e-10, 3, niter=3)},
        # serving: uneven requests over several plans in one prepared batch
        {"name": "batch_32_256_12", **_case("batch", 256, 512, 1e-10, 12)},
    ]


def draw(rng):
    op = rng.choice(["synth", "synth", "synth", "adjoint", "adjoint", "grad", "exact", "exact_adjoint", "spin",
                     "analyze", "batch"])
    top = {"synth": 800, "adjoint": 800, "grad": 700, "exact": 300, "exact_adjoint": 300, "spin": 300,
           "analyze": 300, "batch": 256}[op]
    nside = int(round(math.exp(rng.uniform(math.log(16), math.log(top)))))
    lmax = max(4, int(nside * rng.uniform(1.5, 2.5)))
    nmaps = rng.choice([1, 1, 2, 3, 4, 5, 8, 8, 11])
    eps = rng.choice([1e-10, 1e-10, 1e-12])
    if op in ("exact", "exact_adjoint"):
        return _case("synth" if op == "exact" else "adjoint", nside, lmax, 0.0, min(nmaps, 4))
    if op == "analyze":
        return _case(op, nside, lmax, eps, min(nmaps, 4), niter=rng.choice([0, 1, 3]))
    if op == "spin":
        return _case(op, nside, lmax, eps, min(nmaps, 4))
    if op == "grad":
        return _case(op, nside, lmax, eps, min(nmaps, 4))
    if op == "batch":
        return _case(op, max(nside, 64), 2 * max(nside, 64), 1e-10, rng.randint(4, 12))
    return _case(op, nside, lmax, eps, min(nmaps, 8) if nside > 500 else nmaps)


# ------------------------------------------------------------------ inputs
def _l_of(lmax, dev):
    m = torch.arange(lmax + 1, device=dev)
    l = torch.arange(lmax + 1, device=dev)
    keep = l[None, :] >= m[:, None]                # [m][l], rows in order give the m-major layout
    return l[None, :].expand(lmax + 1, -1)[keep], m[:, None].expand(-1, lmax + 1)[keep]


def _alm(lmax, shape, gen):
    """Gaussian coefficients with C_l = 1/(l+1)^2, Im a_l0 = 0."""
    l, m = _l_of(lmax, "cuda")
    x = torch.randn(*shape, l.numel(), 2, generator=gen, device="cuda", dtype=torch.float64)
    x *= (math.sqrt(0.5) / (l + 1.0))[:, None]
    x[..., 1] *= m > 0
    return torch.view_as_complex(x)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _requests(case):
    """(nside, maps) of a batch's requests: grids from 1/8 to all of the case's size."""
    out = []
    for i in range(case["nmaps"]):
        out.append((max(16, case["nside"] >> (3 - i % 4)), 1 + (5 * i) % 8))
    return out


class _Batch:
    """A prepared batch and the buffers it is bound to."""

    def __init__(self, plans, alms, maps):
        self.plans, self.alms, self.maps = plans, alms, maps
        self.handle = sh.shtb_batch_create(list(zip(plans, alms, maps)))

    def __del__(self):
        try:
            torch.cuda.synchronize()
            sh.shtb_batch_destroy(self.handle)
        except Exception:
            pass


_batch_plans = {}


def _batch_state(case, gen):
    key = (case["nside"], case["lmax"], case["eps"])
    if key not in _batch_plans:
        _batch_plans.clear()
        _batch_plans[key] = {n: sh.Plan(n, 2 * n, case["eps"], gpu_build=True)
                             for n in sorted({n for n, _ in _requests(case)})}
    plans = _batch_plans[key]
    req = _requests(case)
    alms = [_alm(2 * n, (k,), gen) for n, k in req]
    maps = [torch.empty((k, 12 * n * n), device="cuda", dtype=torch.float64) for n, k in req]
    return {"op": "batch", "batch": _Batch([plans[n] for n, _ in req], alms, maps)}


def prepare(case, seed):
    gen = _gen(seed)
    op, nside, lmax, nmaps = case["op"], case["nside"], case["lmax"], case["nmaps"]
    if op == "batch":
        return _batch_state(case, gen)
    plan = _plan(nside, lmax, case["eps"], 2 if op == "spin" else 0)
    s = {"op": op, "plan": plan}
    npix = 12 * nside * nside
    if op == "synth":
        s["alm"] = _alm(lmax, (nmaps,), gen)
    elif op == "spin":
        a = _alm(lmax, (nmaps, 2), gen)
        l, _ = _l_of(lmax, "cuda")
        s["alm"] = a * (l >= 2)
    elif op in ("adjoint", "analyze"):
        s["map"] = torch.randn(nmaps, npix, generator=gen, device="cuda", dtype=torch.float64)
        s["niter"] = case.get("niter", 0)
    elif op == "grad":
        s["alm"] = _alm(lmax, (nmaps,), gen).requires_grad_()
        s["data"] = 0.1 * torch.randn(nmaps, npix, generator=gen, device="cuda", dtype=torch.float64)
    return s


def run(state):
    op = state["op"]
    if op == "batch":
        sh.shtb_batch_run(state["batch"].handle)
        return state["batch"].maps
    plan = state["plan"]
    if op == "synth":
        return plan.synthesize(state["alm"])
    if op == "spin":
        return plan.synthesize_spin(state["alm"])
    if op == "adjoint":
        return plan.adjoint(state["map"])
    if op == "analyze":
        return plan.analyze(state["map"], niter=state["niter"])
    maps = sh.synthesize(state["alm"], plan)
    loss = 0.5 * (maps - state["data"]).square().sum()
    grad, = torch.autograd.grad(loss, state["alm"])
    return {"maps": maps.detach(), "grad": grad}


# -------------------------------------------------------------------- work
def _operator(nside, lmax, eps):
    """(elements, stored) one pass of the Legendre operator needs: all of it
    uncompressed (recurrence tables, not the elements, are read), about
    L^2 log L compressed."""
    dense = 0.6 * lmax * lmax * nside
    if eps <= 0:
        return dense, 32.0 * lmax * lmax / 2
    n = min(dense, lmax * 2.0 * nside * max(40.0, 160.0 + 70.0 * math.log2(lmax / 1024.0)))
    return n, 8.0 * n


def _work1(nside, lmax, eps, fields, ops):
    elems, stored = _operator(nside, lmax, eps)
    npix, nalm = 12.0 * nside * nside, (lmax + 1) * (lmax + 2) / 2.0
    flops = fields * ops * (4.0 * elems + 2.5 * npix * math.log2(4.0 * nside))
    return {"bytes": ops * stored + fields * ops * (8.0 * npix + 16.0 * nalm), "flops": flops}


def work(case):
    op, nside, lmax, eps, nmaps = (case[k] for k in ("op", "nside", "lmax", "eps", "nmaps"))
    if op == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for n in sorted({n for n, _ in _requests(case)}):
            w = _work1(n, 2 * n, eps, sum(k for q, k in _requests(case) if q == n), 1)
            total = {k: total[k] + w[k] for k in total}
        return total
    if op == "spin":
        w = _work1(nside, lmax, eps, 2 * nmaps, 1)
        elems, stored = _operator(nside, lmax, eps)
        return {"bytes": w["bytes"] + stored, "flops": w["flops"] + 2 * nmaps * 4.0 * elems}
    return _work1(nside, lmax, eps, nmaps, {"grad": 2, "analyze": 1 + 2 * case.get("niter", 0)}.get(op, 1))


# ------------------------------------------------------------------- exact
def _grid(nside):
    """z, sin^2 of the half-rings (z >= 0), north to equator, each from an
    exact integer ratio, and (pixels, half-pixel shift) of every ring."""
    i = torch.arange(1, 2 * nside + 1, device="cuda", dtype=torch.float64)
    polar = i < nside
    d = i * i / (3.0 * nside * nside)                # 1 - z on the polar rings
    z = torch.where(polar, 1.0 - d, (4.0 * nside - 2.0 * i) / (3.0 * nside))
    s2 = torch.where(polar, d * (2.0 - d), 1.0 - z * z)
    rings = []
    for k in range(1, 4 * nside):
        j = min(k, 4 * nside - k)
        rings.append((4 * j, 1) if j < nside else (4 * nside, 1 if (k + nside) % 2 == 0 else 0))
    return z, s2, rings


def _legendre(nside, lmax):
    """Yields (l, Ptilde_l^m, Ptilde_{l-1}^m) for l = 0..lmax as [m <= l][half-ring]."""
    _, s2, _ = _grid(nside)
    i = torch.arange(1, 2 * nside + 1, device="cuda", dtype=torch.float64)
    d = torch.where(i < nside, i * i / (3.0 * nside * nside), (2.0 * i - nside) / (3.0 * nside))     # 1 - z
    m = torch.arange(lmax + 1, device="cuda", dtype=torch.float64)
    k = m.clamp(min=1.0)
    # log2 |P_m^m|, kept as a mantissa and a number of factors 2^-600
    step = torch.where(m > 0, torch.log2((2 * k + 1) / (2 * k)), torch.zeros_like(m))
    lg = 0.5 * (math.log2(1.0 / (4.0 * math.pi)) + torch.cumsum(step, 0))[:, None] + 0.5 * m[:, None] * torch.log2(s2)
    n = torch.floor(-lg / 600.0).clamp(min=0.0)
    start = torch.exp2(lg + 600.0 * n) * (1.0 - 2.0 * (m % 2))[:, None]
    cur, prev = torch.zeros_like(lg), torch.zeros_like(lg)
    down = 2.0 ** -600
    for l in range(lmax + 1):
        if l:
            mm = m[:l]
            al = torch.sqrt((4.0 * l * l - 1.0) / (l * l - mm * mm))[:, None]
            be = torch.sqrt(((l - 1.0) ** 2 - mm * mm).clamp(min=0.0) / max(1.0, 4.0 * (l - 1.0) ** 2 - 1.0))[:, None]
            nxt = al * ((cur[:l] - d * cur[:l]) - be * prev[:l])      # z P as P - (1 - z) P
            prev[:l] = cur[:l]
            cur[:l] = nxt
            if l % 16 == 0:
                big = (cur[:l].abs() > 2.0 ** 300) & (n[:l] > 0)
                cur[:l] = torch.where(big, cur[:l] * down, cur[:l])
                prev[:l] = torch.where(big, prev[:l] * down, prev[:l])
                n[:l] -= big.to(torch.float64)
        cur[l] = start[l]
        on = n[: l + 1] == 0
        yield l, cur[: l + 1] * on, prev[: l + 1] * on


def _index(l, lmax, count):
    m = torch.arange(count, device="cuda")
    return m * (2 * lmax + 1 - m) // 2 + l


def _real(a):
    """[n][nalm] complex -> [2n][nalm] real, pairs (re, im)."""
    return torch.view_as_real(a).movedim(-1, 1).reshape(2 * a.shape[0], -1)


def _complex(x):
    return torch.complex(x[0::2], x[1::2])


def _rings_to_map(qn, qs, nside, lmax):
    """q_m on the north half-rings (equator last) and their mirrors,
    [n][m][half-ring] complex -> maps [n][npix]."""
    _, _, rings = _grid(nside)
    nm = qn.shape[0]
    out = torch.empty(nm, 12 * nside * nside, device="cuda", dtype=torch.float64)
    m = torch.arange(lmax + 1, device="cuda")
    starts, p = [], 0
    for J, _ in rings:
        starts.append(p)
        p += J
    for k, (J, s) in enumerate(rings):
        r = k if k < 2 * nside else len(rings) - 1 - k
        q = (qn if k < 2 * nside else qs)[:, :, r]
        ang = ((m * s) % (2 * J)).to(torch.float64) * (math.pi / J)
        q = q * torch.polar(torch.full_like(ang, 2.0), ang)
        q[:, 0] = 0.5 * q[:, 0].real
        pad = -(lmax + 1) % J
        c = torch.nn.functional.pad(torch.view_as_real(q), (0, 0, 0, pad))
        c = torch.view_as_complex(c.reshape(nm, -1, J, 2).sum(1).contiguous())
        out[:, starts[k]: starts[k] + J] = torch.fft.ifft(c, dim=1).real * J
    return out


def _map_to_rings(f, nside, lmax):
    """The transpose of _rings_to_map: (F north, F south) [n][m][half-ring]."""
    _, _, rings = _grid(nside)
    Z = 2 * nside
    gn = torch.zeros(f.shape[0], lmax + 1, Z, device="cuda", dtype=torch.complex128)
    gs = torch.zeros_like(gn)
    m = torch.arange(lmax + 1, device="cuda")
    p = 0
    for k, (J, s) in enumerate(rings):
        F = torch.fft.fft(f[:, p: p + J], dim=1)[:, m % J]
        ang = ((m * s) % (2 * J)).to(torch.float64) * (math.pi / J)
        F = F * torch.polar(torch.ones_like(ang), -ang)
        (gn if k < Z else gs)[:, :, k if k < Z else len(rings) - 1 - k] = F
        p += J
    return gn, gs


def _synth(alm, nside, lmax):
    a = _real(alm)
    Z = 2 * nside
    qn = torch.zeros(a.shape[0], lmax + 1, Z, device="cuda", dtype=torch.float64)
    qs = torch.zeros_like(qn)
    for l, P, _ in _legendre(nside, lmax):
        al = a[:, _index(l, lmax, l + 1)][:, :, None]
        sg = 1.0 - 2.0 * ((l + torch.arange(l + 1, device="cuda")) % 2).to(torch.float64)[:, None]
        qn[:, : l + 1].addcmul_(al, P)
        qs[:, : l + 1].addcmul_(al, P * sg)
    return _rings_to_map(_complex(qn), _complex(qs), nside, lmax)


def _adjoint(f, nside, lmax):
    gn, gs = _map_to_rings(f, nside, lmax)
    even, odd = gn + gs, gn - gs
    gn, gs = (torch.view_as_real(x).movedim(-1, 1).reshape(2 * f.shape[0], lmax + 1, -1).contiguous()
              for x in (even, odd))
    out = torch.zeros(2 * f.shape[0], (lmax + 1) * (lmax + 2) // 2, device="cuda", dtype=torch.float64)
    for l, P, _ in _legendre(nside, lmax):
        v = torch.empty(out.shape[0], l + 1, device="cuda", dtype=torch.float64)
        for t, g in ((0, gn), (1, gs)):
            k0 = (l + t) % 2
            v[:, k0::2] = torch.einsum("nmr,mr->nm", g[:, k0: l + 1: 2], P[k0::2])
        v[:, 1:] *= 2.0
        v[1::2, 0] = 0.0
        out[:, _index(l, lmax, l + 1)] = v
    return _complex(out)


def _analyze(f, nside, lmax, niter):
    w = 4.0 * math.pi / (12.0 * nside * nside)
    h = torch.full(((lmax + 1) * (lmax + 2) // 2,), 0.5, device="cuda", dtype=torch.float64)
    h[: lmax + 1] = 1.0
    a = h * _adjoint(w * f, nside, lmax)
    for _ in range(niter):
        a = a + h * _adjoint(w * (f - _synth(a, nside, lmax)), nside, lmax)
    return a


def _spin(alm, nside, lmax):
    """Q, U of (E, B) pairs: Q_m = -sum (a_E F+ + i a_B F-), U_m = -sum (a_B F+ - i a_E F-)."""
    n = alm.shape[0]
    aE, aB = _real(alm[:, 0]), _real(alm[:, 1])
    z, s2, _ = _grid(nside)
    q = {k: torch.zeros(2 * n, lmax + 1, 2 * nside, device="cuda", dtype=torch.float64)
         for k in ("Ep", "En", "Bp", "Bn")}
    qs = {k: torch.zeros_like(v) for k, v in q.items()}
    for l, P, P1 in _legendre(nside, lmax):
        if l < 2:
            continue
        m = torch.arange(l + 1, device="cuda", dtype=torch.float64)[:, None]
        nl = 2.0 / math.sqrt((l + 2.0) * (l + 1.0) * l * (l - 1.0))
        lo = torch.sqrt((2.0 * l + 1.0) / (2.0 * l - 1.0) * (l * l - m * m)) * P1
        Fp = nl * (z / s2 * lo - ((l - m * m) / s2 + 0.5 * l * (l - 1.0)) * P)
        Fm = nl * m / s2 * (lo - (l - 1.0) * z * P)
        sg = 1.0 - 2.0 * ((l + torch.arange(l + 1, device="cuda")) % 2).to(torch.float64)[:, None]
        for a, x in ((aE, "E"), (aB, "B")):
            al = a[:, _index(l, lmax, l + 1)][:, :, None]
            q[x + "p"][:, : l + 1].addcmul_(al, Fp)
            q[x + "n"][:, : l + 1].addcmul_(al, Fm)
            qs[x + "p"][:, : l + 1].addcmul_(al, Fp * sg)
            qs[x + "n"][:, : l + 1].addcmul_(al, -Fm * sg)
    out = []
    for d in (q, qs):
        c = {k: _complex(v) for k, v in d.items()}
        out.append((-(c["Ep"] + 1j * c["Bn"]), -(c["Bp"] - 1j * c["En"])))
    Q = _rings_to_map(out[0][0], out[1][0], nside, lmax)
    U = _rings_to_map(out[0][1], out[1][1], nside, lmax)
    return torch.stack([Q, U], dim=1)


def exact(case, seed):
    op, nside, lmax = case["op"], case["nside"], case["lmax"]
    with torch.no_grad():
        if op == "batch":
            gen = _gen(seed)
            return [_synth(_alm(2 * n, (k,), gen), n, 2 * n) for n, k in _requests(case)]
        gen, npix, nmaps = _gen(seed), 12 * nside * nside, case["nmaps"]
        if op == "spin":
            a = _alm(lmax, (nmaps, 2), gen)
            return _spin(a * (_l_of(lmax, "cuda")[0] >= 2), nside, lmax)
        if op in ("adjoint", "analyze"):
            f = torch.randn(nmaps, npix, generator=gen, device="cuda", dtype=torch.float64)
            return _adjoint(f, nside, lmax) if op == "adjoint" else _analyze(f, nside, lmax, case["niter"])
        a = _alm(lmax, (nmaps,), gen)
        maps = _synth(a, nside, lmax)
        if op == "synth":
            return maps
        data = 0.1 * torch.randn(nmaps, npix, generator=gen, device="cuda", dtype=torch.float64)
        return {"maps": maps, "grad": _adjoint(maps - data, nside, lmax)}
