"""What a user of the sampler has it do, as measurable cases: field draws over the range of grids,
spectra, precisions and outputs that the workloads, tests and benchmark use, a batch of uneven
requests, HEALPix grids, and plans made for one draw.

listed() gives the cases, draw(rng) more of the same ranges, prepare() what a program holds before
the call (plans, seeds, output buffers), run() one pass, work() the bytes and operations it cannot
do without, exact() the same field in 64 bits from the method's equations (Creasey & Lang, arXiv
1709.10314), in plain torch."""
import math
import random

import numpy as np
import torch

from paper_1709_10314_gb300 import (SMERF_ORDER_PAPER, SMERF_RECUR_FP64, SMERF_TABLES_FP32, SMERF_TABLES_FP64, Batch,
                                    Plan, create_plans)

# Spectrum factors kappa of the repository's workloads for p = 1, 2, 3
KAPPA = {1: (100.0,), 2: (20.0, 50.0), 3: (20.0, 50.0, 120.0)}


def _case(name, kind, n_theta, n_phi, p, n, recur="fp32", tables="fp64", H=0, paper=False, **more):
    c = dict(kind=kind, n_theta=n_theta, n_phi=n_phi, p=p, n=n, recur=recur, tables=tables, H=H, paper=paper, **more)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the plain method: one FP64 realisation of a small grid in Alg. 2's order (a unit test, a
        # notebook, a single draw inside another program's loop): the smallest call
        _case("plain-64x128-fp64", "field", 64, 128, 1, 1, recur="fp64", paper=True, kappa1=10.0),
        # one realisation on one-degree latitudes (an odd ring count): a stochastic-forcing or
        # ensemble-perturbation step that draws one field per call
        _case("single-181x512-p2", "field", 181, 512, 2, 1, tables="fp32"),
        # the paper's simulation example (Sec. 5): many FP64 realisations of a tiny grid with the
        # complex kappa-hat spectrum 1/(10 + l^2 (l+1)^2), for Monte-Carlo covariances
        _case("sec5-32x64-fp64", "field", 32, 64, 2, 20001, recur="fp64", khat=True),
        # the throughput workload: 64 realisations, FP64 tables, FP32 recursion
        _case("ensemble-1024x2048-p2", "field", 1024, 2048, 2, 64),
        # the same grid and spectrum in the FP64 recursion mode (reference runs, precision studies)
        _case("ensemble-1024x2048-p2-fp64", "field", 1024, 2048, 2, 16, recur="fp64"),
        # three spectrum factors
        _case("ensemble-1024x2048-p3", "field", 1024, 2048, 3, 64),
        # the precision-sweep grid
        _case("ensemble-4096x8192-p1", "field", 4096, 8192, 1, 16),
        # the large single grid, the benchmark's default: the largest call
        _case("large-16384x32768-p1", "field", 16384, 32768, 1, 4, tables="fp32", H=24, kappa1=300.0),
        # a service's uneven batch: 256 requests of different grids, spectra and counts in one call
        _case("uneven-batch-256", "batch", 0, 0, 0, 256),
        # HEALPix (Nside 128: 511 rings of 4 to 512 points): the grid of sky maps
        _case("healpix-128-p1", "healpix", 511, 512, 1, 16, tables="fp32"),
        # a spectrum that changes from draw to draw (parameter inference): plan, then one field
        _case("newplan-1024x2048-p2", "newplan", 1024, 2048, 2, 1),
        # the field into page-locked host memory, for a consumer on the CPU
        _case("host-1024x2048-p2", "host", 1024, 2048, 2, 16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["field"] * 7 + ["batch", "healpix", "healpix", "newplan", "host"])
    if kind == "batch":
        return _case(None, "batch", 0, 0, 0, rng.randint(20, 256), gen=rng.randrange(1 << 20))
    if kind == "healpix":
        nside = _log_int(rng, 3, 256)
        n_phi = 8
        while n_phi < 4 * nside:
            n_phi *= 2
        p = rng.choice([1, 1, 2])
        n = max(1, min(64, _log_int(rng, 1, 2e7 / (12 * nside * nside))))
        return _case(None, "healpix", 4 * nside - 1, n_phi, p, n, recur=rng.choice(["fp32", "fp32", "fp64"]), tables="fp32")
    if kind == "newplan":
        lg = rng.randint(6, 12)
        return _case(None, "newplan", _log_int(rng, 2 ** (lg - 2), 2 ** lg), 2 ** lg, rng.choice([1, 2]), rng.randint(1, 4),
                     tables=rng.choice(["fp64", "fp32"]))
    lg = rng.randint(6, 15)
    n_theta = _log_int(rng, max(9, 2 ** (lg - 3)), 2 ** (lg - 1) + 1)
    p = rng.choice([1, 2] if lg > 12 else [1, 2, 3])
    if p == 2:
        n_theta = min(n_theta, 2 ** 13 - 1)
    recur = "fp64" if lg <= 13 and rng.random() < 0.3 else "fp32"
    most = 3e7 if recur == "fp64" else 4e8
    n = max(1, min(2000, _log_int(rng, 1, max(1.0, most / (n_theta * 2 ** lg)))))
    return _case(None, kind, n_theta, 2 ** lg, p, n, recur=recur, tables=rng.choice(["fp64", "fp32"]),
                 H=rng.choice([0, 0, 0, 12, 24]), paper=n_theta < 200 and rng.random() < 0.2)


# ------------------------------------------------------------------ inputs
def _key(seed):
    """The Philox key of a case's first realisation."""
    return (int(seed) * 0x9E3779B97F4A7C15 + 12345) & (2 ** 62 - 1)


def _spectrum(case, seed):
    """kappa-hat values of the case (kappa squared, or Sec. 5's complex pair)."""
    if case.get("khat"):
        return [1j * 10 ** 0.5, -1j * 10 ** 0.5]
    kappa = list(KAPPA[case["p"]])
    if "kappa1" in case:
        kappa[0] = case["kappa1"]
    if case["kind"] == "newplan":  # the next proposal of an inference run
        rng = random.Random(int(seed))
        kappa = [k * math.exp(rng.uniform(-0.1, 0.1)) for k in kappa]
    return [k * k for k in kappa]


def _flags(case):
    return ((SMERF_RECUR_FP64 if case["recur"] == "fp64" else 0) | (SMERF_ORDER_PAPER if case["paper"] else 0) |
            (SMERF_TABLES_FP64 if case["tables"] == "fp64" else SMERF_TABLES_FP32))


def _healpix(nside):
    """Colatitude, point count and first longitude of the rings (Gorski et al. 2005)."""
    th, n, phi0 = [], [], []
    for k in range(1, 4 * nside):
        i = min(k, 4 * nside - k)
        if i < nside:
            z, m, p0 = 1 - i * i / (3.0 * nside * nside), 4 * i, math.pi / (4 * i)
        else:
            z, m, p0 = 4 / 3 - 2 * i / (3.0 * nside), 4 * nside, math.pi / (4 * nside) * ((i - nside + 1) % 2)
        t = math.acos(z)
        th.append(t if k <= 2 * nside else math.pi - t)
        n.append(m)
        phi0.append(p0)
    th[2 * nside - 1] = 0.5 * math.pi
    return th, n, phi0


def _requests(case, seed):
    """The uneven batch: grids of 128 to 1024 rings, p 1 or 2, 1 to 8 realisations each."""
    rng = random.Random(case.get("gen", 12345))
    reqs = []
    for i in range(case["n"]):
        n_theta, p = rng.choice([128, 256, 512, 1024]), rng.choice([1, 2])
        kappa = sorted(rng.uniform(5.0, 200.0) for _ in range(p))
        if p == 2 and kappa[1] ** 2 - kappa[0] ** 2 < 1e-3 * kappa[1] ** 2:
            kappa[1] *= 1.01
        reqs.append(dict(kappa=kappa, A=1.0, n_theta=n_theta, n_phi=2 * n_theta, n=rng.randint(1, 8),
                         seed=(_key(seed) + 1000 * i) & (2 ** 62 - 1)))
    return reqs


def _plan(case, seed):
    kh = _spectrum(case, seed)
    th = _healpix((case["n_theta"] + 1) // 4) if case["kind"] == "healpix" else None
    args = dict(A=1.0, n_theta=case["n_theta"], n_phi=case["n_phi"], flags=_flags(case), anchor_spacing=case["H"])
    if case.get("khat"):
        return Plan(khat=kh, **args)
    plan = Plan([math.sqrt(v) for v in kh], theta=th[0] if th else None, **args)
    if th:
        plan.set_rings(th[1], th[2])
    return plan


def prepare(case, seed):
    state = dict(kind=case["kind"], n=case["n"], seed=_key(seed))
    if case["kind"] == "batch":
        reqs = _requests(case, seed)
        plans = create_plans(reqs)
        counts = [q["n"] for q in reqs]
        sizes = [p.points * n for p, n in zip(plans, counts)]
        out = torch.empty(sum(sizes), device="cuda")
        views = [v.view(n, p.n_theta, p.n_phi) for v, n, p in zip(out.split(sizes), counts, plans)]
        return dict(state, batch=Batch(plans, counts), seeds=[q["seed"] for q in reqs], views=views, out=out)
    if case["kind"] == "newplan":
        return dict(state, case=case, proposal=seed)
    plan = _plan(case, seed)
    if case["kind"] == "host":
        out = torch.empty(case["n"], case["n_theta"], case["n_phi"], dtype=plan.dtype, pin_memory=True)
    elif case["n"] * plan.points > 1 << 24:  # a program keeps its large fields' buffer
        shape = (case["n"], plan.points) if plan.ring_points else (case["n"], case["n_theta"], case["n_phi"])
        out = torch.empty(shape, dtype=plan.dtype, device="cuda")
    else:
        out = None
    return dict(state, plan=plan, out=out)


def run(state):
    if state["kind"] == "batch":
        state["batch"].sample(state["seeds"], state["views"])
        # the next request set waits for this one's (the staging memory is one set of descriptors)
        torch.cuda.current_stream().synchronize()
        return state["out"]
    if state["kind"] == "newplan":
        plan = _plan(state["case"], state["proposal"])
        out = plan.sample(state["seed"], state["n"])
        torch.cuda.current_stream().synchronize()  # before the plan goes
        plan.close()
        return out
    if state["kind"] == "host":
        return state["plan"].sample_host(state["seed"], state["n"], out=state["out"])
    return state["plan"].sample(state["seed"], state["n"], out=state["out"])


def work(case):
    """Field written once, tables A and B read once (p^2 + p (p+1) / 2 values per mode and ring, in
    the recursion's type; written once where the plan is made); noise, recursion and FFT operations
    of every mode, realisation and ring."""
    if case["kind"] == "batch":
        per = [dict(case, kind="field", n_theta=q["n_theta"], n_phi=q["n_phi"], p=len(q["kappa"]), n=q["n"])
               for q in _requests(case, 0)]
        w = [work(c) for c in per]
        return {"bytes": sum(v["bytes"] for v in w), "flops": sum(v["flops"] for v in w)}
    p, n, nc = case["p"], case["n"], case["n_phi"] // 2
    size = 8 if case["recur"] == "fp64" else 4
    points = case["n_theta"] * case["n_phi"]
    if case["kind"] == "healpix":
        points = sum(_healpix((case["n_theta"] + 1) // 4)[1])
    entries = p * p + p * (p + 1) // 2
    ops = 20 * p + 12 * p + 2 * entries + 10 + 3.5 * math.log2(nc)
    return {"bytes": size * (n * points + case["n_theta"] * nc * entries), "flops": ops * n * case["n_theta"] * nc}


# ------------------------------------------------------------------ the same in 64 bits
def _hyp(k2, mu, x):
    """2F1(-l, l+1; 1+mu; x), -l (l+1) = k2, by its series (mu and x broadcast)."""
    t = torch.ones(torch.broadcast_shapes(mu.shape, x.shape), dtype=torch.complex128 if isinstance(k2, complex) else torch.float64,
                   device=x.device)
    s = t.clone()
    for n in range(100000):
        t = t * ((n * (n + 1) + k2) * x / ((n + 1 + mu) * (n + 1)))
        s = s + t
        if n % 16 == 15 and bool((t.abs() <= 1e-18 * s.abs()).all()):
            return s
    raise ArithmeticError("the series does not end")


def _hmat(kh, m, x):
    """H_{q,i} = prod_{j=m}^{m+q-1} (j(j+1) + kh_i)/(j+1) F^i_{m+q}(x) / F^i_m(x): P^{m+q} / P^m without t^q."""
    M = len(kh)
    cols = []
    for k in kh:
        f0 = _hyp(k, m, x)
        r, col = torch.ones_like(m), [torch.ones_like(f0)]
        for q in range(1, M):
            j = m + q - 1
            r = r * ((j * (j + 1) + k) / (j + 1))
            col.append(r * _hyp(k, m + q, x) / f0)
        cols.append((torch.stack(col, -1), f0))
    return torch.stack([c for c, _ in cols], -1), torch.stack([f for _, f in cols], -1)


def _steps(kh, m, th):
    """Transition Phi and conditional covariance Q of the steps th[0] -> th[1] -> ... toward the
    pole (Eqs. (trans_matrix), (innov_matrix)): Phi = U(z2) U(z1)^-1 and Q the integral of the driven
    last component's responses, U the solutions regular at that pole."""
    M, dev = len(kh), m.device
    gx, gw = (torch.as_tensor(v, device=dev) for v in np.polynomial.legendre.leggauss(16))
    powers = torch.arange(M, device=dev, dtype=torch.float64)
    kmax = max(abs(k) for k in kh) ** 0.5
    phi, cov = [], []
    a = 0
    while a < len(th) - 1:
        u = [math.log(math.tan(0.5 * t)) for t in th[a:a + 2]]
        rho = 2 * (m + M - 1) + 2 * kmax * math.sin(th[a]) + 1
        panels = int(math.ceil(float((torch.minimum(torch.full_like(m, u[0] - u[1]), 46 / (2 * m + 1e-9)) * rho).max()) / 8)) + 1
        b = min(len(th) - 1, a + max(1, int(6e6 / (panels * 16 * len(m)))))
        t = torch.as_tensor(th[a:b + 1], device=dev, dtype=torch.float64)
        u = torch.log(torch.tan(0.5 * t))
        x = torch.sin(0.5 * t) ** 2
        H1, F1 = _hmat(kh, m, x[:-1, None])
        H2, F2 = _hmat(kh, m, x[1:, None])
        du = (u[:-1] - u[1:])[:, None]
        scale = F2 / F1  # column i of U(z2) U(z1)^-1
        t1, t2 = torch.exp(u[:-1])[:, None, None], torch.exp(u[1:])[:, None, None]
        A = (H2 * scale[..., None, :]) @ torch.linalg.inv(H1)
        phi.append((A * (t2 ** powers)[..., :, None] / (t1 ** powers)[..., None, :]).real * torch.exp(-m * du)[..., None, None])
        V = torch.minimum(du, 46 / (2 * m + 1e-9))  # the weight (t2 / t)^2m ends the integral
        Q = 0.0
        for j in range(panels):
            v = V[:, None, :] * ((j + 0.5 * (gx + 1)) / panels)[None, :, None]  # [step, node, mode]
            w = V[:, None, :] * (0.5 * gw / panels)[None, :, None]
            ts = torch.exp(u[1:, None, None] + v)
            Hs, Fs = _hmat(kh, m, ts * ts / (1 + ts * ts))
            e = torch.zeros(M, 1, device=dev, dtype=Hs.dtype)
            e[M - 1] = 1
            h = torch.linalg.solve(Hs, e.expand(*Hs.shape[:-1], 1)) * (F2[:, None] / Fs)[..., None]
            f = (H2[:, None] @ h)[..., 0].real * (torch.exp(u[1:])[:, None, None, None] ** powers) / ts[..., None] ** (M - 1)
            w = w * torch.exp(-2 * m * v)
            Q = Q + torch.einsum("snm,snmp,snmq->smpq", w, f, f)
        cov.append(Q / (2 * math.pi))
        a = b
    if not phi:
        z = torch.zeros(0, len(m), M, M, device=dev, dtype=torch.float64)
        return z, z
    return torch.cat(phi), torch.cat(cov)


def _start(kh, m, th):
    """Covariance of the state at the start ring (Eq. (Jmatrix_efficient)): partial fractions of
    Green's functions, whose Wronskian comes from P^{m+1} / P^m on both sides."""
    M = len(kh)
    t, x = math.tan(0.5 * th), torch.tensor(math.sin(0.5 * th) ** 2, device=m.device, dtype=torch.float64)
    if M == 1:
        pad = lambda h, k, y: torch.stack([torch.ones_like(m), (m * (m + 1) + k) / (m + 1) * _hyp(k, m + 1, y) / _hyp(k, m, y)], -1)  # noqa: E731
        north, south = [pad(None, kh[0], x)], [pad(None, kh[0], 1 - x)]
    else:
        Hn, Hs = _hmat(kh, m, x)[0], _hmat(kh, m, 1 - x)[0]
        north, south = [Hn[..., i] for i in range(M)], [Hs[..., i] for i in range(M)]
    J = 0.0
    for i, k in enumerate(kh):
        b = 1.0
        for j, k2 in enumerate(kh):
            b = b / (k2 - k) if j != i else b
        n = north[i] * torch.tensor([t ** q for q in range(north[i].shape[-1])], device=m.device, dtype=torch.float64)
        s = south[i] * torch.tensor([(-1 / t) ** q for q in range(north[i].shape[-1])], device=m.device, dtype=torch.float64)
        g = b / (2 * math.pi * math.sin(th) * (n[..., 1] - s[..., 1]))
        J = J + g[..., None, None] * n[..., :M, None] * s[..., None, :M]
    J = J.real if torch.is_tensor(J) and J.is_complex() else J
    return 0.5 * (J + J.mT)


def _chol(S):
    """Lower Cholesky factors of covariances of any scale (0 where one is below 1e-250)."""
    M = S.shape[-1]
    L = torch.zeros_like(S)
    for j in range(M):
        d = S[..., j, j] - (L[..., j, :j] ** 2).sum(-1)
        ok = d > 1e-250
        r = torch.sqrt(torch.where(ok, d, torch.ones_like(d)))
        L[..., j, j] = torch.where(ok, r, torch.zeros_like(d))
        for i in range(j + 1, M):
            s = S[..., i, j] - (L[..., i, :j] * L[..., j, :j]).sum(-1)
            L[..., i, j] = torch.where(ok, s / r, torch.zeros_like(d))
    return L


def _normals(key, n, ring, per, dev):
    """[n][per] normals of rings' Philox4x32-10 calls (j, ring, 0, 0) under keys key + r, Box-Muller."""
    mask = 0xFFFFFFFF

    def mul(c, k):  # 32 x 32 -> (high, low), the factors below 2^32
        lo = (c & 0xFFFF) * k
        hi = (c >> 16) * k + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    calls = (per + 3) // 4
    keys = [(key + r) & (2 ** 64 - 1) for r in range(n)]
    k0 = torch.tensor([k & mask for k in keys], device=dev)[:, None, None]
    k1 = torch.tensor([k >> 32 for k in keys], device=dev)[:, None, None]
    c = [torch.arange(calls, device=dev)[None, None, :], ring[None, :, None], torch.zeros(1, 1, 1, dtype=torch.int64, device=dev),
         torch.zeros(1, 1, 1, dtype=torch.int64, device=dev)]
    for r in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ ((k0 + r * 0x9E3779B9) & mask), l1, h0 ^ c[3] ^ ((k1 + r * 0xBB67AE85) & mask), l0]
    c = [v.expand(n, len(ring), calls).double() for v in c]
    out = []
    for a, b in ((c[0], c[1]), (c[2], c[3])):
        rad, ang = torch.sqrt(-2 * torch.log((a + 0.5) * 2.0 ** -32)), 2 * math.pi * ((b + 0.5) * 2.0 ** -32)
        out += [rad * torch.cos(ang), rad * torch.sin(ang)]
    return torch.stack(out, -1).reshape(n, len(ring), -1)[..., :per]


def _field(kh, theta, n_phi, H, key, n):
    """Modes g [n][ring][n_phi/2 + 1] (complex; the last one's real part is the Nyquist chain)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    M, n_theta, Nc = len(kh), len(theta), n_phi // 2
    k0 = n_theta // 2
    m = torch.arange(Nc + 1, device=dev, dtype=torch.float64)
    half = torch.where(m > 0, 0.5, 1.0).double().sqrt()[:, None, None]  # the Re and Im chains share the variance
    sign = torch.tensor([(-1.0) ** q for q in range(M)], device=dev, dtype=torch.float64)
    g = torch.zeros(n, n_theta, Nc + 1, dtype=torch.complex128, device=dev)

    def noise(rings):  # [ring][n][mode][part][M]: slot s is mode s, slot 0 the m = 0 and Nyquist chains
        v = _normals(key, n, rings, 2 * M * Nc, dev).view(n, len(rings), Nc, 2, M).transpose(0, 1)
        full = torch.zeros(len(rings), n, Nc + 1, 2, M, dtype=torch.float64, device=dev)
        full[:, :, :Nc] = v
        full[:, :, Nc, 0] = v[:, :, 0, 1]
        full[:, :, 0, 1] = 0
        return full

    def put(rings, x):
        g[:, rings] = torch.complex(x[..., 0, 0], x[..., 1, 0]).transpose(0, 1)

    def mv(T, x):  # [.., mode, M, M] x [.., n, mode, part, M]
        return torch.einsum("...mpq,...nmcq->...nmcp", T, x)

    at = lambda ks: torch.as_tensor(ks, device=dev, dtype=torch.int64)  # noqa: E731
    x0 = mv(_chol(_start(kh, m, theta[k0])) * half, noise(at([k0]))[0])
    put(at([k0]), x0[None])
    for c in (0, 1):
        ks = list(range(k0, -1, -1)) if c == 0 else list(range(k0, n_theta))
        phi, Q = _steps(kh, m, [theta[k] if c == 0 else math.pi - theta[k] for k in ks])
        flip = torch.ones_like(sign) if c == 0 else sign
        length = len(ks) - 1
        na = length // H if H else 0
        x = x0 * flip
        anchors = [x]
        eye = torch.eye(M, device=dev, dtype=torch.float64).expand(Nc + 1, M, M)
        if na:
            P = phi[:na * H].view(na, H, Nc + 1, M, M)
            C = Q[:na * H].view(na, H, Nc + 1, M, M)
            psi, S, bridge = eye.expand(na, Nc + 1, M, M), torch.zeros_like(P[:, 0]), [None] * H
            for h in range(H - 1, 0, -1):  # from ring h of each segment to its right anchor
                S = S + psi @ C[:, h] @ psi.mT
                psi = psi @ P[:, h]
                # gain K = Q psi^T (psi Q psi^T + S)^-1, scaled by the diagonal; 0 where nothing is left
                W = psi @ C[:, h - 1] @ psi.mT + S
                d = torch.diagonal(W, dim1=-2, dim2=-1)
                ok = (d > 1e-250).all(-1)[..., None]
                r = torch.rsqrt(torch.where(ok, d, torch.ones_like(d)))
                Wn = torch.where(ok[..., None], W * r[..., :, None] * r[..., None, :], torch.eye(M, device=dev, dtype=torch.float64))
                K = torch.linalg.solve(Wn, (psi @ C[:, h - 1]) * r[..., :, None]).mT * r[..., None, :]
                K = torch.where(ok[..., None], K, torch.zeros_like(K))
                I = eye - K @ psi
                bridge[h] = (I @ P[:, h - 1], K, I @ C[:, h - 1] @ I.mT + K @ S @ K.mT)
            psi, S = psi @ P[:, 0], S + psi @ C[:, 0] @ psi.mT
            B = _chol(S) * half
            for j in range(na):
                x = mv(psi[j], x) + mv(B[j], noise(at([ks[(j + 1) * H]]))[0] * flip)
                anchors.append(x)
                put(at([ks[(j + 1) * H]]), x[None])
            left, right = torch.stack(anchors[:-1]), torch.stack(anchors[1:])
            for h in range(1, H):
                rings = at([ks[j * H + h] for j in range(na)])
                a, K, V = bridge[h]
                left = mv(a, left) + mv(K, right) + mv(_chol(V) * half, noise(rings) * flip)
                put(rings, left)
        for pos in range(na * H + 1, length + 1):
            x = mv(phi[pos - 1], x) + mv(_chol(Q[pos - 1]) * half, noise(at([ks[pos]]))[0] * flip)
            put(at([ks[pos]]), x[None])
    return g


def exact(case, seed):
    if case["kind"] == "batch" or case["n"] * case["n_theta"] * case["n_phi"] > 2.5e8:
        return None  # over about 20 seconds
    kh, n_theta, n_phi = _spectrum(case, seed), case["n_theta"], case["n_phi"]
    rings = _healpix((n_theta + 1) // 4) if case["kind"] == "healpix" else None
    theta = rings[0] if rings else [math.pi * (k + 0.5) / n_theta for k in range(n_theta)]
    H = 0 if case["paper"] else case["H"] or 16  # the default anchor spacing
    g = _field(kh, theta, n_phi, H if H < n_theta else 0, _key(seed), case["n"])
    if not rings:
        return torch.fft.irfft(g, n=n_phi, dim=-1) * n_phi
    out = []
    m = torch.arange(n_phi // 2 + 1, device=g.device)
    for k in range(n_theta):  # the field at the ring's own points: the spectrum folded to their number
        nk = rings[1][k]
        shift = torch.polar(torch.ones_like(m, dtype=torch.float64), m.double() * rings[2][k])
        c = g[:, k] * shift
        c[:, -1] = 0.5 * g[:, k, -1].real * shift[-1]
        full = torch.zeros(case["n"], nk, dtype=torch.complex128, device=g.device)
        full.index_add_(1, m % nk, c)
        full.index_add_(1, (-m[1:]) % nk, c[:, 1:].conj())
        out.append(torch.fft.ifft(full).real * nk)
    return torch.cat(out, 1)
