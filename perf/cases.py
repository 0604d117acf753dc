"""The work a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  ``kind`` says which public call it makes:

``solve``     ``Plan.solve`` of an FFT plan (constant aspect ratios), into buffers the caller keeps, as a
              hydrodynamics code calls it once per time step;
``host``      ``Plan.solve_host``: the same through pinned host buffers, as a code whose fields live on the host does;
``batch``     ``Batch.solve``: many independent discs of uneven grids (a parameter survey), one graph launch;
``semi``      ``Plan.solve`` of a semi-spectral plan (flaring discs, H = H(r));
``replan``    a semi-spectral plan built, solved once and closed: what a code does whose H(r) evolves;
``direct``    ``Plan.solve`` of a direct plan (H = H(r, phi)), any grid size;
``indirect``  ``Plan.indirect``: the indirect term's two sums per fluid, once per time step.

The discs are the benchmark's: log-normal surface density (5-cell correlation) on r^-1 with m = 2..4 spirals,
a 1 % dust fluid when ``St`` > 0 with H_d = H_g sqrt(alpha / (alpha + St)), radii 0.1 to 5 (0.2 to 2.5 for the
smallest).  Direct plans get an elliptically modulated H(r, phi), semi-spectral ones a flaring H(r).
"""
import math

import torch

from paper_2506_10812_gb300 import Batch, Plan

ALPHA = 1e-3
ALL = ("phi", "gr", "gphi")
ACCEL = ("gr", "gphi")
BATCH_SHAPES = ((128, 256), (256, 512), (512, 1024), (1024, 2048))


def _case(name, kind, nr, nphi, h=0.05, St=0.0, f64=False, accel=False, r_in=0.1, r_out=5.0, flare=0.0, discs=0):
    c = {"kind": kind, "nr": nr, "nphi": nphi, "h": h, "St": St, "f64": f64, "accel": accel, "r_in": r_in, "r_out": r_out,
         "flare": flare, "discs": discs}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a quick look or a unit test of a hydro code: launches and latency
        _case("gas 64x128", "solve", 64, 128, r_in=0.2, r_out=2.5),
        # the ordinary two-fluid disc of a parameter study, every output
        _case("gas+dust 256x512", "solve", 256, 512, St=0.1),
        # a production two-fluid run's step: the accelerations of both fluids
        _case("gas+dust 1024x2048 accel", "solve", 1024, 2048, St=0.01, accel=True),
        # the headline: a high-resolution gas disc, potential and accelerations
        _case("gas 2048x4096", "solve", 2048, 4096),
        # codes that run in double precision, as the method's paper does
        _case("gas 1024x2048 f64", "solve", 1024, 2048, f64=True),
        # a code whose fields live in host memory
        _case("host gas 1024x2048", "host", 1024, 2048),
        # a survey: a dozen uneven gas + dust discs stepped together
        _case("batch of 12", "batch", 0, 0, h=0.03, St=0.1, accel=True, discs=12),
        # flaring discs: one step, and the step after H(r) has changed
        _case("semi gas 512x1024", "semi", 512, 1024, flare=0.25),
        _case("replan gas+dust 128x256", "replan", 128, 256, St=0.1, flare=0.25),
        # scale heights that depend on azimuth too, on an ordinary and on an odd grid, in both precisions
        _case("direct gas+dust 128x256", "direct", 128, 256, St=0.1, flare=0.25),
        _case("direct gas 61x150 f64", "direct", 61, 150, f64=True, flare=0.125),
        # the indirect term of a two-fluid step
        _case("indirect gas+dust 1024x2048", "indirect", 1024, 2048, St=0.1),
    ]


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "solve", "direct", "direct", "semi", "replan", "host", "batch", "indirect"))
    h = round(math.exp(rng.uniform(math.log(0.03), math.log(0.1))), 4)
    St = rng.choice((0.0, 0.0, 0.01, 0.1, 1.0))
    f64 = rng.random() < 0.25
    accel = rng.random() < 0.5
    flare = rng.choice((0.0, 0.125, 0.25, 0.5))
    if kind == "batch":
        return _case("", kind, 0, 0, h=h, St=St or 0.1, accel=True, discs=rng.randint(2, 12))
    if kind == "direct":   # any size; a pass costs no more than the largest listed one
        cells = math.exp(rng.uniform(math.log(500), math.log(9000 if f64 else 32000 if St == 0 else 20000)))
        nr = max(5, round(math.sqrt(cells / 2) * rng.uniform(0.6, 1.6)))
        return _case("", kind, nr, max(8, round(cells / nr)), h=h, St=St, f64=f64, accel=accel, flare=flare)
    lr = rng.randint(4, 9 if kind in ("semi", "replan") else 11)
    if kind == "replan":
        lr, f64 = min(lr, 8 if St == 0 else 7), False
    lp = lr + rng.choice((0, 1, 1, 1, 2))
    if kind == "semi" and (St or f64):
        lr, lp = min(lr, 8), min(lp, 9)
    if f64 and kind != "indirect":
        lr, lp = min(lr, 10), min(lp, 11)
    lp = max(5, min(lp, 12 if kind != "replan" else 9))
    return _case("", kind, 1 << lr, 1 << lp, h=h, St=St, f64=f64, accel=accel, flare=flare)


# ------------------------------------------------------------------ inputs
def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _grid(c):
    du = math.log(c["r_out"] / c["r_in"]) / c["nr"]
    r = c["r_in"] * torch.exp((torch.arange(c["nr"], dtype=torch.float64, device="cuda") + 0.5) * du)
    phi = (torch.arange(c["nphi"], dtype=torch.float64, device="cuda") + 0.5) * (2 * math.pi / c["nphi"])
    return r, phi, du, 2 * math.pi / c["nphi"]


def _sigma(c, seed):
    """(gas, dust or None) in the case's type: the log-normal disc with spirals."""
    g = _rng(seed)
    nr, nphi = c["nr"], c["nphi"]
    r, phi, _, _ = _grid(c)
    w = torch.randn((2 * nr, nphi), generator=g, device="cuda", dtype=torch.float64)
    kx, ky = torch.fft.fftfreq(2 * nr, device="cuda")[:, None], torch.fft.rfftfreq(nphi, device="cuda")[None, :]
    filt = torch.exp(-(math.pi * 5.0) ** 2 * (kx * kx + ky * ky).double())
    f = torch.fft.irfft2(torch.fft.rfft2(w) * filt, s=(2 * nr, nphi))[:nr]
    f = f / f.std()
    psi = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * 2 * math.pi
    arg = phi[None, :] - torch.log(r / c["r_in"])[:, None] / math.tan(math.radians(15.0))
    sp = 1.0 + sum(0.05 * torch.cos(m * arg + psi[m - 2]) for m in (2, 3, 4))
    sig = torch.exp(0.3 * f - 0.045) * sp / r[:, None]
    dt = torch.float64 if c["f64"] else torch.float32
    sd = None
    if c["St"]:
        u = torch.rand((nr, nphi), generator=g, device="cuda", dtype=torch.float64) * 2 - 1
        sd = (0.01 * sig * (1.0 + 0.01 * u)).to(dt).contiguous()
    return sig.to(dt).contiguous(), sd


def _settle(St):
    return math.sqrt(ALPHA / (ALPHA + St)) if St else 0.0


def _heights(c, seed):
    """H of each fluid: a flaring profile, and for direct plans an azimuthal modulation, in the case's type."""
    r, phi, _, _ = _grid(c)
    H = (c["h"] * r ** (1.0 + c["flare"]))[:, None].expand(c["nr"], c["nphi"])
    if c["kind"] == "direct":
        p = torch.rand(2, generator=_rng(seed + 1), device="cuda", dtype=torch.float64) * 2 * math.pi
        H = H * (1.0 + 0.15 * torch.cos(phi + p[0]) + 0.05 * torch.cos(3 * phi + p[1]))[None, :]
    H = H.to(torch.float64 if c["f64"] else torch.float32).contiguous()
    return H, (H * _settle(c["St"])).contiguous() if c["St"] else None


def _comps(c):
    return ACCEL if c["accel"] else ALL


def _keys(c):
    return [k + "_" + f for f in (("g", "d") if c["St"] else ("g",)) for k in _comps(c)]


def _plan(c, Hg=None, Hd=None):
    dt = torch.float64 if c["f64"] else torch.float32
    how = {"semi": "semispectral", "replan": "semispectral", "direct": "direct"}.get(c["kind"], "fft")
    if how == "fft":
        return Plan(c["nr"], c["nphi"], c["r_in"], c["r_out"], c["h"], c["h"] * _settle(c["St"]) or None, dtype=dt)
    return Plan(c["nr"], c["nphi"], c["r_in"], c["r_out"], c["h"], c["h"] * _settle(c["St"]) or None, dtype=dt,
                method=how, H_g=Hg, H_d=Hd)


def _members(c):
    """The discs of a batch: the four grids in turn, aspect ratios and Stokes numbers spread over their ranges."""
    out = []
    for k in range(c["discs"]):
        nr, nphi = BATCH_SHAPES[(3 * k + 1) % 4]
        out.append(_case("", "solve", nr, nphi, h=c["h"] * (1 + 0.05 * k), St=(c["St"], 0.01, 1.0)[k % 3], accel=True))
    return out


def _buffers(c, host=False):
    dt = torch.float64 if c["f64"] else torch.float32
    kw = {"pin_memory": True} if host else {"device": "cuda"}
    return {k: torch.empty((c["nr"], c["nphi"]), dtype=dt, **kw) for k in _keys(c)}


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        members = _members(c)
        plans = [_plan(m) for m in members]
        sig = [_sigma(m, seed + 1000 * k) for k, m in enumerate(members)]
        outs = [_buffers(m) for m in members]
        batch = Batch(plans, [s[0] for s in sig], [s[1] for s in sig], outs, streams=12)
        return {"c": c, "batch": batch, "outs": outs}
    sg, sd = _sigma(c, seed)
    if c["kind"] == "replan":
        Hg, Hd = _heights(c, seed)
        return {"c": c, "H": (Hg, Hd), "sg": sg, "sd": sd, "out": _buffers(c)}
    plan = _plan(c, *_heights(c, seed)) if c["kind"] in ("semi", "direct") else _plan(c)
    if c["kind"] == "host":
        pin = lambda t: None if t is None else t.cpu().pin_memory()  # noqa: E731
        return {"c": c, "plan": plan, "sg": pin(sg), "sd": pin(sd), "out": _buffers(c, host=True)}
    return {"c": c, "plan": plan, "sg": sg, "sd": sd, "out": _buffers(c)}


def run(state):
    kind = state["c"]["kind"]
    if kind == "batch":
        state["batch"].solve()
        return state["outs"]
    if kind == "indirect":
        return state["plan"].indirect(state["sg"], state["sd"])
    if kind == "host":
        return state["plan"].solve_host(state["sg"], state["sd"], outputs=_comps(state["c"]), out=state["out"])
    if kind == "replan":
        with _plan(state["c"], *state["H"]) as plan:
            return plan.solve(state["sg"], state["sd"], out=state["out"])
    return state["plan"].solve(state["sg"], state["sd"], out=state["out"])


# -------------------------------------------------------------------- work
def work(case):
    """Compulsory bytes (fields and plan tables read once, outputs written once) and nominal operations."""
    c = case
    if c["kind"] == "batch":
        parts = [work(m) for m in _members(c)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    nr, nphi, ns = c["nr"], c["nphi"], 2 if c["St"] else 1
    esz, nc = 8 if c["f64"] else 4, len(_comps(c))
    cells = nr * nphi
    fields = (ns + ns * nc) * cells * esz
    if c["kind"] == "indirect":
        return {"bytes": ns * cells * esz + 16 * ns, "flops": 4 * ns * cells}
    if c["kind"] == "direct":   # per pair about 40: geometry, one rsqrt, two short polynomials, three sums
        return {"bytes": fields + ns * cells * esz, "flops": 40 * ns * ns * cells * cells}
    rows = 2.5 * nphi * math.log2(nphi) * nr * (ns + ns * nc)
    if c["kind"] in ("semi", "replan"):
        tab = ns * ns * nc * (nphi // 2) * nr * nr * 2 * esz
        flops = rows + 8 * ns * ns * nc * (nphi // 2) * nr * nr
        if c["kind"] == "semi":
            return {"bytes": fields + tab, "flops": flops}
        full = tab // nc * 3   # the plan builds every component: 40 operations a sample, then the transforms
        return {"bytes": fields + full + tab, "flops": flops + ns * ns * nr * nr * nphi * (40 + 7.5 * math.log2(nphi))}
    tab = ns * ns * nc * (nphi // 2 + 1) * (nr + 2) * 2 * esz
    cols = (nphi // 2) * (5 * 2 * nr * math.log2(2 * nr) * (ns + ns * nc) + 8 * 2 * nr * ns * ns * nc)
    return {"bytes": fields + tab, "flops": rows + cols}


# ------------------------------------------------------- 64-bit references
def _bessel(x):
    """(e^x K0(x), e^x (K1(x) - K0(x))): torch's scaled functions, and Hankel's expansions with their difference
    taken term by term from x = 30 on, where it would cancel."""
    a = x.clamp(max=30.0)
    k0, k1 = torch.special.scaled_modified_bessel_k0(a), torch.special.scaled_modified_bessel_k1(a)
    q = 1.0 / x.clamp(min=30.0)
    t0, t1, s0, sd = torch.ones_like(q), torch.ones_like(q), torch.ones_like(q), torch.zeros_like(q)
    for k in range(14):
        o = (2 * k + 1) ** 2
        t0, t1 = t0 * q * (-o / (8.0 * (k + 1))), t1 * q * ((4.0 - o) / (8.0 * (k + 1)))
        s0, sd = s0 + t0, sd + (t1 - t0)
    s, big = torch.sqrt(0.5 * math.pi * q), x >= 30.0
    return torch.where(big, s * s0, k0), torch.where(big, s * sd, k1 - k0)


def _pairs(r, phi, i, j, src_r, src_j, di, dphi, H2):
    """Phi, g_r and g_phi of target rows i, columns j from unit masses: -K_Phi, -K_r, -K_phi of the pair sum."""
    dj = (j - src_j).double()
    sp2 = torch.sin(0.5 * dphi * dj) ** 2
    sh2 = torch.sinh(0.5 * di) ** 2
    s2 = 4.0 * r * src_r * (sh2 + sp2)
    me = s2 == 0
    k0, D = _bessel(torch.where(me, torch.ones_like(s2), s2 / (8.0 * H2)))
    f = torch.where(me, torch.zeros_like(D), -D / (8.0 * math.sqrt(math.pi) * H2 * torch.sqrt(H2))) * src_r
    p = torch.where(me, torch.zeros_like(D), -k0 / (2.0 * math.sqrt(math.pi) * torch.sqrt(H2)))
    return p, f * (torch.expm1(di) + 2.0 * sp2), f * torch.sin(dphi * dj)


def _exact_direct(c, sig, H):
    """The pair sum itself, over blocks of targets."""
    r, phi, du, dphi = _grid(c)
    nr, nphi = c["nr"], c["nphi"]
    n = nr * nphi
    idx = torch.arange(n, device="cuda")
    ii, jj = idx // nphi, idx % nphi
    rr, ns = r[ii], len(sig)
    out = [[torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)] for _ in range(ns)]
    step = max(1, (1 << 23) // n)
    for t0 in range(0, n, step):
        t = idx[t0:t0 + step, None]
        di = (ii[t] - ii[None, :]).double() * du
        for a in range(ns):
            mass = (sig[a].double().reshape(-1) * rr * rr * du * dphi)[None, :]
            for b in range(ns):
                H2 = 0.5 * (H[a].double().reshape(-1)[None, :] ** 2 + H[b].double().reshape(-1)[t] ** 2)
                for q, w in enumerate(_pairs(rr[t], phi, ii[t], jj[t], rr[None, :], jj[None, :], di, dphi, H2)):
                    out[b][q][t0:t0 + step] += (w * mass).sum(1)
    return [[o.reshape(nr, nphi) for o in f] for f in out]


def _exact_rows(c, sig, H):
    """H = H(r): per target row, the circular convolution in phi of every source row, by FFT along phi."""
    r, phi, du, dphi = _grid(c)
    nr, nphi, ns = c["nr"], c["nphi"], len(sig)
    j = torch.arange(nphi, device="cuda")[None, None, :]
    rows = torch.arange(nr, device="cuda")
    out = [[torch.zeros((nr, nphi), dtype=torch.float64, device="cuda") for _ in range(3)] for _ in range(ns)]
    F = [torch.fft.rfft(s.double() * (r * r * du * dphi)[:, None], dim=1) for s in sig]
    step = max(1, (1 << 23) // (nr * nphi))
    for i0 in range(0, nr, step):
        i = rows[i0:i0 + step, None, None]
        di = (i - rows[None, :, None]).double() * du
        for a in range(ns):
            for b in range(ns):
                H2 = 0.5 * (H[a][:, 0].double()[None, :, None] ** 2 + H[b][:, 0].double()[i] ** 2)
                for q, w in enumerate(_pairs(r[i], phi, i, j, r[None, :, None], 0 * j, di, dphi, H2)):
                    out[b][q][i0:i0 + step] += torch.fft.irfft((torch.fft.rfft(w, dim=2) * F[a][None]).sum(1), n=nphi, dim=1)
    return out


def _exact_lattice(c, sig):
    """Constant aspect ratios: the zero-padded 2-D FFT convolution with the lattice kernels, sources times r and
    kernels times e^Delta (an identity that keeps the rounding even over the radii)."""
    r, phi, du, dphi = _grid(c)
    nr, nphi, ns = c["nr"], c["nphi"], len(sig)
    di = torch.cat([torch.arange(nr, device="cuda"), torch.arange(-nr, 0, device="cuda")]).double()[:, None] * du
    sp = torch.sin(0.5 * dphi * torch.arange(nphi, device="cuda").double())[None, :]
    spsi = torch.sin(dphi * torch.arange(nphi, device="cuda").double())[None, :]
    hs = [c["h"], c["h"] * _settle(c["St"])]
    out = [[torch.zeros((nr, nphi), dtype=torch.float64, device="cuda") for _ in range(3)] for _ in range(ns)]
    F = [torch.fft.rfft2(s.double() * r[:, None], s=(2 * nr, nphi)) for s in sig]
    for a in range(ns):
        for b in range(ns):
            h2 = 0.5 * (hs[a] ** 2 * torch.exp(-di) + hs[b] ** 2 * torch.exp(di))
            X = 0.5 * (torch.sinh(0.5 * di) ** 2 + sp * sp) / h2
            X[0, 0] = 1.0
            k0, D = _bessel(X)
            e = -du * dphi * torch.exp(-0.5 * di)
            D = e * D / (8.0 * math.sqrt(math.pi) * h2 * torch.sqrt(h2))
            for q, K in enumerate((e * k0 / (2.0 * math.sqrt(math.pi) * torch.sqrt(h2)),
                                   D * (torch.expm1(di) + 2.0 * sp * sp), D * spsi)):
                K[0, 0] = 0.0
                K[nr] = 0.0
                y = torch.fft.irfft2(F[a] * torch.fft.rfft2(K), s=(2 * nr, nphi))[:nr]
                out[b][q] += y if q == 0 else y / r[:, None]
    return out


def _exact_indirect(c, sig):
    r, phi, du, dphi = _grid(c)
    rows = []
    for s, h in zip(sig, (c["h"], c["h"] * _settle(c["St"]))):
        k = float(_bessel(torch.tensor([0.25 / (h * h)], dtype=torch.float64, device="cuda"))[1])
        w = math.sqrt(2.0) * du * dphi * k / (4.0 * math.sqrt(math.pi) * h ** 3)
        col = s.double().sum(0)
        rows.append(torch.stack([(col * torch.cos(phi)).sum(), (col * torch.sin(phi)).sum()]) * w)
    return torch.stack(rows)


def _named(c, fields):
    return {k + "_" + f: fields[b][ALL.index(k)] for b, f in enumerate(("g", "d")[:len(fields)]) for k in _comps(c)}


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        out = []
        for k, m in enumerate(_members(c)):
            out.append(_named(m, _exact_lattice(m, [s for s in _sigma(m, seed + 1000 * k) if s is not None])))
        return out
    sig = [s for s in _sigma(c, seed) if s is not None]
    if c["kind"] == "indirect":
        return _exact_indirect(c, sig)
    if c["kind"] in ("semi", "replan", "direct"):
        H = [x for x in _heights(c, seed) if x is not None]
        if c["kind"] == "direct":
            return _named(c, _exact_direct(c, sig, H))
        return _named(c, _exact_rows(c, sig, H))
    return _named(c, _exact_lattice(c, sig))
