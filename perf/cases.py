"""What this library is timed on: photon bunches of air showers, through the
calls a shower program makes.

A case names the call, the precision, how many track steps of how many
showers it brings, their zenith angle, the telescope array, the option that
is switched on and the refraction tables' shape:

* ``hits``     generate_propagate (or the replay of its CUDA graph), the
               records packed and put in order: the production path;
* ``trace``    segment_yield and trace_bunches, every bunch returned: what a
               study of single bunches or a validation run does;
* ``readout``  the differentiable telescope read-out and its gradients: one
               step of a fit of the atmosphere or of the emission geometry;
* ``steps``    generate_steps: parameterised showers made on the device.

Records leave the library in the order in which the warps finish, so a
program that wants the same file from the same seed puts them in order of
their keys; ``hits`` does that on the device after packing them.

The steps are shower-shaped and drawn on the GPU from the seed: depths from
the Greisen profile, lateral offsets exponential (50 m), energies
log-uniform 20 MeV - 5 GeV, angles Gaussian (3 degrees at 50 MeV, falling
as 1 / E), lengths 1 - 20 m.
"""
import math

import numpy as np
import torch

import paper_2006_14927_gb300 as P
from paper_2006_14927_gb300.autograd import telescope_readout

H_OBS = 2200.0
H_MAX = 60000.0
N_FINE = 10000
BUNCH = 5.0
LAM1, LAM2 = 300.0, 600.0
C_LIGHT = 0.299792458
X0_RAD, E_CRIT, X_SEA, H_SCALE, H_START = 36.7, 85.0, 1030.0, 8000.0, 30000.0
BUNCHES_PER_STEP = 30          # mean over the showers drawn here


def _case(name, call, precision, steps, showers=1, zenith=0.0, array="hex19", option="none",
          heights=1000, zeniths=64, table_zenith=70.0, replay=False):
    return dict(name=name, call=call, precision=precision, steps=steps, showers=showers,
                zenith=zenith, array=array, option=option, heights=heights, zeniths=zeniths,
                table_zenith=table_zenith, replay=replay)


def listed():
    return [
        # the smallest call: a handful of steps over one telescope, double precision
        _case("plain_1k_fp64", "hits", "fp64", 1000, array="single"),
        # a low-energy shower, the bulk of an event list by number: launches count
        _case("shower_10gev", "hits", "fp32", 20011),
        # one 1 TeV vertical shower over a small array, the ordinary event
        _case("shower_1tev", "hits", "fp32", 2_000_000),
        # the same in double precision, a tenth of the steps: the reference run
        _case("shower_100gev_fp64", "hits", "fp64", 200_003),
        # a batch of uneven showers over a wide array in one launch, replayed from its graph
        _case("batch_256", "hits", "fp32", 20_000_000, showers=256, zenith=40.0, array="km100",
              replay=True),
        # a shower at 60 degrees through fine tables: long slant paths
        _case("inclined_60deg", "hits", "fp32", 3_000_017, zenith=60.0, array="km100",
              heights=4000, zeniths=256, table_zenith=75.0),
        # atmospheric extinction on: a survival draw per bunch
        _case("transmission", "hits", "fp32", 499_979, zenith=20.0, option="transmission"),
        # a wavelength-dependent index of refraction
        _case("dispersion", "hits", "fp32", 300_007, zenith=20.0, option="dispersion"),
        # a spherical atmosphere at large zenith angle
        _case("curved_70deg", "hits", "fp32", 300_007, zenith=70.0, array="km100",
              option="curved", table_zenith=80.0),
        # every bunch of a short step list
        _case("trace_30k", "trace", "fp32", 30_011),
        # a fit step: read-out of a 300 GeV shower and its gradients
        _case("readout_300gev", "readout", "fp32", 100_000),
        # shower steps made on the device
        _case("steps_2m", "steps", "fp32", 2_000_000, showers=8, zenith=40.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choices(("hits", "trace", "readout", "steps"), (6, 1.5, 1.5, 1))[0]
    precision = rng.choices(("fp32", "fp64"), (3, 1))[0]
    f64 = precision == "fp64"
    c = dict(call=call, precision=precision, showers=1, option="none", replay=False)
    c["array"] = rng.choice(("single", "hex19", "km100"))
    c["zenith"] = round(rng.choice((0.0, rng.uniform(0.0, 40.0), rng.uniform(40.0, 60.0))), 3)
    if call == "hits":
        c["option"] = rng.choices(("none", "profile", "transmission", "dispersion", "curved",
                                   "fallback"), (8, 1, 1.5, 1, 1, 1))[0]
        top = 2_000_000 if c["option"] == "none" else 300_000
        c["steps"] = _log_int(rng, 300, top // 10 if f64 else top)
        c["showers"] = rng.choice((1, 1, 1 + c["steps"] // 20_000))
        c["replay"] = rng.random() < 0.3
    elif call == "trace":
        c["steps"] = _log_int(rng, 100, 10_000 if f64 else 50_000)
    elif call == "readout":
        c["steps"] = _log_int(rng, 1000, 100_000)
    else:
        c["steps"] = _log_int(rng, 1000, 2_000_000)
        c["showers"] = rng.randint(1, 64)
    fine = c["zenith"] > 50.0
    c["heights"], c["zeniths"] = (4000, 256) if fine else (1000, 64)
    c["table_zenith"] = 80.0 if c["option"] == "curved" else (75.0 if fine else 70.0)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _atmosphere():
    """US-standard (Linsley) layers; the fifth continues the fourth at 100 km."""
    a = [-186.555305, -94.919, 0.61289, 0.0, 0.0]
    b = [1222.6562, 1144.9069, 1305.5948, 540.1778, 1.0]
    c = [9941.8638, 8781.5355, 6361.4304, 7721.7016, 1.0e7]
    a[4] = a[3] + b[3] * math.exp(-100000.0 / c[3]) - b[4] * math.exp(-100000.0 / c[4])
    top = -c[4] * math.log(-a[4] / b[4])
    return dict(h_bound=[0.0, 4000.0, 10000.0, 40000.0, 100000.0, top], a=a, b=b, c=c,
                n0_minus_1=2.83e-4)


def _telescopes(array):
    rng = np.random.Generator(np.random.PCG64(7))
    if array == "single":
        return np.array([[0.0, 0.0, 0.0, 12.0]])
    if array == "hex19":       # centre and two rings, pitch 120 m, radii 6 - 12 m
        pts = [(120.0 * (q + 0.5 * r), 120.0 * math.sqrt(0.75) * r)
               for q in range(-2, 3) for r in range(-2, 3) if abs(q + r) <= 2]
        return np.column_stack([np.array(pts), np.zeros(19), rng.uniform(6.0, 12.0, 19)])
    radii = np.array([23.0] * 5 + [12.0] * 35 + [6.0] * 60)      # 100 over 2 x 2 km
    out = []
    for r in radii:
        while True:
            x, y = rng.uniform(-1000.0, 1000.0, 2)
            if all(math.hypot(x - t[0], y - t[1]) > r + t[3] + 2.0 for t in out):
                out.append((x, y, 0.0, r))
                break
    return np.array(out)


def _transmission():
    """Rayleigh and aerosol optical depths above H_OBS, 16 x 121 nodes."""
    lam, h = np.linspace(250.0, 700.0, 16), np.linspace(H_OBS, H_MAX, 121)
    ray = 0.36 * (lam / 400.0) ** -4.0
    aer = 0.10 * (lam / 400.0) ** -1.3
    tau = (ray[:, None] * (np.exp(-H_OBS / 8400.0) - np.exp(-h / 8400.0)) +
           aer[:, None] * (np.exp(-H_OBS / 1200.0) - np.exp(-h / 1200.0)))
    return dict(tau=tau, lambda_nm=(250.0, 700.0), height_m=(H_OBS, H_MAX))


def _dispersion():
    """Edlen's 1966 standard air over 300 - 600 nm, relative to 400 nm."""
    def n1(lam):
        s2 = (1000.0 / lam) ** 2
        return 8342.13 + 2406030.0 / (130.0 - s2) + 15997.0 / (38.9 - s2)
    u = np.linspace(1.0 / LAM1, 1.0 / LAM2, 9)
    return n1(1.0 / u) / n1(400.0)


def _showers(case, rng):
    """Energies, directions, cores and step counts (proportional to energy)."""
    n, k = case["steps"], case["showers"]
    zen = math.radians(case["zenith"])
    if k == 1:
        return [dict(e0_mev=min(max(0.5 * n, 1.0e4), 2.0e7), zenith=zen,
                     azimuth=rng.uniform(0.0, 2.0 * math.pi) if zen else 0.0,
                     core_x=0.0, core_y=0.0, n=n)]
    e0 = np.exp(rng.uniform(math.log(1.0e4), math.log(1.0e7), k))
    cnt = np.maximum((n * e0 / e0.sum()).astype(np.int64), max(1, min(1000, n // (4 * k))))
    cnt[np.argmax(cnt)] += n - cnt.sum()
    return [dict(e0_mev=float(e0[s]), zenith=float(rng.uniform(0.0, zen)),
                 azimuth=float(rng.uniform(0.0, 2.0 * math.pi)),
                 core_x=float(rng.uniform(-1000.0, 1000.0)),
                 core_y=float(rng.uniform(-1000.0, 1000.0)), n=int(cnt[s])) for s in range(k)]


def _tracks(case, showers, seed):
    """Step arrays on the GPU, shower after shower, in the ABI's types."""
    dev, f8 = "cuda", torch.float64
    g = torch.Generator(device=dev).manual_seed(seed)
    k, n = len(showers), case["steps"]

    def col(v):
        return torch.tensor(v, dtype=f8, device=dev)

    def uni(lo, hi):
        return torch.rand(n, generator=g, device=dev, dtype=f8) * (hi - lo) + lo

    zen, az = col([s["zenith"] for s in showers]), col([s["azimuth"] for s in showers])
    ax, ay, az_ = torch.sin(zen) * torch.cos(az), torch.sin(zen) * torch.sin(az), -torch.cos(zen)
    cz = -az_
    cx, cy = col([s["core_x"] for s in showers]), col([s["core_y"] for s in showers])
    y = torch.log(col([s["e0_mev"] for s in showers]) / E_CRIT)
    sh = torch.repeat_interleave(torch.arange(k, device=dev),
                                 torch.tensor([s["n"] for s in showers], device=dev),
                                 output_size=n)
    # depths from the Greisen profile by inversion of its sampled integral
    t_g = X_SEA * math.exp(-H_OBS / H_SCALE) / cz / X0_RAD
    m = 2048
    t = t_g[:, None] * (torch.arange(1, m + 1, device=dev, dtype=f8) / m)
    pdf = torch.exp(t * (1.0 - 1.5 * torch.log(3.0 * t / (t + 2.0 * y[:, None]))))
    cdf = torch.cumsum(pdf, 1)
    cdf = cdf / cdf[:, -1:]
    flat = (cdf + torch.arange(k, device=dev, dtype=f8)[:, None]).reshape(-1)
    at = torch.searchsorted(flat, uni(0.0, 1.0) + sh).clamp_(max=k * m - 1)
    depth = torch.minimum(t.reshape(-1)[at] - uni(0.0, 1.0) * (t_g / m)[sh], t_g[sh])
    h = H_SCALE * torch.log(X_SEA / (depth.clamp_(min=1e-6) * X0_RAD * cz[sh]))
    s = (h.clamp_(max=H_START - 1.0) - H_OBS) / cz[sh]
    r, psi = -50.0 * torch.log(1.0 - uni(0.0, 1.0)), uni(0.0, 2.0 * math.pi)
    # transverse basis: b1 horizontal, b2 = axis x b1
    rho = torch.sqrt(ax * ax + ay * ay)
    flatax = rho < 1e-9
    b1x = torch.where(flatax, torch.ones_like(rho), ay / rho.clamp(min=1e-9))
    b1y = torch.where(flatax, torch.zeros_like(rho), -ax / rho.clamp(min=1e-9))
    b2x, b2y, b2z = -az_ * b1y, az_ * b1x, ax * b1y - ay * b1x
    lx, ly = r * torch.cos(psi), r * torch.sin(psi)
    ekin = 20.0 * torch.exp(uni(0.0, math.log(250.0)))
    sig = math.radians(3.0) * (50.0 / ekin)
    nx = torch.randn(n, generator=g, device=dev, dtype=f8) * sig
    ny = torch.randn(n, generator=g, device=dev, dtype=f8) * sig
    dx = ax[sh] + nx * b1x[sh] + ny * b2x[sh]
    dy = ay[sh] + nx * b1y[sh] + ny * b2y[sh]
    dz = az_[sh] + ny * b2z[sh]
    norm = torch.sqrt(dx * dx + dy * dy + dz * dz)
    s_ref = (H_START - H_OBS) / cz
    fd = torch.float32 if case["precision"] == "fp32" else f8
    return dict(x0=cx[sh] - s * ax[sh] + lx * b1x[sh] + ly * b2x[sh],
                y0=cy[sh] - s * ay[sh] + lx * b1y[sh] + ly * b2y[sh],
                z0=H_OBS - s * az_[sh] + ly * b2z[sh],
                t0=(s_ref[sh] - s) / C_LIGHT, len=uni(1.0, 20.0), ekin=ekin,
                ux=(dx / norm).to(fd), uy=(dy / norm).to(fd), uz=(dz / norm).to(fd),
                shower=sh.to(torch.int32), t_ref=s_ref / C_LIGHT)


def _room(case):
    """Records an event buffer holds, and for a trace its bunches."""
    return (5 * case["steps"]) // 2 + 4000 if case["call"] == "hits" else 40 * case["steps"] + 4000


def prepare(case, seed):
    prec = P.CHER_FP32_BULK if case["precision"] == "fp32" else P.CHER_FP64
    rng = np.random.Generator(np.random.PCG64(seed))
    atm = _atmosphere()
    ctx = P.Context(atm, H_OBS, _telescopes(case["array"]), BUNCH, LAM1, LAM2, N_FINE)
    if case["option"] == "curved":
        ctx.set_curved(6.371e6)
    ctx.build_refraction_tables(case["heights"], case["zeniths"], case["table_zenith"], H_MAX)
    if case["option"] == "transmission":
        ctx.set_transmission(_transmission())
    elif case["option"] == "dispersion":
        ctx.set_dispersion(_dispersion())
    elif case["option"] == "fallback":
        ctx.set_fallback(min(case["table_zenith"] + 8.0, 85.0))
    showers = _showers(case, rng)
    st = dict(call=case["call"], ctx=ctx, prec=prec, seed=int(rng.integers(1 << 62)))
    if case["call"] == "steps":
        st["showers"] = showers
        st["out"] = ctx.generate_steps(showers, st["seed"], prec)
        return st
    st["tracks"] = _tracks(case, showers, seed)
    st["room"] = _room(case)
    if case["call"] == "hits":
        # buffers sized by a counting call without room for records
        count = ctx.alloc_hits(1, prec)
        ctx.generate_propagate(st["tracks"], st["seed"], prec, count)
        ctx.sync_status(count)
        out = ctx.alloc_hits(max(1, int(count.count.max())), prec)
        total = int(count.count.sum())
        dev, ft = "cuda", out.pos.dtype
        st["out"] = out
        st["packed"] = dict(pos=torch.zeros((total, 4), dtype=ft, device=dev),
                            tim=torch.zeros((total, 4), dtype=ft, device=dev),
                            key=torch.zeros(total, dtype=torch.int64, device=dev),
                            offset=torch.zeros(ctx.n_tel + 1, dtype=torch.int64, device=dev))
        # the event's records in order, in buffers of one size for every event
        room = st["room"]
        if total > room:
            raise ValueError("more records than the event buffers hold")
        st["event"] = dict(pos=torch.zeros((room, 4), dtype=ft, device=dev),
                           tim=torch.zeros((room, 4), dtype=ft, device=dev),
                           key=torch.zeros(room, dtype=torch.int64, device=dev))
        # (the four values of a record move as 16-byte elements)
        st["ordered"] = [(st["packed"]["key"], st["event"]["key"][:total])]
        for k in ("pos", "tim"):
            pair = [v.view(torch.complex128) for v in (st["packed"][k], st["event"][k][:total])]
            st["ordered"].append([v.view(-1) for v in pair] if ft == torch.float32 else pair)
        if case["option"] == "profile":
            st["profile"] = torch.zeros((len(showers), 120), dtype=torch.float64, device=dev)
            st["axis_cos"] = torch.tensor([math.cos(s["zenith"]) for s in showers],
                                          dtype=torch.float64, device=dev)
        elif case["replay"]:
            st["graph"] = ctx.graph(st["tracks"], st["seed"], prec, out)
    elif case["call"] == "readout":
        st["atm"] = atm
        params = torch.tensor(atm["a"] + atm["b"] + atm["c"], dtype=torch.float64)
        st["params"] = params.requires_grad_(True)
        for k in ("x0", "y0", "z0", "ux", "uy", "uz"):
            st["tracks"][k].requires_grad_(True)
        st["gD"] = torch.tensor(rng.normal(size=ctx.n_tel), device="cuda")
        st["gT"] = torch.tensor(0.1 * rng.normal(size=ctx.n_tel), device="cuda")
        st["tables"] = {"atm": dict(h_bound=list(atm["h_bound"]), a=list(atm["a"]),
                                    b=list(atm["b"]), c=list(atm["c"]),
                                    n0_minus_1=atm["n0_minus_1"])}
    return st


def run(state):
    ctx, prec = state["ctx"], state["prec"]
    if state["call"] == "steps":
        return ctx.generate_steps(state["showers"], state["seed"], prec, out=state["out"])
    tr = state["tracks"]
    if state["call"] == "trace":
        nb, w = ctx.segment_yield(tr, prec)
        # (the last offset is the room of the event buffers, not the total)
        off = torch.full((nb.numel() + 1,), state["room"], dtype=torch.int64, device=nb.device)
        off[0] = 0
        torch.cumsum(nb[:-1], 0, dtype=torch.int64, out=off[1:-1])
        r = ctx.trace_bunches(tr, state["seed"], prec, off)
        return dict(r, nb=nb, w=w)
    if state["call"] == "readout":
        D, T = telescope_readout(ctx, tr, state["params"], state["atm"], state["seed"], prec,
                                 state=state["tables"])
        leaves = [state["params"]] + [tr[k] for k in ("x0", "y0", "z0", "ux", "uy", "uz")]
        grads = torch.autograd.grad((D, T), leaves, (state["gD"], state["gT"]))
        return dict(D=D, T=T, grads=list(grads))
    out, res = state["out"], {}
    if "graph" in state:
        state["graph"].launch()
    elif "profile" in state:
        state["profile"].zero_()
        ctx.generate_propagate(tr, state["seed"], prec, out, profile=state["profile"],
                               axis_cos=state["axis_cos"])
        res["profile"] = state["profile"]
    else:
        ctx.generate_propagate(tr, state["seed"], prec, out)
    rec = ctx.pack_records(out, state["packed"])
    # stable: a bunch that crosses several spheres keeps their order; a long
    # list of less than 2^23 steps sorts by 32 bits of (step, bunch of the step)
    key = rec["key"]
    if 200_000 < tr["x0"].numel() < 1 << 23:
        key = ((key >> 24) | (key & 0xFF)).to(torch.int32)
    at = torch.sort(key, stable=True)[1]
    for src, dst in state["ordered"]:
        torch.index_select(src, 0, at, out=dst)
    ev = state["event"]
    res.update(count=out.count, stats=out.stats, offset=rec["offset"], key=ev["key"],
               pos=ev["pos"], tim=ev["tim"])
    return res


def work(case):
    n = case["steps"]
    wide = case["precision"] == "fp64"
    step, record = (76, 72) if wide else (64, 40)
    bunches = BUNCHES_PER_STEP * n
    if case["call"] == "steps":      # written once; some 120 operations a step
        return {"bytes": n * step, "flops": 120 * n}
    # the yield of each step (113 operations), and 215 operations for each
    # bunch that has to come back
    if case["call"] == "trace":
        return {"bytes": n * (step + 12) + bunches * (record + 4), "flops": 113 * n + 215 * bunches}
    if case["call"] == "readout":
        return {"bytes": 2 * n * step + n * 48, "flops": 2 * 113 * n}
    return {"bytes": n * step + 0.6 * n * record, "flops": 113 * n + 215 * 0.6 * n}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
_M0, _M1, _W0, _W1, _LOW = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85, 0xFFFFFFFF


def _mul(a, b):
    """High and low words of a 32 x 32 bit product."""
    p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
    m = p0 + ((p1 & 0xFFFF) << 16)
    return (p1 >> 16) + (m >> 32), m & _LOW


def _philox(c, seed):
    k0, k1 = seed & _LOW, seed >> 32
    for r in range(10):
        h0, l0 = _mul(_M0, c[0])
        h1, l1 = _mul(_M1, c[2])
        c = (h1 ^ c[1] ^ ((k0 + r * _W0) & _LOW), l1, h0 ^ c[3] ^ ((k1 + r * _W1) & _LOW), l0)
    return [(w.double() + 0.5) / 4294967296.0 for w in c]


class _Exact:
    """The method in 64 bits over its two interpolation tables, differentiable
    in the atmosphere's parameters (15: a, b, c of the five layers)."""

    def __init__(self, case, params):
        self.p, self.hb = params, _atmosphere()["h_bound"]
        self.H, self.Z = case["heights"], case["zeniths"]
        dev = params.device
        self.eta_obs_exact = self.eta(torch.tensor(H_OBS, dtype=torch.float64, device=dev))
        self.dh = H_MAX / (N_FINE - 1)
        self.fine = self.eta(torch.arange(N_FINE, device=dev, dtype=torch.float64) * self.dh)
        self.eta_obs = self.lookup(torch.tensor(H_OBS, dtype=torch.float64, device=dev))
        self.qmax = math.sin(math.radians(case["table_zenith"])) ** 2
        self.dht, self.dq = (H_MAX - H_OBS) / (self.H - 1), self.qmax / (self.Z - 1)
        # corrections to the straight line, integrated piece by piece
        x, w = np.polynomial.legendre.leggauss(12)
        grid = H_OBS + np.arange(self.H) * self.dht
        edge = np.unique(np.concatenate([grid, [b for b in self.hb if H_OBS < b < H_MAX]]))
        mid, half = 0.5 * (edge[1:] + edge[:-1]), 0.5 * (edge[1:] - edge[:-1])
        node = torch.tensor(mid[:, None] + half[:, None] * x, device=dev)
        wt = torch.tensor(half[:, None] * w, device=dev)[..., None]
        e = self.eta(node)[..., None]
        q = torch.arange(self.Z, device=dev, dtype=torch.float64) * self.dq
        so, co = torch.sqrt(q), torch.sqrt(1.0 - q)
        rm1 = (self.eta_obs_exact - e) / (1.0 + e)
        r, rr = 1.0 + rm1, rm1 * (2.0 + rm1)
        cs = torch.sqrt(1.0 - q * r * r)
        gx = rr * co ** 2 / ((r * co + cs) * cs)
        gl = e * co ** 3 / cs + q * rr * co ** 2 / ((co + cs) * cs)
        at = torch.tensor(np.searchsorted(edge, grid), device=dev)
        zero = torch.zeros((1, self.Z), dtype=torch.float64, device=dev)
        self.ax, self.al = (torch.cat([zero, torch.cumsum((v * wt).sum(1), 0)])[at]
                            for v in (gx, gl))

    def eta(self, h):
        b, c = self.p[5:10], self.p[10:15]
        e = torch.zeros_like(h)
        for i in range(5):
            inside = (h >= self.hb[i]) & (h < self.hb[i + 1])
            e = torch.where(inside, 2.83e-4 * (b[i] / c[i]) * torch.exp(-h / c[i]) / (b[0] / c[0]), e)
        return e

    def lookup(self, h):
        x = h.clamp(0.0, H_MAX) / self.dh
        k = x.detach().long().clamp(max=N_FINE - 2)
        return self.fine[k] + (x - k) * (self.fine[k + 1] - self.fine[k])

    def table(self, T, fj, fk):
        j, k = fj.detach().long().clamp(0, self.H - 2), fk.detach().long().clamp(0, self.Z - 2)
        a, b = fj - j, fk - k
        v0 = T[j, k] + a * (T[j + 1, k] - T[j, k])
        v1 = T[j, k + 1] + a * (T[j + 1, k + 1] - T[j, k + 1])
        return v0 + b * (v1 - v0)

    def counts(self, tr):
        """(sin^2 of the cone, 1 + g, index, photons, bunches) of every step."""
        g = tr["ekin"] * (1.0 / 0.51099895)
        e = self.lookup(tr["z0"] + 0.5 * tr["len"] * tr["uz"])
        s2 = (e * (2.0 + e) * (1.0 + g) ** 2 - (1.0 + e) ** 2) / (g * (2.0 + g) * (1.0 + e) ** 2)
        K = 2.0 * math.pi * 7.2973525693e-3 * (1.0e9 / LAM1 - 1.0e9 / LAM2)
        N = tr["len"] * K * s2.clamp(min=0.0)
        return s2, g, e, N, torch.ceil(N.detach() / BUNCH).long()

    def bunches(self, tr, sel, j, seed):
        """Bunch j of each selected step."""
        t = {k: v[sel] for k, v in tr.items() if k != "t_ref"}
        s2, g, e, N, nb = self.counts(t)
        u0, u1, u2, _ = _philox((sel & _LOW, sel >> 32, j, torch.zeros_like(j)), seed)
        beta = torch.sqrt(g * (2.0 + g)) / (1.0 + g)
        cosc, sinc = 1.0 / (beta * (1.0 + e)), torch.sqrt(s2)
        ux, uy, uz = t["ux"], t["uy"], t["uz"]
        rho2 = ux * ux + uy * uy
        steep = rho2 <= 1e-20
        rho = torch.sqrt(torch.where(steep, torch.ones_like(rho2), rho2))
        e1x = torch.where(steep, torch.ones_like(rho), -uy / rho)
        e1y = torch.where(steep, torch.zeros_like(rho), ux / rho)
        cp, sp = torch.cos(2.0 * math.pi * u1), torch.sin(2.0 * math.pi * u1)
        px = cosc * ux + sinc * (cp * e1x - sp * uz * e1y)
        py = cosc * uy + sinc * (cp * e1y + sp * uz * e1x)
        pz = cosc * uz + sinc * sp * (ux * e1y - uy * e1x)
        fl = (j + u0) / nb * t["len"]
        he = t["z0"] + fl * uz
        dH = he - H_OBS
        se2 = px * px + py * py
        rat = (1.0 + self.lookup(he)) / (1.0 + self.eta_obs)
        q = se2 * rat * rat
        status = torch.where(~(q <= self.qmax), 4, 0)
        status = torch.where(~(he <= H_MAX), 3, status)
        status = torch.where(~(he >= H_OBS), 2, status)
        status = torch.where(~(pz < 0), 1, status)
        q, dHc = q.clamp(max=self.qmax), dH.clamp(0.0, H_MAX - H_OBS)
        sec = 1.0 / torch.sqrt(1.0 - q)
        A = self.table(self.ax, dHc / self.dht, q / self.dq)
        Al = self.table(self.al, dHc / self.dht, q / self.dq)
        se = torch.sqrt(se2)
        so, hx, hy = se * rat, px / se, py / se
        D = so * sec * (dH + A * sec * sec)
        X, Y = t["x0"] + fl * ux + D * hx, t["y0"] + fl * uy + D * hy
        t_arr = (t["t0"] - tr["t_ref"][t["shower"].long()] + fl / (beta * C_LIGHT) +
                 sec * (dH + Al * sec * sec) / C_LIGHT)
        lam = 1.0 / (1.0 / LAM1 - u2 * (1.0 / LAM1 - 1.0 / LAM2))
        return dict(X=X, Y=Y, cx=so * hx, cy=so * hy, cz=-1.0 / sec, t=t_arr, he=he,
                    w=N / nb, lam=lam, status=status)


def _all_bunches(nb, lo, hi):
    """(step, j) of every bunch of the steps lo..hi."""
    n = nb[lo:hi]
    step = torch.repeat_interleave(torch.arange(lo, hi, device=nb.device), n)
    first = torch.cumsum(n, 0) - n
    return step, torch.arange(step.numel(), device=nb.device) - first[step - lo]


def _exact_hits(case, M, tr, seed, tel):
    nb = M.counts(tr)[4]
    parts = []
    for lo in range(0, case["steps"], 20_000):
        step, j = _all_bunches(nb, lo, min(lo + 20_000, case["steps"]))
        o = M.bunches(tr, step, j, seed)
        for k, (tx, ty, tz, r) in enumerate(tel):
            dx, dy, dz = tx - o["X"], ty - o["Y"], tz
            q0, q1 = dy * o["cz"] - dz * o["cy"], dz * o["cx"] - dx * o["cz"]
            q2 = dx * o["cy"] - dy * o["cx"]
            hit = (o["status"] == 0) & (q0 * q0 + q1 * q1 + q2 * q2 <= r * r)
            s = {m: v[hit] for m, v in o.items()}
            sl = tz / s["cz"]
            tt = s["t"] + sl * (1.0 + M.eta_obs) / C_LIGHT
            parts.append(((step[hit] << 32) + j[hit],
                          torch.stack([s["X"] + sl * s["cx"] - tx, s["Y"] + sl * s["cy"] - ty,
                                       s["cx"], s["cy"]], 1),
                          torch.stack([tt, s["he"], s["w"], s["lam"]], 1),
                          torch.full_like(step[hit], k)))
    key, pos, tim, at = (torch.cat(v) for v in zip(*parts))
    order = torch.sort(at, stable=True)[1]
    order = order[torch.sort(key[order], stable=True)[1]]
    pad = _room(case) - order.numel()
    pos, tim = (torch.nn.functional.pad(v[order], (0, 0, 0, pad)) for v in (pos, tim))
    return dict(count=None, stats=None, offset=None, key=None, pos=pos, tim=tim)


def _exact_readout(case, M, tr, seed, st, sigma=1.0):
    tel = torch.tensor(_telescopes(case["array"]), device="cuda")
    with torch.no_grad():
        nb = M.counts(tr)[4]
        near = []
        for lo in range(0, case["steps"], 50_000):
            step, j = _all_bunches(nb, lo, min(lo + 50_000, case["steps"]))
            o = M.bunches(tr, step, j, seed)
            r2 = (o["X"][:, None] - tel[:, 0]) ** 2 + (o["Y"][:, None] - tel[:, 1]) ** 2
            ok = (o["status"] == 0) & (r2 < 36.0 * sigma * sigma).any(1)
            near.append((step[ok], j[ok]))
        step, j = (torch.cat(v) for v in zip(*near))
    o = M.bunches(tr, step, j, seed)
    r2 = (o["X"][:, None] - tel[:, 0]) ** 2 + (o["Y"][:, None] - tel[:, 1]) ** 2
    G = torch.exp(-r2 / (2.0 * sigma ** 2)) / (2.0 * math.pi * sigma ** 2)
    G = torch.where(r2.detach() < 36.0 * sigma * sigma, G, torch.zeros_like(G)) * o["w"][:, None]
    D, U = G.sum(0), (G * o["t"][:, None]).sum(0)
    T = torch.where(D > 0, U / D.clamp(min=1e-300), torch.zeros_like(U))
    leaves = [M.p] + [tr[k] for k in ("x0", "y0", "z0", "ux", "uy", "uz")]
    grads = torch.autograd.grad((D, T), leaves, (st["gD"], st["gT"]))
    return dict(D=D.detach(), T=T.detach(), grads=list(grads))


def _exact_steps(showers, seed):
    """The parameterised showers of generate_steps."""
    cols = {k: [] for k in ("x0", "y0", "z0", "t0", "len", "ekin", "ux", "uy", "uz")}
    x, w = np.polynomial.legendre.leggauss(8)
    first, t_ref = 0, []
    for s in showers:
        cz, y = math.cos(s["zenith"]), math.log(s["e0_mev"] / E_CRIT)
        t_g = X_SEA * math.exp(-H_OBS / H_SCALE) / cz / X0_RAD
        edge = np.linspace(0.0, t_g, 1024)
        t = 0.5 * (edge[1:] + edge[:-1])[:, None] + 0.5 * (edge[1] - edge[0]) * x
        F = np.concatenate([[0.0], np.cumsum((np.exp(t * (1.0 - 1.5 * np.log(3.0 * t / (t + 2.0 * y)))) * w).sum(1))])
        F = torch.tensor(F / F[-1], device="cuda")
        g = torch.arange(first, first + s["n"], device="cuda")
        first += s["n"]
        zero, one = torch.zeros_like(g), torch.ones_like(g)
        u = (_philox((g & _LOW, g >> 32, zero, one), seed) + _philox((g & _LOW, g >> 32, one, one), seed))
        a = (torch.searchsorted(F, u[0], right=True) - 1).clamp(0, 1022)
        depth = (a + (u[0] - F[a]) / (F[a + 1] - F[a])) * (t_g / 1023.0)
        h = (H_SCALE * torch.log(X_SEA / (depth * X0_RAD * cz))).clamp(max=H_START - 1.0)
        up = (h - H_OBS) / cz
        r, psi = -50.0 * torch.log(u[1]), 2.0 * math.pi * u[2]
        sz = math.sin(s["zenith"])
        A = (sz * math.cos(s["azimuth"]), sz * math.sin(s["azimuth"]), -cz)
        rho = math.hypot(A[0], A[1])
        b1 = (A[1] / rho, -A[0] / rho, 0.0) if rho > 1e-12 else (1.0, 0.0, 0.0)
        b2 = (A[1] * b1[2] - A[2] * b1[1], A[2] * b1[0] - A[0] * b1[2], A[0] * b1[1] - A[1] * b1[0])
        core = (s["core_x"], s["core_y"], H_OBS)
        for d, k in enumerate(("x0", "y0", "z0")):
            cols[k].append(core[d] - up * A[d] + r * (torch.cos(psi) * b1[d] + torch.sin(psi) * b2[d]))
        e = 20.0 * torch.exp(u[3] * math.log(250.0))
        sig = math.radians(3.0) * 50.0 / e * torch.sqrt(-2.0 * torch.log(u[4]))
        n1, n2 = sig * torch.cos(2.0 * math.pi * u[5]), sig * torch.sin(2.0 * math.pi * u[5])
        v = [A[d] + n1 * b1[d] + n2 * b2[d] for d in range(3)]
        norm = torch.sqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
        for d, k in enumerate(("ux", "uy", "uz")):
            cols[k].append(v[d] / norm)
        s_ref = (H_START - H_OBS) / cz
        cols["t0"].append((s_ref - up) / C_LIGHT)
        cols["len"].append(1.0 + 19.0 * u[6])
        cols["ekin"].append(e)
        t_ref.append(s_ref / C_LIGHT)
    res = {k: torch.cat(v) for k, v in cols.items()}
    return dict(res, shower=None, t_ref=torch.tensor(t_ref, dtype=torch.float64))


def exact(case, seed):
    # a crossing that FP32 decides the other way would move every record
    # after it, so the records have a value for FP64 only; the options have
    # their own oracles in the tests
    if case["call"] == "hits" and (case["option"] != "none" or case["precision"] != "fp64"):
        return None
    rng = np.random.Generator(np.random.PCG64(seed))
    showers = _showers(case, rng)
    draw_seed = int(rng.integers(1 << 62))
    if case["call"] == "steps":
        return _exact_steps(showers, draw_seed)
    atm = _atmosphere()
    tr = {k: v.double() if v.is_floating_point() else v for k, v in _tracks(case, showers, seed).items()}
    params = torch.tensor(atm["a"] + atm["b"] + atm["c"], dtype=torch.float64, device="cuda")
    tel = _telescopes(case["array"])
    if case["call"] == "readout":
        params.requires_grad_(True)
        for k in ("x0", "y0", "z0", "ux", "uy", "uz"):
            tr[k].requires_grad_(True)
        st = dict(gD=torch.tensor(rng.normal(size=len(tel)), device="cuda"),
                  gT=torch.tensor(0.1 * rng.normal(size=len(tel)), device="cuda"))
        return _exact_readout(case, _Exact(case, params), tr, draw_seed, st)
    M = _Exact(case, params)
    if case["call"] == "hits":
        return _exact_hits(case, M, tr, draw_seed, tel)
    nb = M.counts(tr)[4]
    step, j = _all_bunches(nb, 0, case["steps"])
    o = M.bunches(tr, step, j, draw_seed)
    pos = torch.stack([o["X"], o["Y"], o["cx"], o["cy"]], 1)
    tim = torch.stack([o["t"], o["he"], o["w"], o["lam"]], 1)
    fell = o["status"] != 0                     # no ground point, no arrival time
    pos[fell] = 0.0
    tim[fell, 0] = 0.0
    pos, tim = (torch.nn.functional.pad(v, (0, 0, 0, _room(case) - step.numel()))
                for v in (pos, tim))
    w = torch.where(nb > 0, M.counts(tr)[3] / nb.clamp(min=1), torch.zeros_like(tr["len"]))
    return dict(pos=pos, tim=tim, status=None, nhit=None, first_hit=None, nb=None, w=w)
