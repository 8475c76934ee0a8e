"""The work that users of libfstat have it do, as timed cases.

Every case goes through the public binding (`paper_0904_1826_gb300`): contexts,
SFT loads, template banks, compute, toplists, the batch, the stack-slide and
the proposal network.  Inputs are white complex Gaussian SFTs (E|X|^2 = 1) of
one or two detectors with a few weak continuous-wave signals, made on the GPU
from the seed alone; timing and antenna formulas are written out here in FP64.

A search returns its toplist's 2F values and the whole 2F map.  Which of two
templates whose 2F agree to FP32 rounding comes first is rounding's choice, so
the indices are compared where the 2F values are given: in `toplist`.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_0904_1826_gb300 as fs

T = 1800.0            # SFT length, s
T0 = 8.0e8            # first SFT start, s
LN2 = math.log(2.0)
# detectors: latitude, longitude, azimuth of the x-arm (rad)
DETS = ((math.radians(46.45), 0.0, math.radians(36.0)), (math.radians(30.56), 0.0, math.radians(72.0)))


# ------------------------------------------------------------------ cases

def _search(name, **kw):
    """A search: SFTs of `n_det` detectors, a bank, and the options a context takes."""
    c = dict(kind="search", name=name, n_det=2, n_sft=1200, f_base=100.0, n_sky=100, sky="lattice", n_f=1800, n_fdot=10,
             df_bins=1.0, topk=1000, form="c64", kahan=False, cover=0.0, n_sig=4)
    c.update(kw)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest call: one detector, 60 SFTs, a fine frequency grid around one candidate
        _search("follow_up", n_det=1, n_sft=60, n_sky=4, n_f=200, n_fdot=1, df_bins=1.0 / 120.0, topk=20, n_sig=1),
        # the work unit: 1 Hz, 10 spindowns, two detectors of 1200 SFTs, part of the sky
        _search("workunit", n_sky=4000, n_sig=8),
        # 16-bit storage of a work unit with odd sizes at a higher frequency
        _search("workunit_f16", n_sft=1151, f_base=217.0, n_sky=250, n_f=1733, n_fdot=7, form="f16", topk=500),
        # the learned proposal's coarse map: a regular sky grid, one spindown
        _search("coarse_map", n_sft=800, f_base=120.0, n_sky=2048, sky="grid", n_f=900, n_fdot=1, topk=100),
        # its refinement: a patch of the sky 8 times finer in sky and frequency
        _search("fine_patch", n_sft=800, f_base=120.0, n_sky=2048, sky="patch", n_f=256, n_fdot=1, df_bins=0.125, topk=1),
        # compensated sums over the SFTs, for the candidates that are published
        _search("compensated", n_sft=601, n_sky=100, n_f=901, n_fdot=4, kahan=True, topk=100),
        # SFTs with gaps in frequency: each SFT covers its own part of the band
        _search("partial_cover", n_sky=300, n_f=1800, n_fdot=5, cover=0.2),
        # a new segment of data from the host: load, whiten, search a small sky patch, read everything back
        dict(kind="reload", name="new_data", n_sft=1200, f_base=100.0, n_sky=48, n_f=1800, n_fdot=3, topk=200, half=32),
        # several work units of unlike shapes in one call
        dict(kind="batch", name="batch", n_wu=6, wu_seed=3, n_sky=400, n_sft=1600, n_f=1100, topk=100),
        # the semicoherent sum over eight segments that have been searched
        dict(kind="slide", name="stack_slide", n_seg=8, n_sft=150, f_base=100.0, n_sky=2000, n_f=1800, n_fdot=10),
        # the proposal network: steps of training, then the scores of one map's patches
        dict(kind="network", name="network", n_in=8192, hidden=256, batch=256, steps=8, patches=232),
        # the candidates of a 2F map that another program holds
        dict(kind="toplist", name="toplist", n=60_000_000, k=1000, shift=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["follow_up", "workunit", "workunit", "workunit_16", "grid", "patch", "compensated", "cover",
                       "reload", "batch", "slide", "network", "toplist"])
    if kind == "follow_up":
        n = rng.randint(20, 200)
        return _search(None, n_det=rng.randint(1, 2), n_sft=n, n_sky=rng.randint(1, 12), n_f=rng.randint(50, 400),
                       n_fdot=rng.randint(1, 3), df_bins=1.0 / (2 * n), topk=20, n_sig=1,
                       f_base=float(rng.randint(50, 400)))
    if kind in ("workunit", "workunit_16"):
        form = rng.choice(["f16", "bf16"]) if kind == "workunit_16" else "c64"
        c = _search(None, n_det=rng.randint(1, 2), n_sft=rng.randint(150, 1200), f_base=float(rng.randint(50, 400)),
                    n_sky=_log(rng, 60, 4000 if form == "c64" else 400), n_f=rng.randint(180, 1800),
                    n_fdot=rng.randint(2, 10), form=form, topk=rng.choice([1, 100, 1000]))
        return c
    if kind == "grid":
        return _search(None, n_sft=rng.randint(200, 900), f_base=float(rng.randint(50, 400)), n_sky=_log(rng, 200, 4096),
                       sky="grid", n_f=rng.randint(150, 1000), n_fdot=rng.randint(1, 2), topk=100)
    if kind == "patch":
        return _search(None, n_sft=rng.randint(200, 900), f_base=float(rng.randint(50, 400)), n_sky=_log(rng, 100, 2048),
                       sky="patch", n_f=rng.randint(64, 512), n_fdot=rng.randint(1, 2), df_bins=rng.choice([0.125, 0.25, 0.5]),
                       topk=rng.choice([1, 50]))
    if kind == "compensated":
        return _search(None, n_det=rng.randint(1, 2), n_sft=rng.randint(100, 900), n_sky=_log(rng, 10, 150),
                       n_f=rng.randint(100, 1200), n_fdot=rng.randint(1, 5), kahan=True, topk=100,
                       f_base=float(rng.randint(50, 400)))
    if kind == "cover":
        return _search(None, n_sft=rng.randint(200, 1200), n_sky=_log(rng, 30, 300), n_f=rng.randint(200, 1800),
                       n_fdot=rng.randint(1, 6), cover=rng.uniform(0.05, 0.6), topk=100, f_base=float(rng.randint(50, 400)))
    if kind == "reload":
        return dict(kind="reload", n_sft=rng.randint(200, 1300), f_base=float(rng.randint(50, 400)), n_sky=rng.randint(8, 64),
                    n_f=rng.randint(200, 1800), n_fdot=rng.randint(1, 4), topk=100, half=rng.randint(8, 60))
    if kind == "batch":
        return dict(kind="batch", n_wu=rng.randint(2, 8), wu_seed=rng.randint(0, 999), n_sky=_log(rng, 100, 500),
                    n_sft=rng.randint(300, 1700), n_f=rng.randint(200, 1400), topk=100)
    if kind == "slide":
        return dict(kind="slide", n_seg=rng.randint(2, 10), n_sft=rng.randint(20, 150), f_base=float(rng.randint(50, 300)),
                    n_sky=_log(rng, 100, 2000), n_f=rng.randint(300, 1800), n_fdot=rng.randint(1, 10))
    if kind == "network":
        return dict(kind="network", n_in=rng.choice([1024, 4096, 8192]), hidden=rng.choice([64, 128, 256]),
                    batch=rng.randint(32, 512), steps=rng.randint(1, 8), patches=rng.randint(16, 1024))
    return dict(kind="toplist", n=_log(rng, 10_000, 80_000_000), k=rng.randint(1, 5000), shift=rng.randint(0, 3))


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + stream) % (1 << 62))


def _rand(seed, stream, n):
    return np.random.default_rng([int(seed) % (1 << 32), stream]).random(n)


def _times(seed, stream, n, duty=0.7):
    """n SFT starts on the SFT grid, each slot kept with probability `duty`."""
    keep = np.nonzero(_rand(seed, stream, 2 * n + 64) < duty)[0][:n]
    assert keep.size == n
    return T0 + T * keep.astype(np.float64)


def _sky(seed, kind, n, f_base):
    if kind == "lattice":           # golden-spiral lattice over the whole sphere
        i = np.arange(n, dtype=np.float64)
        return np.stack([np.mod(2 * math.pi * i / ((1 + math.sqrt(5.0)) / 2), 2 * math.pi),
                         np.arcsin(1.0 - (2 * i + 1.0) / n)], 1)
    n_d = 32 if n >= 1024 else max(1, int(math.sqrt(n / 2)))
    n_a = -(-n // n_d)
    a, s = (np.arange(n_a) + 0.5) / n_a, (np.arange(n_d) + 0.5) / n_d
    if kind == "grid":              # cell centres over the whole sphere
        A, S = np.meshgrid(2 * math.pi * a, -1.0 + 2.0 * s, indexing="ij")
    else:                           # one patch of a quarter of the circle in alpha, half of sin(delta)
        q = int(_rand(seed, 7, 1)[0] * 8)
        A, S = np.meshgrid(0.5 * math.pi * (a + q % 4), -1.0 + s + q // 4, indexing="ij")
    return np.stack([A.ravel(), np.arcsin(S.ravel())], 1)[:n]


def _timing(det, t_start, sky, t_ref):
    """dtau, tdot, a, b [n_sky, n_sft] (FP64, on the GPU) of one detector."""
    lat, lon, az = det
    d = dict(dtype=torch.float64, device="cuda")
    t = torch.as_tensor(t_start, **d) + 0.5 * T
    sky = torch.as_tensor(sky, **d)
    c, au, re_ = 299792458.0, 1.495978707e11, 6.371e6
    w_o, w_r = 2 * math.pi / 3.15581498e7, 2 * math.pi / 86164.0905
    ob = math.radians(23.4393)
    ce, se, cl, sl = math.cos(ob), math.sin(ob), math.cos(lat), math.sin(lat)
    th, ph = w_o * t, lon + w_r * t
    sth, cth, sph, cph = torch.sin(th), torch.cos(th), torch.sin(ph), torch.cos(ph)
    r = torch.stack([au * cth + re_ * cl * cph, au * ce * sth + re_ * cl * sph, au * se * sth + re_ * sl])
    v = torch.stack([-au * w_o * sth - re_ * w_r * cl * sph, au * w_o * ce * cth + re_ * w_r * cl * cph, au * w_o * se * cth])
    e = torch.stack([-sph, cph, torch.zeros_like(t)])
    n = torch.stack([-sl * cph, -sl * sph, torch.full_like(t, cl)])
    u, y = math.cos(az) * n + math.sin(az) * e, -math.sin(az) * n + math.cos(az) * e
    al, de = sky[:, 0], sky[:, 1]
    z = torch.zeros_like(al)
    nn = torch.stack([torch.cos(de) * torch.cos(al), torch.cos(de) * torch.sin(al), torch.sin(de)], 1)
    X = torch.stack([-torch.sin(al), torch.cos(al), z], 1)
    Y = torch.stack([-torch.sin(de) * torch.cos(al), -torch.sin(de) * torch.sin(al), torch.cos(de)], 1)
    ux, uy, yx, yy = X @ u, Y @ u, X @ y, Y @ y
    a = 0.5 * (ux * ux - yx * yx) - 0.5 * (uy * uy - yy * yy)
    b = ux * uy - yx * yy
    return (t - t_ref) + (nn @ r) / c, 1.0 + (nn @ v) / c, a, b


def _data(seed, n_det, n_sft, f_base, n_f, n_sig, fd_lo, margin=8):
    """SFTs: list of (detector, t_start, bins [n_sft, n_bins, 2] FP32 on the GPU), first bin, bins."""
    k0 = int(round(f_base * T))
    k_lo, n_bins = k0 - margin, n_f + 2 * margin
    dets = []
    for i in range(n_det):
        t = _times(seed, 20 + i, n_sft)
        x = torch.randn((n_sft, n_bins, 2), generator=_gen(seed, 1 + i), device="cuda") * math.sqrt(0.5)
        dets.append((DETS[i], t, x))
    p = _rand(seed, 60, 8 * max(1, n_sig))
    for s in range(n_sig):
        q = p[8 * s:8 * s + 8]
        sky = np.array([[2 * math.pi * q[0], math.asin(2 * q[1] - 1)]])
        f, fd, rho = (k0 + n_f * (0.1 + 0.8 * q[2])) / T, fd_lo * q[3], 5.0 + 25.0 * q[4]
        ca, cb = complex(math.cos(6.28 * q[5]), math.sin(6.28 * q[5])), 0.5 * complex(math.cos(6.28 * q[6]), math.sin(6.28 * q[6]))
        tm = [_timing(d[0], d[1], sky, T0) for d in dets]
        power = sum(float((torch.abs(a[0] * ca + b[0] * cb) ** 2).sum()) for _, _, a, b in tm)
        for (d, t, x), (dtau, tdot, a, b) in zip(dets, tm):
            kh = (f + fd * dtau[0]) * tdot[0] * T
            cyc = torch.remainder(f * dtau[0] + 0.5 * fd * dtau[0] ** 2, 1.0)
            amp = (rho / math.sqrt(power)) * (a[0] * ca + b[0] * cb) * torch.exp(2j * math.pi * cyc)
            k = torch.arange(k_lo, k_lo + n_bins, dtype=torch.float64, device="cuda")
            z = amp[:, None] * torch.sinc(kh[:, None] - k) * (1.0 - 2.0 * torch.remainder(k, 2.0))
            x += torch.view_as_real(z).float()
    return dets, k_lo, n_bins


def _fdots(n):
    return -1e-9 * np.arange(n, dtype=np.float64) / max(n - 1, 1)


def _cover(seed, frac, n, n_f):
    """Covered frequency ranges: a fraction of the SFTs cover a run of 50-100 % of the band."""
    u = _rand(seed, 90, 3 * n).reshape(3, n)
    w = np.where(u[0] < frac, np.floor(n_f * (0.5 + 0.5 * u[1])), n_f).astype(np.int32)
    lo = np.floor((n_f - w) * u[2]).astype(np.int32)
    return lo, lo + w


def _batch_specs(case, seed):
    out = []
    for w in range(case["n_wu"]):
        r = np.random.default_rng([case["wu_seed"], w])     # the shapes are the case's, the data the seed's
        out.append(dict(n_det=int(r.integers(1, 3)), n_sft=max(20, int(case["n_sft"] * r.uniform(0.2, 1.0)) // 2),
                        f_base=float(r.integers(50, 400)), n_sky=max(8, int(case["n_sky"] * r.uniform(0.3, 1.0))),
                        n_f=max(30, int(case["n_f"] * r.uniform(0.15, 1.0))), n_fdot=int(r.integers(1, 13)),
                        seed=int(seed) * 64 + w))
    return out


class _Bank:
    def __init__(self, sky, f0, df, n_f, fdot):
        self.sky, self.f0, self.df, self.n_f, self.fdot, self.t_ref = sky, f0, df, n_f, fdot, T0
        self.n_sky, self.n_fdot = sky.shape[0], fdot.shape[0]


class _Wu:
    """A batch's workunit as the binding takes it."""

    def __init__(self, spec):
        dets, self.k_lo, self.n_bins = _data(spec["seed"], spec["n_det"], spec["n_sft"], spec["f_base"], spec["n_f"], 2, -1e-9)
        self.T = T
        self.detectors = [type("Det", (), dict(lat=d[0], lon=d[1], az=d[2], t_start=t, n_sft=len(t),
                                               bins=torch.view_as_complex(x).cpu().numpy())) for d, t, x in dets]
        self.bank = _Bank(_sky(0, "lattice", spec["n_sky"], 0), spec["f_base"], 1.0 / T, spec["n_f"], _fdots(spec["n_fdot"]))


def _search_inputs(case, seed):
    band = int(math.ceil(case["n_f"] * case["df_bins"]))
    dets, k_lo, n_bins = _data(seed, case["n_det"], case["n_sft"], case["f_base"], max(band, 32), case["n_sig"], -1e-9)
    bank = _Bank(_sky(seed, case["sky"], case["n_sky"], case["f_base"]), case["f_base"], case["df_bins"] / T, case["n_f"],
                 _fdots(case["n_fdot"]))
    cover = _cover(seed, case["cover"], case["n_det"] * case["n_sft"], case["n_f"]) if case["cover"] else None
    return dets, k_lo, n_bins, bank, cover


def _slide_inputs(case, seed):
    dets, k_lo, n_bins = _data(seed, 2, case["n_sft"] * case["n_seg"], case["f_base"], case["n_f"], 2, -1e-9)
    edges = [case["n_sft"] * s for s in range(case["n_seg"] + 1)]
    sky, fd = _sky(seed, "lattice", case["n_sky"], 0), _fdots(case["n_fdot"])
    return dets, k_lo, edges, sky, fd


def _network_inputs(case, seed):
    I, H, B = case["n_in"], case["hidden"], case["batch"]

    def rn(stream, *shape):
        return torch.randn(shape, generator=_gen(seed, stream), device="cuda")

    par = {"W1": rn(1, I, H) * math.sqrt(2.0 / I), "b1": rn(2, H) * 0.01, "W2": rn(3, H, H) * math.sqrt(2.0 / H),
           "b2": rn(4, H) * 0.01, "w3": rn(5, H) * math.sqrt(1.0 / H), "b3": rn(6, 1) * 0.01}
    # excess power max(2F - 16, 0) / 16 of noise and a few loud cells: mostly zeros
    def cells(stream, n):
        x = -2.0 * torch.log(torch.rand((n, I), generator=_gen(seed, stream), device="cuda").clamp_min(1e-12)) * 2.0
        return (torch.relu(x - 16.0) / 16.0).to(torch.bfloat16)

    X = [cells(10 + s, B) for s in range(case["steps"])]
    y = [(torch.rand(B, generator=_gen(seed, 40 + s), device="cuda") < 0.25).float() for s in range(case["steps"])]
    return par, X, y, cells(9, case["patches"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "search":
        dets, k_lo, n_bins, bank, cover = _search_inputs(case, seed)
        g = fs.FStat(0, dterms=8, bins_form=case["form"], topk=case["topk"], kahan=case["kahan"])
        for i, (d, t, x) in enumerate(dets):
            fs.fstat_set_sfts(g.ctx, i, d[0], d[1], d[2], T, k_lo, t, x)
        g.set_bank(bank)
        if cover is not None:
            fs.fstat_set_coverage(g.ctx, *cover)
        n = bank.n_sky * bank.n_fdot * bank.n_f
        return dict(kind=kind, g=g, n=n, k=min(case["topk"], n), out=torch.empty(n, device="cuda"))
    if kind == "reload":
        dets, k_lo, n_bins = _data(seed, 2, case["n_sft"], case["f_base"], case["n_f"], 3, -1e-9)
        host = []
        for i, (d, t, x) in enumerate(dets):     # coloured, non-stationary noise
            lev = 0.5 + torch.rand(len(t), 1, 1, generator=_gen(seed, 70 + i), device="cuda")
            slope = 1.0 + 0.3 * torch.linspace(0, 1, n_bins, device="cuda")[None, :, None]
            host.append((d, t, torch.view_as_complex(x * lev * slope).cpu().numpy()))
        bank = _Bank(_sky(seed, "lattice", case["n_sky"], 0), case["f_base"], 1.0 / T, case["n_f"], _fdots(case["n_fdot"]))
        g = fs.FStat(0, topk=case["topk"])
        fs.fstat_set_noise_floor(g.ctx, case["half"])
        return dict(kind=kind, g=g, host=host, k_lo=k_lo, bank=bank, k=case["topk"])
    if kind == "batch":
        g = fs.FStat(0, topk=case["topk"])
        wus = [_Wu(s) for s in _batch_specs(case, seed)]
        for w in wus:
            fs.fstat_batch_add(g.ctx, w)
        return dict(kind=kind, g=g, n=[w.bank.n_sky * w.bank.n_fdot * w.bank.n_f for w in wus], k=case["topk"])
    if kind == "slide":
        dets, k_lo, edges, sky, fd = _slide_inputs(case, seed)
        segs = []
        for s in range(case["n_seg"]):
            g = fs.FStat(0, topk=1)
            ts = [t[edges[s]:edges[s + 1]] for _, t, _ in dets]
            mid = 0.5 * (min(t[0] for t in ts) + max(t[-1] for t in ts) + T)
            for i, (d, t, x) in enumerate(dets):
                fs.fstat_set_sfts(g.ctx, i, d[0], d[1], d[2], T, k_lo, ts[i], x[edges[s]:edges[s + 1]].contiguous())
            fs.fstat_set_templates(g.ctx, sky, case["f_base"] - 8.0 / T, 1.0 / T, case["n_f"] + 16, fd, mid)
            g.compute()
            segs.append(g)
        out = torch.empty(case["n_sky"] * case["n_fdot"] * case["n_f"], device="cuda")
        return dict(kind=kind, segs=segs, ctxs=[g.ctx for g in segs], out=out, f0=case["f_base"], n_f=case["n_f"])
    if kind == "network":
        par, X, y, P = _network_inputs(case, seed)
        m = fs.MLP(case["n_in"], case["hidden"], max(case["batch"], case["patches"]))
        par = {k: v.cpu().numpy() for k, v in par.items()}
        m.set_params(par)
        return dict(kind=kind, m=m, par=par, X=[x.view(torch.int16) for x in X], y=y, P=P.view(torch.int16))
    n = case["n"] + case["shift"]
    v = torch.empty(n, device="cuda").exponential_(0.5, generator=_gen(seed, 1))     # 2F of noise: a chi^2 of 4
    v += torch.empty(n, device="cuda").exponential_(0.5, generator=_gen(seed, 2))
    k = min(case["k"], case["n"])
    return dict(kind=kind, v=v[case["shift"]:], k=k, idx=torch.empty(k, dtype=torch.int64, device="cuda"),
                val=torch.empty(k, device="cuda"))


def run(state):
    kind = state["kind"]
    if kind == "search":
        g = state["g"]
        g.compute()
        _, top = g.toplist(state["k"])
        fs.fstat_get_2f(g.ctx, 0, state["n"], out=state["out"])
        return {"top": top, "twoF": state["out"]}
    if kind == "reload":
        g = state["g"]
        for i, (d, t, x) in enumerate(state["host"]):
            fs.fstat_set_sfts(g.ctx, i, d[0], d[1], d[2], T, state["k_lo"], t, x)
        g.set_bank(state["bank"])
        g.compute()
        _, top = g.toplist(state["k"])
        return {"top": top, "twoF": g.twoF()}
    if kind == "batch":
        g = state["g"]
        fs.fstat_batch_compute(g.ctx)
        return {"top": [fs.fstat_batch_get_toplist(g.ctx, i, min(state["k"], n))[1] for i, n in enumerate(state["n"])],
                "twoF": [fs.fstat_batch_get_2f(g.ctx, i, 0, n) for i, n in enumerate(state["n"])]}
    if kind == "slide":
        outside = fs.fstat_stackslide(state["ctxs"], state["f0"], 1.0 / T, state["n_f"], T0, state["out"])
        return {"sum": state["out"], "outside": outside}
    if kind == "network":
        m = state["m"]
        for x, y in zip(state["X"], state["y"]):
            m.train_step(x, y, 1.0, 1e-5, want_loss=False)
        return {"params": m.get_params(), "grads": m.get_grads(), "logits": m.forward(state["P"])}
    fs.fstat_toplist_noalloc(state["v"], state["k"], state["idx"], state["val"])
    return {"idx": state["idx"], "val": state["val"]}


# ------------------------------------------------------------------ work

def _search_work(n_sft, n_bins, n_sky, n_f, n_fdot, elem=8):
    """The SFTs read and the 2F written once; per template and SFT the direct kernel sum: 16 bins of a
    complex value times a real weight (4) and its offset (1), and 20 for the twiddle and the two sums."""
    n_t = float(n_sky) * n_f * n_fdot
    return n_sft * n_bins * float(elem) + 4.0 * n_t, 100.0 * n_t * n_sft


def work(case):
    kind = case["kind"]
    if kind == "search":
        band = max(32, int(math.ceil(case["n_f"] * case["df_bins"])))
        b, f = _search_work(case["n_det"] * case["n_sft"], band + 16, case["n_sky"], case["n_f"], case["n_fdot"],
                            8 if case["form"] == "c64" else 4)
        return {"bytes": b, "flops": f}
    if kind == "reload":
        b, f = _search_work(2 * case["n_sft"], case["n_f"] + 16, case["n_sky"], case["n_f"], case["n_fdot"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        w = [_search_work(s["n_det"] * s["n_sft"], s["n_f"] + 16, s["n_sky"], s["n_f"], s["n_fdot"])
             for s in _batch_specs(case, 0)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "slide":
        n = float(case["n_sky"]) * case["n_fdot"] * case["n_f"]
        return {"bytes": 4.0 * n * (case["n_seg"] + 1), "flops": n * case["n_seg"]}
    if kind == "network":
        I, H, B, P = case["n_in"], case["hidden"], case["batch"], case["patches"]
        par = I * H + H * H + 3.0 * H + 1
        # a step reads its batch, the weights and both moments and writes weights and moments; then weights and gradients are read out
        return {"bytes": case["steps"] * (2.0 * B * I + 24.0 * par) + 8.0 * par + 2.0 * P * I,
                "flops": case["steps"] * 6.0 * B * (I * H + H * H) - case["steps"] * 2.0 * B * I * H + 2.0 * P * (I * H + H * H)}
    return {"bytes": 4.0 * case["n"] + 12.0 * case["k"], "flops": float(case["n"])}


# ------------------------------------------------------------------ in 64 bits

def _stored(x, form):
    """The values that 16-bit storage with a scale per SFT stands for."""
    if form == "c64":
        return x
    s = x.abs().amax(dim=(1, 2)) * 2.0 ** -14
    s = torch.where(s > 0, s, torch.ones_like(s))[:, None, None]
    return (x / s).to(torch.float16 if form == "f16" else torch.bfloat16).double() * s.double()


def _fstat64(dets, k_lo, bank, weights=None, cover=None):
    """2F [n_sky * n_fdot * n_f] in FP64: the direct sum of 16 bins."""
    dd = dict(dtype=torch.float64, device="cuda")
    X = torch.cat([torch.view_as_complex(x.double().contiguous()) for _, _, x in dets])
    N, nb = X.shape
    Xp = torch.nn.functional.pad(torch.view_as_real(X), (0, 0, 64, 64))
    Xr, Xi = Xp[..., 0].contiguous().reshape(-1), Xp[..., 1].contiguous().reshape(-1)
    W = nb + 128
    f = bank.f0 + bank.df * torch.arange(bank.n_f, **dd)
    fd = torch.as_tensor(bank.fdot, **dd)
    j = torch.arange(bank.n_f, device="cuda")
    cov = None if cover is None else ((j[None] >= torch.as_tensor(cover[0], device="cuda")[:, None])
                                      & (j[None] < torch.as_tensor(cover[1], device="cuda")[:, None])).double()
    rowbase = (torch.arange(N, device="cuda") * W)[:, None]
    out = torch.empty((bank.n_sky, bank.n_fdot, bank.n_f), **dd)
    sw = None if weights is None else torch.sqrt(weights)
    for s in range(bank.n_sky):
        tm = [_timing(d, t, bank.sky[s:s + 1], bank.t_ref) for d, t, _ in dets]
        dtau, tdot, a, b = (torch.cat([q[i][0] for q in tm]) for i in range(4))
        if sw is not None:
            a, b = a * sw, b * sw
        if cov is None:
            A, B, C = (a * a).sum(), (b * b).sum(), (a * b).sum()
        else:
            A, B, C = (a * a) @ cov, (b * b) @ cov, (a * b) @ cov
        D = A * B - C * C
        for d in range(bank.n_fdot):
            kh = (f[None] + (fd[d] * dtau)[:, None]) * (tdot * T)[:, None]
            cyc = torch.remainder(f[None] * dtau[:, None] + (0.5 * fd[d] * dtau * dtau)[:, None], 1.0)
            k0 = torch.floor(kh)
            kap = kh - k0
            base = k0.long() - k_lo + 64
            zr, zi = torch.zeros_like(kh), torch.zeros_like(kh)
            for k in range(-7, 9):
                w = torch.sinc(kap - k) * (1.0 if k % 2 == 0 else -1.0)
                p = (base + k).clamp_(0, W - 1) + rowbase
                zr += w * Xr[p]
                zi += w * Xi[p]
            sign = 1.0 - 2.0 * torch.remainder(k0, 2.0)
            c, q = torch.cos(2 * math.pi * cyc) * sign, torch.sin(2 * math.pi * cyc) * sign
            if cov is not None:
                c, q = c * cov, q * cov
            yr, yi = c * zr + q * zi, c * zi - q * zr
            far, fai, fbr, fbi = a @ yr, a @ yi, b @ yr, b @ yi
            v = 2.0 * (B * (far ** 2 + fai ** 2) + A * (fbr ** 2 + fbi ** 2) - 2.0 * C * (far * fbr + fai * fbi)) / D
            out[s, d] = torch.clamp_min(v, 0.0)
    return out.reshape(-1)


def _whiten64(dets, half):
    """Whitened bins and noise weights: running median of |X|^2 over 2 half + 1 bins, divided by ln 2."""
    new, sbar = [], []
    for d, t, x in dets:
        x = torch.view_as_real(torch.from_numpy(x)).cuda()
        p = (x[..., 0] * x[..., 0] + x[..., 1] * x[..., 1]).double()
        n = p.shape[1]
        S = torch.empty_like(p)
        cnt = torch.tensor([min(n - 1, k + half) - max(0, k - half) + 1 for k in range(n)], device="cuda")
        for i in range(0, p.shape[0], 64):
            q = torch.nn.functional.pad(p[i:i + 64], (half, half), value=math.inf).unfold(1, 2 * half + 1, 1).sort(dim=2).values
            ix = cnt[None, :, None].expand(q.shape[0], n, 1)
            S[i:i + 64] = 0.5 * (q.gather(2, (ix - 1) // 2) + q.gather(2, ix // 2))[..., 0] / LN2
        new.append((d, t, x.double() / torch.sqrt(S)[..., None]))
        sbar.append(S.mean(dim=1))
    w = 1.0 / torch.cat(sbar)
    return new, w / w.mean()


def _top(v, k):
    return torch.topk(v, k).values


def exact(case, seed):
    kind = case["kind"]
    if kind == "search":
        if case["n_sky"] * case["n_f"] * case["n_fdot"] * float(case["n_det"] * case["n_sft"]) > 1.2e10:
            return None     # over about 20 s in 64 bits
        dets, k_lo, _, bank, cover = _search_inputs(case, seed)
        v = _fstat64([(d, t, _stored(x, case["form"])) for d, t, x in dets], k_lo, bank, cover=cover)
        return {"top": _top(v, min(case["topk"], v.numel())), "twoF": v}
    if kind == "reload":
        s = prepare(case, seed)
        white, w = _whiten64(s["host"], case["half"])
        v = _fstat64(white, s["k_lo"], s["bank"], weights=w)
        return {"top": _top(v, case["topk"]), "twoF": v}
    if kind == "batch":
        specs = _batch_specs(case, seed)
        if sum(s["n_sky"] * s["n_f"] * s["n_fdot"] * float(s["n_det"] * s["n_sft"]) for s in specs) > 1.2e10:
            return None
        vs = []
        for s in specs:
            w = _Wu(s)
            dets = [((d.lat, d.lon, d.az), d.t_start, torch.view_as_real(torch.from_numpy(d.bins)).cuda()) for d in w.detectors]
            vs.append(_fstat64(dets, w.k_lo, w.bank))
        return {"top": [_top(v, min(case["topk"], v.numel())) for v in vs], "twoF": vs}
    if kind == "toplist":
        v = prepare(case, seed)["v"].double()
        top = torch.topk(v, case["k"] if case["k"] < v.numel() else v.numel()).values
        return {"idx": None, "val": top}
    # slide: 64-bit maps of all its segments take minutes; network: its operands are 16-bit by
    # definition of the call, and training steps amplify the last bit of a small gradient
    return None
