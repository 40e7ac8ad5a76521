"""The work that users of the library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` gives the standing cases, ``draw(rng)`` one more
of the same ranges, ``prepare(case, seed)`` what a program has in hand before the call (inputs on
the GPU and the experiment's handle), ``run(state)`` one pass through the public entry points,
``work(case)`` the bytes and operations a pass cannot do without, and ``exact(case, seed)`` the
same outputs in 64 bits from plain torch.

Kinds of work (``do``):
  cycle     an ensemble handed over, one data-assimilation cycle (forecast and analysis), the
            analysed ensemble taken back: ``letkf_set_deviation``, ``letkf_cycle``,
            ``letkf_get_deviation`` on device buffers.  Handing the ensemble over makes every
            pass the same work; it is what a program does that keeps its ensemble itself.
  analyze   the same with the analysis alone (``letkf_analyze``): the program has its own model
  forecast  the ensemble advanced without an analysis (spin-up, free runs): ``lbm_forecast``
  group     several small ensembles cycled as one batch: ``letkf_group_cycle``
  eigh      the batched symmetric eigensolver on its own: ``letkf_eigh_batch_ws``
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_03310_gb300 import letkf as L

DEV = "cuda"
CX = (-1, 0, 1, -1, 0, 1, -1, 0, 1)
CY = (-1, -1, -1, 0, 0, 0, 1, 1, 1)
WQ = tuple(a / 36.0 for a in (1, 4, 1, 4, 16, 4, 1, 4, 1))
VARS = {"uv": L.LETKF_OBS_U | L.LETKF_OBS_V, "ruv": L.LETKF_OBS_RHO | L.LETKF_OBS_U | L.LETKF_OBS_V,
        "v": L.LETKF_OBS_V}


def _cycle(name, nx, ny, k, **more):
    c = dict(name=name, do="cycle", nx=nx, ny=ny, k=k, tau=0.52, steps=100, network="regular",
             stride=4, vars="uv", sigma=0.01, radius=12.0, loc="gauss", infl=1.0,
             precision="fp32", spread=2e-4, scale=12.0, force=1e-5, yo="device")
    c.update(more)
    return c


GROUP_K = "16,24,32,40,48,56,64,20,16,24,32,40,48,56,64,20"


def listed():
    return [
        # the quick-start experiment: a Taylor-Green-sized flow, eight members, host observations
        _cycle("cycle_tgv32_k8", 32, 32, 8, tau=0.6, steps=50, radius=3.0, spread=5e-3, scale=3.0,
               force=0.0, yo="host"),
        # a small served experiment (short forecasts, accurate observations: large Gram matrices)
        _cycle("cycle_serve128_k16", 128, 128, 16, tau=0.55, steps=25, radius=4.0, sigma=1e-3,
               spread=2e-3, scale=16.0, force=0.0),
        # forced turbulence, sparse observations, the standing mid-size experiment
        _cycle("cycle_turb256_k32", 256, 256, 32, stride=8, radius=8.0, spread=2.2e-3, scale=8.0),
        # the same turbulence at scale, observed every fourth point, in both precisions
        _cycle("cycle_turb1024_k64", 1024, 1024, 64, force=1e-5 / 16),
        _cycle("cycle_turb1024_k64_mixed", 1024, 1024, 64, force=1e-5 / 16, precision="mixed"),
        # an early cycle on a ragged grid: wide spread, density observed too, Gaspari-Cohn,
        # inflation, an ensemble size off the powers of two; the analysis alone
        _cycle("analyze_ragged250_k40_gc", 250, 187, 40, do="analyze", stride=3, vars="ruv",
               radius=5.0, loc="gc", infl=1.05, spread=5e-3, scale=6.0),
        # the analysis shape of the large experiment with the spread of its first cycles
        _cycle("analyze_256_k64_wide", 256, 256, 64, do="analyze", spread=5e-3, scale=10.0),
        # the largest ensembles, on a clustered network with an observation-free band
        _cycle("analyze_clustered192_k128", 192, 160, 128, do="analyze", network="clustered",
               stride=2, radius=4.0, spread=5e-3, scale=16.0),
        # the mixed form on an odd-sized grid with few observations
        _cycle("cycle_ragged301_k24_mixed", 301, 215, 24, tau=0.55, steps=25, stride=5,
               radius=6.0, spread=3e-3, precision="mixed"),
        # spin-up: an ensemble advanced by an odd number of steps on a grid of odd width
        dict(name="forecast_ragged509_k20", do="forecast", nx=509, ny=380, k=20, tau=0.52,
             steps=25, spread=5e-3, scale=8.0, force=1e-5),
        # sixteen small ensembles of mixed sizes cycled as one batch on a clustered network
        dict(name="group_16x64", do="group", nx=64, ny=64, ks=GROUP_K, tau=0.55, steps=25,
             network="clustered", stride=2, radius=2.0, sigma=0.01, spread=5e-3, scale=3.0),
        # the batched eigensolver: 128 x 128 matrices with their eigenvectors
        dict(name="eigh_16384_k32", do="eigh", n=16384, k=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.06:
        return dict(do="eigh", n=_log_int(rng, 500, 30000), k=rng.randint(8, 64))
    if u < 0.12:
        ks = ",".join(str(rng.randint(12, 64)) for _ in range(rng.randint(3, 12)))
        return dict(do="group", nx=rng.randint(40, 96), ny=rng.randint(40, 96), ks=ks, tau=0.55,
                    steps=rng.randint(10, 40), network="clustered", stride=2,
                    radius=rng.choice([2.0, 3.0]), sigma=0.01, spread=5e-3, scale=3.0)
    if u < 0.24:
        return dict(do="forecast", nx=_log_int(rng, 48, 1024), ny=_log_int(rng, 48, 1024),
                    k=rng.randint(8, 64), tau=rng.choice([0.52, 0.55, 0.6]),
                    steps=rng.randint(5, 60), spread=5e-3, scale=8.0,
                    force=rng.choice([0.0, 1e-5]))
    c = _cycle("", _log_int(rng, 32, 1024), _log_int(rng, 32, 1024),
               rng.choice([8, 16, 24, 32, 32, 40, 48, 64, 64, rng.randint(5, 64), 100, 128]))
    del c["name"]
    if rng.random() < 0.35:
        c["do"] = "analyze"
    if rng.random() < 0.7:  # grid edges that are multiples of 4, as most programs choose them
        c["nx"], c["ny"] = (max(32, v // 4 * 4) for v in (c["nx"], c["ny"]))
    c["tau"] = rng.choice([0.52, 0.55, 0.6])
    c["steps"] = rng.choice([10, 25, 25, 50, 100, rng.randint(5, 60)])
    c["stride"] = rng.choice([3, 4, 4, 5, 8])
    c["radius"] = rng.choice([3.0, 4.0, 5.0, 6.0, 8.0, 12.0])
    c["spread"] = math.exp(rng.uniform(math.log(2e-4), math.log(5e-3)))
    c["scale"] = rng.choice([6.0, 8.0, 12.0, 16.0])
    c["sigma"] = rng.choice([0.01, 0.01, 0.003])
    c["force"] = rng.choice([0.0, 1e-6])
    c["precision"] = rng.choice(["fp32", "fp32", "mixed"])
    c["loc"] = rng.choice(["gauss", "gauss", "gc"])
    c["vars"] = rng.choice(["uv", "uv", "uv", "ruv", "v"])
    c["infl"] = rng.choice([1.0, 1.0, 1.05])
    c["yo"] = rng.choice(["device", "device", "host"])
    if rng.random() < 0.2:
        c["network"], c["stride"], c["radius"] = "clustered", 2, min(c["radius"], 4.0)
    while _cost_s(c) > 0.1:  # no costlier than the largest listed case
        c["nx"], c["ny"] = max(32, int(c["nx"] * 0.8)), max(32, int(c["ny"] * 0.8))
        if c["nx"] == 32 and c["ny"] == 32:
            break
    return c


def _cost_s(c):
    """A rough upper estimate of a pass, in seconds: only draw() uses it."""
    npts, k = c["nx"] * c["ny"], c["k"]
    t = npts * _mean_local(c) * len(c["vars"]) * k * k / 25e12
    t += npts * (3e-6 if k > 64 else k * k * k * 6e-13)
    if c["do"] == "cycle":
        t += c["steps"] * npts * k * 9e-12
    return t


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _field(nx, ny, rms, scale, gen):
    """A smooth divergence-free velocity field of the given RMS and correlation length."""
    noise = torch.randn((ny, nx), generator=gen, device=DEV, dtype=torch.float64)
    kx = 2 * math.pi * torch.fft.rfftfreq(nx, device=DEV, dtype=torch.float64)[None, :]
    ky = 2 * math.pi * torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None]
    psi = torch.fft.rfft2(noise) * torch.exp(-0.25 * scale * scale * (kx * kx + ky * ky))
    u = torch.fft.irfft2(1j * ky * psi, s=(ny, nx))
    v = torch.fft.irfft2(-1j * kx * psi, s=(ny, nx))
    f = rms * math.sqrt(2.0) / math.sqrt(float((u * u + v * v).mean()))
    return u * f, v * f


def _equilibrium(u, v, rho):
    """Deviations g = f_eq(rho, u) - w of one member, [9, ny, nx] in 64 bits."""
    base = 1.0 - 1.5 * (u * u + v * v)
    out = []
    for q in range(9):
        cu = CX[q] * u + CY[q] * v
        out.append(WQ[q] * (rho * (base + 3.0 * cu + 4.5 * cu * cu) - 1.0))
    return torch.stack(out)


def _flow(case, k, seed):
    """(ensemble deviations [k, 9, ny, nx] FP32, truth's [1, 9, ny, nx]): a smooth flow and
    members that differ from it by smooth perturbations of the case's spread."""
    nx, ny, gen = case["nx"], case["ny"], _gen(seed)
    tu, tv = _field(nx, ny, 0.02, max(4.0, min(nx, ny) / 8.0), gen)
    one = torch.ones((ny, nx), dtype=torch.float64, device=DEV)
    g = torch.empty((k, 9, ny, nx), dtype=torch.float32, device=DEV)
    for m in range(k):
        u, v = _field(nx, ny, case["spread"], case["scale"], gen)
        r, _ = _field(nx, ny, 0.1 * case["spread"], case["scale"], gen)
        g[m] = _equilibrium(tu + u, tv + v, one + r).float()
    return g, _equilibrium(tu, tv, one).float()[None]


def _force(case):
    """Kolmogorov forcing F_x = amp sin(4 * 2 pi y / ny), [2, ny, nx] FP32, or None."""
    if not case.get("force"):
        return None
    ny, nx = case["ny"], case["nx"]
    f = np.zeros((2, ny, nx), np.float32)
    f[0] = (case["force"] * np.sin(8.0 * np.pi * np.arange(ny) / ny))[:, None]
    return f


def _network(case):
    """Observation points [L][2]: every stride-th point, or a dense patch (every stride-th) in
    a sparse background (every 8 * stride-th) with a band that has none."""
    nx, ny, s = case["nx"], case["ny"], case["stride"]
    if case["network"] == "regular":
        pts = [(x, y) for y in range(0, ny, s) for x in range(0, nx, s)]
    else:
        keep = {(x, y) for y in range(0, ny, 4 * s) for x in range(0, nx, 4 * s)}
        keep |= {(x, y) for y in range(4, ny // 2, s) for x in range(4, nx // 2, s)}
        lo, hi = int(0.6 * ny), int(0.9 * ny)
        pts = sorted((p for p in keep if not lo <= p[1] < hi), key=lambda p: (p[1], p[0]))
    return np.asarray(pts, dtype=np.int32).reshape(-1, 2)


def _observe(g, net, names):
    """h(x) of every member at the observation points: [members, L, V], g = f - w, its type."""
    xs, ys = (torch.from_numpy(net[:, i].astype(np.int64)).to(g.device) for i in (0, 1))
    p = g[:, :, ys, xs]
    rho = 1.0 + p.sum(1)
    j = [sum(c[q] * p[:, q] for q in range(9) if c[q]) for c in (CX, CY)]
    of = {"r": rho, "u": j[0] / rho, "v": j[1] / rho}
    return torch.stack([of[n] for n in names], dim=-1)


def _lbm(g, tau, steps, force):
    """The D2Q9 BGK steps of deviations g (in g's own type), plain torch."""
    f = None if force is None else torch.from_numpy(force).to(g.device).to(g.dtype)
    for _ in range(steps):
        rho = 1.0 + g.sum(1)
        u = sum(CX[q] * g[:, q] for q in range(9) if CX[q]) / rho
        v = sum(CY[q] * g[:, q] for q in range(9) if CY[q]) / rho
        base = 1.0 - 1.5 * (u * u + v * v)
        out = torch.empty_like(g)
        for q in range(9):
            cu = CX[q] * u + CY[q] * v
            eq = WQ[q] * (rho * (base + 3.0 * cu + 4.5 * cu * cu) - 1.0)
            s = g[:, q] + (eq - g[:, q]) / tau
            if f is not None:
                s = s + 3.0 * WQ[q] * (CX[q] * f[0] + CY[q] * f[1])
            out[:, q] = torch.roll(s, shifts=(CY[q], CX[q]), dims=(1, 2))
        g = out
    return g


def _observations(case, truth, net, seed):
    """Noisy observations of the truth at the analysis time, [L * V] FP32."""
    if case["do"] != "analyze":
        truth = _lbm(truth, case["tau"], case["steps"], _force(case))
    y = _observe(truth.double(), net, case.get("vars", "uv"))[0]
    noise = torch.randn(y.shape, generator=_gen(seed + 7919), device=DEV, dtype=torch.float64)
    return (y + case["sigma"] * noise).float().reshape(-1).contiguous()


def _experiment(case, k, net):
    names = case.get("vars", "uv")
    var = np.full(len(net) * len(names), case["sigma"] ** 2, dtype=np.float32)
    return L.Experiment(
        case["nx"], case["ny"], k, case["tau"], net, var, obs_vars=VARS[names],
        loc_radius=case["radius"], force=_force(case), infl=case.get("infl", 1.0),
        precision=L.LETKF_MIXED if case.get("precision") == "mixed" else L.LETKF_FP32,
        loc_kind=L.LETKF_LOC_GC if case.get("loc") == "gc" else L.LETKF_LOC_GAUSS)


def _matrices(case, seed):
    """Symmetric matrices (k - 1) I + Y^T Y of full rank, [n, k, k] FP32."""
    n, k = case["n"], case["k"]
    y = torch.randn((n, 2 * k, k), generator=_gen(seed), device=DEV) * 0.7
    q = torch.bmm(y.transpose(1, 2).double(), y.double())
    q += (k - 1) * torch.eye(k, device=DEV, dtype=torch.float64)
    return q.float().contiguous()


# ---------------------------------------------------------------- prepare and run

def prepare(case, seed):
    s = {"case": case, "do": case["do"]}
    if case["do"] == "eigh":
        n, k = case["n"], case["k"]
        s["q"] = _matrices(case, seed)
        s["lam"] = torch.empty((n, k), device=DEV)
        s["vec"] = torch.empty((n, k, k), device=DEV)
        s["bytes"] = L.letkf_eigh_workspace_bytes(n, k)
        s["ws"] = torch.empty(s["bytes"] + 256, dtype=torch.uint8, device=DEV)
        return s
    ks = [int(v) for v in case["ks"].split(",")] if case["do"] == "group" else [case["k"]]
    net = _network(case) if case["do"] != "forecast" else np.zeros((0, 2), np.int32)
    s["exps"], s["g0"], s["yo"], s["out"] = [], [], [], []
    for i, k in enumerate(ks):
        g0, truth = _flow(case, k, seed * 64 + i)
        if case["do"] == "forecast":
            e = L.Experiment(case["nx"], case["ny"], k, case["tau"], net,
                             np.zeros(0, np.float32), force=_force(case))
        else:
            yo = _observations(case, truth, net, seed * 64 + i)
            s["yo"].append(yo.cpu().numpy() if case.get("yo") == "host" else yo)
            e = _experiment(case, k, net)
        s["exps"].append(e)
        s["g0"].append(g0)
        s["out"].append(torch.empty_like(g0))
    torch.cuda.synchronize()
    if case["do"] == "forecast":
        e, g0 = s["exps"][0], s["g0"][0]
        e.set_deviation(g0)
        s["steps"] = case["steps"]
    return s


def _take_back(e, out):
    L.letkf_get_deviation(e.h, out.data_ptr(), 0, e.k, L.LETKF_DEVICE)


def run(s):
    do, case = s["do"], s["case"]
    if do == "eigh":
        base = (s["ws"].data_ptr() + 255) // 256 * 256
        rc = L.letkf_eigh_batch_ws(case["n"], case["k"], s["q"].data_ptr(), s["lam"].data_ptr(),
                                   s["vec"].data_ptr(), 0, base, s["bytes"],
                                   torch.cuda.current_stream().cuda_stream)
        if rc != L.LETKF_OK:
            raise L.LetkfError(rc, "letkf_eigh_batch_ws")
        return {"eigval": s["lam"], "evec": s["vec"]}
    if do == "group":
        for e, g0 in zip(s["exps"], s["g0"]):
            e.set_deviation(g0)
        L.letkf_group_cycle(s["exps"], case["steps"], s["yo"])
        for e, out in zip(s["exps"], s["out"]):
            _take_back(e, out)
        return s["out"]
    e, out = s["exps"][0], s["out"][0]
    if do == "forecast":  # the ensemble stays on the handle from one pass to the next
        e.forecast(case["steps"])
    else:
        e.set_deviation(s["g0"][0])
        if do == "cycle":
            e.cycle(case["steps"], s["yo"][0])
        else:
            e.analyze(s["yo"][0])
    _take_back(e, out)
    return out


# ---------------------------------------------------------------- what a pass cannot do without

def _mean_local(case):
    """Local observation points per grid point, averaged (an estimate from the density)."""
    cells = case["nx"] * case["ny"]
    s = case["stride"]
    n_obs = cells / (s * s) if case["network"] == "regular" else cells * (0.25 + 0.05) / (s * s)
    return n_obs * min(1.0, math.pi * 40.0 / 3.0 * case["radius"] ** 2 / cells)


def work(case):
    """Bytes: the ensemble in and out once, observations and forcing in.  Operations: 130 per
    node and D2Q9 step; the products dy dy^T and dy d of every observation point (the upper
    triangle) and, per grid point and local observation point, one multiply-add for each of
    their entries; three products of the ten rows [dX; c] with the k x k matrix per point."""
    if case["do"] == "eigh":
        n, k = case["n"], case["k"]
        return {"bytes": 4.0 * n * k * (2 * k + 1), "flops": 9.0 * n * k ** 3}
    total = {"bytes": 0.0, "flops": 0.0}
    npts = case["nx"] * case["ny"]
    for k in ([int(v) for v in case["ks"].split(",")] if case["do"] == "group" else [case["k"]]):
        total["bytes"] += 2.0 * 36.0 * npts * k + (8.0 * npts if case.get("force") else 0.0)
        if case["do"] != "analyze":
            total["flops"] += 130.0 * case["steps"] * npts * k
        if case["do"] != "forecast":
            total["flops"] += npts * (_mean_local(case) * k * (k + 3) + 60.0 * k * k)
    return total


# ---------------------------------------------------------------- 64-bit results

def _weights(case, y0, y1, net):
    """Localization weights of the grid rows [y0, y1) to every observation point, FP64."""
    nx, ny, r = case["nx"], case["ny"], case["radius"]
    ox, oy = (torch.from_numpy(net[:, i].astype(np.int64)).to(DEV) for i in (0, 1))
    x = torch.arange(nx, device=DEV).repeat(y1 - y0)
    y = torch.arange(y0, y1, device=DEV).repeat_interleave(nx)
    dx = (ox[None] - x[:, None] + nx // 2) % nx - nx // 2
    dy = (oy[None] - y[:, None] + ny // 2) % ny - ny // 2
    d2 = (dx * dx + dy * dy).double()
    if case.get("loc") == "gc":
        z = d2.sqrt() / (math.sqrt(10.0 / 3.0) * r)
        near = (((-0.25 * z + 0.5) * z + 0.625) * z - 5.0 / 3.0) * z * z + 1.0
        zf = z.clamp(1.0, 2.0)
        far = ((((zf / 12.0 - 0.5) * zf + 0.625) * zf + 5.0 / 3.0) * zf - 5.0) * zf + 4.0 \
            - 2.0 / (3.0 * zf)
        w = torch.where(z <= 1.0, near, far)
    else:
        w = torch.exp(-d2 / (2.0 * r * r))
    return torch.where(d2 < 40.0 * r * r / 3.0, w, torch.zeros_like(w))


def _inverse_root(q):
    """q^(-1/2) of symmetric positive definite q [n, k, k] by the coupled Newton-Schulz
    iteration (Higham, Functions of Matrices, 2008, section 6.7)."""
    k = q.shape[-1]
    eye = torch.eye(k, device=q.device, dtype=q.dtype)
    s = q.abs().sum(-1).amax(-1)[:, None, None]
    y, z = q / s, eye.expand_as(q).contiguous()
    for _ in range(60):
        t = 1.5 * eye - 0.5 * torch.bmm(z, y)
        y, z = torch.bmm(y, t), torch.bmm(t, z)
        if float((t - eye).abs().max()) < 1e-14 * k:
            break
    return z / s.sqrt()


def _transform(a, c, x, infl):
    """Analysis blocks [n, 9, k] of the forecast blocks x from A [n, k, k] and c [n, k]."""
    k = a.shape[-1]
    q = a + ((k - 1) / infl) * torch.eye(k, device=a.device, dtype=a.dtype)
    root = _inverse_root(q)
    wbar = torch.bmm(root, torch.bmm(root, c[:, :, None]))
    mean = x.mean(-1, keepdim=True)
    dx = x - mean
    return mean + torch.bmm(dx, wbar) + math.sqrt(k - 1) * torch.bmm(dx, root)


def _analysis(case, g, yo, net):
    """The analysed ensemble of g [k, 9, ny, nx] (64 bits)."""
    k, nx, ny = g.shape[0], case["nx"], case["ny"]
    names = case.get("vars", "uv")
    yf = _observe(g, net, names)
    ybar = yf.mean(0)
    rinv = 1.0 / float(np.float32(case["sigma"] ** 2))
    dy = (yf - ybar).permute(1, 2, 0)                       # [L, V, k]
    d = yo.double().reshape(-1, len(names)) - ybar          # [L, V]
    i, j = torch.triu_indices(k, k, device=DEV)
    pairs = rinv * torch.einsum("lvp,lvp->lp", dy[:, :, i], dy[:, :, j])
    proj = rinv * torch.einsum("lvk,lv->lk", dy, d)
    z = torch.cat([pairs, proj], dim=1)
    out = torch.empty_like(g)
    rows = max(1, int(1.5e8 // (nx * max(k * k * 6, len(net) * 4))))
    for y0 in range(0, ny, rows):
        y1 = min(ny, y0 + rows)
        ac = _weights(case, y0, y1, net) @ z
        a = torch.zeros((ac.shape[0], k, k), dtype=g.dtype, device=DEV)
        a[:, i, j] = ac[:, :len(i)]
        a[:, j, i] = ac[:, :len(i)]
        x = g[:, :, y0:y1].permute(2, 3, 1, 0).reshape(-1, 9, k)
        xa = _transform(a, ac[:, len(i):], x, case.get("infl", 1.0))
        out[:, :, y0:y1] = xa.reshape(y1 - y0, nx, 9, k).permute(3, 2, 0, 1)
    return out


def exact(case, seed):
    if case["do"] == "eigh":
        return None  # the eigenvalues come in the solver's own order, the vectors up to a sign
    group = case["do"] == "group"
    ks = [int(v) for v in case["ks"].split(",")] if group else [case["k"]]
    npts, k = case["nx"] * case["ny"], max(ks)
    net = None if case["do"] == "forecast" else _network(case)
    ops = len(ks) * (0 if net is None else npts * (1.0 * len(net) * k * k + 80.0 * k ** 3))
    moved = 0 if case["do"] == "analyze" else len(ks) * case["steps"] * npts * k * 9 * 8 * 30.0
    if ops > 8e12 or moved > 3e13:
        return None  # over about 20 seconds
    outs = []
    for i, k in enumerate(ks):
        g, truth = _flow(case, k, seed * 64 + i)
        g = g.double()
        if case["do"] != "analyze":
            g = _lbm(g, case["tau"], case["steps"], _force(case))
        if net is not None:
            g = _analysis(case, g, _observations(case, truth, net, seed * 64 + i), net)
        outs.append(g)
    return outs if group else outs[0]
