"""Timed cases of the w-projection gridder: imaging, gridding, prediction, sky gradients, weighting.

A case names an operation of the package ("op") and the observation it runs on: a station layout
whose baselines are tracked over `times` steps of `dt` seconds, `chans` channels between `f0` and
`f1` MHz, `pols` polarisations, a grid of side `n`, and a kernel table of `planes` w-planes with
odd supports from `s_lo` to `s_hi` and oversampling `beta`.  prepare() makes what an imaging
program holds before the call (device inputs, kernel table, grid, work list), run() makes one pass
through the package's entry points, and exact() redoes the pass in plain 64-bit torch.
"""
import math

import numpy as np
import torch

import paper_1403_4209_gb300 as wg

C0 = 299792458.0
TAPER = 7                       # bandwidth of the prolate spheroidal taper, in cells
MODES = {"stokes_i": wg.IMAGE_STOKES_I, "per_pol": wg.IMAGE_PER_POL, "stokes_linear": wg.IMAGE_STOKES_LINEAR}
_DEFAULTS = {"op": "image", "layout": "gauss", "stations": 64, "times": 600, "dt": 1.0, "chans": 4, "f0": 120.0,
             "f1": 180.0, "pols": 4, "n": 2048, "planes": 32, "s_lo": 8, "s_hi": 64, "beta": 8, "compress": True,
             "flag": 0.0, "vis": "c64", "store": "f32", "comp": False, "mode": "stokes_i", "interleave": False,
             "cross": False, "groups": 1, "plan": ""}


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # a snapshot of a small array imaged at w = 0, one polarisation, no compression: launches count
        _case("image_snapshot_w0", layout="disk", stations=32, times=256, dt=10.0, chans=1, f0=150.0, f1=150.0, pols=1,
              n=512, planes=1, s_lo=7, s_hi=7, compress=False),
        # a few seconds of a quad-polarised array, as a monitoring loop images them: the smallest call
        _case("image_seconds_quad", stations=24, times=20, chans=2, n=512, planes=8, s_lo=8, s_hi=20),
        # an hour at 1 s in 16 channels, 116 M records: the w-projection imaging step at full size, under
        # the work decomposition its autotuner picks
        _case("image_hour_16ch", times=3600, chans=16, plan="256x256r"),
        # gridding alone of a ten-minute scan, the default work decomposition
        _case("grid_scan_quad", op="grid"),
        # channel groups of a long-baseline array appended to one work list, gridded in one launch and
        # imaged at 8192^2, one polarisation, supports up to 129
        _case("image_batch_8k", layout="log", stations=256, times=120, dt=2.0, chans=4, f0=230.0, f1=260.0, pols=1, n=8192,
              planes=64, s_hi=128, groups=2, plan="256x256r"),
        # model visibilities of a scan from a gridded sky model (a major cycle's predict step)
        _case("predict_scan_quad", op="degrid"),
        # one step of fitting a sky image to visibilities: forward model, then the gradient
        _case("sky_gradient", op="sky", dt=6.0, n=1024, planes=16, s_hi=32),
        # half-precision visibilities and kernel table, compensated flushes
        _case("grid_half_compensated", op="grid", times=300, vis="half", store="f16", comp=True),
        # a subband split into narrow channels, gridded onto one continuum grid, parallel hands only
        _case("image_interleaved", times=300, chans=16, f0=150.0, f1=150.183, pols=2, interleave=True),
        # w-stacking: many cheap gridded planes, and a finaliser that transforms each of them
        _case("image_wstack", op="wstack", times=900, chans=2, pols=1, planes=16, mode="stokes_i"),
        # Briggs weights of a scan
        _case("weights_robust", op="weight", times=1200),
        # an awkward observation: odd counts, flags, a grid side that is no power of two, oversampling 5,
        # full-Stokes imaging with the cross hands swapped
        _case("image_ragged_stokes", stations=37, times=211, dt=4.0, chans=3, n=1500, planes=11, s_lo=7, s_hi=47, beta=5,
              flag=0.05, cross=True, mode="stokes_linear"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth_even(n):
    """the smallest even integer >= n whose prime factors are at most 7"""
    n += n & 1
    while True:
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 2


def draw(rng):
    while True:
        op = rng.choice(["image", "image", "grid", "grid", "degrid", "degrid", "sky", "weight", "wstack"])
        layout = rng.choice(["disk", "gauss", "gauss", "log"])
        n = _smooth_even(_log_int(rng, 400, 1400 if op == "wstack" else 4200))
        planes = 1 if layout == "disk" else _log_int(rng, 4, 16 if op == "wstack" else 48)
        s_lo = rng.choice([7, 8, 9, 11])
        s_hi = s_lo if planes == 1 else min(_log_int(rng, 16, 100), n // 8)
        f0 = rng.uniform(60.0, 250.0)
        chans = 1 if op == "wstack" else _log_int(rng, 1, 16)
        c = _case(op=op, layout=layout, stations=_log_int(rng, 8, 90), times=_log_int(rng, 12, 1500),
                  dt=float(rng.choice([1, 2, 4, 6, 10])), chans=chans, f0=round(f0, 3),
                  f1=round(f0 + (chans - 1) * rng.choice([0.0122, 0.2, 3.0]), 4), pols=rng.choice([1, 2, 4, 4]), n=n,
                  planes=planes, s_lo=s_lo, s_hi=max(s_hi, s_lo), beta=rng.choice([4, 5, 8, 8]), compress=rng.random() < 0.85,
                  flag=rng.choice([0.0, 0.0, 0.02, 0.05]), plan=rng.choice(["", "", "256x256r", "128x256r", "64x128"]))
        if op in ("image", "grid"):
            c["store"] = rng.choice(["f32", "f32", "f32", "f16", "bf16"])
            c["vis"] = rng.choice(["c64", "c64", "c64", "half"])
            c["comp"] = rng.random() < 0.15
        if op == "image":
            c["mode"] = rng.choice(["stokes_i", "stokes_i", "per_pol", "stokes_linear"])
            c["interleave"] = rng.random() < 0.2
            c["cross"] = c["pols"] == 4 and rng.random() < 0.5
            if chans % 2 == 0 and not c["interleave"] and rng.random() < 0.3:
                c["groups"] = 2
        records = c["stations"] * (c["stations"] - 1) // 2 * c["times"] * chans
        mean_s2 = sum(s * s for s in _supports(c)) / planes
        grids = n * n * c["pols"] * (planes if op == "wstack" else 1 if c["interleave"] else chans)
        if records * c["pols"] * mean_s2 <= 3e10 and 2e3 <= records <= 3e7 and grids <= 1.5e8:
            return c


# ---- the observation --------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _supports(c):
    k = c["planes"]
    out = []
    for i in range(k):
        s = int(math.ceil(c["s_lo"] + (c["s_hi"] - c["s_lo"]) * (i / (k - 1) if k > 1 else 0.0) - 1e-9))
        out.append(s + 1 - s % 2)
    return out


def _geometry(c, seed):
    """uvw [rows, 3] in metres (baseline-major, time-minor) on the device, frequencies [C] in Hz, cell
    size and largest |w| in wavelengths (every footprint fits the grid)."""
    rng = np.random.default_rng([int(seed), c["stations"], c["times"]])
    n = c["stations"]
    if c["layout"] == "disk":
        r, t = 1000.0 * np.sqrt(rng.random(n)), 2 * np.pi * rng.random(n)
    elif c["layout"] == "log":
        r, t = 10.0 ** rng.uniform(math.log10(50.0), math.log10(5000.0), n), 2 * np.pi * rng.random(n)
    else:
        r, t = 1500.0 / math.sqrt(2.0 * math.log(20.0)) * np.sqrt(-2.0 * np.log(1.0 - rng.random(n))), 2 * np.pi * rng.random(n)
    e, no, up = r * np.cos(t), r * np.sin(t), rng.normal(0.0, 1.0, n)
    lat, dec = math.radians(52.9), math.radians(45.0 + 5.0 * rng.uniform(-1, 1))
    xyz = np.stack([-math.sin(lat) * no + math.cos(lat) * up, e, math.cos(lat) * no + math.sin(lat) * up], 1)
    i, j = np.triu_indices(n, 1)
    dev = _device()
    b = torch.as_tensor(xyz[j] - xyz[i], device=dev)
    h0 = rng.uniform(-0.3, 0.3)
    h = torch.as_tensor(h0 + 7.2921159e-5 * c["dt"] * (np.arange(c["times"]) - c["times"] / 2), device=dev)
    sh, ch = torch.sin(h)[None], torch.cos(h)[None]
    x, y, z = b[:, 0:1], b[:, 1:2], b[:, 2:3]
    sd, cd = math.sin(dec), math.cos(dec)
    uvw = torch.stack([sh * x + ch * y, -sd * ch * x + sd * sh * y + cd * z, cd * ch * x - cd * sh * y + sd * z], -1).reshape(-1, 3).contiguous()
    freq = np.linspace(c["f0"] * 1e6, c["f1"] * 1e6, c["chans"])
    lam = freq.max() / C0
    du = 2.0 * float(uvw[:, :2].abs().max()) * lam / (c["n"] - max(_supports(c)) - 2)
    return uvw, torch.as_tensor(freq, device=dev), du, float(uvw[:, 2].abs().max()) * lam


def _visibilities(c, seed, uvw, freq):
    """five point sources within a degree plus noise, complex64 [rows, C, P]; weights; flags"""
    dev, (rows, C, P) = uvw.device, (uvw.shape[0], freq.shape[0], c["pols"])
    g = torch.Generator(device=dev)
    g.manual_seed(1000003 * int(seed) + 17)
    rng = np.random.default_rng([int(seed), 5])
    vis = torch.empty((rows, C, P), dtype=torch.complex64, device=dev)
    torch.view_as_real(vis).normal_(0.0, 0.01, generator=g)
    lim = math.radians(1.0)
    for flux, l, m in zip(rng.uniform(0.1, 1.0, 5), rng.uniform(-lim, lim, 5), rng.uniform(-lim, lim, 5)):
        path = uvw[:, 0] * l + uvw[:, 1] * m + uvw[:, 2] * (math.sqrt(1 - l * l - m * m) - 1)
        for ch in range(C):
            turns = path * (freq[ch] / C0)
            ph = ((turns - torch.round(turns)) * (-2 * math.pi)).float()
            v = torch.polar(torch.full_like(ph, float(flux)), ph)
            for p in {0, P - 1}:
                vis[:, ch, p] += v
    if c["flag"] > 0 or c["op"] == "weight":
        weight = torch.empty((rows, C, P), device=dev).uniform_(0.5, 1.5, generator=g)
    else:
        weight = torch.ones((rows, C, P), device=dev)
    flag = torch.zeros((rows, C, P), dtype=torch.uint8, device=dev)
    if c["flag"] > 0:
        draws = torch.empty((rows, C, P), device=dev).uniform_(generator=g)
        whole = torch.empty((rows, C, 1), device=dev).uniform_(generator=g)
        flag = ((draws < c["flag"]) | (whole < c["flag"])).to(torch.uint8)
    return vis, weight, flag


def _half(vis):
    """complex half visibilities with one float32 scale per channel"""
    amax = torch.view_as_real(vis).abs().amax(dim=(0, 2, 3))
    scale = torch.where(amax > 0, amax / 60000.0, torch.ones_like(amax))
    out = torch.view_as_real(vis)
    out = (out / scale[None, :, None, None]).to(torch.float16)
    return torch.view_as_complex(out), scale


def _sky(c, seed, C, P, dev):
    """an image of point sources on a smooth blob, float32 [C, P, N, N]"""
    n = c["n"]
    g = torch.Generator(device=dev)
    g.manual_seed(7 * int(seed) + 3)
    x = torch.arange(n, device=dev, dtype=torch.float32) - n / 2
    blob = torch.exp(-(x[:, None] ** 2 + (x[None, :] + n / 16) ** 2) / (2 * (n / 24) ** 2))
    img = 0.01 * blob.expand(C, P, n, n).clone()
    at = torch.randint(n // 4, 3 * n // 4, (2, 40), generator=g, device=dev)
    img[:, :, at[0], at[1]] += torch.rand((C, P, 40), generator=g, device=dev)
    return img


def prepare(case, seed):
    c = dict(_DEFAULTS, **case)
    uvw, freq, du, w_max = _geometry(c, seed)
    vis, weight, flag = _visibilities(c, seed, uvw, freq)
    rows, C, P, n = uvw.shape[0], c["chans"], c["pols"], c["n"]
    s = {"case": c, "op": c["op"]}
    tab = wg.ConvTable.build(du, c["planes"], w_max, c["beta"], TAPER, supports=_supports(c), store=c["store"],
                             stacking=c["op"] == "wstack")
    s["tab"] = tab
    # images are kept weighted by the correction they were divided by, so that the noise is flat over the field:
    # towards its edges the taper falls to 1e-4, and the plain quotient there is rounding noise
    corr = _corr(c, uvw.device)
    s["taper"] = (corr[:, None] * corr[None, :]).float()
    if c["op"] == "sky":
        s["model"] = wg.SkyModel(tab, uvw, freq, weight, flag, n, du, compress=c["compress"])
        s["vis"] = vis
        s["image"] = _sky(c, seed, C, P, uvw.device).requires_grad_(True)
        return s
    gridch = 1 if c["interleave"] else C * c["planes"] if c["op"] == "wstack" else C
    grid = wg.Grid(n, du, P, gridch, compensated=c["comp"])
    s["grid"] = grid
    step = C // c["groups"]
    s["batches"] = []
    for a in range(0, C, step):
        v, sc = vis[:, a:a + step].contiguous(), None
        if c["vis"] == "half":
            v, sc = _half(v)
        s["batches"].append((a, wg.VisBatch(uvw, freq[a:a + step].contiguous(), v, weight[:, a:a + step].contiguous(),
                                            flag[:, a:a + step].contiguous(), vis_scale=sc)))
    work = wg.WorkList(rows * step, step, P, max_entries=rows * C if c["groups"] > 1 else None)
    s["work"] = work
    if c["plan"]:
        seg, slots = c["plan"].rstrip("r").split("x")
        work.plan(tab, int(seg), int(slots), fixed_r=c["plan"].endswith("r"))
    if c["op"] == "degrid":
        wg.vis_compress(grid, tab, s["batches"][0][1], work, compress=c["compress"])
        wg.image_to_grid(grid, tab, _sky(c, seed, C, P, uvw.device))
    return s


def run(state):
    s, c = state, state["case"]
    if s["op"] == "sky":
        s["image"].grad = None
        pred = s["model"](s["image"] * s["taper"])      # the unknowns are the flat-noise image
        res = pred - s["vis"]
        (res.real.square().sum() + res.imag.square().sum()).backward()
        return {"vis": pred.detach(), "gradient": s["image"].grad}
    grid, tab, work, batches = s["grid"], s["tab"], s["work"], s["batches"]
    if s["op"] == "degrid":
        return {"vis": wg.degrid_vis(grid, tab, batches[0][1], work)}
    if s["op"] == "weight":
        return {"weight": wg.vis_weight(grid, tab, batches[0][1], "robust", 0.0)}
    grid.zero()
    if len(batches) > 1:
        work.clear()
        for chan0, b in batches:
            wg.vis_compress(grid, tab, b, work, compress=c["compress"], cross_swap=c["cross"], append=True, chan0=chan0)
    else:
        wg.vis_compress(grid, tab, batches[0][1], work, compress=c["compress"], interleave=c["interleave"],
                        cross_swap=c["cross"], wstack=s["op"] == "wstack")
    wg.grid_vis(grid, tab, work)
    # the normaliser is a view of the library's memory, freed with the grid: a program that keeps it copies it
    out = {"grid": grid.data, "normaliser": grid.normaliser().clone()}
    if s["op"] == "wstack":
        out["image"] = wg.grid_correct(grid, tab, mode=wg.IMAGE_WSTACK).mul_(s["taper"])
    elif s["op"] == "image":
        out["image"] = wg.grid_correct(grid, tab, mode=MODES[c["mode"]]).mul_(s["taper"])
    return out


# ---- the same in 64 bits ------------------------------------------------------------------------
def _psi(x):
    """psi_0(c, x), c = pi TAPER / 2, scaled to 1 at 0: the even Legendre series of the prolate operator's
    eigenfunction with the smallest eigenvalue"""
    c2, m = (math.pi * TAPER / 2) ** 2, 60
    k = 2.0 * np.arange(m)
    d = k * (k + 1) + c2 * (2 * k * k + 2 * k - 1) / ((2 * k - 1) * (2 * k + 3))
    e = c2 * (k + 1) * (k + 2) / ((2 * k + 3) * np.sqrt((2 * k + 1) * (2 * k + 5)))
    vec = np.linalg.eigh(np.diag(d) + np.diag(e[:-1], 1) + np.diag(e[:-1], -1))[1][:, 0]
    coef = np.zeros(2 * m)
    coef[::2] = vec * np.sqrt(k + 0.5)
    val = np.polynomial.legendre.legval
    return val(np.asarray(x, dtype=np.float64), coef) / val(0.0, coef)


def _table64(c, du, w_max, dev):
    """per plane: sub-kernels [beta^2, S, S] complex128 (ordered frac_v, frac_u)"""
    sup, beta, K = _supports(c), c["beta"], c["planes"]
    nk = 64
    while nk < 2 * max(sup):
        nk *= 2
    M = beta * nk
    eta = 2.0 * (np.arange(nk) - nk // 2) / nk
    t = _psi(eta)
    t[0] = 0.0
    t, l = torch.as_tensor(t, device=dev), torch.as_tensor(eta / (2 * du), device=dev)
    r2 = l[:, None] ** 2 + l[None, :] ** 2
    inside = r2 < 1.0
    nm1 = torch.where(inside, -r2 / (1 + torch.sqrt((1 - r2).clamp(min=0))), torch.zeros_like(r2))
    amp = torch.where(inside, t[:, None] * t[None, :], torch.zeros_like(r2))
    lo, subs = -((beta - 1) // 2), []
    for k in range(K):
        w = 0.0 if K == 1 or c["op"] == "wstack" else w_max * (k / (K - 1)) * (k / (K - 1))
        pad = torch.zeros((M, M), dtype=torch.complex128, device=dev)
        o = M // 2 - nk // 2
        x = w * nm1
        pad[o:o + nk, o:o + nk] = torch.polar(amp, 2 * math.pi * (x - torch.round(x)))
        f = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(pad))) / amp.sum()
        S, h = sup[k], (sup[k] - 1) // 2
        at = beta * (torch.arange(S, device=dev)[None, :] - h) - (torch.arange(beta, device=dev)[:, None] + lo) + M // 2
        ok = (at >= 0) & (at < M)
        at = at.clamp(0, M - 1)                                       # [beta, S]
        sub = f[at[:, None, :, None], at[None, :, None, :]]           # [fv, fu, i, j]
        sub = sub * (ok[:, None, :, None] & ok[None, :, None, :])
        subs.append(sub.reshape(beta * beta, S, S))
    return subs


def _place(c, du, w_max, uvw, freq, flag, chans):
    """per record [rows, len(chans)]: griddable, take-conjugate, cell (x, y), plane, sub-kernel"""
    beta, K, N = c["beta"], c["planes"], c["n"]
    sup = torch.as_tensor(_supports(c), device=uvw.device)
    lam = freq[chans] / C0
    sc = lam * (beta / du)
    neg = uvw[:, 2] < 0
    s = torch.where(neg, -1.0, 1.0)[:, None]
    q = [torch.ceil((s * uvw[:, a:a + 1]) * sc - 0.5).to(torch.int64) for a in (0, 1)]
    xc = [torch.div(2 * a + beta - 1, 2 * beta, rounding_mode="floor") for a in q]
    lo = -((beta - 1) // 2)
    fu, fv = q[0] - beta * xc[0] - lo, q[1] - beta * xc[1] - lo
    if K > 1:
        tm = (torch.arange(1, K + 1, dtype=torch.float64, device=uvw.device) - 0.5) / (K - 1)
        b = w_max * (tm * tm)
        w = uvw[:, 2:3].abs() * lam
        k = torch.searchsorted(b[:K - 1].contiguous(), w.contiguous(), right=True)
        ok = w < b[K - 1]
    else:
        k, ok = torch.zeros_like(q[0]), torch.ones_like(q[0], dtype=torch.bool)
    S = sup[k]
    h = (S - 1) // 2
    x, y = N // 2 + xc[0], N // 2 + xc[1]
    ok &= (x - h >= 0) & (y - h >= 0) & (x + h < N) & (y + h < N) & (flag[:, chans] == 0).any(-1)
    return ok, neg[:, None].expand_as(ok), x, y, k, fv * beta + fu


def _entries(c, seed, sum_vis=True):
    """unique (grid channel, cell, sub-kernel) groups of the griddable records: keys and the record ->
    group map, group positions and planes"""
    uvw, freq, du, w_max = _geometry(c, seed)
    N, K, b2, C = c["n"], c["planes"], c["beta"] ** 2, c["chans"]
    vis, weight, flag = _visibilities(c, seed, uvw, freq)
    ok, neg, x, y, k, sub = _place(c, du, w_max, uvw, freq, flag, list(range(C)))
    ch = torch.arange(C, device=uvw.device)[None, :].expand_as(k)
    gch = torch.zeros_like(k) if c["interleave"] else ch * K + k if c["op"] == "wstack" else ch
    key = ((((gch * N + y) * N + x) * b2 + sub) * K + k)[ok]
    uniq, inv = torch.unique(key, return_inverse=True)
    ent = {"k": uniq % K, "sub": uniq // K % b2, "x": uniq // (K * b2) % N, "y": uniq // (K * b2 * N) % N,
           "g": uniq // (K * b2 * N * N)}
    return uvw, freq, du, w_max, vis, weight, flag, ok, neg, ch, k, sub, ent, inv


def _chunks(c, ent, tab, per):
    """(entries, sample values [m, S, S], flat pixel index [m, S, S] within the grid) plane by plane"""
    N = c["n"]
    for k, S in enumerate(_supports(c)):
        at = torch.nonzero(ent["k"] == k)[:, 0]
        h, o = (S - 1) // 2, torch.arange(S, device=at.device)
        for e in torch.split(at, max(1, per // (S * S))):
            if e.numel():
                row = (ent["g"][e] * N + ent["y"][e] - h)[:, None] + o
                yield e, tab[k][ent["sub"][e]], row[:, :, None] * N + (ent["x"][e] - h)[:, None, None] + o


def _weighted(c, vis, weight, flag, neg, unweighted=False):
    wf = torch.ones_like(weight, dtype=torch.float64) if unweighted else weight.double() * (1 - flag.double())
    q = vis.to(torch.complex128)
    if c["cross"]:
        swap = [0, 2, 1, 3]
        wf = torch.where(neg[..., None], wf[..., swap], wf)
        q = torch.where(neg[..., None], q[..., swap], q)
    return wf, wf * torch.where(neg[..., None], q.conj(), q)


def _grid64(c, ent, inv, q, tab, gridch, P):
    gam = torch.zeros((ent["k"].numel(), P, 2), dtype=torch.float64, device=q.device)
    gam.index_add_(0, inv, torch.view_as_real(q.contiguous()))
    gam = torch.view_as_complex(gam)
    grid = torch.zeros((gridch * c["n"] ** 2, P, 2), dtype=torch.float64, device=q.device)
    for e, ker, pix in _chunks(c, ent, tab, 8 << 20):
        val = ker[..., None] * gam[e][:, None, None, :]
        grid.index_add_(0, pix.reshape(-1), torch.view_as_real(val.reshape(-1, P)))
    return torch.view_as_complex(grid).reshape(gridch, c["n"], c["n"], P)


def _corr(c, dev):
    n = c["n"]
    k = np.arange(n) - n // 2
    return torch.as_tensor(_psi(2.0 * k / n) * np.sinc(k / (n * c["beta"])), device=dev)


def _fft(x, inverse):
    f = torch.fft.ifft2(torch.fft.ifftshift(x, dim=(-2, -1)), norm="forward") if inverse else \
        torch.fft.fft2(torch.fft.ifftshift(x, dim=(-2, -1)))
    return torch.fft.fftshift(f, dim=(-2, -1))


def exact(case, seed):
    c = dict(_DEFAULTS, **case)
    C, P, K, N = c["chans"], c["pols"], c["planes"], c["n"]
    records = c["stations"] * (c["stations"] - 1) // 2 * c["times"] * C
    if records > 2e7 or N > 4300 or (c["op"] != "weight" and records * P * sum(s * s for s in _supports(c)) / K > 4e10):
        return None
    uvw, freq, du, w_max, vis, weight, flag, ok, neg, ch, k, sub, ent, inv = _entries(c, seed)
    if c["vis"] == "half":
        parts = []
        for a in range(0, C, C // c["groups"]):
            v, sc = _half(vis[:, a:a + C // c["groups"]].contiguous())
            parts.append(torch.view_as_complex(torch.view_as_real(v).double()) * sc.double()[None, :, None])
        vis = torch.cat(parts, 1)
    if c["op"] == "weight":
        wf = weight.double() * (1 - flag.double())
        dev = uvw.device
        _, _, x, y, _, _ = _place(c, du, w_max, uvw, freq, flag, list(range(C)))
        cell = ((ch * N + y) * N + x)[ok]
        dens = torch.zeros((C * N * N, P), dtype=torch.float64, device=dev)
        dens.index_add_(0, cell, wf[ok])
        f2 = 25.0 * wf[ok].sum(0) / dens.square().sum(0)
        out = weight.double().clone()
        out[ok] = weight.double()[ok] / (1 + dens[cell] * f2)
        return {"weight": out}
    tab = _table64(c, du, w_max, uvw.device)
    zeta = torch.stack([t.real.sum((1, 2)) for t in tab])
    icorr = 1.0 / _corr(c, uvw.device)
    cc = icorr[:, None] * icorr[None, :]
    taper = (1.0 / cc).float().double()
    if c["op"] in ("degrid", "sky"):
        img = _sky(c, seed, C, P, uvw.device)
        lead = taper if c["op"] == "sky" else 1.0
        grid = _fft(img.double() * lead * cc, False).permute(0, 2, 3, 1).reshape(-1, P)
        m = torch.zeros((ent["k"].numel(), P), dtype=torch.complex128, device=uvw.device)
        for e, ker, pix in _chunks(c, ent, tab, 8 << 20):
            m[e] = (ker.conj()[..., None] * grid[pix]).sum((1, 2))
        pred = torch.zeros(vis.shape, dtype=torch.complex128, device=uvw.device)
        mr, ng = m[inv], neg[ok][:, None]
        pred[ok] = torch.where(ng, mr.conj(), mr)
        if c["op"] == "degrid":
            return {"vis": pred}
        _, q = _weighted(c, 2 * (pred - vis.to(torch.complex128)), weight, flag, neg, unweighted=True)
        back = _grid64(c, ent, inv, q[ok], tab, C, P)
        return {"vis": pred, "gradient": _fft(back.permute(0, 3, 1, 2), True).real * cc * taper}
    gridch = 1 if c["interleave"] else C * K if c["op"] == "wstack" else C
    wf, q = _weighted(c, vis, weight, flag, neg)
    grid = _grid64(c, ent, inv, q[ok], tab, gridch, P)
    terms = wf[ok] * zeta[k[ok], sub[ok]][:, None]
    slot = (torch.zeros_like(ch) if c["interleave"] else ch * K if c["op"] == "wstack" else ch)[ok]
    norm = torch.zeros((gridch, P), dtype=torch.float64, device=uvw.device).index_add_(0, slot, terms)
    out = {"grid": grid, "normaliser": norm}
    if c["op"] == "grid":
        return out
    inv_n = torch.where(norm != 0, 1 / norm, torch.zeros_like(norm))[:, :, None, None]
    if c["op"] == "wstack":
        lm = (torch.arange(N, dtype=torch.float64, device=uvw.device) - N // 2) / (N * du)
        r2 = lm[:, None] ** 2 + lm[None, :] ** 2
        nm1 = -r2 / (1 + torch.sqrt((1 - r2).clamp(min=0)))
        acc = torch.zeros((C, P, N, N), dtype=torch.complex128, device=uvw.device)
        for g in range(gridch):
            x = (w_max * ((g % K) / (K - 1)) ** 2 if K > 1 else 0.0) * nm1
            acc[g // K] += _fft(grid[g].permute(2, 0, 1), True) * torch.polar((r2 < 1).double(), 2 * math.pi * (x - torch.round(x)))
        out["image"] = acc.real * cc * taper * inv_n[::K]
        return out
    z = _fft(grid.permute(0, 3, 1, 2), True) * cc * taper * inv_n
    if c["mode"] == "stokes_i":
        out["image"] = 0.5 * (z[:, 0] + z[:, P - 1]).real
    elif c["mode"] == "per_pol" or P == 1:
        out["image"] = z.real
    elif P == 2:
        out["image"] = 0.5 * torch.stack([z[:, 0] + z[:, 1], z[:, 0] - z[:, 1]], 1).real
    else:
        out["image"] = 0.5 * torch.stack([(z[:, 0] + z[:, 3]).real, (z[:, 0] - z[:, 3]).real, (z[:, 1] + z[:, 2]).real,
                                          (z[:, 1] - z[:, 2]).imag], 1)
    return out


_WORK = {}


def work(case):
    """bytes: every input read once and every output written once; flops: 8 per grid-point update of the
    compressed entries (one complex multiply-add a polarisation), plus 5 n log2 n a transform."""
    c = dict(_DEFAULTS, **case)
    key = repr(sorted(kv for kv in c.items() if kv[0] != "name"))
    if key in _WORK:
        return _WORK[key]
    C, P, K, N = c["chans"], c["pols"], c["planes"], c["n"]
    rows = c["stations"] * (c["stations"] - 1) // 2 * c["times"]
    uvw, freq, du, w_max = _geometry(c, 0)
    s2 = torch.as_tensor([s * s for s in _supports(c)], device=uvw.device)
    points = 0
    one = torch.zeros((rows, 1, 1), dtype=torch.uint8, device=uvw.device)
    for ch in ([list(range(C))] if c["interleave"] else [[a] for a in range(C)]):
        ok, _, x, y, k, sub = _place(c, du, w_max, uvw, freq, one.expand(rows, C, 1), ch)
        code = (((y * N + x) * c["beta"] ** 2 + sub) * K + k).reshape(-1)
        new = torch.ones_like(code, dtype=torch.bool)
        if c["compress"]:
            new[1:] = code[1:] != code[:-1]
        points += int((s2[k].reshape(-1) * (new & ok.reshape(-1))).sum())
    rec, gch = rows * C, 1 if c["interleave"] else C * (K if c["op"] == "wstack" else 1)
    visb = 4 if c["vis"] == "half" else 8
    table = 8 * c["beta"] ** 2 * int(s2.sum())
    grid = 8 * N * N * P * gch
    fft = 5.0 * N * N * math.log2(N * N)
    if c["op"] == "weight":
        w = {"bytes": 24 * rows + rec * P * 9, "flops": 8.0 * rec * P}
    elif c["op"] == "degrid":
        w = {"bytes": grid + table + 24 * rows + rec * P * 8, "flops": 8.0 * P * points}
    elif c["op"] == "sky":
        w = {"bytes": 2 * (4 * N * N * P * C) + table + 24 * rows + rec * P * 17, "flops": 16.0 * P * points + 2 * P * C * fft}
    else:
        img = 0 if c["op"] == "grid" else 4 * N * N * C * (1 if c["mode"] == "stokes_i" and c["op"] == "image" else P)
        img = img // C if c["interleave"] else img
        n_fft = 0 if c["op"] == "grid" else gch * (1 if c["mode"] == "stokes_i" and c["op"] == "image" else P)
        w = {"bytes": 24 * rows + rec * P * (visb + 5) + table + grid + img, "flops": 8.0 * P * points + n_fft * fft}
    _WORK[key] = w
    return w
