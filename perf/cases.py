"""The work that programs have this framework do, as cases that can be timed and checked.

Each case is one call sequence of a user's program through the public entry points
(`Plan`, its methods and `smeared_psf`), on synthetic observations of the shapes that the
repository's configurations use: a 16-antenna compact array, the 64-antenna array (32
antennas within 1 km, 32 within 8 km) with fixed or baseline-dependent averaging, and the
many-channel setting of the PSF-width survey.  The antenna layout of a case is fixed, as a
telescope's is; the seed sets the hour angle at which the track starts, the sky positions,
the cotangents and the images.

`exact` evaluates the definitions (P = sum_k W_k Re(D_k exp(2 pi i u_k . dl)) with the bin
average, Method 1 or Method 2 as D) in float64 with plain torch.
"""
import math
import types

import numpy as np
import torch

import paper_2009_07010_gb300 as psf

C_LIGHT = 299792458.0
OMEGA_E = 7.2921150e-5
ARCSEC = math.pi / (180.0 * 3600.0)
DEG = math.pi / 180.0
WTERM = 1   # PSF_WTERM: (l0, m0, n0 - 1) in the smearing


# ---------------------------------------------------------------- the cases
def _case(name, task, array, minutes, tavg, nchan, favg, f0, df, prec, method, npos, npix, cell, radius, flags=0,
          iters=0):
    c = {"task": task, "array": array, "minutes": minutes, "tavg": tavg, "nchan": nchan, "favg": favg,
         "f0": f0, "df": df, "prec": prec, "method": method, "npos": npos, "npix": npix, "cell": cell,
         "radius": radius, "flags": flags, "iters": iters}
    return dict(c, name=name) if name else c


def _family(kind, name=None, rng=None):
    """One case of a family: its listed sizes, or with `rng` sizes drawn from its range."""
    r = rng

    def pick(listed, lo=None, hi=None, step=1, log=False, of=None):
        if r is None:
            return listed
        if of is not None:
            return r.choice(of)
        v = math.exp(r.uniform(math.log(lo), math.log(hi))) if log else r.uniform(lo, hi)
        return int(round(v / step)) * step

    if kind == "small_fp32":
        # the smallest call, in the default precision: one cutout of a compact array's hour
        return _case(name, "cutout", pick("disk16", of=["disk8", "disk12", "disk16"]), pick(60, 20, 75), 10, 4, 1,
                     1.4e9, 1e6, "fp32", pick("exact", of=["exact", "uv", "img"]), pick(1, 1, 3),
                     pick(64, 24, 96, 2), 2.0, 0.02)
    if kind == "small_step":
        # the same call on the tensor cores: the exact cutout and both approximations to it
        return _case(name, "step", pick("disk16", of=["disk8", "disk12", "disk16"]), pick(60, 20, 75), 10, 4, 1,
                     1.4e9, 1e6, pick("tc_fp16", of=["tc_fp16", "tc_bf16"]), "exact", 1,
                     pick(64, of=[64, 96, 128]), 2.0, 0.02)
    if kind == "step":
        # the benchmark's step: one 128 x 128 cutout of the 4 h MeerKAT-shaped observation
        return _case(name, "step", "mk64", pick(240, 30, 230, log=True), 8, 16, 1, 856e6, 0.836e6, "tc_fp16", "exact",
                     1, pick(128, of=[64, 128]), 1.5, 0.03)
    if kind == "batch_exact":
        # exact PSFs of many directions (one per bright source), baseline-dependent averaging
        return _case(name, "batch", "mk64", pick(120, 20, 110, log=True), 0, 8, 1, 856e6, 0.836e6,
                     pick("tc_fp16", of=["tc_fp16", "tc_bf16"]), "exact", pick(256, 64, 250), pick(64, of=[32, 64]),
                     1.5, 0.017)
    if kind == "batch_mixed":
        # an approximation for directions with cutouts of several sizes (32 to 256 pixels)
        return _case(name, "batch", "mk64", pick(60, 10, 55, log=True), 0, 8, 1, 856e6, 0.836e6, "tc_fp16",
                     pick("uv", of=["uv", "img"]), pick(512, 100, 500), 0, 1.5, 0.017)
    if kind == "split":
        # split precision with the w term: a few cutouts of a size that fills no tile
        return _case(name, "cutout", "mk64", pick(30, 10, 40), 8, 16, 1, 856e6, 0.836e6,
                     pick("tc_bf16x3", of=["tc_fp16x3", "tc_bf16x3"]), pick("exact", of=["exact", "uv"]),
                     pick(2, 1, 3), pick(100, 34, 126, 2), 1.5, 0.03, WTERM)
    if kind == "fp32_ragged":
        # the FP32 form at a larger, ragged size
        return _case(name, "cutout", "mk64", pick(20, 5, 20), 8, 16, 1, 856e6, 0.836e6, "fp32",
                     pick("exact", of=["exact", "uv"]), pick(2, 1, 2), pick(150, 66, 150, 2), 1.5, 0.03)
    if kind == "survey":
        # the PSF-width survey: exact PSFs at several distances, 20 to 40 raw channels per
        # output channel
        favg, tavg = (20, 10) if r is None else r.choice([(20, 10), (40, 20)])
        return _case(name, "batch", "mk64", pick(120, 30, 120), tavg, 120, favg, 1.397e9, 50e3, "tc_fp16", "exact",
                     pick(73, 40, 73), 64, 1.0, 0.075)
    if kind == "grad":
        # a training step on positions and weights: forward and adjoint on the tensor cores
        return _case(name, "grad", "mk64", pick(30, 8, 28, log=True), 0, 8, 1, 856e6, 0.836e6, "tc_fp16",
                     pick("exact", of=["exact", "uv"]), pick(96, 33, 96), pick(64, of=[32, 64]), 1.5, 0.017)
    if kind == "grad_fp32":
        # the same in FP32 on a small array
        return _case(name, "grad", pick("disk16", of=["disk8", "disk12", "disk16"]), pick(60, 20, 60), 10, 4, 1, 1.4e9,
                     1e6, "fp32", pick("exact", of=["exact", "uv"]), pick(4, 1, 4), pick(48, 24, 64, 2), 2.0, 0.02)
    if kind == "grid":
        # gridded Method 2 over a field of directions (the table is kept by the plan)
        return _case(name, "grid", "mk64", pick(60, 20, 60), 8, 16, 1, 856e6, 0.836e6, "tc_fp16", "img_grid",
                     pick(4096, 1, 4000, log=True), pick(128, of=[32, 64, 128]), 1.5, 0.03)
    if kind == "clean":
        # CLEAN with the gridded PSF at every peak
        n = pick(2048, of=[512, 1024, 2048])
        return _case(name, "clean", "mk64", pick(60, 20, 60), 8, 16, 1, 856e6, 0.836e6, "tc_fp16", "img_grid", n,
                     pick(128, of=[64, 128]), 1.5, 0.03, 0, pick(512, 50, 500, log=True))
    raise ValueError(kind)


_LISTED = [("one_cutout_compact_fp32", "small_fp32"), ("step_compact_fp16", "small_step"),
           ("step_meerkat_4h_fp16", "step"), ("batch_256x64_exact_fp16", "batch_exact"),
           ("batch_mixed_512_uv_fp16", "batch_mixed"), ("cutouts_100_wterm_bf16x3", "split"),
           ("cutouts_150_fp32", "fp32_ragged"), ("survey_73x64_exact_fp16", "survey"),
           ("train_96x64_fp16", "grad"), ("train_4x48_fp32", "grad_fp32"), ("grid_4096x128", "grid"),
           ("clean_2048_grid", "clean")]


def listed():
    return [_family(kind, name) for name, kind in _LISTED]


def draw(rng):
    return _family(rng.choice([kind for _, kind in _LISTED]), None, rng)


# ---------------------------------------------------------------- inputs
def _antennas(array):
    """East and north coordinates in metres, the same for every seed."""
    g = np.random.default_rng(20200914)

    def disk(n, radius):
        q, phi = radius * np.sqrt(g.random(n)), 2.0 * np.pi * g.random(n)
        return np.stack([q * np.cos(phi), q * np.sin(phi)], axis=1)

    if array == "mk64":
        return np.concatenate([disk(32, 1000.0), disk(32, 8000.0)])
    return disk(int(array[4:]), 1000.0)


def _baselines(array):
    enu = _antennas(array)
    p, q = np.triu_indices(enu.shape[0], k=1)
    return enu[q] - enu[p]


def _tavg(case):
    b = _baselines(case["array"])
    if case["tavg"]:
        return np.full(b.shape[0], case["tavg"], np.int32)
    blen = np.hypot(b[:, 0], b[:, 1])
    return np.clip(np.rint(8.0 * np.median(blen) / np.maximum(blen, 1e-9)), 2, 30).astype(np.int32)


def _nvis(case):
    return int((case["minutes"] * 60 // _tavg(case).astype(np.int64)).sum()) * (case["nchan"] // case["favg"])


def _uvw(case, seed):
    """Baseline tracks in metres, float64 [nbl, ntime, 3] on the GPU: 1 s samples around
    transit plus the seed's hour angle (latitude -30.7 deg, declination -30 deg)."""
    b = torch.from_numpy(_baselines(case["array"])).cuda()
    e, n = b[:, :1], b[:, 1:]
    nt = case["minutes"] * 60
    ha0 = np.random.default_rng([seed, 1]).uniform(-0.3, 0.3)
    H = ha0 + OMEGA_E * (torch.arange(nt, dtype=torch.float64, device="cuda")[None, :] - 0.5 * nt + 0.5)
    sl, cl = math.sin(-30.7 * DEG), math.cos(-30.7 * DEG)
    sd, cd = math.sin(-30.0 * DEG), math.cos(-30.0 * DEG)
    X, Y, Z = -sl * n, e, cl * n
    sh, ch = torch.sin(H), torch.cos(H)
    return torch.stack([sh * X + ch * Y, -sd * ch * X + sd * sh * Y + cd * Z, cd * ch * X - cd * sh * Y + sd * Z],
                       dim=2)


def _observation(case, seed):
    nt, nc = case["minutes"] * 60, case["nchan"]
    return types.SimpleNamespace(
        uvw_m=_uvw(case, seed).cpu().numpy(), time_s=np.arange(nt) - 0.5 * nt + 0.5,
        freq_hz=case["f0"] + (np.arange(nc) + 0.5) * case["df"], chan_width_hz=np.full(nc, case["df"]),
        tavg=_tavg(case), favg=case["favg"], weights=None)


def _positions(case, seed):
    """Directions (l0, m0), float32-representable, within `radius` of the phase centre."""
    g = np.random.default_rng([seed, 2])
    n = case["npos"] if case["task"] != "clean" else 1
    lm = g.uniform(-case["radius"], case["radius"], (n, 2))
    return lm.astype(np.float32).astype(np.float64)


def _sizes(case):
    if case["npix"]:
        return np.full(case["npos"], case["npix"], np.int32)
    return np.random.default_rng(3).choice(np.array([32, 64, 128, 256], np.int32), case["npos"])


def _dirty(case, seed):
    """A dirty image: sources of widths near the PSF's, and noise."""
    n = case["npos"]
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7 + 5)
    img = 0.05 * torch.randn((n, n), generator=g, device="cuda")
    q = np.random.default_rng([seed, 4])
    ax = torch.arange(-24, 24, device="cuda", dtype=torch.float32)
    for _ in range(120):
        x, y = (int(v) for v in q.integers(32, n - 32, 2))
        sx, sy = q.uniform(2.0, 4.0, 2)
        a = float(min(100.0, 1.0 / q.uniform(1e-3, 1.0) ** 1.2))
        img[y - 24:y + 24, x - 24:x + 24] += a * torch.exp(-0.5 * ((ax[None, :] / sx) ** 2 + (ax[:, None] / sy) ** 2))
    return img


def prepare(case, seed):
    s = types.SimpleNamespace(case=case, cell=case["cell"] * ARCSEC)
    obs = _observation(case, seed)
    lm = _positions(case, seed)
    s.plan = psf.Plan(obs, prec=case["prec"], flags=case["flags"])
    if case["task"] == "clean":
        s.dirty = _dirty(case, seed)
        s.residual, s.model = torch.empty_like(s.dirty), torch.zeros_like(s.dirty)
        return s
    if case["task"] == "grad":
        g = torch.Generator(device="cuda").manual_seed(int(seed) * 7 + 6)
        s.lm = torch.from_numpy(lm.astype(np.float32)).requires_grad_()
        s.W = (0.5 + torch.rand(s.plan.nvis, generator=g, device="cuda")).requires_grad_()
        s.cotangent = torch.randn(case["npos"] * case["npix"] ** 2, generator=g, device="cuda")
        return s
    s.batch = psf.Batch(lm, _sizes(case), s.cell)
    s.out = [torch.empty(s.batch.total(), device="cuda") for _ in range(3 if case["task"] == "step" else 1)]
    return s


# ---------------------------------------------------------------- one pass
def _checked_part(case):
    """Leading positions of a batch whose values `exact` gives (all, but for large batches)."""
    if case["task"] != "batch":
        return case["npos"]
    budget, n = 1.2e12, 0
    for size in _sizes(case):
        budget -= float(_nvis(case)) * size * size
        if budget < 0:
            break
        n += 1
    return max(1, n)


def _split(case, out):
    """A batch's output: the cutouts of the leading positions, and the others."""
    n = _checked_part(case)
    at = int((_sizes(case)[:n].astype(np.int64) ** 2).sum())
    return (out[:at], out[at:]) if n < case["npos"] else out


def run(s):
    c = s.case
    if c["task"] == "step":
        s.plan.exact(s.batch, out=s.out[0])
        s.plan.approx_uv_img(s.batch, out_uv=s.out[1], out_img=s.out[2])
        return tuple(s.out)
    if c["task"] == "clean":
        s.residual.copy_(s.dirty)
        s.model.zero_()
        r, m, pix, flux = s.plan.clean(s.residual, s.cell, c["npix"], method="img_grid", gain=0.1, threshold=0.0,
                                       max_iter=c["iters"], model=s.model, centre=(0.03, 0.03))
        return r, m, pix, flux
    if c["task"] == "grad":
        s.lm.grad = s.W.grad = None
        out = psf.smeared_psf(s.plan, c["method"], s.lm, c["npix"], s.cell, W=s.W)
        out.backward(s.cotangent)
        return out.detach(), s.lm.grad, s.W.grad
    s.plan.forward(c["method"], s.batch, out=s.out[0])
    return _split(c, s.out[0])


# ---------------------------------------------------------------- what it cannot do without
def work(case):
    K = float(_nvis(case))
    px = float((_sizes(case).astype(np.float64) ** 2).sum()) if case["task"] != "clean" else 0.0
    # 4 flops per pixel and visibility, 2 where the weights are real (Methods 1 and 2);
    # records of a bin's samples and centre, weight and uv per visibility, output pixels
    per = {"exact": 4.0, "uv": 2.0, "img": 2.0, "img_grid": 0.0}[case["method"]]
    nout = case["nchan"] // case["favg"]
    nbl = _baselines(case["array"]).shape[0]
    records = 16.0 * nbl * case["minutes"] * 60 + K * (48.0 / nout + 4.0)
    if case["task"] == "step":
        return {"bytes": records + 12.0 * px, "flops": 8.0 * K * px}
    if case["task"] == "grad":
        return {"bytes": 2 * records + 8.0 * K + 12.0 * px, "flops": (per + 4.0) * K * px}
    if case["task"] == "grid":
        N = case["npix"]
        return {"bytes": 4.0 * px + 16.0 * N * N, "flops": case["npos"] * N * N * (2.5 * math.log2(N * N) + 20.0)}
    if case["task"] == "clean":
        n, N, it = case["npos"], case["npix"], case["iters"]
        return {"bytes": 16.0 * n * n + 20.0 * N * N * it, "flops": it * N * N * (2.5 * math.log2(N * N) + 22.0)}
    return {"bytes": records + 4.0 * px, "flops": per * K * px}


# ---------------------------------------------------------------- float64 values
def _groups(case, uvw):
    """Visibilities in groups of baselines with one averaging length n, in blocks: yields
    (first visibility of each bin [B], bin samples [B, n, 3], edge delta [B, 3])."""
    tavg, nt, nout = _tavg(case), case["minutes"] * 60, case["nchan"] // case["favg"]
    first = np.concatenate([[0], np.cumsum(nt // tavg.astype(np.int64))])[:-1]
    for n in np.unique(tavg):
        n = int(n)
        idx = np.nonzero(tavg == n)[0]
        nb = nt // n
        per = max(1, (1 << 21) // (nb * n * nout))
        for i in range(0, len(idx), per):
            sel = idx[i:i + per]
            x = uvw[torch.from_numpy(sel).cuda(), :nb * n].reshape(len(sel) * nb, n, 3)
            k = torch.from_numpy(((first[sel][:, None] + np.arange(nb)) * nout).reshape(-1)).cuda()
            edge = (x[:, -1] - x[:, 0]) * (n / (n - 1.0))
            yield k, x, edge


def _channels(case):
    nout, favg = case["nchan"] // case["favg"], case["favg"]
    f = torch.from_numpy(case["f0"] + (np.arange(case["nchan"]) + 0.5) * case["df"]).cuda().view(nout, favg)
    return f, f.mean(1), case["df"] * favg


def _D(case, method, x, edge, dirs, lm):
    """Decorrelation (re, im) [B, nout] of the bins for one direction (l0, m0, n0 - 1)."""
    f, nu, dnu = _channels(case)
    ub = x.mean(1)
    if method == "exact":
        Xs = x @ dirs                                              # [B, n] metres
        ds = Xs - Xs.mean(1, keepdim=True)
        off = f[0] - nu[0]
        a = -2 * math.pi / C_LIGHT
        ph = a * Xs[:, :, None] * off                              # the raw channels of any output channel
        amp = torch.special.sinc(case["df"] * Xs / C_LIGHT)
        gr, gi = amp * torch.cos(ph).mean(2), amp * torch.sin(ph).mean(2)
        re, im = [], []
        for v in nu:
            c, s = torch.cos(a * v * ds), torch.sin(a * v * ds)
            re.append((c * gr - s * gi).mean(1))
            im.append((c * gi + s * gr).mean(1))
        return torch.stack(re, 1), torch.stack(im, 1)
    if method == "uv":
        A = (edge @ dirs)[:, None] * nu / C_LIGHT
        B = (ub @ dirs)[:, None] * dnu / C_LIGHT
        B = B.expand_as(A)
    else:
        u, v = ub[:, :1] * nu / C_LIGHT, ub[:, 1:2] * nu / C_LIGHT
        A = OMEGA_E * x.shape[1] * (u * lm[1] - v * lm[0])
        B = dnu / nu * torch.hypot(u, v) * torch.hypot(lm[0], lm[1])
    return torch.special.sinc(A) * torch.special.sinc(B), None


def _dirs(case, lm):
    if not case["flags"] & WTERM:
        return torch.stack([lm[0], lm[1], torch.zeros_like(lm[0])])
    r2 = lm[0] * lm[0] + lm[1] * lm[1]
    return torch.stack([lm[0], lm[1], -r2 / (1 + torch.sqrt(1 - r2))])


def _phasors(t, N):
    """cos, sin [N, K] of 2 pi t_k (i - N/2), i = 0 .. N-1."""
    i = torch.arange(N, dtype=torch.float64, device="cuda")[:, None] - N // 2
    M = 16
    lo, hi = torch.arange(M, dtype=torch.float64, device="cuda")[:, None], i[::M]
    a, b = 2 * math.pi * t * lo, 2 * math.pi * torch.remainder(t * hi, 1.0)
    ca, sa, cb, sb = torch.cos(a), torch.sin(a), torch.cos(b)[:, None], torch.sin(b)[:, None]
    c, s = (cb * ca - sb * sa).flatten(0, 1), (cb * sa + sb * ca).flatten(0, 1)
    return c[:N], s[:N]


def _gemm(a, b):
    """a [N, K] b [M, K]^T, K in 128 parts so that the product fills the device."""
    K = a.shape[1]
    k = K // 128 * 128
    r = a[:, k:] @ b[:, k:].T
    if k:
        r = r + torch.bmm(a[:, :k].reshape(a.shape[0], 128, -1).transpose(0, 1),
                          b[:, :k].reshape(b.shape[0], 128, -1).permute(1, 2, 0)).sum(0)
    return r


def _cutouts64(case, seed, methods, lms, sizes, W=None, uvw=None):
    """float64 cutouts [len(methods)][position] of the definition."""
    uvw = _uvw(case, seed) if uvw is None else uvw
    cell, nu = case["cell"] * ARCSEC, _channels(case)[1]
    out = [[torch.zeros((int(N), int(N)), dtype=torch.float64, device="cuda") for N in sizes] for _ in methods]
    for k, x, edge in _groups(case, uvw):
        ub = x.mean(1)
        kk = k[:, None] + torch.arange(len(nu), device="cuda")
        w = float(x.shape[1] * case["favg"]) if W is None else W[kk].double()
        tu, tv = ((ub[:, d:d + 1] * nu / C_LIGHT * cell).reshape(-1) for d in (0, 1))
        tw = {int(N): (_phasors(tu, int(N)), _phasors(tv, int(N))) for N in set(int(v) for v in sizes)}
        for p, lm in enumerate(lms):
            (ca, sa), (cb, sb) = tw[int(sizes[p])]
            for m, method in enumerate(methods):
                re, im = _D(case, method, x, edge, _dirs(case, lm), lm)
                re = (w * re).reshape(-1)
                cr, ci = cb * re, sb * re
                if im is not None:
                    im = (w * im).reshape(-1)
                    cr, ci = cr - sb * im, ci + cb * im
                out[m][p] += _gemm(cr, ca) - _gemm(ci, sa)
    return out


def _grid64(case, seed, lms):
    """Gridded Method 2: F^-1{F{P} D} on the cutout's Fourier grid, D from the cells' mean
    intervals and fractional bandwidths."""
    N, cell = case["npix"], case["cell"] * ARCSEC
    uvw = _uvw(case, seed)
    _, nu, dnu = _channels(case)
    z = torch.zeros(2, dtype=torch.float64, device="cuda")
    P = _cutouts64(case, seed, ["uv"], [z], [N], uvw=uvw)[0][0]
    acc = torch.zeros((3, N * N), dtype=torch.float64, device="cuda")
    tot = torch.zeros(3, dtype=torch.float64, device="cuda")
    for _, x, _ in _groups(case, uvw):
        ub = x.mean(1)
        a, b = (torch.floor(ub[:, d:d + 1] * nu / C_LIGHT * (N * cell) + 0.5).long() for d in (0, 1))
        w = torch.full(a.shape, float(x.shape[1] * case["favg"]), dtype=torch.float64, device="cuda")
        for i, v in enumerate((w, w * x.shape[1], w * (dnu / nu))):
            tot[i] += v.sum()
            for s in (1, -1):
                q = torch.remainder(s * b + N // 2, N) * N + torch.remainder(s * a + N // 2, N)
                acc[i].index_add_(0, q.reshape(-1), v.reshape(-1))
    has = acc[0] > 0
    dt, rr = (torch.where(has, acc[i] / acc[0].clamp(min=1e-300), tot[i] / tot[0]).view(N, N) for i in (1, 2))
    S = torch.fft.fft2(torch.fft.ifftshift(P))                     # cells in the transform's order
    n = torch.fft.ifftshift(torch.arange(N, device="cuda") - N // 2).double()
    dt, rr = torch.fft.ifftshift(dt), torch.fft.ifftshift(rr)
    du = 1.0 / (N * cell)
    a, b = n[None, :], n[:, None]
    out = []
    for lm in lms:
        D = torch.special.sinc(OMEGA_E * dt * du * (a * lm[1] - b * lm[0])) * torch.special.sinc(
            rr * du * torch.hypot(a, b) * torch.hypot(lm[0], lm[1]))
        out.append(torch.fft.fftshift(torch.fft.ifft2(S * D).real))
    return out


def _gradients64(case, seed, lms, W, R):
    """dL/d(l0, m0) and dL/dW of L = sum R P."""
    uvw = _uvw(case, seed)
    N, cell, nu = case["npix"], case["cell"] * ARCSEC, _channels(case)[1]
    gW = torch.zeros(_nvis(case), dtype=torch.float64, device="cuda")
    g = torch.zeros((len(lms), 2), dtype=torch.float64, device="cuda")
    R = R.double().view(len(lms), N, N)
    for k, x, edge in _groups(case, uvw):
        ub = x.mean(1)
        kk = (k[:, None] + torch.arange(len(nu), device="cuda")).reshape(-1)
        w = W[kk].double()
        tu, tv = ((ub[:, d:d + 1] * nu / C_LIGHT * cell).reshape(-1) for d in (0, 1))
        (ca, sa), (cb, sb) = _phasors(tu, N), _phasors(tv, N)
        for p, lm0 in enumerate(lms):
            tr, ti = R[p] @ ca, R[p] @ sa                           # [j, K]
            hr, hi = (cb * tr - sb * ti).sum(0), (cb * ti + sb * tr).sum(0)
            lm = lm0.clone().requires_grad_()
            with torch.enable_grad():
                re, im = _D(case, case["method"], x, edge, _dirs(case, lm), lm)
                v = re.reshape(-1) * hr - (0.0 if im is None else im.reshape(-1) * hi)
                loss = (w * v).sum()
            g[p] += torch.autograd.grad(loss, lm)[0]
            gW[kk] += v.detach()
    return g, gW


def exact(case, seed):
    if case["task"] == "clean":
        return None          # a loop of argmax decisions, no value of its own
    lms = torch.from_numpy(_positions(case, seed)).cuda()
    sizes = _sizes(case)
    if case["task"] == "grid":
        return torch.cat([v.reshape(-1) for v in _grid64(case, seed, lms)])
    if case["task"] == "step":
        return tuple(v[0].reshape(-1) for v in _cutouts64(case, seed, ["exact", "uv", "img"], lms, sizes))
    if case["task"] == "grad":
        s = prepare(case, seed)
        W, R = s.W.detach(), s.cotangent
        s.plan.close()
        out = _cutouts64(case, seed, [case["method"]], lms, sizes, W)[0]
        g, gW = _gradients64(case, seed, lms, W, R)
        return torch.cat([v.reshape(-1) for v in out]), g.cpu(), gW
    n = _checked_part(case)
    out = torch.cat([v.reshape(-1) for v in _cutouts64(case, seed, [case["method"]], lms[:n], sizes[:n])[0]])
    return (out, None) if n < case["npos"] else out
