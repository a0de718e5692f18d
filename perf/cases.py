"""The work that users of this framework have it do, as measurable cases.

A case is one call (or one training step) through the public entry points:
gridding, degridding, a dirty image, a w-stacked dirty image, or a
chi-squared step of differentiable imaging.  The arrays are Earth-rotation
tracks of antennas in a disk or in a spiral with a dense core, as in the
repository's synthetic observations; grid sizes, supports, plane counts,
storage kinds and visibility counts are those of its configurations and of
its serving stream (1e4 to 1e7 visibilities a job).  Inputs come from the
seed alone and are made on the GPU.

``exact`` restates the method (prolate-spheroidal taper times w-screen,
nearest-neighbour index selection, gridding and its adjoint, correction) in
64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

import paper_2111_04141_gb300 as gw
from paper_2111_04141_gb300 import autograd as gwa
from paper_2111_04141_gb300 import imaging

C0 = 299_792_458.0
DEV = "cuda"
STORE = {"bf16": torch.bfloat16, "f16": torch.float16}

# Fields every case has; a listed or drawn case overrides some of them.
#   op       grid | degrid | dirty | wstack | chisq
#   ant, times, chan   antennas, time steps, channels: ant (ant - 1) / 2 x times rows
#   field    field of view, radians; the array is scaled to fill the uv grid
#   planes   w-planes (1: 2-D); smin, smax: kernel support of the first and last
#   weighted per-visibility weights; shuffled: rows in random order
BASE = dict(op="grid", ant=64, times=1, chan=1, pol=1, n=1024, smin=7, smax=7, beta=8, planes=1,
            field=0.4, spiral=False, store="c64", weighted=False, shuffled=False, layers=0)


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the 2-D workload of the tests and the benchmark: 3,840 visibilities,
        # a call whose cost is latency and launches
        _case("grid_2d_small", ant=16, times=32, n=256, field=0.2),
        # its adjoint: predicting a few thousand visibilities
        _case("degrid_2d_small", op="degrid", ant=16, times=32, n=256, field=0.2),
        # small serving job: one polarisation, unsorted rows, 30 thousand visibilities
        _case("grid_serve_1024", ant=64, times=15, n=1024, planes=16, smax=33, field=0.3,
              shuffled=True),
        # ordinary serving job: 4 channels x 4 polarisations, 264 thousand visibilities
        _case("degrid_serve_2048", op="degrid", ant=96, times=14, chan=4, pol=4, n=2048, planes=16,
              smax=41, field=0.5),
        # ragged sizes: grid side no multiple of any tile, 3 polarisations, other
        # oversampling, weights, 5 channels
        _case("grid_ragged_weighted", ant=50, times=77, chan=5, pol=3, n=1502, smin=5, smax=45,
              beta=4, planes=9, field=0.35, weighted=True),
        # the benchmark's headline: 4-pol w-projection, 8.26 million visibilities
        _case("grid_wproj_4096", ant=64, times=256, chan=16, pol=4, n=4096, planes=32, smax=63,
              field=0.634),
        # its adjoint (prediction of the same visibilities)
        _case("degrid_wproj_4096", op="degrid", ant=64, times=256, chan=16, pol=4, n=4096,
              planes=32, smax=63, field=0.634),
        # 16-bit storage at scale: spiral array, 8192^2 x 4, 128 planes, support to
        # 127, a run of the observation's time steps
        _case("grid_bf16_8192", ant=256, times=12, chan=8, pol=4, n=8192, planes=128, smax=127,
              field=0.3, spiral=True, store="bf16"),
        _case("degrid_f16_8192", op="degrid", ant=256, times=4, chan=8, pol=4, n=8192, planes=128,
              smax=127, field=0.3, spiral=True, store="f16"),
        # differentiable imaging: chi-squared and its gradient, 4.2 million
        # visibilities, 1 pol, one support of 31
        _case("chisq_2048", op="chisq", ant=128, times=516, n=2048, smin=31, smax=31, planes=16,
              field=0.185),
        # 2-D dirty image, 4 polarisations: gridding, FFT, correction.  Support 5:
        # the correction of wider tapers (h up to 5000 at the edge for support 7)
        # turns the FP32 rounding of the transform into the image's border
        _case("dirty_2d_4096", op="dirty", ant=64, times=256, chan=16, pol=4, n=4096, smin=5,
              smax=5, field=0.634),
        # w-stacked dirty image of one polarisation
        _case("wstack_2048", op="wstack", ant=64, times=128, chan=4, pol=1, n=2048, smin=5, smax=5,
              field=0.3, layers=16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["grid"] * 5 + ["degrid"] * 4 + ["chisq", "dirty", "wstack"])
    pol = rng.choice([1, 1, 2, 3, 4, 4])
    n = 2 * int(_log(rng, 128, 4096))
    planes, smin, smax = 1, rng.choice([5, 7, 7, 7, 9]), 0
    store = "c64"
    if op in ("grid", "degrid"):
        store = rng.choice(["c64"] * 6 + ["bf16", "f16"])
        if rng.random() < 0.75:
            planes = int(_log(rng, 4, 64))
    if op == "chisq":
        planes, smin, pol, n = int(_log(rng, 4, 16)), rng.choice([15, 21, 31]), 1, min(n, 2048)
    if op == "wstack":
        pol, n = min(pol, 2), min(n, 2048)
    if op in ("dirty", "wstack"):
        smin = 5                    # see the listed dirty image
    smax = smin
    if planes > 1 and op != "chisq":
        smax = min(2 * int(_log(rng, 8, 64)) + 1, (n // 6) | 1)
        smax = max(smax, smin)
    chan = rng.choice([1, 1, 3, 4, 8, 16])
    # visibilities: 4 thousand to 8 million, at most about 1e10 tap updates
    most = min(8e6, 1e10 / (0.4 * smax * smax * pol), 2e6 if op in ("chisq", "wstack") else 8e6)
    nvis = _log(rng, 4e3, max(most, 8e3))
    ant = int(_log(rng, 12, 160))
    bl = ant * (ant - 1) // 2
    while bl * chan > nvis and ant > 8:
        ant -= 1
        bl = ant * (ant - 1) // 2
    return _case(op=op, ant=ant, times=max(1, int(nvis / (bl * chan))), chan=chan, pol=pol, n=n,
                 smin=smin, smax=smax, beta=rng.choice([4, 8, 8, 16]) if smax <= 63 else 8,
                 planes=planes, field=round(rng.uniform(0.15, 0.65), 3), store=store,
                 spiral=rng.random() < 0.3, weighted=op in ("grid", "dirty") and rng.random() < 0.25,
                 shuffled=rng.random() < 0.5, layers=rng.choice([4, 8, 16]) if op == "wstack" else 0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _coords(c, seed):
    """uvw [rows, 3] metres and frequencies [chan] Hz (float64, on the GPU), the
    cell and the largest |w| in wavelengths."""
    r = np.random.default_rng(seed)
    a = c["ant"]
    enu = np.zeros((a, 3))
    if c["spiral"]:
        core = a // 2
        enu[:core, :2] = r.normal(0.0, 0.03, (core, 2))
        k = np.arange(a - core)
        rad = 0.08 * 12.5 ** (k / max(1, a - core - 1))
        th = 2 * np.pi * (k % 3) / 3 + 1.2 * np.log(rad / 0.08)
        rad = rad * (1 + 0.03 * r.normal(size=a - core))
        enu[core:, 0], enu[core:, 1] = rad * np.cos(th), rad * np.sin(th)
    else:
        rad, th = np.sqrt(r.random(a)), 2 * np.pi * r.random(a)
        enu[:, 0], enu[:, 1] = rad * np.cos(th), rad * np.sin(th)
    i, j = np.triu_indices(a, k=1)
    e, nn = torch.from_numpy(enu[j] - enu[i]).to(DEV).T[:2]
    lat = dec = math.radians(-30.0)
    ha = math.pi / 3 * (2.0 * torch.arange(c["times"], dtype=torch.float64, device=DEV) /
                        c["times"] - 1.0)
    sh, ch = torch.sin(ha)[:, None], torch.cos(ha)[:, None]
    x, y, z = -nn * math.sin(lat), e, nn * math.cos(lat)
    u = sh * x + ch * y
    v = -math.sin(dec) * ch * x + math.sin(dec) * sh * y + math.cos(dec) * z
    w = math.cos(dec) * ch * x - math.cos(dec) * sh * y + math.sin(dec) * z
    uvw = torch.stack([u.reshape(-1), v.reshape(-1), w.reshape(-1)], 1)
    f = np.linspace(120e6, 180e6, c["chan"]) if c["chan"] > 1 else np.array([150e6])
    # the longest |u|, |v| lands 0.45 N - S_max / 2 pixels from the centre
    reach = (0.45 * c["n"] - 0.5 * c["smax"]) / c["field"] * C0 / f.max()
    uvw = uvw * (reach / float(uvw[:, :2].abs().max()))
    wmax = float(uvw[:, 2].abs().max()) * f.max() / C0
    if c["shuffled"]:
        uvw = uvw[torch.from_numpy(r.permutation(uvw.shape[0])).to(DEV)]
    return uvw.contiguous(), torch.from_numpy(f).to(DEV), c["field"] / c["n"], wmax


def _inputs(c, seed):
    uvw, freq, cell, wmax = _coords(c, seed)
    g = torch.Generator(device=DEV).manual_seed(seed)
    s = dict(uvw=uvw, freq=freq, cell=cell, wmax=wmax)
    shape = (uvw.shape[0], c["chan"], c["pol"])
    if c["op"] == "degrid":     # a model grid
        s["grid"] = torch.randn((c["pol"], c["n"], c["n"]), dtype=torch.complex64, device=DEV,
                                generator=g)
    else:                       # CN(0, 1) visibilities
        s["vis"] = torch.randn(shape, dtype=torch.complex64, device=DEV, generator=g)
        if c["store"] != "c64":
            s["vis"] = torch.view_as_real(s["vis"]).to(STORE[c["store"]])
    if c["weighted"]:
        s["weight"] = torch.rand(shape, device=DEV, generator=g) * 1.5 + 0.25
    if c["op"] == "chisq":      # point sources in the central quarter of the field
        m = c["n"] // 4
        s["sky"] = torch.zeros((1, m, m), device=DEV)
        at = torch.randint(0, m * m, (200,), device=DEV, generator=g)
        s["sky"].view(-1)[at] = torch.rand(200, device=DEV, generator=g) * 0.9 + 0.1
        s["vis"] *= 3.0
    return s


def _plan(c, s):
    planes = c["planes"]
    return gw.Plan(grid_n=c["n"], cell_rad=s["cell"], support_min=c["smin"], support_max=c["smax"],
                   oversample=c["beta"], n_wplanes=planes, npol=c["pol"],
                   w_max_lambda=s["wmax"] if planes > 1 else 0.0, vis_dtype=c["store"],
                   table_dtype=c["store"])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], s["plan"] = case, _plan(case, s)
    return s


def _pad(sky, n):
    e = (n - sky.shape[-1]) // 2
    return torch.nn.functional.pad(sky, (e, n - sky.shape[-1] - e) * 2)


SIGMA = 0.7


def run(s):
    c, p, uvw, freq = s["case"], s["plan"], s["uvw"], s["freq"]
    op = c["op"]
    if op == "grid":
        return p.grid(uvw, freq, s["vis"], weight=s.get("weight"))
    if op == "degrid":
        return p.degrid(uvw, freq, s["grid"])
    if op == "dirty":
        return imaging.dirty_image(p, uvw, freq, s["vis"], weight=s.get("weight"))
    if op == "wstack":
        return imaging.dirty_image_wstack(p, uvw, freq, s["vis"], c["layers"], -s["wmax"],
                                          s["wmax"])
    sky = s["sky"].detach().requires_grad_(True)
    loss = gwa.chisq(p, uvw, freq, _pad(sky, c["n"]), s["vis"], SIGMA)
    loss.backward()
    return {"loss": loss.detach(), "grad": sky.grad}


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def _support(p, c):
    if c["planes"] == 1:
        return c["smin"]
    y = c["smin"] * (c["planes"] - 1) + (c["smax"] - c["smin"]) * p
    return 2 * (y // (2 * (c["planes"] - 1))) + 1


def _planes(w, c, wmax):
    """The plane nearest in sqrt|w| (ties up) of w in wavelengths."""
    j = torch.arange(c["planes"] - 1, dtype=torch.float64, device=w.device)
    t = (j + 0.5) / float(c["planes"] - 1)
    return torch.searchsorted(t * t * wmax, w.abs().contiguous(), right=True)


def _taps(c):
    """Mean S^2 over the visibilities (of one seed's tracks)."""
    if c["planes"] == 1 or c["smin"] == c["smax"]:
        return float(c["smin"] ** 2)
    uvw, freq, _, wmax = _coords(dict(c, times=min(c["times"], 16), shuffled=False), 0)
    p = _planes(uvw[:, 2:3] * (freq / C0)[None, :], c, wmax)
    s2 = torch.tensor([_support(q, c) ** 2 for q in range(c["planes"])], device=p.device)
    return float(s2[p].double().mean())


def work(case):
    c = case
    rows = c["ant"] * (c["ant"] - 1) // 2 * c["times"]
    nv, px = rows * c["chan"], c["n"] ** 2 * c["pol"]
    vis = nv * c["pol"] * (8 if c["store"] == "c64" else 4)
    taps = nv * _taps(c) * c["pol"]
    fft = 5 * px * 2 * math.log2(c["n"])
    b, f = rows * 24 + vis + 8 * px + (nv * c["pol"] * 4 if c["weighted"] else 0), 8 * taps
    if c["op"] == "dirty":
        f += fft
    elif c["op"] == "wstack":
        f += c["layers"] * (fft + 8 * px)
    elif c["op"] == "chisq":        # the sky and its gradient, not full grids
        b, f = rows * 24 + vis + 8 * px // 16, 2 * (f + fft)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # grids and visibilities: FP32 sums in any order
    if case["store"] == "bf16":
        return {"rel": 1e-2}        # both operands carry 8 bits
    if case["store"] == "f16":
        return {"rel": 1.2e-3}      # 11 bits
    if case["op"] in ("dirty", "wstack"):
        # the correction multiplies the rounding of the transform by up to
        # h(l) h(m) at the border
        return {"rel": 1e-3}
    return {"rel": 2e-6}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _pswf(c, x):
    """psi_0(c, x) up to a constant: the lowest even eigenvector of the prolate
    operator in normalised Legendre polynomials."""
    m = int(c) + 40
    k = 2.0 * np.arange(m)
    d = k * (k + 1) + c * c * (2 * k * (k + 1) - 1) / ((2 * k + 3) * (2 * k - 1))
    o = c * c * (k + 2) * (k + 1) / ((2 * k + 3) * np.sqrt((2 * k + 1) * (2 * k + 5)))
    vec = np.linalg.eigh(np.diag(d) + np.diag(o[:-1], 1) + np.diag(o[:-1], -1))[1][:, 0]
    coef = np.zeros(2 * m)
    coef[::2] = vec * np.sqrt(k + 0.5)
    v = np.polynomial.legendre.legval(x, coef)
    return v / np.polynomial.legendre.legval(0.0, coef)


def _offsets(S, beta):
    """Fine offsets t - o / beta of a support: first one, and all of them."""
    f0 = -beta * (S // 2) - beta // 2 + 1
    return f0, (torch.arange(beta * S, dtype=torch.float64, device=DEV) + f0) / beta


class _Kernels:
    def __init__(self, c, s):
        self.c, beta = c, c["beta"]
        half = 0.5 * c["field"]
        kap = (2 * math.pi * s["wmax"] * half * half / math.sqrt(1 - 2 * half * half)
               if c["planes"] > 1 else 0.0)
        q = int(0.75 * (kap + math.pi * (c["smax"] / 2 + 1 + c["smin"] / 2))) + 50
        x, wt = np.polynomial.legendre.leggauss(q)
        tap = _pswf(math.pi * c["smin"] / 2, x)
        self.x = torch.from_numpy(x).to(DEV)
        self.tw = torch.from_numpy(tap * wt).to(DEV)
        r2 = half * half * (self.x[:, None] ** 2 + self.x[None, :] ** 2)
        self.nm1 = -r2 / (1 + torch.sqrt(1 - r2))
        self.wmax = s["wmax"]
        S = c["smin"]
        f0, off = _offsets(S, beta)
        c1 = torch.cos(math.pi * off[:, None] * self.x[None, :]) @ self.tw
        self.norm = float(c1[torch.arange(-(S // 2), S // 2 + 1) * beta - f0].sum())
        self.c1, self.off = c1 / self.norm, off

    def plane(self, p):
        """[beta S, beta S] kernel over the fine offsets (v, u)."""
        P = self.c["planes"]
        _, off = _offsets(_support(p, self.c), self.c["beta"])
        e = torch.cos(math.pi * off[:, None] * self.x[None, :]) * self.tw[None, :]
        e = e.to(torch.complex128)
        w = self.wmax * (p / (P - 1)) ** 2 if P > 1 else 0.0
        ph = 2 * math.pi * w * self.nm1
        return e @ torch.polar(torch.ones_like(ph), ph) @ e.T / self.norm ** 2

    def corrector(self):
        n, beta = self.c["n"], self.c["beta"]
        l = (torch.arange(n, dtype=torch.float64, device=DEV) - n // 2) / n
        ch = torch.cos(2 * math.pi * l[:, None] * self.off[None, :]) @ self.c1 / beta
        return 1.0 / (ch * torch.sinc(l / beta))


def _records(c, s):
    """Pixel, offset, plane, sign of every visibility that stays on the grid."""
    beta, n = c["beta"], c["n"]
    sc = s["freq"] / C0
    field = n * s["cell"]
    uvw = s["uvw"]

    def axis(m):
        q = torch.floor(((m[:, None] * sc[None, :]) * field + n // 2) * beta + 0.5).long()
        k = torch.div(q + beta // 2, beta, rounding_mode="floor")
        return k.reshape(-1), (q - k * beta).reshape(-1)

    ku, ou = axis(uvw[:, 0].contiguous())
    kv, ov = axis(uvw[:, 1].contiguous())
    wl = (uvw[:, 2:3] * sc[None, :]).reshape(-1)
    if c["planes"] > 1:
        p = _planes(wl, c, s["wmax"])
        conj = wl < 0
    else:
        p, conj = torch.zeros_like(ku), torch.zeros_like(ku, dtype=torch.bool)
    sup = torch.tensor([_support(q, c) for q in range(c["planes"])], device=DEV)
    h = torch.div(sup[p], 2, rounding_mode="floor")
    ok = (ku - h >= 0) & (ku + h < n) & (kv - h >= 0) & (kv + h < n)
    return ku, kv, ou, ov, p, conj, ok, wl


def _chunks(c, rec, kern):
    """(ids, flat pixels [m, S^2], kernel values [m, S^2]) of all valid records."""
    ku, kv, ou, ov, p, conj, ok, _ = rec
    beta, n = c["beta"], c["n"]
    for q in range(c["planes"]):
        ids = torch.nonzero(ok & (p == q)).reshape(-1)
        if not len(ids):
            continue
        S = _support(q, c)
        f0, _ = _offsets(S, beta)
        K = kern.plane(q)
        t = torch.arange(S, device=DEV) - S // 2
        step = max(1, 6_000_000 // (S * S * c["pol"]))
        for a in range(0, len(ids), step):
            i = ids[a:a + step]
            fv = t[None, :] * beta - ov[i][:, None] - f0
            fu = t[None, :] * beta - ou[i][:, None] - f0
            k = K[fv[:, :, None], fu[:, None, :]].reshape(len(i), -1)
            k = torch.where(conj[i][:, None], k.conj(), k)
            px = ((kv[i][:, None] + t)[:, :, None] * n + (ku[i][:, None] + t)[:, None, :])
            yield i, px.reshape(len(i), -1), k


def _grid64(c, rec, kern, vis, layer=None, layers=1):
    n, pol = c["n"], c["pol"]
    out = torch.zeros((layers * n * n, 2 * pol), dtype=torch.float64, device=DEV)
    for i, px, k in _chunks(c, rec, kern):
        if layer is not None:
            px = px + layer[i][:, None] * (n * n)
        val = torch.view_as_real(k[:, :, None] * vis[i][:, None, :])
        out.index_add_(0, px.reshape(-1), val.reshape(-1, 2 * pol))
    g = torch.view_as_complex(out.reshape(layers, n, n, pol, 2)).permute(0, 3, 1, 2)
    return g.contiguous()


def _degrid64(c, rec, kern, grid):
    out = torch.zeros((len(rec[0]), c["pol"]), dtype=torch.complex128, device=DEV)
    flat = grid.reshape(c["pol"], -1).T.contiguous()
    for i, px, k in _chunks(c, rec, kern):
        out[i] = (k.conj()[:, :, None] * flat[px]).sum(1)
    return out


def _sign(n):
    a = 1.0 - 2.0 * (torch.arange(n, device=DEV) % 2).double()
    return a[:, None] * a[None, :]


def exact(case, seed):
    c = case
    rows = c["ant"] * (c["ant"] - 1) // 2 * c["times"]
    if rows * c["chan"] * _taps(c) * (0.5 + 0.5 * c["pol"]) > 4.5e9:
        return None                 # over about 20 seconds
    s = _inputs(c, seed)
    kern, rec = _Kernels(c, s), _records(c, s)
    n, pol = c["n"], c["pol"]
    shape = (rows, c["chan"], pol)
    if c["op"] == "degrid":
        out = _degrid64(c, rec, kern, s["grid"].to(torch.complex128)).reshape(shape)
        return out if c["store"] == "c64" else torch.view_as_real(out)
    vis = s["vis"].double() if c["store"] != "c64" else s["vis"].to(torch.complex128)
    if c["store"] != "c64":
        vis = torch.view_as_complex(vis.contiguous())
    vis = vis.reshape(-1, pol)
    wt = s["weight"].double().reshape(-1, pol) if c["weighted"] else None
    if wt is not None:
        vis = vis * wt
    valid = rec[6]
    if c["op"] == "grid":
        return _grid64(c, rec, kern, vis)[0]
    h = kern.corrector()
    hh = h[:, None] * h[None, :]
    if c["op"] == "dirty":
        g = _grid64(c, rec, kern, vis)[0] * _sign(n)
        img = torch.fft.ifft2(g, norm="forward") * (_sign(n) * hh)
        if wt is None:
            return img / max(float(valid.sum()), 1e-30)
        return img / (wt * valid[:, None]).sum(0)[:, None, None]
    if c["op"] == "wstack":
        L, wmin = c["layers"], -s["wmax"]
        dw = 2 * s["wmax"] / (L - 1)
        layer = torch.floor((rec[7] - wmin) / dw + 0.5).clamp(0, L - 1).long()
        imgs = torch.fft.ifft2(_grid64(c, rec, kern, vis, layer, L) * _sign(n), norm="forward")
        x = (torch.arange(n, dtype=torch.float64, device=DEV) - n // 2) * s["cell"]
        r2 = x[:, None] ** 2 + x[None, :] ** 2
        nm1 = -r2 / (1 + torch.sqrt(1 - r2))
        img = torch.zeros((pol, n, n), dtype=torch.complex128, device=DEV)
        for l in range(L):
            ph = 2 * math.pi * (wmin + l * dw) * nm1
            img += imgs[l] * _sign(n) * torch.polar(torch.ones_like(ph), ph)
        return img * hh / max(float(valid.sum()), 1e-30)
    sky = _pad(s["sky"].double(), n)
    g = torch.fft.fft2(sky * (_sign(n) * hh) + 0j) * _sign(n)
    res = _degrid64(c, rec, kern, g) - vis
    loss = (torch.view_as_real(res) ** 2).sum() / (SIGMA * SIGMA)
    img = torch.fft.ifft2(_grid64(c, rec, kern, res)[0] * _sign(n), norm="forward")
    m = c["n"] // 4
    e = (n - m) // 2
    grad = 2.0 * (img * (_sign(n) * hh)).real / (SIGMA * SIGMA)
    return {"loss": loss, "grad": grad[:, e:e + m, e:e + m]}
