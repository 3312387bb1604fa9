"""What this framework is used for, as cases that can be run and timed: whole reconstructions (dect_reconstruct through
`Solver`), and the single operators a program calls for itself (the projector pair, the per-ray decomposition, the forward
model with its gradient, CDM-FBP).

Sizes are those of the repository's workloads (the 64^2 parallel scan, the 512^2 x 720 x 1024 baggage fan scan, the uneven
batch, the 1024^2 x 1440 x 2048 stack) and odd ones between. Scans are synthetic: ellipses with exact chord lengths, Poisson
counts. `exact` holds plain torch restatements in float64 of what the calls compute.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1905_00934_gb300 import Geometry, Solver, Spectra, autograd, cdm_fbp, dect

E_REF = 100.0  # keV, the photoelectric basis' reference of the baggage workloads
KAPPA = 0.25   # their initial photoelectric image, as a fraction of the Compton image
I0 = 2e5       # photons per ray


def listed():
    return [
        # one small parallel scan, a few iterations: launches and latency
        dict(name="solve_parallel_64", do="solve", beam="parallel", nx=64, ny=64, views=90, bins=96, slices=1, iters=3),
        # the small scan with every vector in float64 and the literal 1 keV basis
        dict(name="solve_f64_64", do="solve", beam="parallel", nx=64, ny=64, views=90, bins=96, slices=1, iters=3,
             storage="f64", e_ref=1.0),
        # one baggage slice by itself
        dict(name="solve_fan_512", do="solve", beam="fan", nx=512, ny=512, views=720, bins=1024, slices=1, iters=3),
        # the benchmark's batch: 8 baggage slices of one scanner
        dict(name="solve_fan_512_x8", do="solve", beam="fan", nx=512, ny=512, views=720, bins=1024, slices=8, iters=3),
        # slices of different sizes in one batch, from the paper's CDM-FBP start, UDM(2)-PCG(2)
        dict(name="solve_uneven", do="solve", beam="fan", nx=448, ny=391, views=540, bins=777, slices=5, iters=2,
             uneven=True, init="cdm_fbp", m=2, n=2),
        # the largest geometry, float16 sinogram storage, continued from a start image
        dict(name="solve_fan_1024_f16", do="solve", beam="fan", nx=1024, ny=1024, views=1440, bins=2048, slices=2, iters=2,
             storage="f16", init="x0"),
        # R and its gradient R^T over a stack of images, through autograd
        dict(name="adjoint_fan_512", do="adjoint", beam="fan", nx=512, ny=512, views=720, bins=1024, images=4),
        # one small image of odd sizes, one channel, R then R^T
        dict(name="adjoint_ragged_93", do="adjoint", beam="parallel", nx=93, ny=70, views=61, bins=131, images=1, offset=0.25),
        # the float64 pair of gradient checks
        dict(name="adjoint_f64_128", do="adjoint", beam="fan", nx=128, ny=128, views=180, bins=256, images=2, dtype="f64"),
        # data fidelity of Eq. 4 and its gradient with respect to both images
        dict(name="fidelity_fan_512", do="fidelity", beam="fan", nx=512, ny=512, views=720, bins=1024),
        # Eq. 13 for every ray of a baggage sinogram
        dict(name="decompose_720x1024", do="decompose", beam="fan", nx=512, ny=512, views=720, bins=1024, iters=10),
        # the comparison method on a baggage slice
        dict(name="cdm_fbp_512", do="cdm_fbp", beam="fan", nx=512, ny=512, views=720, bins=1024, iters=20),
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    do = rng.choice(["solve", "solve", "solve", "adjoint", "adjoint", "fidelity", "decompose", "cdm_fbp"])
    f64 = do in ("solve", "adjoint") and rng.random() < 0.2
    nx = log_uniform(48, 160 if f64 else 900)
    ny = max(32, min(1024, int(nx * rng.uniform(0.7, 1.2))))
    views = max(40, int(max(nx, ny) * rng.uniform(0.8, 1.5)))
    bins = max(48, int(max(nx, ny) * rng.uniform(1.2, 2.2)))
    case = dict(do=do, beam=rng.choice(["parallel", "fan", "fan"]), nx=nx, ny=ny, views=views, bins=bins,
                offset=rng.choice([0.0, 0.0, 0.25]))
    if do == "solve":
        room = 8 * 512 * 512 * 720 / (nx * ny * views)  # slices that cost as much as the benchmark's batch
        case["slices"] = max(1, min(8 if not f64 else 2, int(room / 2), rng.randint(1, 8)))
        case["iters"] = rng.randint(1, 3)
        case["init"] = "pcg" if f64 else rng.choice(["pcg", "pcg", "cdm_fbp", "x0"])
        case["m"], case["n"] = rng.choice([(1, 1), (1, 1), (2, 1), (1, 2)])
        case["storage"] = "f64" if f64 else rng.choice(["f32", "f32", "f16"])
        case["uneven"] = rng.random() < 0.4
    elif do == "adjoint":
        case["images"] = rng.randint(1, 6)
        case["dtype"] = "f64" if f64 else "f32"
    elif do in ("decompose", "cdm_fbp"):
        case["iters"] = rng.randint(1, 20)
    return case


# ---- geometry, spectra and scans -----------------------------------------------------------------

def _geometry(case, nx, ny, views, bins):
    """A detector that just covers the image's circumscribed circle; the fan's source and detector distances are
    those of the baggage scanner (a field of 51.2 cm)."""
    offset = float(case.get("offset", 0.0))
    if case["beam"] == "parallel":
        pixel = 0.1
        pitch = 1.06 * pixel * math.hypot(nx, ny) / bins
        return SimpleNamespace(kind=dect.PARALLEL, nx=nx, ny=ny, pixel_cm=pixel, n_views=views, angle0_rad=0.0,
                               angle_span_rad=math.pi, n_bins=bins, bin_pitch_cm=pitch, bin_offset_cm=offset * pitch,
                               sod_cm=0.0, sdd_cm=0.0)
    sod, sdd = 55.0, 95.0
    pixel = 51.2 / max(nx, ny)
    pitch = 2.0 * sdd * math.tan(math.asin(0.5 * pixel * math.hypot(nx, ny) / sod)) / bins
    return SimpleNamespace(kind=dect.FAN_FLAT, nx=nx, ny=ny, pixel_cm=pixel, n_views=views, angle0_rad=0.0,
                           angle_span_rad=2.0 * math.pi, n_bins=bins, bin_pitch_cm=pitch, bin_offset_cm=offset * pitch,
                           sod_cm=sod, sdd_cm=sdd)


def _geometries(case):
    """One geometry per slice: the same object for the slices of one scan, other sizes for an uneven batch."""
    one = _geometry(case, case["nx"], case["ny"], case["views"], case["bins"])
    out = []
    for b in range(case.get("slices", 1)):
        if not case.get("uneven"):
            out.append(one)
            continue
        f = 1.0 - 0.13 * b if b < 5 else 0.9 - 0.1 * (b - 5)
        out.append(_geometry(case, max(24, int(case["nx"] * f)), max(24, int(case["ny"] * f)),
                             max(32, int(case["views"] * (0.6 + 0.4 * f))), max(40, int(case["bins"] * f))))
    return out


def _tables(case):
    """S_h, S_l, f_KN, f_p: 140 and 80 kVp Kramers spectra behind 2 mm of aluminium, 20 to 140 keV in 1 keV bins."""
    e = 20.0 + np.arange(121)
    a = e / 510.99895
    l = np.log1p(2 * a)
    f_kn = (1 + a) / a**2 * (2 * (1 + a) / (1 + 2 * a) - l / a) + l / (2 * a) - (1 + 3 * a) / (1 + 2 * a) ** 2
    f_p = (case.get("e_ref", E_REF) / e) ** 3
    mu_al = 0.3907 * f_kn  # cm^-1: aluminium's electron density times the cross-section

    def spectrum(kvp):
        s = np.where(e < kvp, (kvp - e) / e, 0.0) * np.exp(-0.2 * mu_al)
        return s / s.sum()

    return spectrum(140.0), spectrum(80.0), f_kn, f_p


def _objects(case, g, rng):
    """Rows {cx, cy, a, b, angle, Compton, photoelectric}: a body, inserts, and a small one of high atomic number."""
    half = 0.5 * g.pixel_cm * min(g.nx, g.ny)
    p_max = 4e-3
    thin = min(1.0, 4.0 / half)  # keeps the longest paths at a few attenuation lengths
    rows = [[0.0, 0.0, 0.85 * half, 0.8 * half, rng.uniform(0, math.pi), 0.2 * thin, 0.5 * p_max * thin]]
    for k in range(9):
        r, t = 0.65 * half * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        if k == 0 and case["beam"] == "fan":
            a, b, c, p = 0.02 * half, 0.04 * half, rng.uniform(1.0, 1.5), rng.uniform(0.1, 0.3)
        else:
            a, b = rng.uniform(0.05, 0.22, 2) * half
            c, p = rng.uniform(-0.1, 0.3) * thin, rng.uniform(-0.4, 1.0) * p_max * thin
        rows.append([r * math.cos(t), r * math.sin(t), a, b, rng.uniform(0, math.pi), c, p])
    return rows


def _rays(g, dev):
    """Origins and unit directions [views, bins] in float64."""
    th = g.angle0_rad + torch.arange(g.n_views, device=dev, dtype=torch.float64) * (g.angle_span_rad / g.n_views)
    c, s = torch.cos(th)[:, None], torch.sin(th)[:, None]
    u = ((torch.arange(g.n_bins, device=dev, dtype=torch.float64) - 0.5 * (g.n_bins - 1)) * g.bin_pitch_cm
         + g.bin_offset_cm)[None, :]
    if g.kind == dect.PARALLEL:
        return u * c, u * s, (-s).expand(-1, g.n_bins), c.expand(-1, g.n_bins)
    sx, sy = (g.sod_cm * c).expand(-1, g.n_bins), (g.sod_cm * s).expand(-1, g.n_bins)
    ex, ey = -g.sdd_cm * c - u * s, -g.sdd_cm * s + u * c
    ln = torch.hypot(ex, ey)
    return sx, sy, ex / ln, ey / ln


def _line_integrals(g, rows, dev):
    px, py, dx, dy = _rays(g, dev)
    out = torch.zeros((2, g.n_views, g.n_bins), device=dev, dtype=torch.float64)
    for cx, cy, a, b, phi, comp, phot in rows:
        c, s = math.cos(phi), math.sin(phi)
        qx, qy = (c * (px - cx) + s * (py - cy)) / a, (-s * (px - cx) + c * (py - cy)) / b
        ex, ey = (c * dx + s * dy) / a, (-s * dx + c * dy) / b
        aa, bb, cc = ex * ex + ey * ey, qx * ex + qy * ey, qx * qx + qy * qy - 1.0
        chord = 2.0 * torch.sqrt(torch.clamp(bb * bb - aa * cc, min=0.0)) / aa
        out[0] += comp * chord
        out[1] += phot * chord
    return torch.clamp(out, min=0.0)


def _image(g, rows, dev):
    """The objects at the pixel centres, [2, ny, nx] float32."""
    x = ((torch.arange(g.nx, device=dev) - 0.5 * (g.nx - 1)) * g.pixel_cm)[None, :]
    y = ((torch.arange(g.ny, device=dev) - 0.5 * (g.ny - 1)) * g.pixel_cm)[:, None]
    img = torch.zeros((2, g.ny, g.nx), device=dev)
    for cx, cy, a, b, phi, comp, phot in rows:
        c, s = math.cos(phi), math.sin(phi)
        m = ((c * (x - cx) + s * (y - cy)) / a) ** 2 + ((-s * (x - cx) + c * (y - cy)) / b) ** 2 <= 1.0
        img[0] += comp * m
        img[1] += phot * m
    return torch.clamp(img, min=0.0)


def _scan(case, g, seed, b, dev):
    """Measurements of slice b: m_h, m_l, w_h, w_l [views, bins] float32; its line integrals and its objects."""
    rng = np.random.default_rng([seed, b])
    rows = _objects(case, g, rng)
    a = _line_integrals(g, rows, dev)
    s_h, s_l, f_kn, f_p = _tables(case)
    t = torch.zeros((2, g.n_views, g.n_bins), device=dev, dtype=torch.float64)
    for k in range(len(f_kn)):
        x = torch.exp(-f_kn[k] * a[0] - f_p[k] * a[1])
        t[0] += s_h[k] * x
        t[1] += s_l[k] * x
    gen = torch.Generator(device=dev)
    gen.manual_seed(1_000_003 * seed + b)
    n = torch.clamp(torch.poisson((I0 * t).float(), generator=gen), min=1.0)
    m = -torch.log(n.double() / I0).float()
    return m[0].contiguous(), m[1].contiguous(), n[0].contiguous(), n[1].contiguous(), a, rows


STORAGE = {"f32": dect.STORE_F32, "f16": dect.STORE_F16, "f64": dect.STORE_F64}


# ---- what a program has in hand, and its call -------------------------------------------------------

def prepare(case, seed):
    dev = torch.device("cuda")
    gs = _geometries(case)
    gen = torch.Generator(device=dev)
    gen.manual_seed(7_919 * seed + 13)
    st = {"case": case}
    if case["do"] == "solve":
        one = None if case.get("uneven") else Geometry(gs[0])
        st["geoms"] = [one or Geometry(g) for g in gs]
        st["spec"] = Spectra(*_tables(case))
        st["data"] = []
        for b, g in enumerate(gs):
            m_h, m_l, w_h, w_l, _, rows = _scan(case, g, seed, b, dev)
            x0 = None
            if case.get("init") == "x0":  # a smooth image from an earlier pass
                x0 = torch.nn.functional.avg_pool2d(_image(g, rows, dev)[None], 5, 1, 2)[0]
                x0[1] = KAPPA * x0[0]
                x0 = x0.contiguous()
            st["data"].append((m_h, m_l, w_h, w_l, x0))
        st["solver"] = Solver(st["geoms"], st["spec"], m_udm=case.get("m", 1), n_pcg=case.get("n", 1), kappa=_kappa(case),
                              storage=STORAGE[case.get("storage", "f32")],
                              init=dect.INIT_CDM_FBP if case.get("init") == "cdm_fbp" else dect.INIT_PCG)
        return st
    g = gs[0]
    st["geo"] = Geometry(g)
    if case["do"] == "adjoint":
        dtype = torch.float64 if case.get("dtype") == "f64" else torch.float32
        rng = np.random.default_rng(seed)
        x = torch.stack([_image(g, _objects(case, g, rng), dev)[k % 2] for k in range(case["images"])])
        x = x.to(dtype) + 0.01 * torch.randn(x.shape, generator=gen, device=dev, dtype=dtype)
        st["x"] = x.contiguous().requires_grad_(case["images"] > 1)
        st["g"] = torch.randn((case["images"], g.n_views, g.n_bins), generator=gen, device=dev, dtype=dtype)
        return st
    st["spec"] = Spectra(*_tables(case))
    m_h, m_l, w_h, w_l, a, rows = _scan(case, g, seed, 0, dev)
    st["m"] = (m_h, m_l, w_h, w_l)
    if case["do"] == "fidelity":  # at an image some way from the data's
        st["x"] = (0.9 * torch.nn.functional.avg_pool2d(_image(g, rows, dev)[None], 3, 1, 1)[0]).contiguous().requires_grad_(True)
    elif case["do"] == "decompose":  # v = R x - u^a near the line integrals, the last iteration's a, the damping's start
        v = (a * (1.0 + 0.02 * torch.randn(a.shape, generator=gen, device=dev, dtype=torch.float64))).float()
        st["v"] = (v[0].contiguous(), v[1].contiguous())
        w = (a * (1.0 + 0.05 * torch.randn(a.shape, generator=gen, device=dev, dtype=torch.float64))).float()
        st["start"] = (w[0].contiguous(), w[1].contiguous(), torch.full_like(m_h, 1e-3))
    return st


def _kappa(case):
    return KAPPA if case.get("e_ref", E_REF) == E_REF else 1e-2


def run(st):
    case = st["case"]
    if case["do"] == "solve":  # new measurements, a reconstruction, the images
        sol = st["solver"]
        for b, (m_h, m_l, w_h, w_l, x0) in enumerate(st["data"]):
            sol.set_data(b, m_h, m_l, w_h, w_l, x0)
        sol.reconstruct(case["iters"])
        return [sol.get(b, dect.X) for b in range(len(st["data"]))]
    geo = st["geo"]
    if case["do"] == "adjoint":
        if case["images"] > 1:
            s = autograd.project(st["x"], geo)
            return [s.detach(), torch.autograd.grad(s, st["x"], st["g"])[0]]
        return [geo.project(st["x"]), geo.backproject(st["g"])]
    if case["do"] == "fidelity":
        m_h, m_l, w_h, w_l = st["m"]
        a = autograd.project(st["x"], geo)
        f_h, f_l = autograd.forward_model(a[0], a[1], st["spec"])
        loss = 0.5 * ((w_h * (f_h - m_h) ** 2).sum() + (w_l * (f_l - m_l) ** 2).sum())
        return [f_h.detach(), f_l.detach(), torch.autograd.grad(loss, st["x"])[0]]
    if case["do"] == "decompose":
        a_c, a_p, mu = (t.clone() for t in st["start"])
        status = torch.empty(mu.shape, dtype=torch.uint8, device=mu.device)
        st["spec"].decompose(*st["m"], *st["v"], 1e-3, 1e-3, case["iters"], a_c, a_p, mu, status)
        return [a_c, a_p, mu, status]
    return [cdm_fbp(geo, st["spec"], *st["m"], iters=case["iters"])]


# ---- the work that cannot be left out ------------------------------------------------------------------

def _samples(g):
    """Interpolated samples of one projection: one per ray and column or row (the spacing of the rays at the isocentre)."""
    spacing = g.bin_pitch_cm * (g.sod_cm / g.sdd_cm if g.kind == dect.FAN_FLAT else 1.0) / g.pixel_cm
    return 0.9 * g.n_views * g.nx * g.ny / spacing


def work(case):
    gs = _geometries(case)
    size = 8 if "f64" in (case.get("dtype"), case.get("storage")) else 4
    rays, pix, samples = (sum(f) for f in ([g.n_views * g.n_bins for g in gs], [g.nx * g.ny for g in gs],
                                           [_samples(g) for g in gs]))
    sums = 4 * 2 * 121  # exponential's argument and sums of one evaluation of f with its derivatives, about
    if case["do"] == "solve":
        m, n, it = case.get("m", 1), case.get("n", 1), case["iters"]
        pairs = it * (2 * n + 1) + {"pcg": 21, "cdm_fbp": 1, "x0": 0}[case.get("init", "pcg")] + 1
        fs = it * m + (10 if case.get("init", "pcg") != "x0" else 0)
        return {"bytes": 16 * rays + 2 * size * pix, "flops": pairs * 2 * 4 * samples + 2 * fs * sums * rays}
    if case["do"] == "adjoint":
        k = case["images"]
        return {"bytes": 2 * size * k * (rays + pix), "flops": 2 * k * 4 * samples}
    if case["do"] == "fidelity":
        return {"bytes": 4 * (4 * rays + 2 * rays + 4 * pix), "flops": 4 * 4 * samples + sums * rays}
    if case["do"] == "decompose":
        return {"bytes": (9 + 3) * 4 * rays + rays, "flops": 2 * case["iters"] * sums * rays}
    return {"bytes": 16 * rays + 8 * pix, "flops": 2 * case["iters"] * sums * rays + 2 * 6 * case["views"] * pix}


# ---- the same in float64, in plain torch -----------------------------------------------------------------

class _Exact:
    """R, R^T and the preconditioner of one geometry in float64 (Joseph's projector: a ray is sampled once per column,
    or per row where it is steeper, with linear interpolation between the two nearest pixels)."""

    def __init__(self, g, dev):
        self.g, self.dev = g, dev
        px, py, dx, dy = (t.reshape(-1) for t in _rays(g, dev))
        per_col = dx.abs() >= dy.abs()
        self.parts = []
        for axis, sel in ((0, per_col), (1, ~per_col)):
            i = torch.nonzero(sel).reshape(-1)
            a, b, da, db, n, m = (px, py, dx, dy, g.nx, g.ny) if axis == 0 else (py, px, dy, dx, g.ny, g.nx)
            slope = db[i] / da[i]
            q0 = (b[i] - a[i] * slope) / g.pixel_cm + 0.5 * (m - 1) - 0.5 * (n - 1) * slope
            self.parts.append((axis, i, q0, slope, g.pixel_cm / da[i].abs(), n, m))

    def _at(self, q0, slope, t, m):
        q = q0 + t * slope
        h = torch.floor(q)
        return (h + 1).clamp_(0, m + 1).long(), (h + 2).clamp_(0, m + 1).long(), q - h

    def project(self, x):
        out = torch.zeros((x.shape[0], self.g.n_views * self.g.n_bins), device=self.dev, dtype=torch.float64)
        for axis, i, q0, slope, w, n, m in self.parts:
            im = torch.nn.functional.pad(x if axis == 0 else x.transpose(1, 2), (0, 0, 1, 1)).transpose(1, 2).contiguous()
            acc = torch.zeros((x.shape[0], i.numel()), device=self.dev, dtype=torch.float64)
            for t in range(n):
                lo, hi, f = self._at(q0, slope, t, m)
                acc += (1 - f) * im[:, t][:, lo] + f * im[:, t][:, hi]
            out[:, i] = w * acc
        return out.reshape(-1, self.g.n_views, self.g.n_bins)

    def backproject(self, s):
        s = s.reshape(s.shape[0], -1)
        out = torch.zeros((s.shape[0], self.g.ny, self.g.nx), device=self.dev, dtype=torch.float64)
        for axis, i, q0, slope, w, n, m in self.parts:
            ws = w * s[:, i]
            acc = torch.zeros((s.shape[0], n, m + 2), device=self.dev, dtype=torch.float64)
            for t in range(n):
                lo, hi, f = self._at(q0, slope, t, m)
                acc[:, t].index_add_(1, lo, (1 - f) * ws)
                acc[:, t].index_add_(1, hi, f * ws)
            out += acc[:, :, 1:-1].transpose(1, 2) if axis == 0 else acc[:, :, 1:-1]
        return out

    def responses(self):
        """The circulant preconditioner with and without the D^T D term."""
        g = self.g
        ny, nx = (1 << (2 * n - 1).bit_length() for n in (g.ny, g.nx))
        d = torch.zeros((1, g.ny, g.nx), device=self.dev, dtype=torch.float64)
        d[0, g.ny // 2, g.nx // 2] = 1.0
        grid = torch.zeros((ny, nx), device=self.dev, dtype=torch.float64)
        grid[: g.ny, : g.nx] = self.backproject(self.project(d))[0]
        p = torch.fft.fft2(torch.roll(grid, (-(g.ny // 2), -(g.nx // 2)), (0, 1))).real.clamp(min=0.0)
        wy = 2 * math.pi * torch.arange(ny, device=self.dev, dtype=torch.float64) / ny
        wx = 2 * math.pi * torch.arange(nx, device=self.dev, dtype=torch.float64) / nx
        dd = 4 * torch.sin(wy / 2)[:, None] ** 2 + 4 * torch.sin(wx / 2)[None, :] ** 2
        return 1 / (p + dd + 1), 1 / (p + 1)

    def fbp(self, s):
        """Filtered backprojection with the band-limited ramp; linear interpolation between bins, zero beyond them."""
        g, dev = self.g, self.dev
        fan = g.kind == dect.FAN_FLAT
        scale = g.sod_cm / g.sdd_cm if fan else 1.0
        pitch = g.bin_pitch_cm * scale
        k = torch.arange(g.n_bins, device=dev, dtype=torch.float64)
        if fan:
            u = ((k - 0.5 * (g.n_bins - 1)) * g.bin_pitch_cm + g.bin_offset_cm) * scale
            s = s * (g.sod_cm / torch.sqrt(g.sod_cm**2 + u * u))
        d = k[:, None] - k[None, :]
        h = torch.where(d == 0, 0.25, torch.where(d.remainder(2) == 1, -1 / (math.pi * d.clamp(min=1)) ** 2, 0.0))
        h = torch.tril(h) + torch.tril(h, -1).T
        q = torch.nn.functional.pad(s @ h / pitch * (0.5 if fan else 1.0), (1, 1))
        x = ((torch.arange(g.nx, device=dev, dtype=torch.float64) - 0.5 * (g.nx - 1)) * g.pixel_cm)[None, :]
        y = ((torch.arange(g.ny, device=dev, dtype=torch.float64) - 0.5 * (g.ny - 1)) * g.pixel_cm)[:, None]
        out = torch.zeros((s.shape[0], g.ny, g.nx), device=dev, dtype=torch.float64)
        for v in range(g.n_views):
            th = g.angle0_rad + v * (g.angle_span_rad / g.n_views)
            c, sn = math.cos(th), math.sin(th)
            wgt = (g.sod_cm / (g.sod_cm - x * c - y * sn)) if fan else torch.ones_like(x + y)
            pos = (y * c - x * sn) * wgt * (g.sdd_cm / g.sod_cm) if fan else x * c + y * sn
            kf = (pos - g.bin_offset_cm) / g.bin_pitch_cm + 0.5 * (g.n_bins - 1)
            k0 = torch.floor(kf)
            f = kf - k0
            lo, hi = (k0 + 1).clamp(0, g.n_bins + 1).long(), (k0 + 2).clamp(0, g.n_bins + 1).long()
            out += (wgt * wgt) * ((1 - f) * q[:, v][:, lo] + f * q[:, v][:, hi])
        return out * ((2 * math.pi if fan else math.pi) / g.n_views)


def _model(tab, a, jac=True):
    """f_h, f_l and, with jac, {df_h/da_c, df_h/da_p, df_l/da_c, df_l/da_p} at a [2, ...]."""
    s_h, s_l, f_kn, f_p = tab
    t = [torch.zeros_like(a[0]) for _ in range(6 if jac else 2)]
    for k in range(len(f_kn)):
        x = torch.exp(-float(f_kn[k]) * a[0] - float(f_p[k]) * a[1])
        for i, c in enumerate((s_h[k], s_l[k], s_h[k] * f_kn[k], s_h[k] * f_p[k], s_l[k] * f_kn[k], s_l[k] * f_p[k])):
            if i < len(t) and c:
                t[i].add_(x, alpha=float(c))
    if not jac:
        return -torch.log(t[0]), -torch.log(t[1])
    return -torch.log(t[0]), -torch.log(t[1]), (t[2] / t[0], t[3] / t[0], t[4] / t[1], t[5] / t[1])


def _decompose(tab, meas, v, rho, iters, a, mu):
    """Levenberg-Marquardt on Eq. 13 per ray; a [2, ...], mu: the new ones."""
    m_h, m_l, w_h, w_l = meas

    def cost(f_h, f_l, a):
        return 0.5 * (w_h * (f_h - m_h) ** 2 + w_l * (f_l - m_l) ** 2
                      + rho[0] * (a[0] - v[0]) ** 2 + rho[1] * (a[1] - v[1]) ** 2)

    for _ in range(iters):
        f_h, f_l, (j0, j1, j2, j3) = _model(tab, a)
        r_h, r_l = f_h - m_h, f_l - m_l
        g0 = w_h * r_h * j0 + w_l * r_l * j2 + rho[0] * (a[0] - v[0])
        g1 = w_h * r_h * j1 + w_l * r_l * j3 + rho[1] * (a[1] - v[1])
        b00 = (w_h * j0 * j0 + w_l * j2 * j2 + rho[0]) * (1 + mu)
        b11 = (w_h * j1 * j1 + w_l * j3 * j3 + rho[1]) * (1 + mu)
        b01 = w_h * j0 * j1 + w_l * j2 * j3
        det = b00 * b11 - b01 * b01
        new = torch.stack([a[0] + (g1 * b01 - g0 * b11) / det, a[1] + (g0 * b01 - g1 * b00) / det])
        ok = (cost(*_model(tab, new, jac=False), new) < cost(f_h, f_l, a)) & (det > 0)
        a = torch.where(ok, new, a)
        mu = torch.where(ok, mu * 0.1, mu * 10.0).clamp(1e-10, 1e10)
    return a, mu


def _grad(x):
    y = torch.zeros((2,) + x.shape, device=x.device, dtype=x.dtype)
    y[0, :, :, :-1] = x[:, :, 1:] - x[:, :, :-1]
    y[1, :, :-1, :] = x[:, 1:, :] - x[:, :-1, :]
    return y


def _grad_t(y):
    x = torch.zeros_like(y[0])
    x[:, :, :-1] -= y[0, :, :, :-1]
    x[:, :, 1:] += y[0, :, :, :-1]
    x[:, :-1, :] -= y[1, :, :-1, :]
    x[:, 1:, :] += y[1, :, :-1, :]
    return x


def _solve(case, g, tab, meas, x0, dev):
    """UDM(m)-PCG(n) from the case's start, in float64."""
    R, lam, rho = _Exact(g, dev), 1e-5, [1e-3, 1e-3]
    H, Hn = R.responses()
    meas = tuple(t.double() for t in meas)
    m, n = case.get("m", 1), case.get("n", 1)

    def dot(a, b):
        return (a * b).sum((1, 2), keepdim=True)

    def pcg(x, Rx, r, steps, H, with_grad):
        def M(r):
            return torch.fft.ifft2(H * torch.fft.fft2(r, s=H.shape)).real[:, : g.ny, : g.nx]

        def safe(a, b):
            return torch.where(b > 0, a / torch.where(b > 0, b, 1.0), 0.0)

        p = M(r)
        rs = dot(r, p)
        for k in range(steps):
            q = R.project(p)
            Ap = R.backproject(q) + p + (_grad_t(_grad(p)) if with_grad else 0.0)
            al = safe(rs, dot(p, Ap))
            x, Rx = x + al * p, Rx + al * q
            if k + 1 < steps:
                r = r - al * Ap
                s = M(r)
                new = dot(r, s)
                p, rs = s + safe(new, rs) * p, new
        return x, Rx

    if x0 is not None:
        x = x0.double()
    else:
        abar = float((tab[1] * tab[2]).sum())
        z = torch.zeros_like(meas[0])
        cdm = case.get("init") == "cdm_fbp"
        a, _ = _decompose(tab, meas, (z, z), (0.0, 0.0 if cdm else rho[1]), 10, torch.stack([meas[1] / abar, z]),
                          torch.full_like(z, 1e-3))
        if cdm:
            xc = R.fbp(a[:1].clamp(min=0.0))
        else:
            b = a[:1]
            xc, _ = pcg(torch.zeros((1, g.ny, g.nx), device=dev, dtype=torch.float64), torch.zeros_like(b),
                        R.backproject(b), 10, Hn, False)
        xc = xc.clamp(min=0.0)
        x = torch.cat([xc, _kappa(case) * xc])
    Rx = R.project(x)
    a, y, z = Rx, _grad(x), x
    ua, uy, uz = torch.zeros_like(a), torch.zeros_like(y), torch.zeros_like(z)
    mu = torch.full_like(meas[0], 1e-3)
    for _ in range(case["iters"]):
        a0, y0, z0 = a, y, z
        r = R.backproject(a + ua - Rx) + _grad_t(y + uy - _grad(x)) + z + uz - x
        x, Rx = pcg(x, Rx, r, n, H, True)
        a, mu = _decompose(tab, meas, Rx - ua, rho, m, a, mu)
        t = _grad(x) - uy
        tau = torch.tensor([lam / rho[0], lam / rho[1]], device=dev, dtype=torch.float64)[None, :, None, None]
        y = torch.sign(t) * (t.abs() - tau).clamp(min=0.0)
        z = (x - uz).clamp(min=0.0)
        ua, uy, uz = ua + a - Rx, uy + y - _grad(x), uz + z - x
        for b in range(2):
            pri = ((a - Rx)[b].square().sum() + (y - _grad(x))[:, b].square().sum() + (z - x)[b].square().sum()).sqrt().item()
            dual = rho[b] * ((a - a0)[b].square().sum() + (y - y0)[:, b].square().sum() + (z - z0)[b].square().sum()).sqrt().item()
            f = 2.0 if pri > 10.0 * dual else 0.5 if dual > 10.0 * pri else 1.0
            rho[b] *= f
            ua[b] /= f
            uy[:, b] /= f
            uz[b] /= f
    return x


def exact(case, seed):
    if case["do"] == "solve":
        # projections of a pass, in samples: beyond this the float64 restatement takes longer than is useful
        gs = _geometries(case)
        pairs = 3 * case["iters"] * case.get("n", 1) + (23 if case.get("init", "pcg") == "pcg" else 4)
        if case.get("storage") == "f16" or pairs * sum(_samples(g) for g in gs) > 8e9:
            return None
    dev = torch.device("cuda")
    st = prepare(case, seed)
    tab = _tables(case)
    if case["do"] == "solve":
        return [_solve(case, g, tab, d[:4], d[4], dev) for g, d in zip(gs, st["data"])]
    g = _geometries(case)[0]
    R = _Exact(g, dev)
    if case["do"] == "adjoint":
        return [R.project(st["x"].detach().double()), R.backproject(st["g"].double())]
    meas = tuple(t.double() for t in st["m"])
    if case["do"] == "fidelity":
        f_h, f_l, (j0, j1, j2, j3) = _model(tab, R.project(st["x"].detach().double()))
        e_h, e_l = meas[2] * (f_h - meas[0]), meas[3] * (f_l - meas[1])
        return [f_h, f_l, R.backproject(torch.stack([e_h * j0 + e_l * j2, e_h * j1 + e_l * j3]))]
    if case["do"] == "decompose":
        a, _ = _decompose(tab, meas, tuple(t.double() for t in st["v"]), (1e-3, 1e-3), case["iters"],
                          torch.stack([t.double() for t in st["start"][:2]]), st["start"][2].double())
        return [a[0], a[1], None, None]  # the damping and the status follow from comparisons, not from sums
    z = torch.zeros_like(meas[0])
    a, _ = _decompose(tab, meas, (z, z), (0.0, 0.0), case["iters"],
                      torch.stack([meas[1] / float((tab[1] * tab[2]).sum()), z]), torch.full_like(z, 1e-3))
    return [R.fbp(a.clamp(min=0.0))]
