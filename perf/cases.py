"""The calls that users of this library make, as measurable cases.

Each case is one pass through the public entry points on inputs drawn from a
seed: a pattern on the device (``scatman_voxelise`` + ``scatman_forward``), a
fit step through ``torch.autograd`` (``autograd.msft``), patterns into host
memory (``scatman_acquire_batch``), or a batch of fit requests on the native
server.  Sizes are those of the repository's workloads, tests and benchmark:
grids 24^3 - 128^3, flat detectors 48^2 - 512^2 to 25 - 60 degrees, uniform-q
detectors 128^2 - 2048^2, wavelengths of 6 - 12 voxels, every shape kind.

``exact`` restates the result in plain FP64 torch (direct sums, no code of the
library).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2202_03411_gb300 as sm
from paper_2202_03411_gb300.autograd import msft, params_of
from paper_2202_03411_gb300.serving import Server
from paper_2202_03411_gb300.types import (DETECTOR_FLAT, DETECTOR_UNIFORM_Q, ELLIPSOID, RADIALMAP, SPHERE, SPHHARM,
                                          VOLUMEMAP, Geometry, Shape)

KINDS = {"sphere": SPHERE, "ellipsoid": ELLIPSOID, "harmonics": SPHHARM, "radialmap": RADIALMAP,
         "volumemap": VOLUMEMAP}
SOFT_WIDTH = 0.5
SERVE_SLOTS = 4
SERVE_BUDGET = 32 << 30
SERVE_GRIDS = (48, 64, 96, 128)
SERVE_DETECTORS = (128, 256, 512)


def _case(do, precision, kind, n, det, theta, wavelength, **more):
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    det_nx, det_ny = (det, det) if isinstance(det, int) else det
    return {"do": do, "precision": precision, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "det_nx": det_nx,
            "det_ny": det_ny, "theta": float(theta), "wavelength": float(wavelength), "lmax": 8, "count": 1, **more}


def listed():
    return [
        # the FP64 reference mode on the paper's simplest sample: the smallest call, where latency counts
        {"name": "sphere_32_fp64", **_case("forward", "fp64", "sphere", 32, 64, 30, 8)},
        # the plain FP32 mode and the FP64 accuracy mode on the ellipsoid workload
        {"name": "ellipsoid_96_fp32", **_case("forward", "fp32", "ellipsoid", 96, 256, 45, 10)},
        {"name": "ellipsoid_96_fp64", **_case("forward", "fp64", "ellipsoid", 96, 256, 45, 10)},
        # the benchmark: l <= 8 harmonics, BF16 split phases, 512^2 pixels to 60 degrees
        {"name": "harmonics_128_bf16", **_case("forward", "tc_bf16_split", "harmonics", 128, 512, 60, 10)},
        # a sample box and a detector off every tile boundary, FP16 split phases
        {"name": "ragged_f16", **_case("forward", "tc_f16_split", "ellipsoid", (70, 52, 41), (301, 257), 50, 7)},
        # a voxelised two-material sample (per-cell refractive index)
        {"name": "volumemap_96_bf16", **_case("forward", "tc_bf16_split", "volumemap", 96, 256, 45, 10)},
        # the paper's virtual detector: Fig. 8b's largest case on the tensor cores, a mid one in the paper's FP32
        {"name": "uniform_2048_bf16", **_case("uniform", "tc_bf16_split", "harmonics", 56, 2048, 30, 1, radius=20.0)},
        {"name": "uniform_512_fp32", **_case("uniform", "fp32", "harmonics", 30, 512, 30, 1, radius=10.0)},
        # one step of a shape fit: forward, least-squares loss, gradient of every shape parameter
        {"name": "fit_96_bf16", **_case("fit", "tc_bf16_split", "harmonics", 96, 256, 45, 10, lmax=6)},
        {"name": "fit_48_fp32", **_case("fit", "fp32", "ellipsoid", 48, 128, 45, 10)},
        # patterns for a host program (a data set, a plot): shape parameters in, pinned host images out
        {"name": "batch_128_bf16", **_case("batch", "tc_bf16_split", "harmonics", 128, 512, 60, 10, count=4)},
        # many concurrent fits of mixed grids and detectors on the server
        {"name": "serve_mixed_bf16", **_case("serve", "tc_bf16_split", "mixed", 128, 512, 45, 10, lmax=6, count=12)},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choices(["forward", "fit", "uniform", "batch", "serve"], [10, 5, 2, 2, 2])[0]
    theta, wavelength = round(rng.uniform(25, 60), 2), round(rng.uniform(6, 12), 2)
    if do == "serve":
        return _case("serve", "tc_bf16_split", "mixed", rng.choice([64, 96, 128]), rng.choice([256, 512]), 45, 10,
                     lmax=rng.randint(3, 6), count=rng.randint(4, 12))
    if do == "uniform":
        radius = round(math.exp(rng.uniform(math.log(3), math.log(20))), 2)
        n = int(math.ceil(2.6 * radius)) + 4
        return _case("uniform", rng.choice(["tc_bf16_split", "fp32"]), "harmonics", n,
                     (_log_int(rng, 128, 2048), _log_int(rng, 128, 2048)), 30, 1, radius=radius)
    if do == "fit":
        precision = rng.choices(["tc_bf16_split", "tc_f16_split", "fp32", "fp64"], [4, 2, 3, 1])[0]
        top, pix = (96, 256) if precision.startswith("tc") else (64, 160) if precision == "fp32" else (40, 80)
        kind = rng.choice(["sphere", "ellipsoid", "harmonics"])
    else:
        precision = rng.choices(["tc_bf16_split", "tc_f16_split", "fp32", "fp64"], [5, 2, 2, 1])[0]
        top, pix = (128, 512) if precision.startswith("tc") else (96, 256)
        kind = rng.choice(["sphere", "ellipsoid", "harmonics", "radialmap", "volumemap"])
    base = _log_int(rng, 24, top)
    n = tuple(min(top, max(20, int(base * rng.uniform(0.75, 1.2)))) for _ in range(3))
    side = _log_int(rng, 48, pix)
    det = tuple(min(pix, max(40, int(side * rng.uniform(0.8, 1.25)))) for _ in range(2))
    return _case(do, precision, kind, n, det, theta, wavelength, lmax=rng.randint(3, 8),
                 count=rng.randint(2, 4) if do == "batch" else 1)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _geometry(c):
    if c["do"] == "uniform":
        # Fig. 8b: lengths in wavelengths, the voxel at the detector's Nyquist spacing
        voxel = c["wavelength"] / (2.0 * math.sin(math.radians(c["theta"])))
        return Geometry(c["nx"], c["ny"], c["nz"], voxel, c["wavelength"], c["theta"], c["det_nx"], c["det_ny"],
                        DETECTOR_UNIFORM_Q)
    return Geometry(c["nx"], c["ny"], c["nz"], 1.0, c["wavelength"], c["theta"], c["det_nx"], c["det_ny"],
                    DETECTOR_FLAT)


def _orientation(rng):
    return dict(latitude=math.degrees(math.asin(rng.uniform(-1, 1))), longitude=rng.uniform(-180, 180),
                rotation=rng.uniform(0, 360))


def _alm(rng, lmax, sigma=0.05):
    alm = np.zeros((lmax + 1) ** 2)
    for l in range(1, lmax + 1):
        alm[l * l:(l + 1) ** 2] = rng.normal(0.0, sigma / l, 2 * l + 1)
    return alm


def _shape(kind, n, lmax, rng, radius=None):
    """A random sample of the given kind in a box of n voxels (smallest side)."""
    delta = rng.uniform(1e-3, 2e-2)
    common = dict(delta=delta, beta=delta / 10.0, **_orientation(rng))
    if kind == "sphere":
        return Shape(SPHERE, r=rng.uniform(0.28, 0.4) * n, delta=delta, beta=delta / 10.0)
    if kind == "ellipsoid":
        a, b, c = rng.uniform(0.21, 0.42, 3) * n
        return Shape(ELLIPSOID, a=a, b=b, c=c, **common)
    if kind == "harmonics":
        if radius is not None:          # the Listing-2 shape's degrees, at its mean radius
            return Shape(SPHHARM, R0=radius, lmax=lmax, alm=_alm(rng, lmax, 0.08), **common)
        return Shape(SPHHARM, R0=0.375 * n, lmax=lmax, alm=_alm(rng, lmax), **common)
    if kind == "radialmap":
        nt, npf = 96, 192
        lat = -math.pi / 2 + math.pi * np.arange(nt)[:, None] / nt
        lon = 2 * math.pi * np.arange(npf)[None, :] / npf
        f = np.zeros((nt, npf))
        for _ in range(6):
            a, b = int(rng.integers(1, 4)), int(rng.integers(0, 4))
            p, q = rng.uniform(0, 2 * math.pi, 2)
            f += rng.normal() * np.cos(2 * a * lat + p) * np.cos(b * lon + q)
        return Shape(RADIALMAP, radial_map=0.31 * n * (1.0 + 0.15 * f / np.abs(f).max()), **common)
    m = 40
    v = np.zeros((m, m, m), dtype=bool)
    v[13:27, 13:27, 13:27] = True
    for _ in range(6):
        lo = rng.integers(0, m - 2, 3)
        hi = np.minimum(lo + rng.integers(2, 13, 3), m)
        v[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] = True
    core = (np.abs(np.indices(v.shape) - (m - 1) / 2) <= m / 4).all(axis=0)
    return Shape(VOLUMEMAP, volume_map=v, map_dx=0.71 * n / m, map_delta=np.where(core, 0.02, 0.006),
                 map_beta=np.where(core, 0.004, 0.0005), **common)


def _samples(c, seed):
    """The case's (geometry, shape) pairs."""
    rng = np.random.default_rng([seed, c["nx"], c["det_nx"], c["count"]])
    mix = np.random.default_rng([c["lmax"], c["nx"], c["det_nx"], c["count"]])
    out = []
    for i in range(c["count"]):
        if c["do"] == "serve":
            # the serving mix: every request its own grid, detector and kind, up to the case's sizes
            n = int(mix.choice([g for g in SERVE_GRIDS if g <= c["nx"]]))
            det = int(mix.choice([d for d in SERVE_DETECTORS if d <= c["det_nx"]]))
            g = Geometry(n, n, n, 1.0, c["wavelength"], c["theta"], det, det)
            s = _shape(("sphere", "ellipsoid", "harmonics")[i % 3], 0.8 * n, c["lmax"], rng)
        else:
            g = _geometry(c)
            s = _shape(c["kind"], min(g.nx, g.ny, g.nz), c["lmax"], rng, c.get("radius"))
        out.append((g, s))
    return out


def _k(g):
    """Outgoing directions of the detector's pixels, in units of k0, and whether each exists ([n_pix, 3], [n_pix])."""
    u = (2 * torch.arange(g.det_nx, dtype=torch.float64, device="cuda") + 1 - g.det_nx) / g.det_nx
    v = (2 * torch.arange(g.det_ny, dtype=torch.float64, device="cuda") + 1 - g.det_ny) / g.det_ny
    v, u = torch.meshgrid(v, u, indexing="ij")
    u, v = u.reshape(-1), v.reshape(-1)
    if g.detector == DETECTOR_UNIFORM_Q:
        top = math.sin(math.radians(g.theta_max_deg))
        kx, ky = u * top, v * top
        s2 = kx * kx + ky * ky
        return torch.stack([kx, ky, torch.sqrt((1 - s2).clamp(min=0))], 1), s2 <= 1
    top = math.tan(math.radians(g.theta_max_deg))
    k = torch.stack([u * top, v * top, torch.ones_like(u)], 1)
    return k / k.norm(dim=1, keepdim=True), torch.ones_like(u, dtype=torch.bool)


def _measured(g, shape, rng):
    """A measured pattern to fit: the form factor of a sphere of about the sample's size with counting noise."""
    q = (_k(g)[0] - torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")) * (2 * math.pi / g.wavelength)
    size = {SPHERE: shape.r, ELLIPSOID: (shape.a * shape.b * shape.c) ** (1 / 3)}.get(shape.kind, shape.R0)
    x = q.norm(dim=1).clamp(min=1e-6) * (size * (1 + 0.02 * float(rng.normal())))
    f = 3 * (torch.sin(x) - x * torch.cos(x)) / x ** 3
    top = (2 * shape.delta * 4 / 3 * math.pi * size ** 3 / g.voxel ** 3) ** 2
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    return (torch.poisson(1e4 * f * f, generator=gen) * (top / 1e4)).float()


def _real(c):
    return torch.float64 if c["precision"] == "fp64" else torch.float32


def prepare(c, seed):
    pairs = _samples(c, seed)
    g, s = pairs[0]
    st = {"do": c["do"], "g": g, "shape": s}
    rng = np.random.default_rng([seed, 7])
    if c["do"] == "serve":
        st["server"] = Server(SERVE_BUDGET, slots=SERVE_SLOTS, precision=c["precision"], soft_width=SOFT_WIDTH)
        st["requests"] = [(g, s, _measured(g, s, rng).cpu().numpy()) for g, s in pairs]
        return st
    fit = c["do"] == "fit"
    st["h"] = sm.scatman_create(g, c["precision"], soft=fit, soft_width=SOFT_WIDTH)
    if fit:
        # an optimiser holds the parameters in the precision of the fit
        st["params"] = torch.from_numpy(params_of(s)).to(_real(c)).requires_grad_()
        st["target"] = _measured(g, s, rng).to(_real(c))
    elif c["do"] == "batch":
        st["shapes"] = [s for _, s in pairs]
        st["host"] = torch.empty(c["count"], g.n_pix, dtype=_real(c), pin_memory=True)
    else:
        st["I"] = torch.empty(g.n_pix, dtype=_real(c), device="cuda")
    return st


def run(st):
    if st["do"] == "serve":
        tickets = [st["server"].submit(g, s, t, want_I=True) for g, s, t in st["requests"]]
        out = []
        for ticket, res in tickets:
            status, _ = st["server"].wait(ticket)
            if status != 0:
                raise RuntimeError(f"request failed with status {status}")
            # the fits behind the server keep losses and gradients in FP32, the precision they are computed in
            out.append({"I": res["I"], "loss": res["loss"].astype(np.float32), "grad": res["grad"].astype(np.float32)})
        return out
    if st["do"] == "fit":
        p = st["params"]
        p.grad = None
        I = msft(p, st["h"], st["shape"])
        loss = ((I - st["target"]) ** 2).sum()
        loss.backward()
        return {"I": I.detach(), "loss": loss.detach(), "grad": p.grad}
    if st["do"] == "batch":
        sm.scatman_acquire_batch(st["h"], st["shapes"], st["host"])
        return st["host"]
    sm.scatman_voxelise(st["h"], st["shape"])
    sm.scatman_forward(st["h"], st["I"])
    return st["I"]


def work(c):
    """Bytes: the shape's description in, the results out.  Flops: the band limit of a sample that fills the box
    sets the directions at which its field is needed (two per period along each transverse axis); the sums over y and
    then over x and z at those, eight flops a complex term, twice for a gradient; eight per pixel to interpolate."""
    total = {"bytes": 0.0, "flops": 0.0}
    for g, s in _samples(c, 0):
        sinus = math.sin(math.radians(g.theta_max_deg))
        ky, kx = (2 * n * g.voxel * sinus / g.wavelength + 1 for n in (g.ny, g.nx))
        flops = 8.0 * (ky * g.n_vox + ky * kx * g.nx * g.nz + g.n_pix) + 10.0 * g.n_vox
        size = 8 if c["precision"] == "fp64" else 4
        data = size * g.n_pix + 8 * s.n_params() + sum(a.nbytes for a in (s.radial_map, s.volume_map, s.map_delta,
                                                                          s.map_beta) if a is not None)
        if c["do"] in ("fit", "serve"):
            flops, data = 2 * flops, data + 4 * g.n_pix + 8 * s.n_params()
        total["bytes"] += data
        total["flops"] += flops
    return total


# ---------------------------------------------------------------------------
# The same results in plain FP64 torch
# ---------------------------------------------------------------------------

def _coords(n, voxel):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1) / 2) * voxel


def _rotation(s):
    lon, tilt, rot = (math.radians(v) for v in (s.longitude, 90.0 + s.latitude, s.rotation))

    def about_z(a):
        return np.array([[math.cos(a), -math.sin(a), 0], [math.sin(a), math.cos(a), 0], [0, 0, 1.0]])

    about_y = np.array([[math.cos(tilt), 0, math.sin(tilt)], [0, 1.0, 0], [-math.sin(tilt), 0, math.cos(tilt)]])
    return torch.from_numpy(about_z(lon) @ about_y @ about_z(rot)).cuda()


def _harmonics(lmax, u):
    """Real orthonormal harmonics (with the Condon-Shortley sign) for l = 1 .. lmax at unit vectors u, in alm order."""
    z, rho = u[..., 2], torch.sqrt(u[..., 0] ** 2 + u[..., 1] ** 2)
    safe = torch.where(rho > 0, rho, torch.ones_like(rho))
    e = torch.complex(torch.where(rho > 0, u[..., 0] / safe, torch.ones_like(rho)),
                      torch.where(rho > 0, u[..., 1] / safe, torch.zeros_like(rho)))
    P = {(0, 0): torch.ones_like(z)}
    for m in range(1, lmax + 1):
        P[m, m] = -(2 * m - 1) * rho * P[m - 1, m - 1]
    for m in range(lmax + 1):
        for l in range(m + 1, lmax + 1):
            low = P[l - 2, m] if l >= m + 2 else 0.0
            P[l, m] = ((2 * l - 1) * z * P[l - 1, m] - (l + m - 1) * low) / (l - m)
    powers = [torch.ones_like(e)]
    for m in range(lmax):
        powers.append(powers[-1] * e)
    for l in range(1, lmax + 1):
        for m in range(-l, l + 1):
            k = abs(m)
            norm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - k) / math.factorial(l + k))
            if m == 0:
                yield norm * P[l, 0]
            else:
                yield math.sqrt(2) * norm * P[l, k] * (powers[k].real if m > 0 else powers[k].imag)


def _sample_exact(g, s, p, soft):
    """The slice strengths [z][x][y], differentiable in p = params_of(s) where the occupancy is soft."""
    d = torch.stack(torch.broadcast_tensors(_coords(g.nx, g.voxel)[None, :, None], _coords(g.ny, g.voxel)[None, None],
                                            _coords(g.nz, g.voxel)[:, None, None]), -1)
    d = d - torch.tensor([s.cx, s.cy, s.cz], dtype=torch.float64, device="cuda")
    body = d @ _rotation(s)
    r = body.norm(dim=-1)
    u = torch.where(r[..., None] > 0, body / r.clamp(min=1e-300)[..., None],
                    torch.tensor([0, 0, 1.0], dtype=torch.float64, device="cuda"))
    delta, beta = (p[-2], p[-1]) if p is not None else (torch.tensor(v, dtype=torch.float64) for v in (s.delta, s.beta))
    if s.kind == VOLUMEMAP:
        m = s.volume_map.shape
        cell = torch.floor(body / s.map_dx + torch.tensor(m, dtype=torch.float64, device="cuda") / 2).long()
        ok = ((cell >= 0) & (cell < torch.tensor(m, device="cuda"))).all(-1)
        at = ((cell[..., 0] * m[1] + cell[..., 1]) * m[2] + cell[..., 2]) * ok
        chi = torch.from_numpy(np.ascontiguousarray(s.volume_map)).cuda().reshape(-1)[at].double() * ok
        delta, beta = (torch.from_numpy(a).cuda().reshape(-1)[at] for a in (s.map_delta, s.map_beta))
    else:
        if s.kind == SPHERE:
            rs = (p[0] if p is not None else s.r) + 0 * r
        elif s.kind == ELLIPSOID:
            axes = p[:3] if p is not None else torch.tensor([s.a, s.b, s.c], dtype=torch.float64, device="cuda")
            rs = 1.0 / ((u / axes) ** 2).sum(-1).sqrt()
        elif s.kind == RADIALMAP:
            rm = torch.from_numpy(s.radial_map).cuda()
            nt, npf = rm.shape
            ti = (torch.atan2(body[..., 2], body[..., :2].norm(dim=-1)) + math.pi / 2) * (nt / math.pi)
            tk = torch.remainder(torch.atan2(body[..., 1], body[..., 0]), 2 * math.pi) * (npf / (2 * math.pi))
            i, k = torch.floor(ti).long(), torch.floor(tk).long()
            f, h = ti - i, tk - k
            rs = sum(wi * wk * rm[(i + a) % nt, (k + b) % npf] for a, wi in ((0, 1 - f), (1, f))
                     for b, wk in ((0, 1 - h), (1, h)))
        else:
            R0 = p[-3] if p is not None else s.R0
            alm = p[:-3] if p is not None else torch.from_numpy(s.alm[1:]).cuda()
            rs = R0 * (1 + sum(a * y for a, y in zip(alm, _harmonics(s.lmax, u))))
            top = 0.5 * (min(g.nx, g.ny, g.nz) - 1) * g.voxel - g.voxel
            rs = torch.minimum(torch.maximum(rs, 0.1 * R0 + 0 * rs), torch.full_like(rs, top))
        chi = torch.sigmoid((rs - r) / SOFT_WIDTH) if soft else (r <= rs).double()
    n = torch.complex(1 - delta + 0 * chi, beta + 0 * chi)
    step = chi * (n - 1)
    before = torch.cumsum(step, 0) - step
    k0 = 2 * math.pi / g.wavelength
    return (n * n - 1) * chi * torch.exp(1j * k0 * g.voxel * before)


def _phases(q, n, voxel):
    return torch.exp(-1j * q[:, None] * _coords(n, voxel)[None, :])


def _chunks(g):
    step = max(256, int(1.5e9 / (16 * g.nx * g.nz)))
    return [slice(a, min(a + step, g.n_pix)) for a in range(0, g.n_pix, step)]


def _q(g):
    k, valid = _k(g)
    return (k - torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")) * (2 * math.pi / g.wavelength), valid


def _field_exact(g, rho):
    q, valid = _q(g)
    box = [torch.nonzero(rho.abs().amax(dim=[k for k in range(3) if k != a]) > 0)[:, 0] for a in range(3)]
    if not all(len(b) for b in box):
        return torch.zeros(g.n_pix, dtype=torch.complex128, device="cuda")
    z, x, y = (slice(int(b[0]), int(b[-1]) + 1) for b in box)
    part = rho[z, x, y]
    flat = part.reshape(-1, part.shape[2]).t().contiguous()
    A = torch.empty(g.n_pix, dtype=torch.complex128, device="cuda")
    for c in _chunks(g):
        G = (_phases(q[c, 1], g.ny, g.voxel)[:, y] @ flat).view(-1, part.shape[0], part.shape[1])
        G = torch.bmm(G, _phases(q[c, 0], g.nx, g.voxel)[:, x, None])[..., 0]
        A[c] = (G * _phases(q[c, 2], g.nz, g.voxel)[:, z]).sum(1)
    return A * valid


def _adjoint_exact(g, w):
    """sum_p w_p e^{+i q_p r_v} over the pixels."""
    q, _ = _q(g)
    S = torch.zeros(g.nz * g.nx, g.ny, dtype=torch.complex128, device="cuda")
    for c in _chunks(g):
        left = (w[c, None] * _phases(q[c, 2], g.nz, g.voxel).conj())[:, :, None] * \
            _phases(q[c, 0], g.nx, g.voxel).conj()[:, None, :]
        S += left.reshape(-1, g.nz * g.nx).t() @ _phases(q[c, 1], g.ny, g.voxel).conj()
    return S.view(g.nz, g.nx, g.ny)


def _fit_exact(g, s, p, target):
    p = p.detach().double().cuda().requires_grad_()
    rho = _sample_exact(g, s, p, True)
    A = _field_exact(g, rho.detach())
    I = A.abs() ** 2
    t = target.double().to("cuda")
    S = _adjoint_exact(g, 2 * (I - t) * A)
    (2 * (S.conj() * rho).real.sum()).backward()
    return {"I": I, "loss": ((I - t) ** 2).sum(), "grad": p.grad}


def exact(c, seed):
    pairs = _samples(c, seed)
    rng = np.random.default_rng([seed, 7])
    if c["do"] in ("fit", "serve"):
        out, left = [], 6e12
        for g, s in pairs:
            target = _measured(g, s, rng)
            left -= 16.0 * g.n_pix * g.n_vox
            if left < 0:                    # the rest of a long list of requests would take too long
                out.append(None)
                left += 16.0 * g.n_pix * g.n_vox
                continue
            p = torch.from_numpy(params_of(s))
            r = _fit_exact(g, s, p.to(_real(c)) if c["do"] == "fit" else p, target)
            out.append(r if c["do"] == "fit" else {**r, "loss": r["loss"].reshape(1)})
        return out[0] if c["do"] == "fit" else out
    with torch.no_grad():
        I = [_field_exact(g, _sample_exact(g, s, None, False)).abs() ** 2 for g, s in pairs]
    return torch.stack(I) if c["do"] == "batch" else I[0]
