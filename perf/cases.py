"""Measured cases: what a user of the library has it compute, from one small
map to a paper-scale evaluation.

A case is a specimen (grid, slices, ionized sites and their channels), the
optics, a scan list, a precision and the call that is made:
  map    the map of a specimen whose matrices are built (another H, e.g. the
         next edge, on the same builds);
  eval   the whole evaluation: both builds, then the map;
  sites  both builds, then every site's own contribution;
  fit    one step of a fit through torch.autograd: forward map, squared
         distance to a measured map, gradients;
  cube   the S1 build and the 4D cube;
  qeels  the momentum-resolved map of a built specimen.
Maps are returned as the float32 image that a program stores or compares with
a measured one.  Specimens are synthetic crystals like those of synth/
(Gaussian atoms, one per 2.5 A cell and 2 A slice, 0.078 A pixels; hydrogenic
transition potentials with a random complex amplitude per site and channel),
made here from the seed.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2607_00756_gb300.autograd import coreloss_map
from paper_2607_00756_gb300.context import BipContext

CELL, SLICE = 2.5, 2.0                # A
PX = 10.0 / 128.0                     # A per pixel
CELL_PX = 32                          # pixels per cell

# every case has these fields; a listed case names those that differ
DEFAULTS = dict(
    kind="eval", prec="mixed",
    ny=512, nx=512, nz=100, f=4,      # grid, slices, beam subsampling
    kv=300, alpha=25.0, theta=40.0,   # keV, mrad
    defocus=0.0, cs=0.0,              # A
    rings=4,                          # hex rings of parents, both sides
    recon="magnitude",
    win=64, cells=4, planes=100,      # sites: the central cells x cells columns on that many slices
    nch=3,                            # channels per site
    small_win=0, small_nch=0,         # every second site: its own window and channel count
    raster=True, sy=128, sx=128, step=1.0,   # raster of sy x sx, or sy*sx scattered positions
    box=0,                            # cube: box x box k-pixels (0: the detector disc)
)


def _case(**kw):
    c = dict(DEFAULTS)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: four atoms of a 10 A cell, 16 x 16 scans, the builds at hand
        _case(name="map_small", kind="map", ny=128, nx=128, nz=5, f=2, kv=200, alpha=20.0, rings=2, cells=2, planes=1,
              sy=16, sx=16, step=4.0),
        # the same specimen from its potential, in the library's default precision
        _case(name="eval_small_fp32", prec="fp32", ny=128, nx=128, nz=5, f=2, kv=200, alpha=20.0, rings=2, cells=2,
              planes=1, sy=16, sx=16, step=4.0),
        # paper-like scale, whole evaluation, the mixed path: 1600 sites, 128 x 128 scans
        _case(name="eval_paper_mixed"),
        # the same optics with FP8 operands: 640 sites
        _case(name="eval_512_fp8", prec="fp8", planes=40),
        # the same optics in FP32 (reference-quality maps): 160 sites, 64 x 64 scans
        _case(name="eval_512_fp32", prec="fp32", planes=10, sy=64, sx=64, step=2.0),
        # L-edge-like sites (nine channels) in split BF16, f = 3, scattered scan positions
        _case(name="eval_384_split", prec="split_bf16", ny=384, nx=384, nz=40, f=3, planes=3, nch=9, raster=False,
              sy=64, sx=32),
        # large grid, few sites, every site's own contribution
        _case(name="sites_1024", kind="sites", ny=1024, nx=1024, nz=20, planes=2, sy=64, sx=64),
        # two edges on one specimen: nine channels on 64 px, one channel on 32 px, aberrated probe
        _case(name="map_two_edges", kind="map", ny=384, nx=384, nz=40, f=3, planes=3, nch=9, small_win=32, small_nch=1,
              defocus=30.0, cs=5.0e5, sy=64, sx=64),
        # structure refinement: occupancies, transition potentials, slice potentials
        _case(name="fit_mixed", kind="fit", ny=256, nx=256, nz=40, f=2, kv=200, alpha=20.0, rings=2, planes=4, sy=32,
              sx=32, step=2.0, defocus=25.0, cs=5.0e5),
        # the same in FP32
        _case(name="fit_fp32", kind="fit", prec="fp32", ny=256, nx=256, nz=40, f=2, kv=200, alpha=20.0, rings=2, planes=4,
              sy=32, sx=32, step=2.0, defocus=25.0, cs=5.0e5),
        # 4D cube on a pixelated detector: 128 x 128 k-pixels, 64 x 64 probes, 32 sites
        _case(name="cube_256", kind="cube", ny=256, nx=256, nz=20, f=2, alpha=20.0, planes=2, nch=1, sy=64, sx=64, box=128),
        # momentum-resolved line in FP32: the detector unsubsampled along q_x
        _case(name="qeels_fp32", kind="qeels", prec="fp32", ny=256, nx=256, nz=20, f=2, kv=200, alpha=20.0, rings=3,
              cells=2, planes=4, sy=32, sx=32, step=2.0),
    ]


# --------------------------------------------------------------------------
# drawn cases

# most work a drawn case may have, of the tensor-core and of the FP32 paths (a
# little under the largest listed ones'), in real operations of the contractions
MOST = {"mixed": 8e13, "fp8": 8e13, "split_bf16": 3e13, "fp32": 8e12}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["map", "eval", "eval", "eval", "sites", "fit", "cube", "qeels"])
        prec = rng.choice(["mixed", "mixed", "fp32", "split_bf16", "fp8"])
        if kind in ("cube", "qeels", "fit") and prec == "fp8":
            prec = "mixed"
        if kind in ("cube", "qeels", "fit"):
            n, f = rng.choice([(128, 2), (192, 3), (256, 2), (256, 4)])
        else:
            n, f = rng.choice([(128, 2), (192, 3), (256, 2), (256, 4), (384, 3), (512, 4), (768, 3), (1024, 4)])
        nx = n if rng.random() < 0.7 or n < 256 else rng.choice([n // 2, n])
        if nx // f < 64:
            nx = n
        nz = _log(rng, 5, 100 if n <= 512 else 30)
        c = _case(
            kind=kind, prec=prec, ny=n, nx=nx, nz=nz, f=f, kv=rng.choice([200, 300]),
            alpha=rng.choice([15.0, 20.0, 25.0]), theta=rng.choice([30.0, 40.0]),
            defocus=rng.choice([0.0, 0.0, rng.uniform(10.0, 60.0)]), rings=rng.choice([2, 3, 4]),
            recon="complex" if rng.random() < 0.15 else "magnitude", win=rng.choice([32, 48, 64, 64, 64]),
            cells=rng.choice([2, 2, 3, 4]), planes=min(nz, _log(rng, 1, 40)), nch=rng.choice([1, 3, 3, 4, 9]),
            raster=rng.random() < 0.75, sy=_log(rng, 3, 128), sx=_log(rng, 3, 128), step=rng.choice([1.0, 2.0]))
        c["cells"] = min(c["cells"], min(n, nx) // CELL_PX - 2)
        if kind in ("map", "eval") and c["win"] == 64 and rng.random() < 0.2:
            c["small_win"], c["small_nch"] = 32, 1
        if kind in ("cube", "qeels"):
            c["nz"], c["planes"] = min(nz, 20), min(c["planes"], 4)
        if kind == "cube":
            c["box"] = rng.choice([0, 64, 96])
        B, nd, P = _sizes(c)[:3]
        n_sites = c["cells"] ** 2 * c["planes"]
        columns = n * nx * c["nz"] * (2 * (1 + 3 * c["rings"] * (c["rings"] + 1)) + (nd if kind == "cube" else 0))
        if (work(c)["flops"] <= MOST[prec] * (0.25 if kind in ("fit", "qeels", "cube") else 1.0)
                and columns <= 512 * 512 * 12000 and n_sites * (P if kind != "cube" else 1) <= 3e7
                and (kind != "cube" or P * nd <= 7e7) and (kind != "qeels" or P <= 4096)
                and (kind != "fit" or (B <= 600 and n_sites <= 64))):
            return c


# --------------------------------------------------------------------------
# sizes

def _wavelength(kv):
    e = kv * 1e3
    return 12398.419843320026 / math.sqrt(e * (2 * 510998.95 + e))


def _disc(c, angle, fy, fx):
    """Beams (h_y, h_x) with |q| lambda <= angle and h = 0 mod f, in that order."""
    ly, lx = c["ny"] * PX, c["nx"] * PX
    hy, hx = np.meshgrid(np.arange(-c["ny"] // 2, c["ny"] // 2), np.arange(-c["nx"] // 2, c["nx"] // 2), indexing="ij")
    q = np.sqrt((hy / ly) ** 2 + (hx / lx) ** 2)
    keep = (q * _wavelength(c["kv"]) <= angle * 1e-3 * (1 + 1e-12)) & (hy % fy == 0) & (hx % fx == 0)
    return np.stack([hy[keep], hx[keep]], axis=1)


def _detector(c):
    if c["kind"] == "cube":
        if c["box"]:
            h = np.arange(-(c["box"] // 2), c["box"] - c["box"] // 2)
            return np.stack([g.ravel() for g in np.meshgrid(h, h, indexing="ij")], axis=1)
        return _disc(c, c["theta"], 1, 1)
    return _disc(c, c["theta"], c["f"], 1 if c["kind"] == "qeels" else c["f"])


def _sizes(c):
    """Aperture beams, output beams, scans, (channels, window) of each site."""
    n = c["cells"] ** 2 * c["planes"]
    per = [(c["small_nch"], c["small_win"]) if c["small_win"] and k % 2 else (c["nch"], c["win"]) for k in range(n)]
    return len(_disc(c, c["alpha"], c["f"], c["f"])), len(_detector(c)), c["sy"] * c["sx"], per


def work(case):
    """One pass: the contractions (coupling; then over the scans by the Gram
    matrix or directly, whichever is less), the sweeps' transforms; the
    potential, H and scans read, the outputs written."""
    c = case
    B, nd, P, per = _sizes(c)
    flops = 0.0
    for nch, w in per:
        flops += 8.0 * nd * nch * B * w * w
        gram = 8.0 * B * B * nch * nd + 8.0 * B * B / 2 * min(P, 4 * B)
        flops += 8.0 * nch * nd * B * P if c["kind"] in ("cube", "qeels") and P < 64 else \
            8.0 * nch * nd * B * 64 if c["kind"] in ("cube", "qeels") else min(gram, 8.0 * nch * nd * B * P)
    parents = 1 + 3 * c["rings"] * (c["rings"] + 1)
    cols = {"map": 0, "qeels": 0, "cube": parents + nd}.get(c["kind"], 2 * parents)
    G = c["ny"] * c["nx"]
    sweep = cols * c["nz"] * G * (10.0 * math.log2(G) + 14.0)
    V = 0 if c["kind"] in ("map", "qeels") else 4.0 * G * c["nz"]
    H = sum(8.0 * nch * w * w for nch, w in per)
    out = {"sites": 4.0 * len(per) * P, "cube": 4.0 * P * nd, "qeels": 4.0 * P * 64}.get(c["kind"], 8.0 * P)
    if c["kind"] == "fit":
        flops, sweep, out = 3 * flops, 3 * sweep, out + V + H
    return {"bytes": V + H + 16.0 * P + out, "flops": flops + sweep}


# --------------------------------------------------------------------------
# inputs

def _inputs(c, seed):
    """Atoms, channels, V, H, scans, and what a fit also has, on the GPU where the calls want it."""
    dev = torch.device("cuda")
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 20260757])
    ny, nx, nz = c["ny"], c["nx"], c["nz"]
    cy, cx = ny // CELL_PX, nx // CELL_PX
    grid = np.stack(np.meshgrid(np.arange(nz), np.arange(cy), np.arange(cx), indexing="ij"), -1).reshape(-1, 3)
    yx = (grid[:, 1:] + 0.5) * CELL + rng.uniform(-0.05, 0.05, (len(grid), 2))
    atoms = np.concatenate([yx, grid[:, :1]], axis=1).astype(np.float64)

    # potential: one separable Gaussian per atom (30 V A peak, sigma 0.3 A), periodic
    def axis(pos, n):
        d = torch.arange(n, device=dev, dtype=torch.float64) * PX - torch.as_tensor(pos, device=dev)[..., None]
        d = d - n * PX * torch.round(d / (n * PX))
        return torch.exp(-d * d / (2 * 0.3 ** 2))
    gy = axis(yx[:, 0].reshape(nz, -1), ny)
    gx = axis(yx[:, 1].reshape(nz, -1), nx)
    V = (30.0 * torch.bmm(gy.transpose(1, 2), gx)).float()
    del gy, gx

    # ionized sites: a central square of columns, on evenly spaced slices
    a, b, k = (cy - c["cells"]) // 2, (cx - c["cells"]) // 2, c["cells"]
    on = np.unique((np.arange(c["planes"]) * nz) // c["planes"] + (nz // c["planes"]) // 2)
    ion = np.isin(grid[:, 0], on) & (grid[:, 1] >= a) & (grid[:, 1] < a + k) & (grid[:, 2] >= b) & (grid[:, 2] < b + k)
    per = _sizes(c)[3]
    nch = np.zeros(len(atoms), dtype=np.int32)
    nch[ion] = [p[0] for p in per]

    # transition potentials of channels m around 0 on each site's window
    ids = np.nonzero(ion)[0]
    amp = rng.normal(size=(len(ids), max(p[0] for p in per), 2)) * 0.3 + [1.0, 0.0]
    H = []
    for n_s, w in sorted(set(per)):
        at = [i for i, p in enumerate(per) if p == (n_s, w)]
        t = torch.as_tensor(yx[ids[at]], device=dev)
        off = torch.floor(t / PX + 0.5) - w // 2
        u = torch.arange(w, device=dev, dtype=torch.float64)
        dy = ((off[:, :1] + u) * PX - t[:, :1])[:, :, None]
        dx = ((off[:, 1:] + u) * PX - t[:, 1:])[:, None, :]
        env = torch.exp(-(dy ** 2 + dx ** 2) / (2 * 0.5 ** 2))
        z = torch.as_tensor(amp[at], device=dev)
        parts = []
        for j in range(n_s):
            m = j - n_s // 2
            phi = env * (torch.complex(dx + 0 * dy, m * dy + 0 * dx) / 0.5) ** abs(m)
            parts.append(phi * torch.complex(z[:, j, 0], z[:, j, 1])[:, None, None])
        H += list(zip(at, torch.stack(parts, 1).to(torch.complex64)))
    H.sort(key=lambda v: v[0])
    if c["small_win"]:
        H = torch.cat([h.reshape(-1) for _, h in H])
    else:
        H = torch.cat([h for _, h in H])

    mid = np.array([(a + k / 2) * CELL_PX, (b + k / 2) * CELL_PX])
    if c["raster"]:
        ys = mid[0] + (np.arange(c["sy"]) - c["sy"] / 2) * c["step"]
        xs = mid[1] + (np.arange(c["sx"]) - c["sx"] / 2) * c["step"]
        scans = np.stack(np.meshgrid(ys, xs, indexing="ij"), -1).reshape(-1, 2)
    else:
        scans = mid + rng.uniform(-0.5, 0.5, (c["sy"] * c["sx"], 2)) * (k * CELL_PX)
    s = SimpleNamespace(atoms=atoms, nch=nch, V=V, H=H, scans=np.ascontiguousarray(scans), per=per, ids=ids)
    if c["kind"] == "fit":
        s.target = torch.as_tensor(0.02 * c["planes"] * rng.uniform(0.5, 1.5, len(scans)), device=dev)
        s.occ = torch.as_tensor(rng.uniform(0.8, 1.0, len(ids)), device=dev).float()
    return s


def _config(c):
    return SimpleNamespace(
        ny=c["ny"], nx=c["nx"], ly=c["ny"] * PX, lx=c["nx"] * PX, nz=c["nz"], dz=SLICE, e0=c["kv"] * 1e3,
        alpha=c["alpha"] * 1e-3, theta_det=c["theta"] * 1e-3, defocus=c["defocus"], cs=c["cs"], fy=c["f"], fx=c["f"],
        dfy=0, dfx=1 if c["kind"] == "qeels" else 0, cube_ky=c["box"], cube_kx=c["box"], nrad1=c["rings"], nang1=6,
        nrad2=c["rings"], nang2=6, win=c["win"], recon=c["recon"], prec=c["prec"])


def prepare(case, seed):
    s = _inputs(case, seed)
    s.kind = case["kind"]
    s.bip = BipContext(_config(case))
    if s.kind in ("map", "qeels"):
        s.bip.build(s.V, s.atoms, s.nch)
    s.small = [w for _, w in s.per] if case["small_win"] else None
    if s.small and s.kind == "map":
        s.bip.set_site_windows(s.small)
    if s.kind == "fit":
        s.V.requires_grad_(True)
        s.H.requires_grad_(True)
        s.occ.requires_grad_(True)
    return s


def run(state):
    s = state
    if s.kind == "map":
        return s.bip.map(s.H, s.scans).float()
    if s.kind == "eval":
        s.bip.build(s.V, s.atoms, s.nch)
        if s.small:
            s.bip.set_site_windows(s.small)
        return s.bip.map(s.H, s.scans).float()
    if s.kind == "sites":
        s.bip.build(s.V, s.atoms, s.nch)
        return s.bip.sites(s.H, s.scans)
    if s.kind == "fit":
        m = coreloss_map(s.bip, s.H, s.scans, occ=s.occ, V=s.V, atoms=s.atoms, nch=s.nch)
        dV, dH, docc = torch.autograd.grad(((m - s.target) ** 2).sum(), [s.V, s.H, s.occ])
        return {"map": m.detach().float(), "V": dV, "H": dH, "occ": docc}
    if s.kind == "cube":
        s.bip.build_s1(s.V, s.atoms, s.nch)
        return s.bip.cube(s.V, s.H, s.scans)
    return s.bip.qeels(s.H, s.scans, 1)[1]


# --------------------------------------------------------------------------
# the same in 64 bits

def _parents(h, c):
    """Hex rings of beams: the centre and 6 (1 + i) targets on ring i, each snapped to its nearest beam."""
    q = h / np.array([c["ny"] * PX, c["nx"] * PX])
    R, rings = np.sqrt((q ** 2).sum(1).max()), c["rings"]
    want = [(0.0, 0.0)]
    for i in range(rings):
        want += [(R * (i + 1) / rings * math.sin(t), R * (i + 1) / rings * math.cos(t))
                 for t in 2 * math.pi * np.arange(6 * (1 + i)) / (6 * (1 + i))]
    got = []
    for p in want:
        d = ((q - p) ** 2).sum(1)
        j = int(np.nonzero(d <= d.min() * (1 + 1e-9))[0][0])          # ties: the first in beam order
        if j not in got:
            got.append(j)
    return h[got]


def _half(poly, n, d):
    """The part of a convex polygon with n.x <= d."""
    f = poly @ n - d
    out = []
    for i in range(len(poly)):
        j = (i + 1) % len(poly)
        if f[i] <= 0:
            out.append(poly[i])
        if f[i] * f[j] < 0:
            out.append(poly[i] + f[i] / (f[i] - f[j]) * (poly[j] - poly[i]))
    return np.array(out).reshape(-1, 2)


def _area(p):
    return 0.0 if len(p) < 3 else 0.5 * abs(np.dot(p[:, 1], np.roll(p[:, 0], -1)) - np.dot(p[:, 0], np.roll(p[:, 1], -1)))


def _weights(hp, h, c):
    """Natural-neighbour weights [len(h), len(hp)]; on and outside the hull the linear weights of its nearest edge."""
    L = np.array([c["ny"] * PX, c["nx"] * PX])
    W = np.zeros((len(h), len(hp)))

    def cross(o, a, b):
        return int((a[0] - o[0]) * (b[1] - o[1]) - (a[1] - o[1]) * (b[0] - o[0]))
    pts = sorted(range(len(hp)), key=lambda i: (hp[i, 0], hp[i, 1]))
    hull = []
    for seq in (pts, pts[::-1]):                                      # points on an edge are kept
        part = []
        for i in seq:
            while len(part) >= 2 and cross(hp[part[-2]], hp[part[-1]], hp[i]) < 0:
                part.pop()
            part.append(i)
        hull += part[:-1]
    at = {tuple(p): i for i, p in enumerate(hp)}
    for t, ht in enumerate(h):
        if tuple(ht) in at:
            W[t, at[tuple(ht)]] = 1.0
            continue
        x = ht / L
        edges = list(zip(hull, hull[1:] + hull[:1]))
        if min(cross(hp[i], hp[j], ht) for i, j in edges) <= 0:
            best = None
            for i, j in edges:
                p, e = hp[i] / L, hp[j] / L - hp[i] / L
                s = float(np.clip(np.dot(x - p, e) / np.dot(e, e), 0, 1))
                d = ((x - p - s * e) ** 2).sum()
                if best is None or d < best[0] - 1e-300:
                    best = (d, i, j, s)
            W[t, best[1]] += 1 - best[3]
            W[t, best[2]] += best[3]
            continue
        r = hp / L - x
        r2 = (r ** 2).sum(1)
        order = np.argsort(r2, kind="stable")
        box = 64 * math.sqrt(r2.max())
        cell = box * np.array([[-1.0, -1.0], [-1.0, 1.0], [1.0, 1.0], [1.0, -1.0]])
        for p in order:
            if (cell @ (2 * r[p])).max() > r2[p]:
                cell = _half(cell, 2 * r[p], r2[p])
        reach = np.sqrt((cell ** 2).sum(1).max())
        near = [p for p in order if math.sqrt(r2[p]) <= 2 * reach + math.sqrt(r2[order[0]])]
        for p in near:
            piece = cell
            for j in near:
                if j != p and len(piece) and (piece @ (2 * (r[j] - r[p]))).max() > r2[j] - r2[p]:
                    piece = _half(piece, 2 * (r[j] - r[p]), r2[j] - r2[p])
            W[t, p] = _area(piece) / _area(cell)
    return W


def _sweep(c, V, h, planes, forward):
    """De-tilted columns on the ionized slices: plane waves of the beams h taken
    forward (transmit, propagate) or back from the exit by the transpose."""
    dev = V.device
    ny, nx = c["ny"], c["nx"]
    lam, e = _wavelength(c["kv"]), c["kv"] * 1e3
    sigma = 2 * math.pi / (lam * e) * (510998.95 + e) / (2 * 510998.95 + e)
    fy, fx = (torch.fft.fftfreq(n, 1.0 / n, device=dev, dtype=torch.float64) for n in (ny, nx))
    sign = 1.0 if forward else -1.0
    h = torch.as_tensor(h, device=dev, dtype=torch.float64) * sign

    def phase(n, l, freq, hk):                                        # propagator at the beam's shifted frequencies
        k = torch.remainder(freq[None] + hk[:, None] + n // 2, n) - n // 2
        return torch.polar(torch.ones_like(k), -math.pi * lam * SLICE * (k / l) ** 2)
    Py, Px = phase(ny, ny * PX, fy, h[:, 0])[:, :, None], phase(nx, nx * PX, fx, h[:, 1])[:, None, :]
    x = torch.full((len(h), ny, nx), 1.0 if forward else 1.0 / math.sqrt(ny * nx), dtype=torch.complex128, device=dev)

    def step(x):
        return torch.fft.ifft2(torch.fft.fft2(x) * Py * Px)

    def T(j):
        v = sigma * V[j]
        return torch.complex(torch.cos(v), torch.sin(v))
    out = {}
    if forward:
        for j in range(max(planes) + 1):
            if j in planes:
                out[j] = x
            x = step(x * T(j))
    else:
        for j in range(c["nz"] - 1, min(planes) - 1, -1):
            x = step(x) * T(j)
            if j in planes:
                out[j] = x
    return out


def exact(case, seed):
    c = case
    B, nd, P, per = _sizes(c)
    K = c["win"] ** 2
    cost = sum(8.0 * nd * n * B * w * w for n, w in per) * (4 if c["kind"] == "fit" else 1)
    scan_cost = len(per) * 8.0 * B * (nd * max(p[0] for p in per) if c["kind"] in ("cube", "qeels") else B) * P
    if cost + scan_cost > 1.3e13:
        return None                                                   # over about 20 s in 64 bits
    s = _inputs(c, seed)
    dev = s.V.device
    ny, nx, f = c["ny"], c["nx"], c["f"]
    h1, h2 = _disc(c, c["alpha"], f, f), _detector(c)
    p1 = _parents(h1, c)
    W1 = torch.as_tensor(_weights(p1, h1, c), device=dev)
    if c["kind"] == "cube":
        p2, W2 = None, None
    else:
        p2 = _parents(h2, c)
        W2 = torch.as_tensor(_weights(p2, h2, c), device=dev)

    lam = _wavelength(c["kv"])

    def psi(h):
        q2 = (h[:, 0] / (ny * PX)) ** 2 + (h[:, 1] / (nx * PX)) ** 2
        return np.exp(-1j * (math.pi * lam * c["defocus"] * q2 + 0.5 * math.pi * c["cs"] * lam ** 3 * q2 ** 2))
    norm = math.sqrt(ny * nx * len(_disc(c, c["alpha"], 1, 1)))
    turn = np.outer(h1[:, 0], s.scans[:, 0]) / ny + np.outer(h1[:, 1], s.scans[:, 1]) / nx
    C = torch.as_tensor((f * f * psi(h1) / norm)[:, None] * np.exp(-2j * np.pi * turn), device=dev)
    tau = s.atoms[s.ids, :2] / PX
    plane = s.atoms[s.ids, 2].astype(int)

    def crop(k):
        d = s.scans - tau[k]
        n = np.array([ny, nx])
        d = d - n * np.floor((d + 0.5 * n) / n)
        return torch.as_tensor(((d >= -0.5 * n / f) & (d < 0.5 * n / f)).all(1).astype(np.float64), device=dev)

    def window(x, k, w):
        o = [int(math.floor(t + 0.5)) - w // 2 for t in tau[k]]
        iy, ix = (torch.as_tensor((o[i] + np.arange(w)) % n, device=dev) for i, n in enumerate((ny, nx)))
        return x[:, iy[:, None], ix[None, :]].reshape(x.shape[0], -1), iy, ix

    def tilt(h, iy, ix, sign):
        h = torch.as_tensor(h, device=dev)
        t = (h[:, :1] * iy % ny / ny)[:, :, None] + (h[:, 1:] * ix % nx / nx)[:, None, :]
        t = t.reshape(len(h), -1) * (2 * math.pi * sign)
        return torch.complex(torch.cos(t), torch.sin(t))

    def rebuilt(x, W, h, k, w, sign):
        d, iy, ix = window(x, k, w)
        U = W.to(torch.complex128) @ d
        if c["recon"] == "magnitude":
            U = (W @ d.abs()) * U / U.abs()
        return U * tilt(h, iy, ix, sign)

    def chunks():
        o = 0
        for n, w in per:
            yield o, n, w
            o += n * w * w

    def site(k, H, x1, x2, o, n, w):
        """I_tau on every scan of site k from its planes' columns."""
        A = rebuilt(x1, W1, h1, k, w, 1.0)
        D = rebuilt(x2, W2, h2, k, w, -1.0)
        M = [D @ (H[o + j * w * w:o + (j + 1) * w * w] * A).T for j in range(n)]
        Q = sum(m.conj().T @ m for m in M)
        return f * f * (C.conj() * (Q @ C)).sum(0).real * crop(k)

    H = s.H.to(torch.complex128).reshape(-1)
    V = s.V.double()
    planes = sorted(set(plane.tolist()))
    if c["kind"] == "cube":
        x1 = _sweep(c, V, p1, planes, True)
        out = torch.zeros(P, nd, dtype=torch.float64, device=dev)
        most = max(1, int(4e9 / (16 * ny * nx)))
        for a in range(0, nd, most):
            hq = h2[a:a + most]
            x2 = _sweep(c, V, hq, planes, False)
            for k, (o, n, w) in enumerate(chunks()):
                A = rebuilt(x1[plane[k]], W1, h1, k, w, 1.0)
                d, iy, ix = window(x2[plane[k]], k, w)
                D = d * tilt(hq, iy, ix, -1.0)
                m = crop(k)
                for j in range(n):
                    v = (D @ (H[o + j * w * w:o + (j + 1) * w * w] * A).T) @ C
                    out[:, a:a + most] += ((v.real ** 2 + v.imag ** 2) * m).T
        return out
    if c["kind"] == "fit":
        # gradients site by site, so that only one site's windows live at a time
        V.requires_grad_(True)
        x1, x2 = _sweep(c, V, p1, planes, True), _sweep(c, V, p2, planes, False)
        leaf1 = {j: x.detach().requires_grad_(True) for j, x in x1.items()}
        leaf2 = {j: x.detach().requires_grad_(True) for j, x in x2.items()}
        H.requires_grad_(True)
        occ = s.occ.double()
        parts = []
        with torch.no_grad():
            for k, (o, n, w) in enumerate(chunks()):
                parts.append(site(k, H, leaf1[plane[k]], leaf2[plane[k]], o, n, w))
        m = sum(v * occ[k] for k, v in enumerate(parts))
        g = 2 * (m - s.target)
        docc = torch.stack([(g * v).sum() for v in parts])
        for k, (o, n, w) in enumerate(chunks()):
            (g * occ[k] * site(k, H, leaf1[plane[k]], leaf2[plane[k]], o, n, w)).sum().backward()
        torch.autograd.backward([x1[j] for j in planes] + [x2[j] for j in planes],
                                [leaf1[j].grad for j in planes] + [leaf2[j].grad for j in planes])
        return {"map": m.detach(), "V": V.grad, "H": H.grad.reshape(s.H.shape), "occ": docc}
    x1, x2 = _sweep(c, V, p1, planes, True), _sweep(c, V, p2, planes, False)
    if c["kind"] == "qeels":
        bins = np.unique(h2[:, 1])
        at = torch.as_tensor(np.searchsorted(bins, h2[:, 1]), device=dev)
        out = torch.zeros(len(bins), P, dtype=torch.float64, device=dev)
        for k, (o, n, w) in enumerate(chunks()):
            A = rebuilt(x1[plane[k]], W1, h1, k, w, 1.0)
            D = rebuilt(x2[plane[k]], W2, h2, k, w, -1.0)
            m = crop(k) * f
            for j in range(n):
                v = (D @ (H[o + j * w * w:o + (j + 1) * w * w] * A).T) @ C
                out.index_add_(0, at, (v.real ** 2 + v.imag ** 2) * m)
        return out.T.contiguous()
    parts = (site(k, H, x1[plane[k]], x2[plane[k]], o, n, w) for k, (o, n, w) in enumerate(chunks()))
    if c["kind"] == "sites":
        return torch.stack(list(parts))
    return sum(parts)
