"""Performance cases of the RSP signature and indexing library.

A case is one call (or the two or three calls a program makes together) of the
public Python binding at one size.  The kinds of case, and what each stands for:

  signature  aptidx_compute_signatures on loaded positions and placed ROIs: the
             step every analysis spends most of its time in, on the tensor-core
             path (tiny, single crystal, wide band, large ROIs, 2^11 bins) and on
             the FP32 path
  ingest     a new reconstruction on the device: positions and types loaded,
             ROIs of uneven radii and bands placed, signatures computed
  match      Eq. 3 against a 5-degree orientation set, best orientation per ROI
  topk       Eq. 3 keeping the 1000 best of a dense orientation set
  setup      one more crystal-structure candidate: reference, look-up table, and
             the match of a few ROIs against it
  refine     20 Gauss-Newton steps per ROI from the matched orientations
  refgrad    the differentiable refinement loss, forward and backward
  fsp        reciprocal-space signatures (Eq. 2) on an L^3 grid

Inputs are synthetic: rotated cubic lattices with missing atoms and Gaussian
displacements, signatures with bright poles on a noise floor.
"""
import functools
import math

import numpy as np
import torch

import paper_2009_00735_gb300 as apt
from paper_2009_00735_gb300 import refine as apt_refine

TC = apt.APTIDX_PATH_TC_FP16
PLAIN = apt.APTIDX_PATH_PLAIN_FP32
DEV = "cuda"
LAT = {"bcc": (0.287, [[0, 0, 0], [.5, .5, .5]], 0.287 / math.sqrt(2.0)),
       "fcc": (0.405, [[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]], 0.405 / 2)}


def listed():
    return [
        # the smallest call in use: 16 ROIs of 1 nm, 10242 directions, 2^8 bins (launches and latency)
        dict(name="sig_tiny", kind="signature", path="tc", lattice="fcc", eta=0.5, sigma=0.03, nroi=16, R=1.0,
             m=8, dirs="ico5", band="peak", normalise=True),
        # the benchmark's single crystal: 8192 ROIs of 2 nm, 40962 directions, 2^10 bins, {110} band
        dict(name="sig_crystal", kind="signature", path="tc", lattice="bcc", eta=0.4, sigma=0.04, nroi=8192, R=2.0,
             m=10, dirs="ico6", band="peak", normalise=True),
        # the whole spectrum searched (k = 8..128) instead of one plane family
        dict(name="sig_wide", kind="signature", path="tc", lattice="bcc", eta=0.4, sigma=0.04, nroi=512, R=2.0,
             m=10, dirs="ico6", band="wide", normalise=False),
        # few large ROIs (9000 atoms each) on a direction set without antipodes, an odd number of directions
        dict(name="sig_large", kind="signature", path="tc", lattice="bcc", eta=0.4, sigma=0.04, nroi=61, R=4.0,
             m=11, dirs="spiral20011", band="peak", normalise=False),
        # the FP32 path, which results of the tensor-core path are checked against
        dict(name="sig_fp32", kind="signature", path="plain", lattice="bcc", eta=0.4, sigma=0.04, nroi=512, R=2.0,
             m=10, dirs="ico6", band="peak", normalise=False),
        # a polycrystal read in and analysed: uneven ROIs (R = 1 to 2.5 nm) with their own bands
        dict(name="ingest_poly", kind="ingest", nroi=2000, grains=12, box=26.0, m=10, dirs="ico6"),
        # matching after the single-crystal step, the 3419 orientations of the 5-degree set
        dict(name="match_5deg", kind="match", nroi=4096, ng=3419, n_hat=1000, dirs="ico6"),
        # the 1000 best solutions of a dense orientation set
        dict(name="topk_dense", kind="topk", nroi=192, ng=50000, n_hat=1000, topk=1000, dirs="ico6"),
        # a further candidate structure prepared and tried on a few ROIs
        dict(name="setup_cand", kind="setup", nroi=64, ng=3419, n_hat=1000, dirs="ico6"),
        # refinement after matching
        dict(name="refine_gn", kind="refine", nroi=2048, iters=20, dirs="ico6"),
        # the loss and its gradient inside an optimiser, on a coarser sphere
        dict(name="refine_grad", kind="refgrad", nroi=1000, dirs="ico5"),
        # the reciprocal-space method on the 64^3 grid
        dict(name="fsp_64", kind="fsp", lattice="bcc", eta=0.4, sigma=0.04, nroi=512, R=2.0, L=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_dirs(rng, most=6):
    if rng.random() < 0.6:
        return "ico%d" % rng.randint(4, most)
    return "spiral%d" % _log(rng, 1000, 40000 if most > 5 else 10000)


def draw(rng):
    kind = rng.choice(["signature", "signature", "signature", "signature", "ingest", "match", "topk", "setup",
                       "refine", "refgrad", "fsp"])
    if kind == "signature":
        lat = rng.choice(["bcc", "fcc"])
        path = rng.choice(["tc", "tc", "tc", "plain"])
        wide = rng.random() < 0.25
        R = round(rng.uniform(1.0, 4.5), 3)
        c = dict(kind=kind, path=path, lattice=lat, eta=round(rng.uniform(0.3, 0.8), 3),
                 sigma=round(rng.uniform(0.01, 0.06), 3), R=R, m=rng.choice([8, 9, 10, 10, 10, 11, 12]),
                 dirs=_draw_dirs(rng), band="wide" if wide else "peak", normalise=rng.random() < 0.5)
        if wide and c["m"] < 10:
            c["m"] = 10
        most = 1.5e10 if wide else 1e11
        if path == "plain":
            most = 2e9 if wide else 1e10
        nv = _ndirs(c["dirs"])
        top = max(17, min(8192, int(most / (nv * _atoms(c)))))
        c["nroi"] = _log(rng, 16, top)
        return c
    if kind == "ingest":
        return dict(kind=kind, nroi=_log(rng, 100, 2000), grains=rng.randint(4, 20), box=round(rng.uniform(12, 26), 2),
                    m=rng.choice([9, 10]), dirs=_draw_dirs(rng))
    if kind in ("match", "topk"):
        ng = _log(rng, 500, 4000) if kind == "match" else _log(rng, 2000, 50000)
        c = dict(kind=kind, ng=ng, n_hat=_log(rng, 50, 1000), dirs=_draw_dirs(rng))
        c["nroi"] = _log(rng, 64, max(65, min(4096, int(1e10 / (ng * c["n_hat"])))))
        if kind == "topk":
            c["topk"] = min(ng, _log(rng, 2, 1000))
        return c
    if kind == "setup":
        return dict(kind=kind, nroi=rng.randint(16, 128), ng=_log(rng, 500, 4000), n_hat=_log(rng, 100, 1000),
                    dirs=_draw_dirs(rng))
    if kind == "refine":
        return dict(kind=kind, nroi=_log(rng, 64, 2048), iters=rng.randint(3, 20), dirs=_draw_dirs(rng))
    if kind == "refgrad":
        return dict(kind=kind, nroi=_log(rng, 64, 4000), dirs=_draw_dirs(rng, 5))
    L = rng.choice([64, 64, 128])
    return dict(kind=kind, lattice=rng.choice(["bcc", "fcc"]), eta=round(rng.uniform(0.3, 0.6), 3),
                sigma=round(rng.uniform(0.01, 0.05), 3), nroi=_log(rng, 16, 512) if L == 64 else _log(rng, 8, 64),
                R=round(rng.uniform(1.0, 2.4), 3), L=L)


# ---- inputs ------------------------------------------------------------------------

def _ndirs(name):
    return 10 * 4 ** int(name[3:]) + 2 if name.startswith("ico") else int(name[6:])


@functools.lru_cache(maxsize=8)
def _dirs_np(name):
    """Unit vectors: a geodesic sphere ("icoL", closed under negation) or a
    golden-angle spiral of any number of directions ("spiralN")."""
    if name.startswith("spiral"):
        n = int(name[6:])
        i = np.arange(n) + 0.5
        z = 1.0 - 2.0 * i / n
        r, a = np.sqrt(1.0 - z * z), i * (math.pi * (3.0 - math.sqrt(5.0)))
        return np.stack([r * np.cos(a), r * np.sin(a), z], 1).astype(np.float32)
    t = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([(s * a, u * b, 0.0) for s in (1, -1) for u in (1, -1) for a, b in [(1.0, t)]])
    v = np.concatenate([v, np.roll(v, 1, 1), np.roll(v, 2, 1)])
    d = ((v[:, None] - v[None]) ** 2).sum(-1)
    edge = np.abs(d - 4.0) < 1e-9
    f = np.array([(i, j, k) for i in range(12) for j in range(i) for k in range(j)
                  if edge[i, j] and edge[j, k] and edge[i, k]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    for _ in range(int(name[3:])):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        uniq, inv = np.unique(e, axis=0, return_inverse=True)
        mid = v[uniq[:, 0]] + v[uniq[:, 1]]
        mid /= np.linalg.norm(mid, axis=1, keepdims=True)
        a, b, c = inv.reshape(3, -1) + len(v)
        v = np.concatenate([v, mid])
        f = np.concatenate([np.stack(x, 1) for x in ((f[:, 0], a, c), (f[:, 1], b, a), (f[:, 2], c, b), (a, b, c))])
    return v.astype(np.float32)


def _dirs(name):
    return torch.from_numpy(_dirs_np(name)).to(DEV)


def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + salt)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _quats(g, n):
    q = torch.randn(n, 4, generator=g, device=DEV, dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True)
    return q * torch.where(q[:, :1] < 0, -1.0, 1.0)


def _rot(q):
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(*q.shape[:-1], 3, 3)


def _crystal(g, lattice, rot, hi, eta, sigma):
    """Sites of a rotated lattice in the box [0, hi), a fraction eta kept, displaced."""
    a, basis, _ = LAT[lattice]
    hi = torch.tensor(hi, device=DEV, dtype=torch.float64)
    c = torch.tensor([[x, y, z] for x in (0, 1) for y in (0, 1) for z in (0, 1)], device=DEV, dtype=torch.float64) * hi
    n = (c - hi / 2) @ rot / a
    ax = [torch.arange(int(n[:, d].min()) - 1, int(n[:, d].max()) + 2, device=DEV, dtype=torch.float64) for d in range(3)]
    cells = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)
    out = []
    for b in basis:
        p = (cells + torch.tensor(b, device=DEV, dtype=torch.float64)) @ rot.T * a + hi / 2
        p = p[((p >= 0) & (p < hi)).all(1)]
        out.append(p[_rand(g, len(p)) < eta])
    p = torch.cat(out)
    return p + sigma * torch.randn(p.shape, generator=g, device=DEV, dtype=torch.float64)


def _atoms(c):
    """Mean atoms of a ROI."""
    a, basis, _ = LAT[c["lattice"]]
    return len(basis) / a ** 3 * c["eta"] * 4.0 / 3.0 * math.pi * c["R"] ** 3


def _band(c):
    if c["band"] == "wide":
        return 8, 128
    d = LAT[c["lattice"]][2]
    return _peak_band(d, c["R"], c["m"])


def _peak_band(d, R, m):
    """Frequency bins of plane spacings d -/+ 10 %: k = W / d over the histogram span W."""
    W = 2.0 * (R + R / ((1 << (m - 1)) - 1))
    lo, hi = math.ceil(W / (1.1 * d)), math.floor(W / (0.9 * d))
    return lo, max(hi, lo)


def _roi_box(c):
    """ROI centres on a 1 nm grid and the box that holds them."""
    n = int(math.ceil(c["nroi"] ** (1.0 / 3.0) - 1e-9))
    idx = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)[:c["nroi"]]
    off = c["R"] + 0.5
    hi = [idx[:, d].max() + 2 * off + 0.37 for d in range(3)]
    return np.ascontiguousarray(idx + off), hi


def _poly(c, seed):
    """Poisson-Voronoi grains of f.c.c. Al with 5 % minority atoms (type 1)."""
    g = _gen(seed, 3)
    hi = [c["box"], c["box"], 2 * c["box"]]
    h = torch.tensor(hi, device=DEV, dtype=torch.float64)
    nuclei = _rand(g, c["grains"], 3) * h
    rot = _rot(_quats(g, c["grains"]))
    keep = []
    for i in range(c["grains"]):
        p = _crystal(g, "fcc", rot[i], hi, 0.5, 0.04)
        near = torch.cdist(p, nuclei, compute_mode="donot_use_mm_for_euclid_dist").argmin(1)
        keep.append(p[near == i])
    p = torch.cat(keep).to(torch.float32).contiguous()
    types = (_rand(g, len(p)) < 0.05).to(torch.uint8)
    radii = 1.0 + 1.5 * _rand(g, c["nroi"])
    centres = radii[:, None] + _rand(g, c["nroi"], 3) * (h - 2 * radii[:, None])
    bands = np.array([_peak_band(0.2025, float(r), c["m"]) for r in radii.cpu()], np.int32)
    return p, types, centres.contiguous(), radii, torch.from_numpy(bands).to(DEV)


_CUBE = [[1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1]]


def _bumps(d, width):
    """Bright {100} poles of the given width (degrees) at the unit vectors d."""
    p = torch.tensor(_CUBE, device=DEV, dtype=torch.float64)
    out = torch.zeros(d.shape[:-1], device=DEV, dtype=torch.float64)
    for k in range(6):
        th = torch.arccos((d @ p[k]).clamp(-1.0, 1.0))
        out += torch.exp(-th ** 2 / (2 * math.radians(width) ** 2))
    return out


def _measured(g, name, q):
    """Normalised signatures of ROIs of orientations q: poles on a noise floor."""
    u = _dirs(name).double()
    S = torch.empty(len(q), len(u), device=DEV, dtype=torch.float32)
    for i in range(0, len(q), 256):
        d = u @ _rot(q[i:i + 256])                       # rows R^T u
        s = 0.75 * _bumps(d, 10.0) + 0.25 * torch.rand(d.shape[:-1], generator=g, device=DEV, dtype=torch.float32)
        S[i:i + 256] = (s / s.max(dim=1, keepdim=True).values).float()
    return S


def _reference(name):
    """Reference values on the directions and on the 1-degree elevation-azimuth image."""
    a, b = torch.meshgrid(torch.deg2rad(torch.arange(-90.0, 91.0, device=DEV, dtype=torch.float64)),
                          torch.deg2rad(torch.arange(0.0, 360.0, device=DEV, dtype=torch.float64)), indexing="ij")
    d = torch.stack([a.cos() * b.cos(), a.cos() * b.sin(), a.sin()], -1)
    node, img = _bumps(_dirs(name).double(), 10.0), _bumps(d, 10.0)
    return (node / node.max()).float(), (img / img.max()).float().contiguous()


def _near(g, q, deg):
    """Orientations about `deg` degrees off q (what matching hands to refinement)."""
    w = math.radians(deg) * torch.randn(len(q), 3, generator=g, device=DEV, dtype=torch.float64) / math.sqrt(3.0)
    th = w.norm(dim=1, keepdim=True)
    e = torch.cat([torch.cos(th / 2), torch.sin(th / 2) * w / th], 1)
    return _qmul(e, q)


def _qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _inputs(c, seed):
    """Everything a case is computed from."""
    g = _gen(seed, 1)
    k = c["kind"]
    if k in ("signature", "fsp"):
        centres, hi = _roi_box(c)
        p = _crystal(g, c["lattice"], _rot(_quats(g, 1))[0], hi, c["eta"], c["sigma"])
        return dict(xyz=p.float().contiguous(), centres=torch.from_numpy(centres).to(DEV),
                    radii=torch.full((c["nroi"],), c["R"], device=DEV, dtype=torch.float64))
    if k == "ingest":
        p, t, cen, rad, band = _poly(c, seed)
        return dict(xyz=p, types=t, centres=cen, radii=rad, lo=band[:, 0].contiguous(), hi=band[:, 1].contiguous())
    node, img = _reference(c["dirs"])
    q = _quats(g, c["nroi"])
    x = dict(node=node, img=img, S=_measured(g, c["dirs"], q))
    if k in ("match", "topk", "setup"):
        x["grid"] = _quats(g, c["ng"])
    elif k == "refine":
        x["q0"] = _near(g, q, 2.0)
    else:
        x["q0"] = _near(g, q, 2.0)
        x["omega"] = 0.01 * torch.randn(c["nroi"], 3, generator=g, device=DEV, dtype=torch.float64)
    return x


def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    k = c["kind"]
    ctx = apt.Context(torch.cuda.current_device())
    h = ctx.handle
    s = dict(case=c, ctx=ctx, **x)
    nroi = c["nroi"]
    if k in ("signature", "ingest", "fsp"):
        lo, hi = _band(c) if k == "signature" else (1, 4)
        if k != "ingest":
            apt.aptidx_load_positions(h, x["xyz"])
        apt.aptidx_set_directions(h, _dirs(c.get("dirs", "ico4")))
        apt.aptidx_set_binning(h, c.get("m", 10), lo, hi)
        if k != "ingest":
            apt.aptidx_set_rois(h, x["centres"], x["radii"])
        if k == "fsp":
            s["amp"] = torch.empty(nroi, c["L"], c["L"], c["L"], device=DEV)
        else:
            s["out"] = torch.empty(nroi, _ndirs(c["dirs"]), device=DEV)
            s["n"] = torch.empty(nroi, device=DEV, dtype=torch.int32)
        return s
    apt.aptidx_set_directions(h, _dirs(c["dirs"]))
    if k != "setup":
        apt.aptidx_set_reference(h, 0, x["node"], c.get("n_hat", 1), x["img"])
    if k in ("match", "topk"):
        apt.aptidx_build_lut(h, 0, x["grid"])
    width = (c["topk"],) if k == "topk" else ()
    s["best"] = torch.empty((nroi,) + width, device=DEV, dtype=torch.int32)
    s["score"] = torch.empty((nroi,) + width, device=DEV)
    s["q"] = torch.empty(nroi, 4, device=DEV, dtype=torch.float64)
    s["loss"] = torch.empty(nroi, device=DEV)
    return s


def run(state):
    s, c = state, state["case"]
    h, k = s["ctx"].handle, c["kind"]
    if k == "signature":
        apt.aptidx_compute_signatures(h, TC if c["path"] == "tc" else PLAIN,
                                      apt.APTIDX_NORMALISE_MAX if c["normalise"] else 0, s["out"], None, s["n"])
        return s["out"], s["n"]
    if k == "ingest":
        apt.aptidx_load_positions(h, s["xyz"], s["types"])
        apt.aptidx_set_rois(h, s["centres"], s["radii"], s["lo"], s["hi"], type_mask=0b11)
        apt.aptidx_compute_signatures(h, TC, apt.APTIDX_NORMALISE_MAX, s["out"], None, s["n"])
        return s["out"], s["n"]
    if k == "match":
        apt.aptidx_match(h, 0, s["S"], s["best"], s["score"])
        return s["best"], s["score"]
    if k == "topk":
        apt.aptidx_match_topk(h, 0, s["S"], c["topk"], s["best"], s["score"])
        return s["best"], s["score"]
    if k == "setup":
        apt.aptidx_set_reference(h, 0, s["node"], c["n_hat"], s["img"])
        apt.aptidx_build_lut(h, 0, s["grid"])
        apt.aptidx_match(h, 0, s["S"], s["best"], s["score"])
        return s["best"], s["score"]
    if k == "refine":
        apt.aptidx_refine(h, 0, s["S"], s["q0"], c["iters"], s["q"], s["loss"])
        return s["q"], s["loss"]
    if k == "refgrad":
        omega = s["omega"].clone().requires_grad_(True)
        loss = apt_refine.refine_loss(omega, s["S"], s["q0"], h, 0)
        loss.sum().backward()
        return loss.detach(), omega.grad
    apt.aptidx_compute_fsp(h, s["amp"])
    return s["amp"]


# ---- what a pass cannot do without ----------------------------------------------------

def work(case):
    c, k = case, case["kind"]
    nroi = c["nroi"]
    if k == "ingest":
        vol = 2.0 * c["box"] ** 3
        mean = 4 / 0.405 ** 3 * 0.5 * 4.0 / 3.0 * math.pi * 5.36     # mean of R^3 over [1, 2.5] nm cubed: 5.86
        nv = _ndirs(c["dirs"])
        return {"bytes": 13.0 * vol * 4 / 0.405 ** 3 * 0.5 + nroi * (48.0 + 4.0 * nv) + 12.0 * nv,
                "flops": nroi * nv * (8.0 * mean + 16.0 * (1 << c["m"]))}
    if k in ("signature", "fsp"):
        a, basis, _ = LAT[c["lattice"]]
        _, hi = _roi_box(c)
        n = hi[0] * hi[1] * hi[2] * len(basis) / a ** 3 * c["eta"]
        if k == "fsp":
            pts = nroi * float(c["L"]) ** 3
            return {"bytes": 12.0 * n + 36.0 * nroi + 4.0 * pts, "flops": 8.0 * pts * _atoms(c)}
        lo, hi_k = _band(c)
        nv = _ndirs(c["dirs"])
        return {"bytes": 12.0 * n + nroi * (36.0 + 4.0 * nv) + 12.0 * nv,
                "flops": nroi * nv * (8.0 * _atoms(c) + 4.0 * (hi_k - lo + 1) * (1 << c["m"]))}
    nv = _ndirs(c["dirs"])
    if k in ("match", "topk", "setup"):
        entries = float(c["ng"]) * c["n_hat"]
        b = nroi * (4.0 * nv + 8.0 * c.get("topk", 1)) + 32.0 * c["ng"]
        if k == "setup":
            return {"bytes": b + 16.0 * nv + 4.0 * 181 * 360, "flops": 15.0 * entries + 3.0 * entries * nroi}
        return {"bytes": b + 2.0 * entries, "flops": 3.0 * entries * nroi}
    passes = c["iters"] + 1 if k == "refine" else 1
    return {"bytes": nroi * (4.0 * nv + 100.0) + 12.0 * nv + 4.0 * 181 * 360, "flops": 100.0 * nroi * nv * passes}


# ---- the same results in 64 bits --------------------------------------------------------

def exact(case, seed):
    c, k = case, case["kind"]
    nv = _ndirs(c.get("dirs", "ico4"))
    if k in ("signature", "ingest"):
        atoms = 1400.0 if k == "ingest" else _atoms(c)
        if c["nroi"] * nv * (atoms + (1 << c["m"])) > 2.0e11:
            return None
        return _exact_signatures(c, _inputs(c, seed)), None
    if k == "fsp":
        if 8.0 * c["nroi"] * c["L"] ** 3 * _atoms(c) > 4e12:
            return None
        return _exact_fsp(c, _inputs(c, seed))
    if k in ("match", "topk", "setup"):
        if float(c["ng"]) * c["n_hat"] * (nv + 8 * c["nroi"]) > 5e11:
            return None
        return None, _exact_scores(c, _inputs(c, seed))
    return _exact_refine(c, _inputs(c, seed))


def _f32(x):
    return x.to(torch.float32).to(torch.float64)


def _exact_signatures(c, x):
    """Membership in FP64, the projection and binning rule (FP32 projections by
    definition, floor of the exact product), and the band's largest amplitude of
    an FP64 Fourier transform."""
    u = _dirs(c["dirs"]).double()
    NB, nv = 1 << c["m"], len(u)
    half = NB // 2
    xyz = x["xyz"].double()
    out = torch.empty(c["nroi"], nv, device=DEV, dtype=torch.float64)
    lohi = torch.stack([x["lo"], x["hi"]], 1).tolist() if "lo" in x else [_band(c)] * c["nroi"]
    rows = torch.arange(nv, device=DEV)[:, None] * NB
    for r in range(c["nroi"]):
        R = x["radii"][r]
        d = xyz - x["centres"][r]
        a = _f32(d[(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2] <= R * R])
        scale = _f32((half - 1) / R)
        H = torch.zeros(nv * NB, device=DEV, dtype=torch.int32)
        for j in range(0, len(a), 2048):
            b = a[j:j + 2048]
            s = _f32(u[:, :1] * b[:, 0])
            s = _f32(u[:, 1:2] * b[:, 1] + s)
            s = _f32(u[:, 2:3] * b[:, 2] + s)
            i = (torch.floor(s * scale).to(torch.int64) + half).clamp_(0, NB - 1) + rows
            H += torch.bincount(i.reshape(-1), minlength=nv * NB).to(torch.int32)
        lo, hi = lohi[r]
        out[r] = torch.fft.rfft(H.reshape(nv, NB).double(), dim=1)[:, lo:hi + 1].abs().amax(1)
    if c["kind"] == "ingest" or c["normalise"]:
        out /= out.amax(1, keepdim=True)
    return out


def _exact_fsp(c, x):
    L, km = c["L"], 2.0 * math.pi
    kk = -km + torch.arange(L, device=DEV, dtype=torch.float64) * (2.0 * km / (L - 1))
    xyz = x["xyz"].double()
    out = torch.empty(c["nroi"], L, L, L, device=DEV, dtype=torch.float64)
    for r in range(c["nroi"]):
        d = xyz - x["centres"][r]
        a = d[(d * d).sum(1) <= x["radii"][r] ** 2]
        e = [torch.exp(-2j * math.pi * kk[:, None] * a[:, i]) for i in range(3)]
        for i in range(0, L, 16):
            P = (e[0][i:i + 16, None] * e[1][None]).reshape(-1, len(a))
            out[r, i:i + 16] = (P @ e[2].T).abs().reshape(-1, L, L)
    return out


def _exact_scores(c, x):
    """Eq. 3 over the table of nearest directions (by the FP32 dot product of
    its definition, ties to the lowest index), smallest scores first."""
    u32 = _dirs(c["dirs"])
    u = u32.double()
    top = torch.sort(x["node"], descending=True, stable=True).indices[:c["n_hat"]]
    ref = x["node"][top].double()
    S = x["S"].double()
    keep = torch.full((c["nroi"], 0), math.inf, device=DEV, dtype=torch.float64)
    want = c.get("topk", 1)
    step = max(1, int(2e9 / (8 * c["n_hat"] * max(len(u), 1))))
    for g in range(0, c["ng"], step):
        r = _f32(torch.einsum("gij,kj->gki", _rot(x["grid"][g:g + step]), u[top])).reshape(-1, 3)
        D = r @ u.T
        q, p = torch.nonzero(D >= D.amax(1, keepdim=True) - 5e-7, as_tuple=True)
        d = _f32(u[p, 2] * r[q, 2] + _f32(u[p, 1] * r[q, 1] + _f32(u[p, 0] * r[q, 0])))
        m = torch.full((len(r),), -math.inf, device=DEV, dtype=torch.float64).scatter_reduce(0, q, d, "amax")
        best = torch.full((len(r),), len(u), device=DEV, dtype=torch.int64)
        best = best.scatter_reduce(0, q, torch.where(d == m[q], p, len(u)), "amin").reshape(-1, c["n_hat"])
        del D
        sc = torch.empty(c["nroi"], len(best), device=DEV, dtype=torch.float64)
        for i in range(c["nroi"]):
            sc[i] = ((S[i][best] - ref) ** 2).sum(1)
        keep = torch.sort(torch.cat([keep, sc], 1), dim=1).values[:, :want]
    return keep.reshape(c["nroi"], *((want,) if c["kind"] == "topk" else ()))


def _residuals(S, R, u, img):
    """Residual S - I(R^T u) and the derivative of I with respect to R^T u."""
    cx, cy, cz = (u @ R).unbind(-1)
    rho2 = cx * cx + cy * cy
    rho = rho2.sqrt()
    al, be = torch.rad2deg(torch.atan2(cz, rho)), torch.rad2deg(torch.atan2(cy, cx))
    be = torch.where(be < 0, be + 360.0, be)
    i0 = torch.floor(al + 90.0).clamp(0, 179)
    fj = torch.floor(be)
    ti, tj = al + 90.0 - i0, be - fj
    i0, j0 = i0.long(), (fj.long() % 360)
    j1 = (j0 + 1) % 360
    a, b, d, e = img[i0, j0], img[i0, j1], img[i0 + 1, j0], img[i0 + 1, j1]
    ok = (al.abs() <= 89.0).double()
    r = (S - ((1 - ti) * ((1 - tj) * a + tj * b) + ti * ((1 - tj) * d + tj * e))) * ok
    fi, fjj = (1 - tj) * (d - a) + tj * (e - b), (1 - ti) * (b - a) + ti * (e - d)
    n2 = rho2 + cz * cz
    deg = 180.0 / math.pi
    gx = deg * (-fi * cz * cx / (n2 * rho) - fjj * cy / rho2)
    gy = deg * (-fi * cz * cy / (n2 * rho) + fjj * cx / rho2)
    gz = deg * fi * rho / n2
    zero = torch.zeros_like(r)
    g = torch.stack([torch.where(ok > 0, v, zero) for v in (gx, gy, gz)], -1)
    # dr / d delta of R <- exp([delta]x) R is -(R grad) x u
    return r, -torch.linalg.cross((g @ R.transpose(-1, -2)), u.expand_as(g))


def _expq(w):
    th = w.norm(dim=1, keepdim=True)
    s = torch.where(th > 1e-12, torch.sin(th / 2) / th.clamp_min(1e-300), torch.full_like(th, 0.5))
    return torch.cat([torch.cos(th / 2), s * w], 1)


def _exact_refine(c, x):
    u, img = _dirs(c["dirs"]).double(), x["img"].double()
    n = c["nroi"]
    q, loss, grad = x["q0"].clone(), torch.empty(n, device=DEV, dtype=torch.float64), torch.empty(n, 3, device=DEV, dtype=torch.float64)
    for i in range(0, n, 256):
        S, p = x["S"][i:i + 256].double(), q[i:i + 256]
        if c["kind"] == "refgrad":
            w = x["omega"][i:i + 256]
            p = _qmul(_expq(w), p)
            r, J = _residuals(S, _rot(p / p.norm(dim=1, keepdim=True)), u, img)
            loss[i:i + 256] = (r * r).sum(1)
            gd = 2.0 * (J * r[..., None]).sum(1)
            th = w.norm(dim=1, keepdim=True)
            A, B = (1 - torch.cos(th)) / th ** 2, (th - torch.sin(th)) / th ** 3
            c1 = torch.linalg.cross(w, gd)
            grad[i:i + 256] = gd - A * c1 + B * torch.linalg.cross(w, c1)
            continue
        p = p / p.norm(dim=1, keepdim=True)
        for it in range(c["iters"]):
            r, J = _residuals(S, _rot(p), u, img)
            H = J.transpose(1, 2) @ J
            lam = 1e-6 * H.diagonal(dim1=1, dim2=2).sum(1)
            H = H + lam[:, None, None] * torch.eye(3, device=DEV, dtype=torch.float64)
            d = -torch.linalg.solve(H, (J * r[..., None]).sum(1))
            p = _qmul(_expq(d), p)
            p = p / p.norm(dim=1, keepdim=True)
        r, _ = _residuals(S, _rot(p), u, img)
        q[i:i + 256] = p * torch.where(p[:, :1] < 0, -1.0, 1.0)
        loss[i:i + 256] = (r * r).sum(1)
    return (q, loss) if c["kind"] == "refine" else (loss, grad)
