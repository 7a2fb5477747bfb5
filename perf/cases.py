"""The work this framework is measured on, through its public entry points.

Every case is one pass of something a user's program does repeatedly: assemble a force field, run a
relaxed scan on one, differentiate an image, correlate densities, image one small molecule, image a
batch of molecules.  listed() gives the fixed cases, draw() more of the same ranges, prepare() what a
program holds before the pass, run() the pass, work() what it cannot do without, exact() the same
outputs in 64 bits from plain torch.

Inputs that a stage takes from an earlier one (the grid a scan reads, the positions an adjoint starts
from) are made here with torch, so that a case exercises its own stage alone.  Geometries are the
repository's synthetic ones (synth.py) with every atom displaced and every charge redrawn by the seed.

The whole calls (image, batch) return images that depend on a stopping tolerance: a scan that stops at
|G| < ftol can take one update more or less after any change of rounding in its grid.  They run
with the options a program uses that wants images free of that: the Newton polish for one image; for a
batch, which has no polish, a stiff (metal) tip and a tight tolerance.
"""
import functools
import math

import numpy as np
import torch

from paper_2401_14564_gb300 import afm, batch, pp, synth

K_E = 14.3996454784  # eV A / e^2
EV_A2 = 16.02176634  # 1 eV/A^2 in N/m
KEYS = ("x", "y", "z", "R", "eps", "q")


# ------------------------------------------------------------------ the cases

def _ff(name, shape, atoms, nx, ny, nz, d=0.1, energy=True, interp=0, qzz=0.0):
    c = {"kind": "ff", "shape": shape, "atoms": atoms, "nx": nx, "ny": ny, "nz": nz, "d": d, "energy": energy,
         "interp": interp, "qzz": qzz}
    return dict(c, name=name) if name else c


def _scan(name, kind, atoms, nx, ny, nz, d, sx, sy, sz, interp=0, qzz=0.0):
    c = {"kind": kind, "shape": "flake" if atoms == 60 else "molecule", "atoms": atoms, "nx": nx, "ny": ny, "nz": nz,
         "d": d, "sx": sx, "sy": sy, "sz": sz, "interp": interp, "qzz": qzz}
    return dict(c, name=name) if name else c


def _fft(name, nx, ny, nz, power, accumulate):
    c = {"kind": "fft", "nx": nx, "ny": ny, "nz": nz, "power": power, "accumulate": accumulate}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one benzene-sized molecule, coarse grid, small scan, host to image in three launches: the smallest
        # call of interactive use, where launches and latency count
        {"name": "image_small", "kind": "image", "shape": "molecule", "atoms": 12, "nx": 80, "ny": 80, "nz": 60, "d": 0.2,
         "sx": 40, "sy": 40, "sz": 20, "interp": 0},
        # the grid of one molecule of a dataset, CO tip with its quadrupole, energies kept
        _ff("ff_molecule", "molecule", 40, 176, 160, 60, qzz=-0.05),
        # the flagship image's grid: 60-atom flake at 0.1 A, forces only (all a scan reads)
        _ff("ff_flake", "flake", 60, 256, 256, 200, energy=False),
        # a 500-atom molecule on a periodic 2016-atom bilayer: minimum image, Coulomb cut at 8 A
        _ff("ff_slab", "slab", 2516, 512, 512, 250),
        # an energy-only grid for tricubic interpolation at a coarser spacing, odd in every direction
        _ff("ff_energy_odd", "molecule", 97, 203, 187, 101, d=0.15, interp=1),
        # the flagship relaxed scan and df image on its force grid
        _scan("scan_flake", "scan", 60, 256, 256, 200, 0.1, 256, 256, 40),
        # a ragged scan on a tricubic energy grid at 0.2 A
        _scan("scan_tricubic_odd", "scan", 30, 128, 128, 75, 0.2, 131, 117, 30, interp=1),
        # gradients of one molecule's image (fitting a geometry, charges or the tip): the small adjoint
        _scan("backward_molecule", "backward", 40, 160, 160, 60, 0.1, 128, 128, 20, qzz=-0.05),
        # gradients of the flagship image
        _scan("backward_flake", "backward", 60, 256, 256, 200, 0.1, 256, 256, 40),
        # Hartree electrostatics of one molecule's cell
        _fft("fft_molecule", 128, 128, 128, 1.0, False),
        # the full-density model's Pauli term on a large periodic sheet, added to the grid
        _fft("fft_sheet", 512, 512, 128, 1.05, True),
        # images of a dataset's molecules, 10-80 atoms each, in one launch
        {"name": "batch_dataset", "kind": "batch", "molecules": 64, "first": 1000, "px": 128, "heights": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["image", "ff", "ff", "ff", "scan", "scan", "backward", "fft", "batch"])
    if kind == "image":
        nx, ny = _log(rng, 60, 110), _log(rng, 60, 110)
        return {"kind": "image", "shape": "molecule", "atoms": rng.randint(8, 14), "nx": nx, "ny": ny,
                "nz": rng.randint(50, 70), "d": 0.2, "sx": _log(rng, 20, 64), "sy": _log(rng, 20, 64),
                "sz": rng.randint(14, 24), "interp": 0}
    if kind == "ff":
        if rng.random() < 0.25:
            # a periodic sheet: minimum image and cutoff
            return _ff(None, "sheet", 4 * _log(rng, 30, 400), _log(rng, 96, 400), _log(rng, 96, 400), _log(rng, 40, 160))
        interp = int(rng.random() < 0.3)
        return _ff(None, "molecule", _log(rng, 8, 500), _log(rng, 60, 320), _log(rng, 60, 320), _log(rng, 40, 200),
                   d=rng.choice([0.1, 0.1, 0.15, 0.2]), energy=bool(interp) or rng.random() < 0.6, interp=interp,
                   qzz=rng.choice([0.0, 0.0, -0.05]))
    if kind in ("scan", "backward"):
        interp = int(kind == "scan" and rng.random() < 0.3)
        d = 0.2 if interp else 0.1
        n = (60, 130) if interp else (120, 260)
        return _scan(None, kind, _log(rng, 12, 120), _log(rng, *n), _log(rng, *n), rng.randint(70, 90) if interp else
                     rng.randint(110, 150), d, _log(rng, 30, 256), _log(rng, 30, 256), rng.randint(16, 40), interp,
                     qzz=rng.choice([0.0, -0.05]))
    if kind == "fft":
        return _fft(None, 1 << rng.randint(5, 9), 1 << rng.randint(5, 9), 1 << rng.randint(5, 8),
                    rng.choice([1.0, 1.05, 1.2]), rng.random() < 0.5)
    return {"kind": "batch", "molecules": _log(rng, 2, 64), "first": rng.randint(1000, 1900),
            "px": rng.randint(48, 128), "heights": rng.randint(14, 24)}


# ------------------------------------------------------------------ geometries

@functools.lru_cache(maxsize=512)
def _base(shape, n):
    if shape == "flake":
        return synth.aromatic_flake(60, 42) if n == 60 else synth.aromatic_flake(n, 42)
    if shape == "slab":
        return synth.slab_case()["atoms"]
    if shape == "sheet":
        cells = n // 4
        na = max(1, int(round(math.sqrt(cells * math.sqrt(3.0)))))
        return synth.graphene_sheet(na, max(1, -(-cells // na)), z=0.0)
    return synth.random_molecule(n, n)


@functools.lru_cache(maxsize=2048)
def _dataset(seed):
    return synth.random_molecule(seed)


def _moved(atoms, seed):
    """A neighbouring geometry: every atom displaced by up to 0.05 A along each axis, charges redrawn
    within the same bound and neutral."""
    rng = np.random.default_rng(seed)
    out = dict(atoms)
    n = len(atoms["x"])
    for k in ("x", "y", "z"):
        out[k] = np.asarray(atoms[k]) + rng.uniform(-0.05, 0.05, n)
    q = rng.uniform(-1.0, 1.0, n) * (np.abs(atoms["q"]) > 0)
    charged = np.abs(atoms["q"]) > 0
    if charged.any():
        q[charged] -= q[charged].mean()
        q *= np.abs(atoms["q"]).max() / np.abs(q).max()
    out["q"] = q
    return {k: np.asarray(out[k], dtype=np.float32) for k in KEYS}


def _f32(v):
    return float(np.float32(v))


def _case(case, seed):
    """The framework's case dict (grid, scan, probe, tip, FIRE, df) of one of the cases above."""
    base = _base(case["shape"], case["atoms"])
    atoms = _moved(base, seed)
    d, nx, ny, nz = case["d"], case["nx"], case["ny"], case["nz"]
    probe = synth.default_probe(Qzz=case.get("qzz", 0.0))
    top = float(np.max(base["z"]))
    if case["shape"] == "slab":
        x0 = y0 = z0 = 0.0
        probe = synth.default_probe(coul_rc=8.0, min_image=1)
    elif case["shape"] == "sheet":
        # the grid spans the sheet's period; its spacing follows
        probe = synth.default_probe(coul_rc=8.0, min_image=1)
        x0 = y0 = 0.0
        z0 = top + 1.5
    else:
        x0, y0 = -0.5 * nx * d, -0.5 * ny * d
        z0 = top if case["shape"] == "flake" else top + 2.0
    g = {"nx": nx, "ny": ny, "nz": nz, "x0": _f32(x0), "y0": _f32(y0), "z0": _f32(z0), "dx": _f32(d), "dy": _f32(d),
         "dz": _f32(d), "periodic_xy": 1, "interp": case.get("interp", 0)}
    if case["shape"] == "sheet":
        cells = case["atoms"] // 4
        na = max(1, int(round(math.sqrt(cells * math.sqrt(3.0)))))
        g["dx"], g["dy"] = _f32(na * 2.46 / nx), _f32(max(1, -(-cells // na)) * 2.46 * math.sqrt(3.0) / ny)
    c = {"name": "case", "atoms": atoms, "grid": g, "probe": probe, "tip": synth.default_tip(),
         "fire": synth.default_fire(), "df": synth.default_df()}
    if "sx" in case:
        sx, sy, sz = case["sx"], case["sy"], case["sz"]
        px, py = 0.94 * nx * d / sx, 0.94 * ny * d / sy
        # the probe goes from 2.8 A above the grid's own clearance down, unrelaxed, in 0.1 A steps
        zlow = top + (3.3 if case["kind"] != "image" else 3.5)
        c["scan"] = {"nx": sx, "ny": sy, "nz": sz, "x0": _f32(-0.5 * (sx - 1) * px), "y0": _f32(-0.5 * (sy - 1) * py),
                     "px": _f32(px), "py": _f32(py), "z_top": _f32(zlow + 0.1 * (sz - 1) + 4.0), "dz": _f32(0.1)}
    if case["kind"] == "image":
        c["fire"] = synth.default_fire(polish=4)
    return c


def _batch_cases(case, seed):
    out = []
    for i in range(case["molecules"]):
        m = synth.molecule_case(_dataset(case["first"] + i), f"mol{i}", scan_px=case["px"], nz_scan=case["heights"])
        m["atoms"] = _moved(m["atoms"], seed * 1009 + i)
        m["tip"] = synth.default_tip(kx=5.0, ky=5.0)
        m["fire"] = synth.parity_fire(ftol=1e-6)
        for blk in ("grid", "scan"):
            m[blk] = {k: _f32(v) if isinstance(v, float) else v for k, v in m[blk].items()}
        out.append(m)
    return out


# ------------------------------------------------------------------ the model in plain torch

def _probe64(p):
    return {k: _f32(p[k]) for k in ("R_pp", "eps_pp", "Q", "coul_rc", "core_frac", "Qzz")} | {"min_image": p["min_image"]}


def _pairs(nodes, A, P, period, energy_only=False):
    """(Fx, Fy, Fz, E) at the nodes (three tensors of one shape), summed over the atoms of A (tensors),
    of the probe P; differentiable."""
    dx, dy, dz = (nodes[i].unsqueeze(-1) - A[k] for i, k in enumerate("xyz"))
    if P["min_image"]:
        dx = dx - period[0] * torch.round(dx / period[0]).detach()
        dy = dy - period[1] * torch.round(dy / period[1]).detach()
    R = A["R"] + P["R_pp"]
    e = torch.sqrt(A["eps"] * P["eps_pp"])
    r2 = torch.maximum(dx * dx + dy * dy + dz * dz, (P["core_frac"] * R) ** 2)
    ir2 = 1.0 / r2
    rs = torch.sqrt(ir2)
    u6 = (R * R * ir2) ** 3
    kq = K_E * P["Q"] * A["q"]
    s = 12.0 * e * (u6 * u6 - u6) * ir2
    E = e * (u6 * u6 - 2.0 * u6)
    if P["coul_rc"] > 0:
        rc = P["coul_rc"]
        kq = torch.where(r2 < rc * rc, kq.expand_as(r2), torch.zeros_like(r2))
        s = s + kq * rs * (ir2 - 1.0 / rc ** 2)
        E = E + kq * (rs + r2 * rs / rc ** 2 - 2.0 / rc)
    else:
        s = s + kq * rs * ir2
        E = E + kq * rs
    sz = s
    if torch.is_tensor(P["Qzz"]) or P["Qzz"] != 0.0:
        c5 = 0.5 * K_E * P["Qzz"] * A["q"] * ir2 * ir2 * rs
        s = s + c5 * (15.0 * dz * dz * ir2 - 3.0)
        sz = s - 6.0 * c5
        E = E + c5 * (3.0 * dz * dz - r2)
    if energy_only:
        return E.sum(-1)
    return torch.stack([(s * dx).sum(-1), (s * dy).sum(-1), (sz * dz).sum(-1), E.sum(-1)], -1)


def _axes(g, dtype):
    return [g[o] + torch.arange(g[n], device="cuda", dtype=dtype) * g[d] for o, n, d in
            (("x0", "nx", "dx"), ("y0", "ny", "dy"), ("z0", "nz", "dz"))]


def _atoms(c, dtype):
    return {k: torch.as_tensor(c["atoms"][k], dtype=dtype, device="cuda") for k in KEYS}


def _grid(c, dtype):
    """The case's grid, [nz][ny][nx][4] (or [nz][ny][nx] energies), in slices that fit."""
    g, P, A = c["grid"], _probe64(c["probe"]), _atoms(c, dtype)
    x, y, z = _axes(g, dtype)
    period = (g["nx"] * g["dx"], g["ny"] * g["dy"])
    e_only = g["interp"] == 1
    out = torch.zeros((g["nz"], g["ny"], g["nx"]) + (() if e_only else (4,)), dtype=dtype, device="cuda")
    n = A["x"].numel()
    na = min(n, 64)
    rows = max(1, (1 << 26) // (g["nx"] * na))
    flat = out.view((g["nz"] * g["ny"], g["nx"]) + out.shape[3:])
    for r0 in range(0, flat.shape[0], rows):
        r = torch.arange(r0, min(r0 + rows, flat.shape[0]), device="cuda")
        nodes = (x.expand(r.numel(), -1), y[r % g["ny"]][:, None].expand(-1, g["nx"]),
                 z[r // g["ny"]][:, None].expand(-1, g["nx"]))
        for a0 in range(0, n, na):
            flat[r0:r0 + rows] += _pairs(nodes, {k: v[a0:a0 + na] for k, v in A.items()}, P, period, e_only)
    return out


def _cells(g, p):
    """Cell indices and fractions of the positions p (.., 3) as the grid's interpolation takes them."""
    out = []
    for a, (o, n, d) in enumerate((("x0", "nx", "dx"), ("y0", "ny", "dy"), ("z0", "nz", "dz"))):
        f = (p[..., a] - g[o]) / g[d]
        m = g[n]
        if a < 2 and g["periodic_xy"]:
            f = f - m * torch.floor(f / m)
            i = f.floor().long().clamp(0, m - 1)
            out.append((i, (i + 1) % m, (f - i).clamp(0.0, 1.0)))
        else:
            i = f.floor().long().clamp(0, m - 2)
            out.append((i, i + 1, (f - i).clamp(0.0, 1.0)))
    return out


def _trilinear(ff, g, p, jac=False):
    """Forces of the trilinear interpolant at p (n, 3) and, with jac, dF_a/dp_b (n, 3, 3)."""
    (i0, i1, tx), (j0, j1, ty), (k0, k1, tz) = _cells(g, p)
    flat = ff.view(-1, 4)
    v = [[[flat[(k * g["ny"] + j) * g["nx"] + i, :3] for i in (i0, i1)] for j in (j0, j1)] for k in (k0, k1)]
    tx, ty, tz = tx[:, None], ty[:, None], tz[:, None]

    def lerp(a, b, t):
        return a + (b - a) * t

    F = lerp(*[lerp(*[lerp(v[k][j][0], v[k][j][1], tx) for j in (0, 1)], ty) for k in (0, 1)], tz)
    if not jac:
        return F
    gx = lerp(*[lerp(*[v[k][j][1] - v[k][j][0] for j in (0, 1)], ty) for k in (0, 1)], tz) / g["dx"]
    gy = lerp(*[lerp(v[k][1][0] - v[k][0][0], v[k][1][1] - v[k][0][1], tx) for k in (0, 1)], tz) / g["dy"]
    gz = lerp(*[lerp(v[1][j][0] - v[0][j][0], v[1][j][1] - v[0][j][1], tx) for j in (0, 1)], ty) / g["dz"]
    return F, torch.stack([gx, gy, gz], -1)


def _tricubic(E, g, p):
    """Forces of the cubic-convolution energy interpolant at p (n, 3)."""
    cells = _cells(g, p)
    idx, w, dw = [], [], []
    for a, (i0, i1, t) in enumerate(cells):
        n = g[("nx", "ny", "nz")[a]]
        wrap = (lambda i, n=n: i % n) if a < 2 and g["periodic_xy"] else (lambda i, n=n: i.clamp(0, n - 1))
        idx.append([wrap(i0 - 1), i0, i1, wrap(i1 + 1)])
        w.append([(-t ** 3 + 2 * t ** 2 - t) / 2, (3 * t ** 3 - 5 * t ** 2 + 2) / 2, (-3 * t ** 3 + 4 * t ** 2 + t) / 2,
                  (t ** 3 - t ** 2) / 2])
        dw.append([(-3 * t ** 2 + 4 * t - 1) / 2, (9 * t ** 2 - 10 * t) / 2, (-9 * t ** 2 + 8 * t + 1) / 2,
                   (3 * t ** 2 - 2 * t) / 2])
    flat = E.view(-1)
    at = torch.stack([(idx[2][c] * g["ny"] + idx[1][b]) * g["nx"] + idx[0][a] for c in range(4) for b in range(4)
                      for a in range(4)], -1)
    e = flat[at].view(-1, 4, 4, 4)
    W, D = [torch.stack(u, -1) for u in w], [torch.stack(u, -1) for u in dw]

    def con(x, y, z):
        return torch.einsum("nkji,ni,nj,nk->n", e, x, y, z)

    inside = []
    for a, (o, n, d) in enumerate((("x0", "nx", "dx"), ("y0", "ny", "dy"), ("z0", "nz", "dz"))):
        f = (p[:, a] - g[o]) / g[d]
        ok = torch.ones_like(f) if a < 2 and g["periodic_xy"] else ((f > 0) & (f < g[n] - 1)).to(f.dtype)
        inside.append(ok / g[d])
    return -torch.stack([con(D[0], W[1], W[2]) * inside[0], con(W[0], D[1], W[2]) * inside[1],
                         con(W[0], W[1], D[2]) * inside[2]], -1)


def _springs(tip, dtype):
    k = [_f32(tip[n]) / EV_A2 for n in ("kx", "ky", "kR")]
    R0 = _f32(tip["R0"])
    d0 = torch.tensor([0.0, 0.0, -R0], dtype=dtype, device="cuda")
    return k, R0, d0


def _anchors(s, dtype):
    j, i = torch.meshgrid(torch.arange(s["ny"], device="cuda", dtype=dtype), torch.arange(s["nx"], device="cuda",
                          dtype=dtype), indexing="ij")
    return torch.stack([s["x0"] + i * s["px"], s["y0"] + j * s["py"]], -1).view(-1, 2)


def _df_weights(df, dz):
    """Stencil of the frequency shift, Fz piecewise linear between the heights, from the top down."""
    a, m = 0.5 * df["A_pp"], int(math.ceil(0.5 * df["A_pp"] / dz - 1e-9))
    W = np.zeros(2 * m + 1)
    for j in range(-m, m):
        lo, hi = max(j * dz, -a), min((j + 1) * dz, a)
        if hi <= lo:
            continue
        r = [math.sqrt(max(a * a - u * u, 0.0)) for u in (lo, hi)]
        sn = [math.asin(min(max(u / a, -1.0), 1.0)) for u in (lo, hi)]
        k1 = r[0] - r[1]
        k2 = (0.5 * a * a * sn[1] - 0.5 * hi * r[1]) - (0.5 * a * a * sn[0] - 0.5 * lo * r[0])
        W[j + m] += ((j + 1) * dz * k1 - k2) / dz
        W[j + 1 + m] += (k2 - j * dz * k1) / dz
    pref = -(df["f0"] / (2.0 * df["k"])) * 2.0 / (math.pi * a * a) * EV_A2
    return [pref * w for w in W[::-1]], m


def _fire(force, c, equilibrium=False):
    """The relaxed scan in 64 bits: per column from the top down, FIRE at each height (to 1e-9 eV/A with
    `equilibrium`).  Returns df, fz, pos laid out as the scan's."""
    s, f, dt64 = c["scan"], c["fire"], torch.float64
    (kx, ky, kR), R0, d0 = _springs(c["tip"], dt64)
    kl = torch.tensor([kx, ky, 0.0], dtype=dt64, device="cuda")
    base = _anchors(s, dt64)
    n = base.shape[0]
    tol = 1e-9 if equilibrium else _f32(f["ftol"])
    most = 100000 if equilibrium else f["max_iter"]
    pos = torch.zeros((s["nz"], n, 3), dtype=dt64, device="cuda")
    fz = torch.zeros((s["nz"], n), dtype=dt64, device="cuda")
    col = torch.arange(n, device="cuda")  # columns still running; state of the others is dropped
    e, v = (torch.zeros((n, 3), dtype=dt64, device="cuda") for _ in range(2))
    dt = torch.full((n, 1), _f32(f["dt0"]), dtype=dt64, device="cuda")
    al = torch.full((n, 1), _f32(f["alpha0"]), dtype=dt64, device="cuda")
    k, it, npos = (torch.zeros(n, dtype=torch.long, device="cuda") for _ in range(3))
    step = 0
    while True:
        d = d0 + e
        dn = d.norm(dim=1, keepdim=True)
        rad = -kR * (dn - R0) / dn
        anchor = torch.cat([base[col], (s["z_top"] - k * s["dz"])[:, None]], 1)
        G = rad * d - kl * e + force(anchor + d)
        done = ((G.norm(dim=1) < tol) | (it >= most)) & (k < s["nz"])
        w = done.nonzero().squeeze(1)
        if w.numel():
            fz[k[w], col[w]] = (-rad * d[:, 2:])[w, 0]
            pos[k[w], col[w]] = (anchor + d)[w]
        pw = (G * v).sum(1, keepdim=True)
        later = (it > 0)[:, None]
        up, down = later & (pw > 0), later & ~(pw > 0)
        mix = (1 - al) * v + al * v.norm(dim=1, keepdim=True) * G / G.norm(dim=1, keepdim=True).clamp(min=1e-300)
        grow = up & (npos > f["n_min"])[:, None]
        v = torch.where(up, mix, torch.where(down, torch.zeros_like(v), v))
        dt = torch.where(grow, (dt * _f32(f["f_inc"])).clamp(max=_f32(f["dt_max"])), torch.where(down, dt * _f32(f["f_dec"]), dt))
        al = torch.where(grow, al * _f32(f["f_alpha"]), torch.where(down, torch.full_like(al, _f32(f["alpha0"])), al))
        npos = torch.where(up[:, 0], npos + 1, torch.where(down[:, 0], torch.zeros_like(npos), npos))
        v = v + dt * G / _f32(f["mass"])
        e = torch.where(done[:, None], e, e + dt * v)
        # a finished height: the next one starts from its deflection, at rest
        v = torch.where(done[:, None], torch.zeros_like(v), v)
        dt = torch.where(done[:, None], torch.full_like(dt, _f32(f["dt0"])), dt)
        al = torch.where(done[:, None], torch.full_like(al, _f32(f["alpha0"])), al)
        npos = torch.where(done, torch.zeros_like(npos), npos)
        it = torch.where(done, torch.zeros_like(it), it + 1)
        k = k + done
        step += 1
        if step % 64 == 0:
            live = (k < s["nz"]).nonzero().squeeze(1)
            if not live.numel():
                break
            if live.numel() < 0.7 * col.numel():
                col, e, v, dt, al, npos, it, k = (t[live] for t in (col, e, v, dt, al, npos, it, k))
        # columns already through stay at rest below the scan until they are dropped
        stop = k >= s["nz"]
        e = torch.where(stop[:, None], torch.zeros_like(e), e)
        it = torch.where(stop, torch.zeros_like(it), it)
        v = torch.where(stop[:, None], torch.zeros_like(v), v)
    W, m = _df_weights({q: _f32(x) for q, x in c["df"].items()}, s["dz"])
    df = sum(W[t] * fz[t:t + s["nz"] - 2 * m] for t in range(2 * m + 1))
    shape = (s["ny"], s["nx"])
    return df.view(-1, *shape), fz.view(-1, *shape), pos.view(-1, *shape, 3)


def _settled(ff, c):
    """Positions near the equilibrium of every pixel and height, by damped descent in 32 bits, and the
    points where the lateral stiffness there is above 0.01 eV/A^2: an image's gradient diverges where the
    probe is about to jump, and a fit leaves those pixels out of its loss."""
    s, g, dtp = c["scan"], c["grid"], torch.float32
    (kx, ky, kR), R0, d0 = _springs(c["tip"], dtp)
    kl = torch.tensor([kx, ky, 0.0], dtype=dtp, device="cuda")
    hard = torch.tensor([0.05, 0.05, kR], dtype=dtp, device="cuda")
    out = torch.empty((s["nz"], s["ny"] * s["nx"], 3), dtype=dtp, device="cuda")
    base = _anchors(s, dtp)
    e = torch.zeros((base.shape[0], 3), dtype=dtp, device="cuda")
    firm = torch.empty((s["nz"], s["ny"] * s["nx"]), dtype=torch.bool, device="cuda")
    for k in range(s["nz"]):
        anchor = torch.cat([base, torch.full_like(base[:, :1], s["z_top"] - k * s["dz"])], 1)
        for _ in range(8):
            d = d0 + e
            dn = d.norm(dim=1, keepdim=True)
            G = -kR * (dn - R0) / dn * d - kl * e + _trilinear(ff, g, anchor + d)
            e = e + (0.7 * G / hard).clamp(-0.1, 0.1)
        out[k] = anchor + d0 + e
        _, J = _trilinear(ff, g, out[k], jac=True)
        a, b, h = kx - J[:, 0, 0], ky - J[:, 1, 1], -0.5 * (J[:, 0, 1] + J[:, 1, 0])
        firm[k] = 0.5 * (a + b) - torch.sqrt((0.5 * (a - b)) ** 2 + h * h) > 0.01
    return out.view(s["nz"], s["ny"], s["nx"], 3), firm.view(s["nz"], s["ny"], s["nx"])


def _loss_weights(c, firm, seed):
    """N(0, 1) weights of the df image, zero where any height an output reads is not firm."""
    s = c["scan"]
    m = int(math.ceil(0.5 * c["df"]["A_pp"] / s["dz"] - 1e-9))
    n = s["nz"] - 2 * m
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn((n, s["ny"], s["nx"]), device="cuda", generator=gen)
    for t in range(2 * m + 1):
        w = w * firm[t:t + n]
    return w


def _backward64(c, ff, pos, gdf):
    """Gradients of sum(gdf * df) by the implicit function theorem at pos, in 64 bits."""
    s, g, dt64 = c["scan"], c["grid"], torch.float64
    (kx, ky, kR), R0, d0 = _springs(c["tip"], dt64)
    W, m = _df_weights({q: _f32(x) for q, x in c["df"].items()}, s["dz"])
    npix = s["nx"] * s["ny"]
    gf = torch.zeros((s["nz"], npix), dtype=dt64, device="cuda")
    w = gdf.double().view(-1, npix)
    for t in range(2 * m + 1):
        gf[t:t + w.shape[0]] += W[t] * w
    base = _anchors(s, dt64)
    gbar = torch.zeros((g["nz"] * g["ny"] * g["nx"], 3), dtype=dt64, device="cuda")
    tip = torch.zeros(3, dtype=dt64, device="cuda")
    ff64 = ff.double()
    eye = torch.eye(3, dtype=dt64, device="cuda")
    for k in range(s["nz"]):
        p = pos[k].reshape(-1, 3).double()
        d = p - torch.cat([base, torch.full_like(base[:, :1], s["z_top"] - k * s["dz"])], 1)
        e = d - d0
        dn = d.norm(dim=1)
        ext = (dn - R0) / dn
        ar, br = -kR * ext, -kR * R0 / dn ** 3
        _, J = _trilinear(ff64, g, p, jac=True)
        J = J + ar[:, None, None] * eye + br[:, None, None] * d[:, :, None] * d[:, None, :]
        J = J - torch.diag(torch.tensor([kx, ky, 0.0], dtype=dt64, device="cuda"))
        r = (-ar[:, None] * eye[2] - br[:, None] * d[:, 2:] * d) * gf[k][:, None]
        lam = torch.linalg.solve(J.transpose(1, 2), r)
        tip += torch.stack([(lam[:, 0] * e[:, 0]).sum(), (lam[:, 1] * e[:, 1]).sum(),
                            (gf[k] * ext * d[:, 2] + (lam * d).sum(1) * ext).sum()])
        (i0, i1, tx), (j0, j1, ty), (k0, k1, tz) = _cells(g, p)
        for zc, wz in ((k0, 1 - tz), (k1, tz)):
            for yc, wy in ((j0, 1 - ty), (j1, ty)):
                for xc, wx in ((i0, 1 - tx), (i1, tx)):
                    gbar.index_add_(0, (zc * g["ny"] + yc) * g["nx"] + xc, -lam * (wz * wy * wx)[:, None])
    A = {k: v.requires_grad_(True) for k, v in _atoms(c, dt64).items()}
    P = _probe64(c["probe"])
    P["Q"], P["Qzz"] = (torch.tensor(P[k], dtype=dt64, device="cuda", requires_grad=True) for k in ("Q", "Qzz"))
    at = gbar.abs().amax(1).nonzero().squeeze(1)
    x, y, z = _axes(g, dt64)
    period = (g["nx"] * g["dx"], g["ny"] * g["dy"])
    chunk = max(1, (1 << 25) // A["x"].numel())
    for h in range(0, at.numel(), chunk):
        b = at[h:h + chunk]
        nodes = (x[b % g["nx"]], y[b // g["nx"] % g["ny"]], z[b // (g["nx"] * g["ny"])])
        (_pairs(nodes, A, P, period)[:, :3] * gbar[b]).sum().backward()
    out = {k: A[k].grad for k in KEYS}
    # (the derivative along Qzz is formed only for a tip that has a quadrupole)
    qzz = P["Qzz"].grad if c["probe"]["Qzz"] != 0.0 else torch.zeros_like(P["Q"].grad)
    out["tip"] = torch.cat([tip / EV_A2, P["Q"].grad.view(1), qzz.view(1)])
    return out


def _densities(case, seed):
    """Sample field and tip density of the correlation: sums of Gaussians, periodic in x, y and z."""
    n, d = [case[k] for k in ("nx", "ny", "nz")], 0.1
    L = [v * d for v in n]
    rng = np.random.default_rng(seed)
    count = max(8, min(960, int(0.35 * L[0] * L[1])))
    xyz = rng.random((count, 3)) * L
    pauli = case["power"] != 1.0
    amp = rng.uniform(1.0, 7.0, count) if pauli else rng.uniform(-0.3, 0.3, count)

    def field(at, weight, sigma):
        prof = []
        for a in range(3):
            r = torch.arange(n[a], device="cuda", dtype=torch.float64) * d - torch.as_tensor(at[:, a:a + 1], device="cuda")
            r = r - L[a] * torch.round(r / L[a])
            prof.append(sum(torch.exp(-(r + m * L[a]) ** 2 / (2 * sigma * sigma)) for m in (-1, 0, 1)).float())
        w = torch.as_tensor(weight, device="cuda", dtype=torch.float32) * (2 * math.pi * sigma * sigma) ** -1.5
        zy = (w[:, None, None] * prof[2][:, :, None] * prof[1][:, None, :]).reshape(len(at), -1)
        return (zy.T @ prof[0]).view(n[2], n[1], n[0]).contiguous()

    f = field(xyz, amp if pauli else amp - amp.mean(), 0.5)
    tip = np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 0.3], [0.0, 0.0, -0.3]])
    g = field(tip, [6.0, 0.5, 0.5] if pauli else [0.55, -0.28, -0.27], 0.6)
    return f, g


# ------------------------------------------------------------------ the passes

def prepare(case, seed):
    kind = case["kind"]
    if kind == "fft":
        g = {"nx": case["nx"], "ny": case["ny"], "nz": case["nz"], "x0": 0.0, "y0": 0.0, "z0": 0.0, "dx": 0.1,
             "dy": 0.1, "dz": 0.1, "periodic_xy": 1}
        grid = pp.make_grid(g)
        f, tip = _densities(case, seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        start = torch.randn(pp.pp_ff_floats(grid), device="cuda", generator=gen) * 0.05
        # (with accumulate each pass adds to the grid, as a program adds its terms; it starts at `start` again)
        return {"kind": kind, "f": f, "g": tip, "grid": grid, "start": start, "ff": torch.empty_like(start),
                "ws": torch.empty(pp.pp_fft_workspace(grid) // 4, device="cuda"), "scale": 18.0 if case["power"] != 1.0 else 1.0,
                "power": case["power"], "accumulate": case["accumulate"]}
    if kind == "batch":
        b = batch.Batch(_batch_cases(case, seed), want_pos=False, want_iters=False)
        return {"kind": kind, "batch": b}
    c = _case(case, seed)
    if kind == "ff":
        c["scan"] = {"nx": 1, "ny": 1, "nz": 11, "x0": 0.0, "y0": 0.0, "px": 1.0, "py": 1.0, "z_top": 9.0, "dz": 0.1}
        sim = afm.Simulator(c, ff_energy=case["energy"])
        return {"kind": kind, "sim": sim, "atoms": afm.atoms_to_device(c["atoms"])}
    if kind == "image":
        return {"kind": kind, "sim": afm.Simulator(c), "atoms": afm.atoms_to_device(c["atoms"])}
    sim = afm.Simulator(c, ff_energy=case["interp"] == 1)
    ff = _grid(c, torch.float32)
    sim.ff.copy_(ff.view(-1))
    if kind == "scan":
        return {"kind": kind, "sim": sim}
    pos, firm = _settled(ff, c)
    gdf = _loss_weights(c, firm, seed)
    n = len(c["atoms"]["x"])
    dev = afm.atoms_to_device(c["atoms"])
    grads = {k: torch.empty(n, device="cuda") for k in KEYS}
    grads["tip"] = torch.empty(5, device="cuda")
    return {"kind": kind, "sim": sim, "atoms": dev, "pos": pos.contiguous(), "gdf": gdf, "grads": grads,
            "ws": torch.empty(pp.pp_backward_workspace(sim.grid) // 4 + 4, device="cuda")}


def run(state):
    kind = state["kind"]
    if kind == "fft":
        if state["accumulate"]:
            state["ff"].copy_(state["start"])
        pp.pp_fft_correlate(state["f"], state["g"], state["grid"], state["scale"], state["power"], state["ff"],
                            state["ws"], accumulate=state["accumulate"])
        return state["ff"]
    if kind == "batch":
        b = state["batch"]
        b.run()
        return {"ff": b.ff, "df": b.df, "fz": b.fz}
    sim = state["sim"]
    if kind == "ff":
        sim.make_ff(state["atoms"])
        return sim.ff
    if kind == "image":
        sim.run(state["atoms"])
        return {"df": sim.df, "fz": sim.fz, "pos": sim.pos}
    if kind == "scan":
        sim.relax()
        return {"df": sim.df, "fz": sim.fz, "pos": sim.pos, "iters": sim.iters}
    pp.pp_backward(pp.make_atoms(state["atoms"]), sim.probe, sim.grid, sim.ff, sim.scan, sim.tip, sim.dfp, state["pos"],
                   state["gdf"], pp.make_grads(state["grads"]), state["ws"])
    return state["grads"]


# FP32 operations of one node-atom pair: forces; the energy; the quadrupole
_FORCE, _ENERGY, _QUAD = 26, 4, 12
_FIRE_OPS = 130   # one FIRE update with its trilinear lookup
_UPDATES = 13     # FIRE updates per pixel and height at ftol 1e-4, from the warm start


def work(case):
    kind = case["kind"]
    if kind == "fft":
        n = case["nx"] * case["ny"] * case["nz"]
        # two real fields in, four values per node out (and in, when added); a forward and two inverse
        # complex transforms
        return {"bytes": n * (8 + 16 + (16 if case["accumulate"] else 0)), "flops": 3 * 5 * n * math.log2(n) + 40 * n}
    if kind == "batch":
        by = fl = 0.0
        for m in _batch_cases(case, 0):
            g, s, n = m["grid"], m["scan"], len(m["atoms"]["x"])
            nodes, pts = g["nx"] * g["ny"] * g["nz"], s["nx"] * s["ny"] * s["nz"]
            by += 24 * n + 16 * nodes + 4 * pts + 4 * pts * (s["nz"] - 10) / s["nz"]
            fl += nodes * n * (_FORCE + _ENERGY) + pts * 30 * _FIRE_OPS
        return {"bytes": by, "flops": fl}
    nodes, n = case["nx"] * case["ny"] * case["nz"], case["atoms"]
    e_only = case["interp"] == 1
    if kind == "ff":
        per = (11 if e_only else _FORCE + (_ENERGY if case["energy"] else 0)) + (_QUAD if case["qzz"] else 0)
        return {"bytes": 24 * n + nodes * (4 if e_only else 16), "flops": nodes * n * per}
    pts = case["sx"] * case["sy"] * case["sz"]
    band = min(case["nz"], int((0.1 * case["sz"] + 1.0) / case["d"])) * case["nx"] * case["ny"]
    read = band * (4 if e_only else 16)
    if kind == "scan":
        return {"bytes": read + pts * 24, "flops": pts * _UPDATES * (_FIRE_OPS + (250 if e_only else 0))}
    if kind == "image":
        return {"bytes": 24 * n + nodes * 16 + read + pts * 20,
                "flops": nodes * n * (_FORCE + _ENERGY) + pts * (_UPDATES + 4) * _FIRE_OPS}
    # the touched nodes of the adjoint, contracted with every atom
    touched = min(band, 8 * pts)
    return {"bytes": read + pts * 16 + 48 * n, "flops": pts * 300 + touched * n * 60}


def exact(case, seed):
    kind = case["kind"]
    if kind == "fft":
        f, g = (t.double() for t in _densities(case, seed))
        grid = {"nx": case["nx"], "ny": case["ny"], "nz": case["nz"]}
        d = _f32(0.1)
        p = case["power"]
        if p != 1.0:
            f, g = (t.clamp(min=0.0) ** _f32(p) for t in (f, g))
        S = torch.conj(torch.fft.fftn(g)) * torch.fft.fftn(f)
        S = S * ((18.0 if p != 1.0 else 1.0) * d ** 3)
        out = torch.empty((grid["nz"], grid["ny"], grid["nx"], 4), dtype=torch.float64, device="cuda")
        out[..., 3] = torch.fft.ifftn(S).real
        for c, (axis, name) in enumerate(((2, "nx"), (1, "ny"), (0, "nz"))):
            n = grid[name]
            k = 2 * math.pi * torch.fft.fftfreq(n, d, device="cuda", dtype=torch.float64)
            k[n // 2] = 0.0
            shape = [1, 1, 1]
            shape[axis] = n
            out[..., c] = torch.fft.ifftn(-1j * k.view(shape) * S).real
        out = out.view(-1)
        if case["accumulate"]:
            gen = torch.Generator(device="cuda").manual_seed(seed)
            out = out + (torch.randn(out.numel(), device="cuda", generator=gen) * 0.05).double()
        return out
    if kind == "batch":
        # the packed grids; the images stop at a tolerance, on 64-bit grids of another rounding elsewhere
        cs = _batch_cases(case, seed)
        for m in cs:
            m["grid"]["interp"] = 0
        return {"ff": torch.cat([_grid(m, torch.float64).view(-1) for m in cs]), "df": None, "fz": None}
    if kind == "ff" and case["nx"] * case["ny"] * case["nz"] * case["atoms"] > 6e10:
        return None
    c = _case(case, seed)
    if kind == "ff":
        ff = _grid(c, torch.float64)
        if not case["energy"]:
            ff[..., 3] = 0.0
        return ff.view(-1)
    if kind == "image":
        ff = _grid(c, torch.float64)
        df, fz, pos = _fire(lambda p: _trilinear(ff, c["grid"], p), c, equilibrium=True)
        return {"df": df, "fz": fz, "pos": pos}
    ff = _grid(c, torch.float32)
    if kind == "scan":
        wide, g = ff.double(), c["grid"]
        force = (lambda p: _tricubic(wide, g, p)) if case["interp"] else (lambda p: _trilinear(wide, g, p))
        df, fz, pos = _fire(force, c)
        return {"df": df, "fz": fz, "pos": pos, "iters": None}
    pos, firm = _settled(ff, c)
    return _backward64(c, ff, pos, _loss_weights(c, firm, seed))
