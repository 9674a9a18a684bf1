"""Cases of the coupled free-surface LBM / DEM step and of its learned normal, as a user's program runs them.

What a pass is, by `kind`:
  flume     one output interval of a run: `steps` time steps, the bed height h_b(x), the lattice reduction, and the
            state a restart needs (PDFs, cell types, masses, particle positions and velocities), kept in single
            precision. The flume has a particle bed (random deposition, placed as repeated patches along x), a
            fixed bottom layer and a free surface, flat or wavy (antidunes come with surface waves).
  box       a restart and a short run without a free surface: PDFs in, `steps` time steps, PDFs and velocity out.
  stencils  training surfaces of the learned normal voxelised.
  train     Adam steps of the learned normal.
  infer     the network's raw outputs for a set of stencils.
  spectrum  power spectral density and dominant bedform of a bed-height series.
"""
import math

import numpy as np
import torch

from paper_2301_10674_gb300 import fslbm as F
from paper_2301_10674_gb300 import workloads as W

STORAGE = {"fp32": F.STORE_FP32, "fp16": F.STORE_FP16, "bf16": F.STORE_BF16}
LAM, MU = 0.4, 0.1          # loss weights of the learned normal
PATCH = 128                 # cells of x per bed patch


def flume(name, nx, ny, nz, d, bed, depth, steps, storage, normal, wave, stream, spread=0.1):
    c = {"kind": "flume", "nx": nx, "ny": ny, "nz": nz, "d": d, "spread": spread, "bed": bed, "depth": depth,
         "steps": steps, "storage": storage, "normal": normal, "wave": wave, "stream": stream}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the tiny test flume on the default stream: 33 k cells, a step is launches and latency
        flume("tiny flume fp32", 64, 16, 32, 6.0, 14.0, 12.0, 40, "fp32", "fd", 0.0, "default", 0.0),
        # the mid flume in the plain form, with a wavy surface: an ordinary parameter study
        flume("mid flume fp32", 512, 40, 96, 8.0, 40.0, 30.0, 40, "fp32", "fd", 2.0, "own"),
        # a flume whose extents fit no vector width, on the default stream
        flume("ragged flume fp32", 301, 37, 75, 7.0, 30.0, 26.0, 40, "fp32", "fd", 1.5, "default"),
        # the precision-study flume in its two 16-bit forms
        flume("precision flume bf16", 1024, 64, 128, 8.0, 56.0, 40.0, 40, "bf16", "fd", 2.0, "own"),
        flume("precision flume fp16 learned", 1024, 64, 128, 8.0, 56.0, 40.0, 40, "fp16", "learned", 2.0, "own"),
        # the large flume: the headline form and the reference form
        flume("large flume fp16 learned", 3072, 96, 320, 10.0, 150.0, 110.0, 40, "fp16", "learned", 0.0, "own"),
        flume("large flume fp32", 3072, 96, 320, 10.0, 150.0, 110.0, 40, "fp32", "fd", 0.0, "own"),
        # restart and run of a channel full of liquid between two plates
        {"name": "box fp32", "kind": "box", "nx": 200, "ny": 72, "nz": 90, "storage": "fp32", "steps": 20},
        # one shard of the training surfaces, all four kinds
        {"name": "stencils", "kind": "stencils", "n": 20000},
        # a stretch of training at the usual batch, with the cube symmetries
        {"name": "train", "kind": "train", "n": 200000, "batch": 4096, "steps": 64},
        # a held-out set through the network
        {"name": "infer", "kind": "infer", "n": 66944},
        # h_b(x, t) of a run: a sample every ten steps
        {"name": "spectrum", "kind": "spectrum", "nt": 500, "nx": 3072},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flume"] * 6 + ["box"] * 2 + ["stencils", "train", "infer", "spectrum"])
    if kind == "flume":
        d = rng.choice([6.0, 7.0, 8.0, 10.0])
        nx, ny = _logint(rng, 48, 2048), _logint(rng, 16, 96)
        nz = _logint(rng, 32, 256)
        if rng.random() < 0.5:          # half of the users pick round extents in x
            nx = max(64, nx // 32 * 32)
        bed = max(2.2 * d, round(rng.uniform(0.25, 0.45) * nz, 1)) if nz > 40 else 14.0
        d = min(d, 6.0) if nz <= 40 else d
        depth = round(max(6.0, min(0.8 * (nz - bed), rng.uniform(0.25, 0.4) * nz)), 1)
        depth = min(depth, nz - bed - 4.0)
        return flume(None, nx, ny, nz, d, bed, depth, rng.choice([11, 20, 40]), rng.choice(["fp32", "fp16", "bf16"]),
                     rng.choice(["fd", "learned"]), rng.choice([0.0, 1.0, 2.0]) if depth > 12 else 0.0,
                     rng.choice(["own", "default"]))
    if kind == "box":
        return {"kind": "box", "nx": _logint(rng, 16, 400), "ny": _logint(rng, 8, 96), "nz": _logint(rng, 8, 96),
                "storage": rng.choice(["fp32", "fp16", "bf16"]), "steps": rng.choice([7, 20, 40])}
    if kind == "stencils":
        return {"kind": "stencils", "n": _logint(rng, 100, 40000)}
    if kind == "train":
        return {"kind": "train", "n": _logint(rng, 5000, 500000), "batch": rng.choice([500, 1024, 4096, 10000]),
                "steps": rng.choice([10, 40, 100])}
    if kind == "infer":
        return {"kind": "infer", "n": _logint(rng, 100, 2000000)}
    return {"kind": "spectrum", "nt": _logint(rng, 20, 700), "nx": _logint(rng, 200, 3500)}


# ------------------------------------------------------------------ flume
def _bed(c, seed):
    """A deposition bed: one periodic patch of about PATCH cells, repeated along x. The number of spheres follows from
    the sizes alone (a packing that the deposition reaches)."""
    k = max(1, int(round(c["nx"] / PATCH)))
    width = c["nx"] / k
    want = max(1, int(0.38 * width * c["ny"] * (c["bed"] - 0.65 * c["d"]) / (math.pi / 6.0 * c["d"] ** 3)))
    for again in range(20):
        w = W.Workload(name="patch", nx=width, ny=c["ny"], nz=c["nz"], liquid_height=c["bed"] + c["depth"],
                       diameter=c["d"], polydispersity=c["spread"], bed="rsd", bed_height=c["bed"],
                       spheres_nominal=want, seed=seed + 1000003 * again).generate()
        if w.nspheres == want:
            break
    xyz = np.concatenate([w.xyz + np.array([i * width, 0.0, 0.0]) for i in range(k)])
    return xyz, np.tile(w.radius, k), np.tile(w.fixed, k)


def _workload(c, seed):
    gz, tau = -1e-5, 0.51
    # slope forcing of a flow at Froude number 1.2 (laminar open-channel estimate)
    gx = 3.0 * (tau - 0.5) / 3.0 * 1.2 * math.sqrt(abs(gz) * c["depth"]) / c["depth"] ** 2
    w = W.Workload(name="flume", nx=c["nx"], ny=c["ny"], nz=c["nz"], tau=tau, g=(gx, 0.0, gz),
                   liquid_height=c["bed"] + c["depth"], diameter=c["d"], polydispersity=c["spread"], bed_height=c["bed"])
    w.xyz, w.radius, w.fixed = _bed(c, seed)
    return w


def _network(seed):
    """Learned-normal weights: six units carry the Parker-Youngs gradient, the others small random features."""
    rng = np.random.default_rng(seed)
    w1, w2, w3 = np.zeros((64, 27)), np.zeros((64, 64)), np.zeros((4, 64))
    for q in range(27):
        cq = (q % 3 - 1, q // 3 % 3 - 1, q // 9 - 1)
        wt = {1: 4.0, 2: 2.0, 3: 1.0, 0: 0.0}[sum(v != 0 for v in cq)]
        for a in range(3):
            w1[2 * a, q], w1[2 * a + 1, q] = wt * cq[a] / 16.0, -wt * cq[a] / 16.0
    w1[6:] = rng.uniform(-0.4, 0.4, (58, 27))
    for u in range(6):
        w2[u, u] = 1.0
    w2[6:, 6:] = rng.uniform(-0.3, 0.3, (58, 58))
    for a in range(3):
        w3[a, 2 * a], w3[a, 2 * a + 1] = -1.0, 1.0
    w3[:, 6:] = rng.normal(0.0, 0.003, (4, 58))
    z = np.zeros
    return np.concatenate([w1.ravel(), z(64), w2.ravel(), z(64), w3.ravel(), z(4)]).astype(np.float32)


def _prepare_flume(c, seed):
    w = _workload(c, seed)
    stream = torch.cuda.Stream() if c["stream"] == "own" else None
    sim = F.Simulation.from_workload(w, storage=STORAGE[c["storage"]], stream=stream)
    rng = np.random.default_rng(seed)
    if c["wave"] > 0:
        # surface waves of about 128 cells, a little uneven across the flume
        x, y = np.arange(c["nx"]) + 0.5, np.arange(c["ny"]) + 0.5
        m = max(1, int(round(c["nx"] / 128.0)))
        p = rng.uniform(0.0, 2.0 * math.pi, 2)
        h = w.liquid_height + c["wave"] * np.sin(2.0 * math.pi * m * x / c["nx"] + p[0])[None, :] * \
            (1.0 + 0.3 * np.cos(2.0 * math.pi * y / c["ny"] + p[1]))[:, None]
        sim.init_surface(h)
    if c["normal"] == "learned":
        sim.set_normal_model(_network(seed), mirror=True)
    n, np_ = sim.n, sim.nspheres
    dev, f64, f32 = "cuda", torch.float64, torch.float32
    mask = F.FIELD_PDF | F.FIELD_TYPE | F.FIELD_MASS | F.FIELD_P_X | F.FIELD_P_U | F.FIELD_P_OMEGA
    read = [torch.empty(27, n, dtype=f64, device=dev), torch.empty(n, dtype=torch.uint8, device=dev),
            torch.empty(n, dtype=f64, device=dev)] + [torch.empty(np_, 3, dtype=f64, device=dev) for _ in range(3)]
    kept = [t if t.dtype == torch.uint8 else torch.empty(t.shape, dtype=f32, device=dev) for t in read]
    return {"c": c, "sim": sim, "mask": mask, "read": read, "kept": kept}


def _run_flume(s):
    sim = s["sim"]
    sim.step(s["c"]["steps"])
    bed = sim.bed_height()
    sums = sim.reduce()
    F._check(F.fslbm_get_fields(sim.h, s["mask"], s["read"], on_device=True), "fslbm_get_fields")
    with torch.cuda.stream(sim.stream):
        for a, b in zip(s["read"], s["kept"]):
            if a is not b:
                b.copy_(a)
    names = ("pdf", "type", "mass", "x", "u", "omega")
    return dict(zip(names, s["kept"]), bed=bed, sums=sums)


# ------------------------------------------------------------------ box
_C = [(q % 3 - 1, q // 3 % 3 - 1, q // 9 - 1) for q in range(27)]
_WQ = [{0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216}[sum(v != 0 for v in c)] for c in _C]
BOX_G = (1e-6, 0.0, 0.0)
BOX_OMEGA = 1.0 / 0.53


def _box_start(c, seed):
    """Equilibrium PDFs of a smooth random flow, [27][nz][ny][nx] in 64 bits."""
    rng = np.random.default_rng(seed)
    ax = [torch.arange(m, dtype=torch.float64, device="cuda") + 0.5 for m in (c["nz"], c["ny"], c["nx"])]
    fields = []
    for _ in range(4):
        v = torch.zeros(c["nz"], c["ny"], c["nx"], dtype=torch.float64, device="cuda")
        for _ in range(4):
            k, p = rng.integers(0, 3, 3), rng.uniform(0.0, 2.0 * math.pi, 3)
            g = [torch.cos(2.0 * math.pi * int(k[a]) * ax[a] / len(ax[a]) + p[a]) for a in range(3)]
            v += rng.uniform(-1.0, 1.0) * g[0][:, None, None] * g[1][None, :, None] * g[2][None, None, :]
        fields.append(v)
    rho, u = 1.0 + 2e-3 * fields[0], [0.02 * f for f in fields[1:]]
    uu = sum(v * v for v in u)
    f = torch.empty((27,) + tuple(rho.shape), dtype=torch.float64, device="cuda")
    for q in range(27):
        cu = sum(_C[q][a] * u[a] for a in range(3))
        f[q] = _WQ[q] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
    return f


def _prepare_box(c, seed):
    p = F.fslbm_default_params()
    p.nx, p.ny, p.nz = c["nx"], c["ny"], c["nz"]
    p.bc_flags = F.PERIODIC_X | F.PERIODIC_Y
    p.omega = BOX_OMEGA
    p.g[:] = list(BOX_G)
    p.liquid_height = float(c["nz"] + 2)
    p.storage = STORAGE[c["storage"]]
    sim = F.Simulation(p, torch.cuda.Stream())
    f = _box_start(c, seed)
    read = [torch.empty(27, sim.n, dtype=torch.float64, device="cuda"), torch.empty(3, sim.n, dtype=torch.float64, device="cuda")]
    return {"c": c, "sim": sim, "f": f, "read": read, "kept": [torch.empty(t.shape, dtype=torch.float32, device="cuda") for t in read]}


def _run_box(s):
    sim = s["sim"]
    F._check(F.fslbm_set_fields(sim.h, F.FIELD_PDF, [s["f"]], on_device=True), "fslbm_set_fields")
    sim.step(s["c"]["steps"])
    F._check(F.fslbm_get_fields(sim.h, F.FIELD_PDF | F.FIELD_U, s["read"], on_device=True), "fslbm_get_fields")
    with torch.cuda.stream(sim.stream):
        for a, b in zip(s["read"], s["kept"]):
            b.copy_(a)
    return {"pdf": s["kept"][0], "u": s["kept"][1]}


def _collide64(f, omega, g):
    """D3Q27 cumulant collision in 64 bits: second-order shear parts relax with omega, the trace with rate 1, all
    cumulants of higher order vanish; the body force as a half shift of the velocity."""
    rho = f.sum(0)
    j = [sum(_C[q][a] * f[q] for q in range(27)) for a in range(3)]
    u = [(j[a] + 0.5 * rho * g[a]) / rho for a in range(3)]
    k2 = {}
    for a in range(3):
        for b in range(a, 3):
            k2[a, b] = sum((_C[q][a] - u[a]) * (_C[q][b] - u[b]) * f[q] for q in range(27)) / rho
    d = {1: (1.0 - omega) * (k2[0, 0] - k2[1, 1]), 2: (1.0 - omega) * (k2[0, 0] - k2[2, 2])}
    xx = (1.0 + d[1] + d[2]) / 3.0
    S = {(0, 0): xx, (1, 1): xx - d[1], (2, 2): xx - d[2]}
    for a, b in ((0, 1), (0, 2), (1, 2)):
        S[a, b] = (1.0 - omega) * k2[a, b]
    s = lambda a, b: S[min(a, b), max(a, b)]  # noqa: E731
    # central moments about u, exponents 0..2 per axis
    K = {(i, jj, k): torch.zeros_like(rho) for i in range(3) for jj in range(3) for k in range(3)}
    K[0, 0, 0] = rho
    for a in range(3):
        e = [0, 0, 0]
        e[a] = 1
        K[tuple(e)] = 0.5 * rho * g[a]
        e[a] = 2
        K[tuple(e)] = rho * s(a, a)
    for a, b in ((0, 1), (0, 2), (1, 2)):
        e = [0, 0, 0]
        e[a] = e[b] = 1
        K[tuple(e)] = rho * s(a, b)
        e[a] = e[b] = 2
        K[tuple(e)] = rho * (s(a, a) * s(b, b) + 2.0 * s(a, b) ** 2)
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        e = [1, 1, 1]
        e[a] = 2
        K[tuple(e)] = rho * (s(a, a) * s(b, c) + 2.0 * s(a, b) * s(a, c))
    K[2, 2, 2] = rho * (s(0, 0) * s(1, 1) * s(2, 2) + 2.0 * (s(0, 0) * s(1, 2) ** 2 + s(1, 1) * s(0, 2) ** 2 + s(2, 2) * s(0, 1) ** 2)
                        + 8.0 * s(0, 1) * s(0, 2) * s(1, 2))
    # axis by axis: raw moments (m0, m1, m2) = (k0, k1 + u k0, k2 + 2 u k1 + u^2 k0), then the three populations
    for a in range(3):
        new = {}
        for i in range(3):
            for jj in range(3):
                key = lambda t: tuple(np.insert([i, jj], a, t))  # noqa: E731
                k0, k1, kk = K[key(0)], K[key(1)], K[key(2)]
                m1, m2 = k1 + u[a] * k0, kk + 2.0 * u[a] * k1 + u[a] ** 2 * k0
                new[key(0)], new[key(1)], new[key(2)] = 0.5 * (m2 - m1), k0 - m2, 0.5 * (m2 + m1)
        K = new
    return torch.stack([K[_C[q][0] + 1, _C[q][1] + 1, _C[q][2] + 1] for q in range(27)])


def _exact_box(c, seed):
    f = _box_start(c, seed)
    g = torch.tensor(BOX_G, dtype=torch.float32).double().tolist()
    for _ in range(c["steps"]):
        h = torch.empty_like(f)
        for q in range(27):
            cx, cy, cz = _C[q]
            t = torch.roll(f[q], (cz, cy, cx), (0, 1, 2))
            if cz > 0:                       # halfway bounce-back at the bottom and top plates
                t[0] = f[26 - q][0]
            elif cz < 0:
                t[-1] = f[26 - q][-1]
            h[q] = t
        f = _collide64(h, BOX_OMEGA, g)
    rho = f.sum(0)
    u = torch.stack([(sum(_C[q][a] * f[q] for q in range(27)) - 0.5 * rho * g[a]) / rho for a in range(3)])
    return {"pdf": f.reshape(27, -1), "u": u.reshape(3, -1)}


# ------------------------------------------------------------------ learned normal
def _prepare_stencils(c, seed):
    n = c["n"]
    return {"c": c, "params": torch.from_numpy(W.surface_stencils(n, seed=seed)).cuda(),
            "fill": torch.empty(n, 27, dtype=torch.float32, device="cuda"),
            "target": torch.empty(n, 4, dtype=torch.float32, device="cuda")}


def _run_stencils(s):
    F._check(F.fslbm_mlp_stencils(s["params"], s["c"]["n"], s["fill"], s["target"]), "fslbm_mlp_stencils")
    return {"fill": s["fill"], "target": s["target"]}


def _plane_fill(n, alpha):
    """Volume of the unit cube below n.x = alpha, n >= 0 componentwise, by 16-point Gauss sections along the largest
    component of the area below the line in the other two (exact up to the kinks, refined by 64 panels)."""
    o = torch.argsort(n, dim=-1, descending=True)
    m = torch.gather(n, -1, o)
    a, b, cc = m[..., 0], m[..., 1], m[..., 2]
    # integrate over the two smaller directions the clamped height (alpha - b y - c z) / a
    t = (torch.arange(64, dtype=torch.float64, device=n.device) + 0.5) / 64
    y, z = t[:, None].expand(64, 64).reshape(-1), t[None, :].expand(64, 64).reshape(-1)
    # within a sub-square the height is linear: the clamp only acts in the cut squares, taken by 8 x 8 points
    h = (alpha[..., None] - b[..., None] * y - cc[..., None] * z) / a[..., None]
    v = h.clamp(0.0, 1.0)
    r = (b + cc)[..., None] / a[..., None] / 128
    cut = ((h.abs() < r) | ((h - 1.0).abs() < r)).nonzero()
    if len(cut):
        i = tuple(cut[:, k] for k in range(cut.shape[1] - 1))
        s = ((torch.arange(8, dtype=torch.float64, device=n.device) + 0.5) / 8 - 0.5) / 64
        hh = h[tuple(cut.t())][:, None, None] - (b[i] / a[i])[:, None, None] * s[:, None] - (cc[i] / a[i])[:, None, None] * s[None, :]
        v[tuple(cut.t())] = hh.clamp(0.0, 1.0).mean((1, 2))
    return v.mean(-1)


def _exact_stencils(c, seed):
    n = c["n"]
    if n > 20000:
        return None
    P = torch.from_numpy(W.surface_stencils(n, seed=seed)).cuda()
    fill = torch.zeros(n, 27, dtype=torch.float64, device="cuda")
    C = torch.tensor(_C, dtype=torch.float64, device="cuda")
    n0, e1 = P[:, 1:4], P[:, 9:12]
    pt = P[:, 4:5] * n0
    sub = (torch.arange(64, dtype=torch.float64, device="cuda") + 0.5) / 64 - 0.5
    yy, zz = sub.repeat(64), sub.repeat_interleave(64)
    for kind in range(4):
        idx = (P[:, 0] == kind).nonzero()[:, 0]
        for at in idx.split(64 if kind == 0 else 256 if kind < 3 else 4):
            if kind == 0:
                nn = n0[at][:, None, :].expand(-1, 27, -1)
                beta = (nn * (pt[at][:, None, :] - (C[None] - 0.5))).sum(-1)
                fill[at] = _plane_fill(nn.abs(), beta - nn.clamp(max=0.0).sum(-1))
            elif kind < 3:
                r, sg = P[at, 5], (-1.0 if kind == 1 else 1.0)
                o = (pt[at] + sg * r[:, None] * n0[at])[:, None, :] - C[None]
                h2 = r[:, None, None] ** 2 - (yy - o[..., 1:2]) ** 2 - (zz - o[..., 2:3]) ** 2
                h = h2.clamp(min=0.0).sqrt()
                ch = (torch.minimum(o[..., 0:1] + h, h.new_tensor(0.5)) - torch.maximum(o[..., 0:1] - h, h.new_tensor(-0.5))).clamp(min=0.0)
                v = torch.where(h2 > 0, ch, torch.zeros_like(ch)).mean(-1)
                fill[at] = v if kind == 1 else 1.0 - v
            else:
                A, k, ph = P[at, 6], P[at, 7], P[at, 8]
                for q in range(27):
                    b = C[q] - pt[at]
                    u = (b * e1[at]).sum(-1)[:, None, None] + e1[at, 1:2, None] * yy[None, :, None] + e1[at, 2:3, None] * zz[None, :, None] + e1[at, 0:1, None] * sub
                    w = (b * n0[at]).sum(-1)[:, None, None] + n0[at, 1:2, None] * yy[None, :, None] + n0[at, 2:3, None] * zz[None, :, None] + n0[at, 0:1, None] * sub
                    f = A[:, None, None] * (torch.sin(k[:, None, None] * u + ph[:, None, None]) - torch.sin(ph)[:, None, None])
                    fill[at, q] = (w <= f).double().mean((1, 2))
    target = torch.zeros(n, 4, dtype=torch.float64, device="cuda")
    target[:, :3] = n0
    sph = (P[:, 0] == 1) | (P[:, 0] == 2)
    target[sph, 3] = torch.where(P[sph, 0] == 1, 1.0, -1.0).double() / P[sph, 5]
    sn = P[:, 0] == 3
    A, k, ph = P[sn, 6], P[sn, 7], P[sn, 8]
    fp, fpp = A * k * torch.cos(ph), -A * k * k * torch.sin(ph)
    qn = torch.sqrt(1.0 + fp * fp)
    target[sn, :3] = (n0[sn] - fp[:, None] * e1[sn]) / qn[:, None]
    target[sn, 3] = -fpp / (2.0 * qn ** 3)
    return {"fill": fill, "target": target}


def _planes(n, seed):
    """Fill levels and labels of n planes near a block's centre, from 5^3 points per cell."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nv = torch.randn(n, 3, generator=gen, device="cuda")
    nv = nv / nv.norm(dim=1, keepdim=True)
    s = torch.rand(n, generator=gen, device="cuda") - 0.5
    C = torch.tensor(_C, dtype=torch.float32, device="cuda")
    t = (torch.arange(5, device="cuda") + 0.5) / 5 - 0.5
    sub = torch.cartesian_prod(t, t, t)
    fill = torch.empty(n, 27, device="cuda")
    for q in range(27):
        for a in range(0, n, 1 << 18):
            b = slice(a, a + (1 << 18))
            fill[b, q] = (nv[b] @ (C[q] + sub).t() <= s[b, None]).float().mean(1)
    return fill, torch.cat([nv, torch.zeros(n, 1, device="cuda")], 1)


def _prepare_train(c, seed):
    fill, target = _planes(c["n"], seed)
    theta0 = torch.from_numpy(W.mlp_initial_weights(seed)).cuda()
    return {"c": c, "seed": seed, "fill": fill, "target": target, "theta0": theta0, "theta": torch.empty_like(theta0),
            "curve": torch.empty(c["steps"], dtype=torch.float32, device="cuda")}


def _run_train(s):
    c = s["c"]
    s["theta"].copy_(s["theta0"])
    F._check(F.fslbm_mlp_train(s["theta"], s["fill"], s["target"], c["n"], c["steps"], c["batch"], 2e-3, LAM, MU,
                               s["seed"], True, s["curve"], lr_end=1e-5), "fslbm_mlp_train")
    return {"theta": s["theta"], "loss": s["curve"]}


def _forward64(theta, x):
    at, out = 0, x
    for o, i, last in ((64, 27, False), (64, 64, False), (4, 64, True)):
        w, b = theta[at:at + o * i].reshape(o, i), theta[at + o * i:at + o * i + o]
        at += o * i + o
        out = out @ w.t() + b
        out = out if last else torch.relu(out)
    return out


def _draws(seed, first, count):
    """Outputs first .. first + count of SplitMix64."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.arange(first, first + count, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _exact_train(c, seed):
    if c["batch"] * c["steps"] > 2000000:
        return None
    fill, target = _planes(c["n"], seed)
    fill, target = fill.double(), target.double()
    perms = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))
    src, lab, sgn = np.zeros((48, 27), np.int64), np.zeros((48, 3), np.int64), np.zeros((48, 3))
    for k in range(48):
        p, s = perms[k // 8], [-1 if (k % 8) >> i & 1 else 1 for i in range(3)]
        lab[k], sgn[k] = p, s
        for q in range(27):
            v = [0, 0, 0]
            for i in range(3):
                v[p[i]] = s[i] * _C[q][i]
            src[k, q] = (v[0] + 1) + 3 * (v[1] + 1) + 9 * (v[2] + 1)
    src, lab, sgn = (torch.from_numpy(a).cuda() for a in (src, lab, sgn))
    theta = torch.from_numpy(W.mlp_initial_weights(seed)).cuda().double()
    m, v, curve = torch.zeros_like(theta), torch.zeros_like(theta), []
    for t in range(c["steps"]):
        z = _draws(seed, t * c["batch"], c["batch"])
        i = torch.from_numpy((z % np.uint64(c["n"])).astype(np.int64)).cuda()
        k = torch.from_numpy(((z >> np.uint64(32)) % np.uint64(48)).astype(np.int64)).cuda()
        x = torch.gather(fill[i], 1, src[k])
        nt, kt = sgn[k] * torch.gather(target[i, :3], 1, lab[k]), target[i, 3]
        th = theta.clone().requires_grad_(True)
        y = _forward64(th, x)
        r = y[:, :3].norm(dim=1)
        loss = (1.0 - (y[:, :3] * nt).sum(1) / r + LAM * (y[:, 3] - kt) ** 2 + MU * (r - 1.0) ** 2).mean()
        g, = torch.autograd.grad(loss, th)
        curve.append(loss.detach())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        lr = 2e-3 * (1e-5 / 2e-3) ** (t / max(1, c["steps"] - 1))
        theta = theta - lr * (m / (1.0 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1.0 - 0.999 ** (t + 1))) + 1e-8)
    return {"theta": theta, "loss": torch.stack(curve)}


def _prepare_infer(c, seed):
    fill, _ = _planes(c["n"], seed)
    return {"c": c, "fill": fill, "theta": torch.from_numpy(_network(seed)).cuda(),
            "out": torch.empty(c["n"], 4, dtype=torch.float32, device="cuda")}


def _run_infer(s):
    F._check(F.fslbm_mlp_infer(s["theta"], s["fill"], s["c"]["n"], s["out"]), "fslbm_mlp_infer")
    return s["out"]


# ------------------------------------------------------------------ bed spectrum
def _prepare_spectrum(c, seed):
    """A bed with a few travelling bedforms and roughness."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.arange(c["nt"], dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(c["nx"], dtype=torch.float64, device="cuda")[None, :]
    h = 145.0 + 0.3 * torch.randn(c["nt"], c["nx"], dtype=torch.float64, device="cuda", generator=gen)
    for _ in range(4):
        j, l = int(rng.integers(2, 40)), int(rng.integers(-8, 9))
        h += rng.uniform(0.5, 3.0) * torch.sin(2 * math.pi * (j * x / c["nx"] + l * t / c["nt"]) + rng.uniform(0, 6.28))
    return {"c": c, "h": h, "psd": torch.empty_like(h)}


def _run_spectrum(s):
    c = s["c"]
    rc, peak = F.fslbm_bed_spectrum(s["h"], c["nt"], c["nx"], 1.0, 10.0, s["psd"])
    F._check(rc, "fslbm_bed_spectrum")
    return {"psd": s["psd"], "peak": peak}


def _exact_spectrum(c, seed):
    h = _prepare_spectrum(c, seed)["h"]
    nt, nx = c["nt"], c["nx"]
    psd = torch.fft.fft2(h - h.mean()).abs() ** 2 / (nt * nx)
    top = psd[:, 1:nx // 2 + 1]
    at = int(top.argmax())
    l, j = at // (nx // 2), 1 + at % (nx // 2)
    l = l if l <= nt // 2 else l - nt
    lam, per = nx / j, (nt * 10.0 / abs(l) if l else math.inf)
    cel = (lam / per if l < 0 else -lam / per) if l else 0.0
    return {"psd": psd, "peak": np.array([lam, per, cel, 2.0 * math.sqrt(float(top.max()) / (nt * nx))])}


# ------------------------------------------------------------------ the file's functions
_PREPARE = {"flume": _prepare_flume, "box": _prepare_box, "stencils": _prepare_stencils, "train": _prepare_train,
            "infer": _prepare_infer, "spectrum": _prepare_spectrum}
_RUN = {"flume": _run_flume, "box": _run_box, "stencils": _run_stencils, "train": _run_train, "infer": _run_infer,
        "spectrum": _run_spectrum}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["c"]["kind"]](state)


def exact(case, seed):
    kind = case["kind"]
    if kind == "box":
        return _exact_box(case, seed)
    if kind == "stencils":
        return _exact_stencils(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "infer":
        s = _prepare_infer(case, seed)
        return _forward64(s["theta"].double(), s["fill"].double())
    if kind == "spectrum":
        return _exact_spectrum(case, seed)
    return None


def work(case):
    c, kind = case, case["kind"]
    if kind in ("flume", "box"):
        n, e = c["nx"] * c["ny"] * c["nz"], 4 if c["storage"] == "fp32" else 2
        if kind == "flume":
            # the bed holds about 0.4 of its volume in spheres; liquid above it
            fluid = c["nx"] * c["ny"] * (0.6 * c["bed"] + c["depth"])
            moved = n * (27 * 4 + 1 + 4)                      # the state read out
        else:
            fluid = float(n)
            moved = n * (27 * 8 + 30 * 4)                     # PDFs in, PDFs and velocity out
        return {"bytes": c["steps"] * (fluid * (54 * e + 1) + (n - fluid)) + moved, "flops": c["steps"] * fluid * 500.0}
    if kind == "stencils":
        return {"bytes": c["n"] * (12 * 8 + 31 * 4), "flops": c["n"] * 27 * (0.4 * 4096 * 12 + 0.25 * 4096 * 12)}
    if kind == "train":
        return {"bytes": c["steps"] * (c["batch"] * 31 * 4 + 6212 * 24), "flops": c["steps"] * c["batch"] * 6.0 * 6080}
    if kind == "infer":
        return {"bytes": c["n"] * 31 * 4, "flops": c["n"] * 2.0 * 6080}
    m = c["nt"] * c["nx"]
    return {"bytes": m * 16, "flops": 2.5 * m * math.log2(m)}
