"""The workloads whose speed counts: what a user of the library has it do.

Every case runs through the public binding (``paper_1904_11792_gb300.lbm``):

* ``steps``: one lattice advanced for some steps with in-loop diagnostics,
  whose records are read back after the call (as ``studies.breakup`` does);
  the populations stay on the device in the caller's own buffer.
* ``cylinder``: a small FP64 lattice advanced between readings of its density
  field (as ``studies.surface_tension`` and the coexistence runs do).
* ``sweep``: a batch of uneven ligaments advanced with diagnostics of every
  instance every ``check`` steps (as ``studies.breakup_vs_radius`` does) and
  a checkpoint of every instance's populations at the end.
* ``droplets``: diagnostics with droplet counting and the per-droplet
  statistics of a broken-up state.

``exact`` restates the method in plain FP64 torch on the device: D3Q19,
psi = 1 - exp(-rho), Shan-Chen force, velocity-shift BGK (or the MRT
collision with Guo's forcing) and streaming.
"""
import math
import random

import numpy as np
import torch

from paper_1904_11792_gb300 import lbm

G = -6.0
RHO_L, RHO_V = 2.6489, 0.0732   # flat-interface densities at G = -6, tau = 1
MRT_G, MRT_RHO_L, MRT_RHO_V = -5.3, 2.1085, 0.0778   # the paper's G with the MRT collision
WIDTH = 2.0
Q = 19
ELEM = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2}
TORCH = {"f64": torch.float64, "f32": torch.float32, "f16dev": torch.float16, "bf16dev": torch.bfloat16}


def listed():
    def steps(name, nx, ny, nz, precision, n, pattern="ab", collision="srt", tau=1.0):
        return {"name": name, "kind": "steps", "nx": nx, "ny": ny, "nz": nz, "precision": precision,
                "pattern": pattern, "collision": collision, "tau": tau, "steps": n, "diag": 10}

    return [
        # surface tension from static cylinders (Laplace's law), the smallest
        # calls of the studies: a few thousand FP64 nodes, many short steps
        {"name": "cylinder49_f64", "kind": "cylinder", "nx": 4, "ny": 49, "nz": 49, "tau": 1.0, "steps": 100},
        # the small break-up run of the parity tests, diagnosed every 10 steps
        steps("ligament64_f32", 64, 32, 32, "f32", 100),
        # the FP64 reference run of the precision study
        steps("grid256_f64", 256, 128, 128, "f64", 10),
        # the grid-convergence ligament
        steps("grid256_f32", 256, 128, 128, "f32", 20),
        # a box cut to the ligament's wavelength (2 pi R0 / 0.7 x 4 R0 x 4 R0, R0 = 28): odd row length
        steps("ragged251_f32", 251, 112, 112, "f32", 20),
        # the MRT collision on the same ligament
        steps("mrt256_f32", 256, 128, 128, "f32", 20, collision="mrt"),
        # the precision form: 2-byte deviation storage, two arrays and in place
        steps("precision512_f16dev", 512, 256, 256, "f16dev", 10, tau=0.9),
        steps("inplace512_f16dev", 512, 256, 256, "f16dev", 10, pattern="aa", tau=0.9),
        # the large ligament, the benchmark's workload
        steps("large1024_f32", 1024, 512, 512, "f32", 10),
        # sweeps of uneven ligaments, every instance diagnosed every 100 steps
        # (the break-up study against R0), with a checkpoint at the end
        {"name": "sweep12_f32", "kind": "sweep", "count": 12, "rmax": 16, "precision": "f32", "steps": 1000, "check": 100},
        {"name": "sweep8_f16dev", "kind": "sweep", "count": 8, "rmax": 16, "precision": "f16dev", "steps": 1000,
         "check": 100},
        # droplet counting and statistics after break-up
        {"name": "droplets256_f32", "kind": "droplets", "nx": 256, "ny": 128, "nz": 128, "precision": "f32", "drops": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("steps", "steps", "steps", "steps", "steps", "cylinder", "sweep", "droplets"))
    if kind == "cylinder":
        n = rng.randrange(33, 66)
        return {"kind": kind, "nx": rng.choice((3, 4, 5, 8)), "ny": n, "nz": n, "tau": round(rng.uniform(0.9, 1.0), 3),
                "steps": rng.choice((50, 100, 200))}
    if kind == "sweep":
        return {"kind": kind, "count": rng.randrange(3, 13), "rmax": rng.choice((8, 12, 16)),
                "precision": rng.choice(("f32", "f32", "f16dev", "bf16dev")), "steps": 100 * rng.randrange(5, 11), "check": rng.choice((50, 100))}
    if kind == "droplets":
        ny = _log(rng, 48, 160)
        return {"kind": kind, "nx": _log(rng, 4 * ny, 8 * ny) if ny < 100 else _log(rng, 2 * ny, 4 * ny), "ny": ny,
                "nz": ny + rng.randrange(-7, 8), "precision": rng.choice(("f32", "f32", "f64", "f16dev")),
                "drops": rng.randrange(2, 9)}
    precision = rng.choice(("f32", "f32", "f32", "f16dev", "f16dev", "bf16dev", "f64"))
    pattern = rng.choice(("ab", "ab", "ab", "aa"))
    collision = rng.choice(("srt", "srt", "srt", "mrt"))
    nx, ny = _log(rng, 48, 640), _log(rng, 28, 256)
    if rng.random() < 0.5:
        nx, ny = max(64, nx // 64 * 64), max(32, ny // 8 * 8)   # the sizes people pick
    nz = max(24, ny + rng.randrange(-5, 6)) if rng.random() < 0.5 else ny
    most = 4_200_000 if precision == "f64" else 34_000_000
    while nx * ny * nz > most:
        nx, ny, nz = max(48, nx // 2), max(28, ny // 2), max(24, nz // 2)
    n = 100 if nx * ny * nz < 300_000 else (20 if nx * ny * nz < 6_000_000 else 10)
    return {"kind": "steps", "nx": nx, "ny": ny, "nz": nz, "precision": precision, "pattern": pattern,
            "collision": collision, "tau": round(rng.uniform(0.9, 1.0), 3), "steps": n, "diag": 10}


# ---- inputs -------------------------------------------------------------------

def _fluid(case):
    """(G, liquid density, vapour density) of a case."""
    return (MRT_G, MRT_RHO_L, MRT_RHO_V) if case.get("collision") == "mrt" else (G, RHO_L, RHO_V)


def _ligament(case, seed):
    """The ligament of a case: R0 in nodes, eps and phase drawn from the seed."""
    rng = random.Random(seed)
    half = min(case["ny"], case["nz"]) / 2
    if case["kind"] == "cylinder":
        return dict(R0=rng.uniform(0.3, 0.65) * half, lam=float(case["nx"]), eps=0.0, phase=0.0)
    return dict(R0=rng.uniform(0.36, 0.5) * half, lam=float(case["nx"]), eps=rng.uniform(0.01, 0.05),
                phase=rng.uniform(0.0, 2 * math.pi))


def _instances(case, seed):
    """The uneven batch: R0 in {8, 12, 16} up to rmax, boxes lambda x 4 R0 x 4
    R0 with lambda = round(r R0).  The radii and lengths, which set the work,
    are the case's own; phases, eps and tau come from the seed."""
    size, rng = random.Random(1000 * case["count"] + case["rmax"]), random.Random(seed)
    out = []
    for _ in range(case["count"]):
        R0 = size.choice([r for r in (8, 12, 16) if r <= case["rmax"]])
        nx = int(round(size.uniform(4.5, 12.0) * R0))
        out.append(dict(nx=nx, ny=4 * R0, nz=4 * R0, tau=rng.uniform(0.9, 1.0), G=G, R0=float(R0), lam=float(nx),
                        eps=rng.uniform(0.03, 0.06), phase=rng.uniform(0.0, 2 * math.pi), rho_l=RHO_L, rho_v=RHO_V,
                        width=WIDTH))
    return out


def _drops(case, seed):
    """Centres (along the axis) and radii of the main drops and satellites
    left by a break-up, separated by vapour."""
    rng = random.Random(seed)
    n, nx, room = case["drops"], case["nx"], 0.42 * min(case["ny"], case["nz"])
    cell = nx / n
    out = []
    for k in range(n):
        r = min(room, 0.5 * cell - 3.0) * (rng.uniform(0.75, 0.95) if k % 2 == 0 else rng.uniform(0.3, 0.5))
        r = max(r, 2.5)
        out.append((cell * (k + 0.5) + rng.uniform(-0.5, 0.5), (case["ny"] - 1) / 2 + rng.uniform(-2, 2),
                    (case["nz"] - 1) / 2 + rng.uniform(-2, 2), r))
    return out


def _drop_distance(case, seed):
    """Signed distance to the nearest droplet's surface and that droplet's index, [nz, ny, nx]."""
    f64 = dict(dtype=torch.float64, device="cuda")
    z, y, x = (torch.arange(n, **f64) for n in (case["nz"], case["ny"], case["nx"]))
    best, who = None, None
    for k, (cx, cy, cz, r) in enumerate(_drops(case, seed)):
        dx = (x - cx).abs()
        dx = torch.minimum(dx, case["nx"] - dx)
        d = torch.sqrt(dx[None, None, :] ** 2 + (y - cy)[None, :, None] ** 2 + (z - cz)[:, None, None] ** 2) - r
        if best is None:
            best, who = d, torch.zeros_like(d, dtype=torch.int64)
        else:
            who = torch.where(d < best, k, who)
            best = torch.minimum(best, d)
    return best, who


def _drop_populations(case, seed):
    """FP64 populations of the droplets, with the weak flow of their motion along the axis."""
    d, who = _drop_distance(case, seed)
    rho = RHO_V + 0.5 * (RHO_L - RHO_V) * (1.0 - torch.tanh(2.0 * d / WIDTH))
    rng = random.Random(seed + 1)
    speed = torch.tensor([rng.uniform(-0.02, 0.02) for _ in range(case["drops"])], dtype=torch.float64, device="cuda")
    u = speed[who]
    c, w = _lattice()
    return torch.stack([w[a] * rho * (1 + 3 * c[a][0] * u + 4.5 * (c[a][0] * u) ** 2 - 1.5 * u * u) for a in range(Q)])


class _Lattice:
    """One lattice whose populations live in a buffer of the caller's."""

    def __init__(self, case):
        cfg = lbm.lbm_config_default()
        cfg.nx, cfg.ny, cfg.nz = case["nx"], case["ny"], case["nz"]
        cfg.tau, cfg.G = case.get("tau", 1.0), _fluid(case)[0]
        cfg.precision = lbm.PRECISIONS[case.get("precision", "f64")]
        cfg.pattern = lbm.PATTERNS[case.get("pattern", "ab")]
        cfg.rho_ref = _fluid(case)[2] if case.get("precision", "f64").endswith("dev") else 0.0
        state, psi = lbm.lbm_required_bytes(cfg)
        self.state = torch.empty(state, dtype=torch.uint8, device="cuda")
        self.psi = torch.empty(psi, dtype=torch.uint8, device="cuda")
        cfg.ext_state, cfg.ext_state_bytes = self.state.data_ptr(), state
        cfg.ext_psi, cfg.ext_psi_bytes = self.psi.data_ptr(), psi
        cfg.stream = torch.cuda.current_stream().cuda_stream or 1
        self.shape = (case["nz"], case["ny"], case["nx"])
        self.h = lbm.lbm_create_ex(cfg)
        # after an even number of steps population a of node i is element a N + i of the first array
        n = Q * case["nx"] * case["ny"] * case["nz"] * ELEM[case.get("precision", "f64")]
        self.f = self.state[:n].view(TORCH[case.get("precision", "f64")]).view((Q,) + self.shape)

    def __del__(self):
        if getattr(self, "h", None):
            lbm.lbm_destroy(self.h)
            self.h = None


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        insts = _instances(case, seed)
        b = lbm.Batch(insts, precision=case["precision"])
        b.init()
        return case, b
    lat = _Lattice(case)
    if kind == "droplets":
        lbm.lbm_set_populations(lat.h, _drop_populations(case, seed).cpu().numpy())
        lbm.lbm_set_option(lat.h, "rho_l", RHO_L)
        lbm.lbm_set_option(lat.h, "rho_v", RHO_V)
        return case, lat
    p = _ligament(case, seed)
    lbm.lbm_init_ligament(lat.h, p["R0"], p["lam"], p["eps"], p["phase"], *_fluid(case)[1:], WIDTH)
    if kind == "steps":
        if case["collision"] == "mrt":
            lbm.lbm_set_option(lat.h, "collision", 1)
        lbm.lbm_set_option(lat.h, "diag_interval", case["diag"])
    return case, lat


_REAL = ("mass", "mom", "liquid_volume_w", "min_slice_area_w", "neck_radius", "max_u", "rho_min", "rho_max")
_WHOLE = ("liquid_count", "min_slice_count", "min_slice_x", "numeric_ok")


def _records(recs, whole=_WHOLE):
    """Diagnostics records as an array of their sums and extrema and one of their counts."""
    real = [[v for k in _REAL for v in (r[k] if k == "mom" else (r[k],))] for r in recs]
    return np.array(real, dtype=np.float64), np.array([[r[k] for k in whole] for r in recs], dtype=np.int64)


def run(state):
    case, s = state
    kind = case["kind"]
    if kind == "sweep":
        recs = []
        for _ in range(case["steps"] // case["check"]):
            s.step(case["check"])
            recs += [s.diagnostics(k) for k in range(case["count"])]
        real, whole = _records(recs)
        return {"f": [s.populations(k) for k in range(case["count"])], "real": real, "whole": whole}
    if kind == "cylinder":
        lbm.lbm_step(s.h, case["steps"])
        return {"f": s.f, "rho": lbm.lbm_moments(s.h, s.shape, ("rho",))["rho"]}
    if kind == "droplets":
        real, whole = _records([lbm.lbm_diagnostics(s.h, True).as_dict()],
                               _WHOLE + ("droplets", "droplets_min8", "largest_droplet"))
        count, drops = lbm.lbm_droplets(s.h)
        return {"real": real, "whole": whole, "count": count,
                "drops": np.array([[d.volume_w, d.mass, *d.centroid, *d.resultant] for d in drops]),
                "nodes": np.array([[d.first_node, d.nodes, d.x_slices] for d in drops], dtype=np.int64)}
    lbm.lbm_step(s.h, case["steps"])
    real, whole = _records(lbm.lbm_diag_history(s.h))
    return {"f": s.f, "real": real, "whole": whole}


def work(case):
    """Every step reads and writes each population once; about 250 operations
    update a node.  The droplet statistics read each population once."""
    if case["kind"] == "sweep":
        n = sum(i["nx"] * i["ny"] * i["nz"] for i in _instances(case, 0))
        return {"bytes": 2.0 * Q * ELEM[case["precision"]] * n * case["steps"] + 8.0 * Q * n,
                "flops": 250.0 * n * case["steps"]}
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "droplets":
        return {"bytes": float(Q * ELEM[case["precision"]] * n), "flops": 40.0 * n}
    e = ELEM[case.get("precision", "f64")]
    out = 8.0 * n if case["kind"] == "cylinder" else 0.0
    return {"bytes": 2.0 * Q * e * n * case["steps"] + out, "flops": 250.0 * n * case["steps"]}


# ---- the method in 64 bits ------------------------------------------------------

def _lattice():
    axis = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    diag = [(1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
    c = [(0, 0, 0)]
    for v in axis + diag:
        c += [v, tuple(-k for k in v)]
    return c, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _shift(t, v, sign):
    """t at x - sign v (periodic), t[nz, ny, nx]."""
    moved = [(sign * v[k], 2 - k) for k in range(3) if v[k]]
    return torch.roll(t, [m[0] for m in moved], [m[1] for m in moved]) if moved else t


def _moments(f, c):
    rho = f[0].clone()
    for a in range(1, Q):
        rho += f[a]
    j = []
    for k in range(3):
        s = torch.zeros_like(rho)
        for a in range(1, Q):
            if c[a][k]:
                s += c[a][k] * f[a]
        j.append(s)
    return rho, j


def _mrt_matrix(c):
    v = np.array(c, dtype=np.float64)
    x, y, z = v.T
    s = (v * v).sum(1)
    p, q = 5 * s - 9, 3 * s - 5
    return np.array([np.ones(Q), 19 * s - 30, (21 * s * s - 53 * s + 24) / 2, x, p * x, y, p * y, z, p * z,
                     3 * x * x - s, q * (3 * x * x - s), y * y - z * z, q * (y * y - z * z), x * y, y * z, x * z,
                     (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z])


def _step64(f, G, tau, mrt):
    """One step of populations f[19, nz, ny, nx] (a list of FP64 fields), in place of them."""
    c, w = _lattice()
    rho, j = _moments(f, c)
    psi = 1.0 - torch.exp(-rho)
    F = [torch.zeros_like(rho) for _ in range(3)]
    for a in range(1, Q):
        p = w[a] * _shift(psi, c[a], -1)
        for k in range(3):
            if c[a][k]:
                F[k] += c[a][k] * p
    for k in range(3):
        F[k] *= -G * psi
    shift = 0.5 if mrt else tau
    u = [(j[k] + shift * F[k]) / rho for k in range(3)]
    if mrt:
        M = _mrt_matrix(c)
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        nu = 1.0 / tau
        rates = [0, 1.19, 1.4, 0, 1.2, 0, 1.2, 0, 1.2, nu, 1.4, nu, 1.4, nu, nu, nu, 1.98, 1.98, 1.98]
        cu = [sum(c[a][k] * u[k] for k in range(3) if c[a][k]) + torch.zeros_like(rho) for a in range(Q)]
        ms = []
        for k in range(Q):
            m = sum(float(M[k][a]) * f[a] for a in range(Q) if M[k][a])
            eq = src = 0
            for a in range(Q):
                if M[k][a]:
                    cF = sum(c[a][i] * F[i] for i in range(3) if c[a][i])
                    eq = eq + float(M[k][a]) * w[a] * rho * (1 + 3 * cu[a] + 4.5 * cu[a] ** 2 - 1.5 * uu)
                    src = src + float(M[k][a]) * w[a] * (3 * (cF - uF) + 9 * cu[a] * cF)
            ms.append((m - rates[k] * (m - eq) + (1 - 0.5 * rates[k]) * src) / float((M[k] ** 2).sum()))
        del cu
        new = []
        for a in range(Q):
            new.append(_shift(sum(float(M[k][a]) * ms[k] for k in range(Q) if M[k][a]), c[a], 1))
        return new
    usq = 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    for a in range(Q):
        cu = sum(c[a][k] * u[k] for k in range(3) if c[a][k]) + torch.zeros_like(rho)
        feq = w[a] * rho * (1 + 3 * cu + 4.5 * cu * cu - usq)
        f[a] = _shift(f[a] + (feq - f[a]) / tau, c[a], 1)
    return f


def _shifts(precision, w, rho_v):
    """The deviation shift of each population: w_a rho_v rounded to the storage type."""
    if not precision.endswith("dev"):
        return [0.0] * Q
    return [float(torch.tensor(v * rho_v, dtype=torch.float32).to(TORCH[precision])) for v in w]


def _start64(nx, ny, nz, p, precision, rho_l, rho_v):
    """The ligament's populations as stored: w_a rho, rounded to the storage type."""
    f64 = dict(dtype=torch.float64, device="cuda")
    x, y, z = (torch.arange(n, **f64) for n in (nx, ny, nz))
    R = p["R0"] * (1.0 + p["eps"] * torch.cos(2 * math.pi * x / p["lam"] + p["phase"]))
    r = torch.sqrt((y - 0.5 * (ny - 1))[None, :] ** 2 + (z - 0.5 * (nz - 1))[:, None] ** 2)
    rho = rho_v + 0.5 * (rho_l - rho_v) * (1.0 - torch.tanh(2.0 * (r[:, :, None] - R) / WIDTH))
    w = _lattice()[1]
    s = _shifts(precision, w, rho_v)
    if precision == "f64":
        return [w[a] * rho for a in range(Q)]
    return [((w[a] * rho).float() - s[a]).to(TORCH[precision]).double() + s[a] for a in range(Q)]


def _record64(f, rho_l, rho_v):
    c, _ = _lattice()
    rho, j = _moments(f, c)
    phi = ((rho - rho_v) / (rho_l - rho_v)).clamp(0, 1)
    area = float(phi.sum((0, 1)).min())
    u = torch.sqrt(j[0] ** 2 + j[1] ** 2 + j[2] ** 2) / rho
    return [float(v) for v in (rho.sum(), j[0].sum(), j[1].sum(), j[2].sum(), phi.sum(), area,
                               math.sqrt(area / math.pi), u.max(), rho.min(), rho.max())]


def exact(case, seed):
    kind = case["kind"]
    c, w = _lattice()
    if kind == "sweep":
        out, recs = [], []
        for i in _instances(case, seed):
            f = _start64(i["nx"], i["ny"], i["nz"], i, case["precision"], RHO_L, RHO_V)
            recs.append([])
            for t in range(1, case["steps"] + 1):
                f = _step64(f, G, i["tau"], False)
                if t % case["check"] == 0:
                    recs[-1].append(_record64(f, RHO_L, RHO_V))
            out.append(torch.stack(f).cpu().numpy())
        return {"f": out, "real": np.array([r[t] for t in range(len(recs[0])) for r in recs]), "whole": None}
    if kind == "droplets":
        s = _shifts(case["precision"], w, RHO_V)
        f = _drop_populations(case, seed)
        if case["precision"] != "f64":
            f = [(f[a].float() - s[a]).to(TORCH[case["precision"]]).double() + s[a] for a in range(Q)]
        rho, _ = _moments(f, c)
        _, who = _drop_distance(case, seed)
        liquid = rho > 0.5 * (RHO_L + RHO_V)
        phi = ((rho - RHO_V) / (RHO_L - RHO_V)).clamp(0, 1)
        dims = (case["nx"], case["ny"], case["nz"])
        rows = []
        for k in range(case["drops"]):
            at = torch.nonzero(liquid & (who == k))
            n = at.shape[0]
            if not n:
                continue
            row = [float(phi[tuple(at.T)].sum()), float(rho[tuple(at.T)].sum())]
            place, length = [], []
            for axis in range(3):
                t = 2 * math.pi / dims[axis] * at[:, 2 - axis].double()
                cs, sn = float(torch.cos(t).sum()), float(torch.sin(t).sum())
                place.append(math.atan2(sn, cs) % (2 * math.pi) / (2 * math.pi) * dims[axis])
                length.append(math.hypot(cs, sn) / n)
            first = int((at[:, 2] + dims[0] * (at[:, 1] + dims[1] * at[:, 0])).min())
            rows.append((-n, first, row + place + length))
        rows.sort(key=lambda r: r[:2])
        return {"real": np.array([_record64(f, RHO_L, RHO_V)]), "whole": None, "count": None,
                "drops": np.array([r[2] for r in rows]), "nodes": None}
    precision = case.get("precision", "f64")
    g, rho_l, rho_v = _fluid(case)
    f = _start64(case["nx"], case["ny"], case["nz"], _ligament(case, seed), precision, rho_l, rho_v)
    recs = []
    for t in range(case["steps"]):
        if kind == "steps" and t % case["diag"] == 0:
            recs.append(_record64(f, rho_l, rho_v))
        f = _step64(f, g, case["tau"], case.get("collision") == "mrt")
    if kind == "cylinder":
        return {"f": torch.stack(f), "rho": _moments(f, c)[0].cpu().numpy()}
    s = _shifts(precision, w, rho_v)
    for a in range(Q):
        f[a] -= s[a]
    return {"f": torch.stack(f), "real": np.array(recs), "whole": None}
