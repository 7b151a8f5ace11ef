"""Performance cases: the work this library is used for, through its public entry points.

Every case is a whole call of a user's program: inputs and structure are in hand (prepare), one
pass (run) starts from the initial values, takes a number of steps through the queue and reads the
result back the way the binding offers it (particle arrays stay on the device, where the caller
owns them).  The kinds of work:

  shell    the tiny shell: every step re-activates, lists, diffuses and swaps (launch-bound)
  band     fused diffusion of a narrow band: clear, 7-point, 27-point, swap, sum
  rebuild  a band whose structure changes before every step: deactivate, activate, list, fill, step
  ew       element-wise struct-for programs (saxpy, chained copies, squares with their sum)
  batch    many uneven grids stepped by one launch
  serve    a batch of diffusion jobs of mixed sizes through the continuous-batching server
  pic      particles: deactivate, P2G with activation, grid update, G2P (PIC or APIC with C stored)
  mpm      the same with the fused G2P2G over two grids, C never stored
  tube     MacCormack / RK3 advection of scalar channels through a swirling tube
  vcycle   a four-level V-cycle: restrict, smooth, prolong
"""
import math

import numpy as np
import torch

import paper_2012_08141_gb300 as sg
from paper_2012_08141_gb300.serve import Server

COEF = 0.1
DEV = "cuda"


# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: a 64^3 shell of a few leaves, twenty steps, every step re-activated
        {"name": "shell64", "kind": "shell", "n": 64, "r": 24.0, "h": 2.0, "steps": 20},
        # the headline workload: 512^3 band of 8M voxels, one hundred fused steps
        {"name": "band512", "kind": "band", "n": 512, "r": 200.0, "h": 8.0, "steps": 100},
        # a band far larger than L2, on an odd number of root cells along an edge
        {"name": "band1000", "kind": "band", "n": 1000, "r": 390.0, "h": 8.0, "steps": 40},
        # a moving interface at scale: the structure changes before every step
        {"name": "rebuild1024", "kind": "rebuild", "n": 1024, "r": 400.0, "h": 8.0, "steps": 8},
        # element-wise programs on a medium band with an odd root edge
        {"name": "saxpy440", "kind": "ew", "n": 440, "r": 190.0, "h": 8.0, "program": "saxpy", "steps": 20},
        # sixty-four independent grids of very different sizes in one launch per step
        {"name": "batch64", "kind": "batch", "grids": 64, "lo": 1e3, "hi": 5e6, "steps": 20},
        # a burst of requests served together: mixed sizes and step counts
        {"name": "serve24", "kind": "serve", "jobs": 24, "lo": 1e4, "hi": 3e6, "steps_lo": 10, "steps_hi": 100},
        # the particle workload: 2M particles in three spheres, PIC transfers
        {"name": "pic2m", "kind": "pic", "n": 256, "leaf_log2": 2, "particles": 2_000_000, "affine": False, "steps": 10},
        # a small particle simulation with stored affine matrices on a ragged grid
        {"name": "apic100k", "kind": "pic", "n": 100, "leaf_log2": 2, "particles": 100_003, "affine": True, "steps": 10},
        # MLS-MPM substeps between two binnings: fused G2P2G
        {"name": "mpm2m", "kind": "mpm", "n": 256, "leaf_log2": 2, "particles": 2_000_000, "steps": 10},
        # advection of temperature, colour and density through a tube
        {"name": "tube256", "kind": "tube", "n": 256, "channels": 3, "steps": 6},
        # the multigrid pattern: V-cycles from the 512^3 band
        {"name": "vcycle512", "kind": "vcycle", "n": 512, "r": 200.0, "h": 8.0, "steps": 10},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["shell", "band", "band", "rebuild", "ew", "batch", "serve", "pic", "pic", "mpm", "tube", "vcycle"])
    if kind == "shell":
        n = 8 * rng.randint(6, 14)
        return {"kind": kind, "n": n, "r": round(n * rng.uniform(0.3, 0.42), 2), "h": rng.choice([1.5, 2.0, 3.0]), "steps": rng.randint(10, 20)}
    if kind in ("band", "rebuild", "ew"):
        n = 8 * int(round(_log(rng, 96, 1000) / 8))
        c = {"kind": kind, "n": n, "r": round(n * rng.uniform(0.3, 0.4), 2), "h": rng.choice([4.0, 6.0, 8.0])}
        if kind == "ew":
            c["n"], c["r"] = min(n, 640), round(min(n, 640) * 0.4, 2)
            c["program"] = rng.choice(["saxpy", "copies", "squares"])
        return dict(c, steps=rng.randint(4, 8) if kind == "rebuild" else rng.randint(10, 40))
    if kind == "batch":
        return {"kind": kind, "grids": rng.randint(3, 60), "lo": 1e3, "hi": round(_log(rng, 1e5, 5e6)), "steps": rng.randint(8, 20)}
    if kind == "serve":
        return {"kind": kind, "jobs": rng.randint(4, 24), "lo": 1e4, "hi": round(_log(rng, 1e5, 3e6)), "steps_lo": 10, "steps_hi": rng.randint(20, 100)}
    if kind in ("pic", "mpm"):
        n = 4 * rng.randint(16, 64)
        c = {"kind": kind, "n": n if n % 8 == 0 else n + 4, "leaf_log2": rng.choice([2, 2, 3]), "steps": rng.randint(4, 10),
             "particles": int(min(_log(rng, 2e4, 2e6), 0.12 * n ** 3 + 2e4))}
        return dict(c, affine=rng.random() < 0.5) if kind == "pic" else c
    if kind == "tube":
        return {"kind": kind, "n": 8 * rng.randint(8, 32), "channels": rng.randint(1, 3), "steps": rng.randint(2, 6)}
    n = 64 * rng.randint(2, 8)
    return {"kind": kind, "n": n, "r": round(n * rng.uniform(0.3, 0.4), 2), "h": rng.choice([6.0, 8.0]), "steps": rng.randint(4, 10)}


# ---------------------------------------------------------------------------------------------
# Bands: bounds, sizes, initial values
# ---------------------------------------------------------------------------------------------

def _bounds(r, h):
    """|dist - r| < h as the library takes it: lo2 < D < hi2, D = 4 dist^2."""
    return int(round(4.0 * (r - h) ** 2)), int(round(4.0 * (r + h) ** 2)), True


def _band_for(count, h=8.0):
    """Domain edge and bounds of a band (or ball) of about `count` active voxels."""
    r = math.sqrt(count / (8.0 * math.pi * h))
    if r > 2.0 * h:
        return (int(8 * math.ceil((2.0 * (r + h) + 4.0) / 8)),) + _bounds(r, h)
    r = (3.0 * count / (4.0 * math.pi)) ** (1.0 / 3.0)
    return int(8 * math.ceil((2.0 * r + 4.0) / 8)), 0, int(math.ceil(4.0 * r * r)), False


def _leaf_bound(n, lo2, hi2, L=8):
    """How many leaves the band can touch (a pool size a caller would choose)."""
    d = (2 * np.arange(n, dtype=np.int64) + 1 - n) ** 2
    a = d.reshape(n // L, L)
    lo, hi = a.min(1), a.max(1)
    near = lo[:, None, None] + lo[None, :, None] + lo[None, None, :]
    far = hi[:, None, None] + hi[None, :, None] + hi[None, None, :]
    return max(1, int(np.count_nonzero((near < hi2) & (far >= lo2))))


def _band_grid(n, bounds, fields, scratch=0, sums=1, leaves=None):
    g = sg.Grid(n, 3, fields, max_leaves=leaves or _leaf_bound(n, bounds[0], bounds[1]), max_sums=sums, scratch_mask=scratch)
    g.activate_shell(*bounds)
    g.list_gen()
    return g


def _pinned(count):
    return torch.zeros(max(1, int(count)), dtype=torch.float32).pin_memory().numpy()


def _mix(case, seed):
    """(edge, lo2, hi2, strict) of log-uniform active counts, and step counts."""
    rng = np.random.default_rng(seed)
    m = case["grids"] if case["kind"] == "batch" else case["jobs"]
    # sizes are the case's own (one size mix), values come from the seed
    sizes = np.random.default_rng(7)
    specs = [_band_for(float(c)) for c in np.exp(sizes.uniform(math.log(case["lo"]), math.log(case["hi"]), size=m))]
    steps = [int(s) for s in sizes.integers(case.get("steps_lo", 1), case.get("steps_hi", 1) + 1, size=m)]
    return specs, steps, [int(s) for s in rng.integers(0, 1 << 24, size=m)]


def _spheres(case, seed):
    """Particles uniform in three spheres of the unit cube, N(0, 0.1) velocities."""
    rng = np.random.default_rng(seed)
    n, count = case["n"], case["particles"]
    m = 3.0 / n
    radii = rng.uniform(0.05, 0.15, size=3)
    centers = np.stack([rng.uniform(m + r, 1.0 - m - r, size=3) for r in radii])
    share = np.floor(count * radii ** 3 / (radii ** 3).sum()).astype(int)
    share[0] += count - share.sum()
    which = torch.from_numpy(np.repeat(np.arange(3), share)).to(DEV)
    gen = torch.Generator(DEV).manual_seed(seed)
    which = which[torch.randperm(count, generator=gen, device=DEV)]
    d = torch.randn(count, 3, generator=gen, device=DEV, dtype=torch.float64)
    d /= d.norm(dim=1, keepdim=True)
    rad = torch.from_numpy(radii).to(DEV)[which] * torch.rand(count, generator=gen, device=DEV, dtype=torch.float64) ** (1.0 / 3.0)
    x = (torch.from_numpy(centers).to(DEV)[which] + d * rad[:, None]).float().contiguous()
    v = (0.1 * torch.randn(count, 3, generator=gen, device=DEV)).contiguous()
    C = (5.0 * torch.randn(count, 9, generator=gen, device=DEV)).contiguous() if case["kind"] == "mpm" or case.get("affine") else None
    return x, v, C


DT, GRAVITY, BOUND = 1e-4, 9.8, 3


def _node_bound(case, x):
    """Pool size for the leaves that the particles' stencils can touch while they move a little."""
    L = 1 << case["leaf_log2"]
    R = case["n"] // L
    b = (x * (case["n"] / L)).floor().long().clamp_(0, R - 1)
    grid = torch.zeros(1, 1, R, R, R, device=DEV)
    grid[0, 0, b[:, 0], b[:, 1], b[:, 2]] = 1.0
    return int(torch.nn.functional.max_pool3d(grid, 3, 1, 1).sum().item())


def _tube(n):
    return math.ceil(4.0 * n * n * 0.32 ** 2), math.ceil(4.0 * n * n * 0.45 ** 2)


def _tube_fields(n, cells, seed, channels):
    """Swirl plus axial drift, and smooth scalar channels, at cell centres; phases from the seed."""
    ph = np.random.default_rng(seed).uniform(0, 2 * math.pi, size=3)
    x, y, z = [(cells[..., a].double() + 0.5) / n for a in range(3)]
    tp = 2 * math.pi
    vel = [-2.0 * (y - 0.5), 2.0 * (x - 0.5), torch.full_like(x, 0.3)]
    ch = [0.5 + 0.5 * torch.sin(tp * x + ph[0]) * torch.cos(tp * y),
          0.5 + 0.4 * torch.sin(2 * tp * z + ph[1]) * torch.sin(tp * (x + y)),
          torch.exp(-((x - 0.5) ** 2 + (y - 0.88) ** 2 + (z - 0.5) ** 2) / 0.01) + 0.1 * torch.sin(tp * z + ph[2])]
    return [v.float() for v in vel], [c.float() for c in ch[:channels]]


def _channel(c):
    return 3 + 4 * c, 4 + 4 * c, 5 + 4 * c, 6 + 4 * c


# ---------------------------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------------------------

def prepare(case, seed):
    s = {"case": case, "kind": case["kind"], "seed": seed % (1 << 24)}
    k = case["kind"]
    if k in ("shell", "band", "ew"):
        b = s["bounds"] = _bounds(case["r"], case["h"])
        fields = {"shell": 2, "band": 3, "ew": 5}[k]
        g = s["grid"] = _band_grid(case["n"], b, fields, scratch={"shell": 0, "band": 0b010, "ew": 0b01000}[k], sums=max(1, case["steps"]))
        s["out"] = _pinned(g.num_active())
    elif k == "rebuild":
        # two positions of the moving interface
        s["bands"] = [_bounds(case["r"] + d, case["h"]) for d in (0.0, 1.0)]
        leaves = max(_leaf_bound(case["n"], b[0], b[1]) for b in s["bands"])
        g = s["grid"] = _band_grid(case["n"], s["bands"][(case["steps"] - 1) % 2], 3, scratch=0b010, sums=case["steps"], leaves=leaves)
        s["out"] = _pinned(g.num_active())
    elif k == "batch":
        specs, _, seeds = _mix(case, seed)
        s["grids"], s["slices"], at = [], [], 0
        for (n, lo2, hi2, strict), v in zip(specs, seeds):
            g = _band_grid(n, (lo2, hi2, strict), 3, scratch=0b010)
            g.fill_hash(0, v)
            s["grids"].append(g)
            s["slices"].append((at, at + g.num_active()))
            at = (s["slices"][-1][1] + 3) // 4 * 4
        s["out"] = _pinned(at)
        s["batch"] = sg.Batch(s["grids"], 0, 1, 2, COEF)
    elif k == "serve":
        specs, steps, seeds = _mix(case, seed)
        s["server"] = Server(max_jobs=64, warps_per_cta=4, hbm_reserve=8 << 30, coef=COEF)
        s["jobs"], at = [], 0
        for (n, lo2, hi2, strict), m, v in zip(specs, steps, seeds):
            count = int(_mask(n, lo2, hi2, strict).sum().item())
            s["jobs"].append((_Job(n, lo2, hi2, strict, v), m, at, at + count))
            at = (at + count + 3) // 4 * 4
        s["out"] = _pinned(at)
    elif k in ("pic", "mpm"):
        s["x0"], s["v0"], s["C0"] = _spheres(case, seed)
        s["x"], s["v"] = torch.empty_like(s["x0"]), torch.empty_like(s["v0"])
        leaves = _node_bound(case, s["x0"])
        grids = 2 if k == "mpm" else 1
        s["grids"] = [sg.Grid(case["n"], case["leaf_log2"], 4, max_leaves=leaves) for _ in range(grids)]
        if k == "pic" and case["affine"]:
            s["C"] = torch.empty_like(s["C0"])
    elif k == "tube":
        n, m = case["n"], case["channels"]
        lo2, hi2 = _tube(n)
        R = n // 8
        d = (2 * np.arange(n, dtype=np.int64) + 1 - n) ** 2
        a = d.reshape(R, 8)
        leaves = R * int(np.count_nonzero((a.min(1)[:, None] + a.min(1)[None, :] < hi2) & (a.max(1)[:, None] + a.max(1)[None, :] >= lo2)))
        g = s["grid"] = sg.Grid(n, 3, 3 + 4 * m, max_leaves=leaves, scratch_mask=sum(1 << _channel(c)[2] for c in range(m)))
        g.activate_tube(lo2, hi2)
        b, _ = g.read_structure()
        b = torch.from_numpy(b.astype(np.int64)).to(DEV)
        l = torch.arange(512, device=DEV)
        cells = torch.stack([(b // (R * R))[:, None] * 8 + l // 64, (b // R % R)[:, None] * 8 + l // 8 % 8, (b % R)[:, None] * 8 + l % 8], -1)
        vel, ch = _tube_fields(n, cells, seed, m)
        for a in range(3):
            g.write_field(a, vel[a].cpu().contiguous())
        for c in range(m):
            g.write_field(_channel(c)[0], ch[c].cpu().contiguous())
        count = g.num_active()
        s["outs"] = [_pinned(count) for _ in range(m)]
    elif k == "vcycle":
        b = _bounds(case["r"], case["h"])
        leaves = _leaf_bound(case["n"], b[0], b[1])
        G = s["grids"] = [sg.Grid(case["n"] >> l, 3, 3, max_leaves=leaves) for l in range(4)]
        G[0].activate_shell(*b)
        G[0].fill_hash(0, s["seed"])
        _vcycle(G)  # the first cycle activates the coarse levels
        for g in G:
            g.sync()
        s["out"] = _pinned(G[0].num_active())
    return s


class _Job:
    """The band of one served job, as Server.submit takes it."""

    def __init__(self, n, lo2, hi2, strict, seed):
        self.N, self.lo2, self.hi2, self.lo_strict, self.seed = n, lo2, hi2, strict, seed


def _vcycle(G):
    for l in range(3):
        G[l + 1].clear(1)
        G[l].restrict_to(G[l + 1], 0, 1, 0.125)
        G[l + 1].diffuse7(1, 0, COEF)
    for l in (2, 1, 0):
        G[l].prolong_from(G[l + 1], 0, 0, 0.5)
        G[l].diffuse7(0, 2, COEF)
        G[l].swap(0, 2)
    for g in G:
        g.flush()


def _fused_step(g, slot):
    g.clear(1)
    g.diffuse7(0, 1, COEF)
    g.box27(1, 2)
    g.swap(0, 2)
    g.reduce_sum(0, slot)
    g.flush()


_PROGRAMS = {
    # (fields 0 x, 1 y, 2 z, 3 scratch, 4 gradient)
    "saxpy": lambda g, s: (g.ew(2, 0, 1, 2.0, 1.0), g.ew(1, 2, 0, 0.25, 1.0), g.ew(2, 2, 1, 1.0, 1.0)),
    "copies": lambda g, s: (g.ew(1, 0, alpha=1.0, delta=1.0), g.ew(2, 1, alpha=1.0, delta=4.0), g.ew(0, 0, 2, 0.5, 0.25)),
    "squares": lambda g, s: (g.ew(3, 0, 0, gamma=1.0), g.reduce_sum(3, s), g.ew(4, 4, 0, 1.0, 2.0), g.ew(2, 4, delta=1.0, alpha=0.5)),
}


def run(s):
    c, k = s["case"], s["kind"]
    if k == "shell":
        g = s["grid"]
        g.fill_hash(0, s["seed"])
        for _ in range(c["steps"]):
            g.activate_shell(*s["bounds"])
            g.list_gen()
            g.diffuse7(0, 1, COEF)
            g.swap(0, 1)
            g.flush()
        return {"x": g.read_field_active(0, out=s["out"])}
    if k == "band":
        g = s["grid"]
        g.fill_hash(0, s["seed"])
        for i in range(c["steps"]):
            _fused_step(g, i)
        return {"sums": g.read_sums(c["steps"]), "x": g.read_field_active(0, out=s["out"])}
    if k == "rebuild":
        g = s["grid"]
        for i in range(c["steps"]):
            g.deactivate_all()
            g.activate_shell(*s["bands"][i % 2])
            g.list_gen()
            g.fill_hash(0, (s["seed"] + i) % (1 << 24))
            _fused_step(g, i)
        return {"sums": g.read_sums(c["steps"]), "x": g.read_field_active(0, out=s["out"])}
    if k == "ew":
        g, body = s["grid"], _PROGRAMS[c["program"]]
        g.fill_hash(0, s["seed"])
        g.fill_hash(1, (s["seed"] + 1) % (1 << 24))
        g.ew(4, delta=0.0)
        for i in range(c["steps"]):
            body(g, i)
            g.flush()
        out = {"z": g.read_field_active(2, out=s["out"])}
        if c["program"] == "squares":
            out["sums"] = g.read_sums(c["steps"])
        return out
    if k == "batch":
        for _ in range(c["steps"]):
            s["batch"].step()
        sums = s["batch"].read_sums()
        for g, (a, b) in zip(s["grids"], s["slices"]):
            g.read_field_active(0, out=s["out"][a:b])
        return {"sums": sums, "x": s["out"]}
    if k == "serve":
        srv = s["server"]
        ids = [srv.submit(job, m, out=s["out"][a:b]) for job, m, a, b in s["jobs"]]
        while True:
            st = srv.stats()
            if not st["resident"] and not st["pending"]:
                break
            srv.tick()
        sums = np.array([srv.job(i)["sum"] for i in ids])
        for i in ids:
            srv.release(i)
        return {"sums": sums, "x": s["out"]}
    if k == "pic":
        g, x, v, C = s["grids"][0], s["x"], s["v"], s.get("C")
        x.copy_(s["x0"])
        v.copy_(s["v0"])
        if C is not None:
            C.copy_(s["C0"])
        for _ in range(c["steps"]):
            g.deactivate_all()
            if C is None:
                g.p2g(x, v, 1.0, 0, 1)
            else:
                g.p2g_apic(x, v, C, 1.0, 0, 1)
            g.grid_update(0, 1, DT, GRAVITY, BOUND)
            if C is None:
                g.g2p(x, v, DT, 1)
            else:
                g.g2p_apic(x, v, C, DT, 1)
            g.flush()
        g.sync()
        return {"x": x, "v": v} if C is None else {"x": x, "v": v, "C": C}
    if k == "mpm":
        src, dst = s["grids"]
        x, v = s["x"], s["v"]
        x.copy_(s["x0"])
        v.copy_(s["v0"])
        src.deactivate_all()
        src.p2g_apic(x, v, s["C0"], 1.0, 0, 1)
        src.grid_update(0, 1, DT, GRAVITY, BOUND)
        for _ in range(c["steps"]):
            dst.deactivate_all()
            src.g2p2g(dst, x, v, DT, 1, 1.0, 0, 1)
            dst.grid_update(0, 1, DT, GRAVITY, BOUND)
            dst.flush()
            src, dst = dst, src
        for g in s["grids"]:
            g.sync()
        return {"x": x, "v": v}
    if k == "tube":
        g, dt = s["grid"], 1.0 / c["n"]
        for _ in range(c["steps"]):
            for a in range(c["channels"]):
                q, qh, qt, qn = _channel(a)
                g.advect(qh, q, 0, dt)
                g.advect(qt, qh, 0, -dt)
                g.maccormack(qn, q, qh, qt, 0, dt)
                g.swap(q, qn)
            g.flush()
        return [g.read_field_active(_channel(a)[0], out=s["outs"][a]) for a in range(c["channels"])]
    G = s["grids"]
    G[0].fill_hash(0, s["seed"])
    for _ in range(c["steps"]):
        _vcycle(G)
    return {"x": G[0].read_field_active(0, out=s["out"])}


# ---------------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------------

def _volume(lo2, hi2):
    """Active voxels of a band, to a fraction of a per cent."""
    return 4.0 / 3.0 * math.pi * ((hi2 / 4.0) ** 1.5 - (lo2 / 4.0) ** 1.5)


def work(case):
    """Active voxels' values read once and written once per step, results written out once."""
    k, m = case["kind"], case.get("steps", 1)
    if k in ("batch", "serve"):
        specs, steps, _ = _mix(case, 0)
        vs = [_volume(lo2, hi2) for _, lo2, hi2, _ in specs]
        vox = sum(v * (m if k == "batch" else t) for v, t in zip(vs, steps))
        return {"bytes": 8 * vox + 4 * sum(vs), "flops": 35 * vox}
    if k in ("pic", "mpm"):
        p = case["particles"]
        per = 48 + (72 if case.get("affine") else 0)
        return {"bytes": m * p * per, "flops": m * p * 27 * (34 if k == "mpm" or case.get("affine") else 16)}
    if k == "tube":
        vox = math.pi * (0.45 ** 2 - 0.32 ** 2) * case["n"] ** 3
        ch = case["channels"]
        # velocity, the channels in and out; two backtraces and 3 samples a channel
        return {"bytes": m * vox * 4 * (3 + 2 * ch) + 4 * vox * ch, "flops": m * vox * (2 * 2 * 3 * 15 + 3 * ch * 15)}
    lo2, hi2, _ = _bounds(case["r"], case["h"])
    vox = _volume(lo2, hi2)
    per, flops = {"shell": (8, 8), "band": (8, 35), "rebuild": (8, 35), "ew": (16, 8), "vcycle": (8 * 4, 40)}[k]
    return {"bytes": m * vox * per + 4 * vox, "flops": m * vox * flops}


# ---------------------------------------------------------------------------------------------
# exact: the same definitions in 64 bits with plain torch
# ---------------------------------------------------------------------------------------------

def _mask(n, lo2, hi2, strict):
    """Dense active set of a band."""
    d = (2 * torch.arange(n, device=DEV, dtype=torch.int32) + 1 - n) ** 2
    m = torch.empty(n, n, n, dtype=torch.bool, device=DEV)
    jk = d[:, None] + d[None, :]
    for i in range(n):
        D = jk + d[i]
        m[i] = ((D > lo2) if strict else (D >= lo2)) & (D < hi2)
    return m


def _leaf_order(a, L=8):
    R = a.shape[0] // L
    return a.view(R, L, R, L, R, L).permute(0, 2, 4, 1, 3, 5).reshape(-1)


def _packed(a, mask):
    """Active values in list order: leaves by root index, voxels by mask bit."""
    return _leaf_order(a)[_leaf_order(mask)]


def _hash_values(seed, n, mask=None):
    """The library's documented initial values, top24(splitmix64) * 2^-24, dense (0 outside mask)."""
    def shr(z, b):
        return (z >> b) & ((1 << (64 - b)) - 1)

    def i64(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    out = torch.empty(n, n, n, dtype=torch.float64, device=DEV)
    plane = torch.arange(n * n, device=DEV, dtype=torch.int64).view(n, n)
    for i in range(n):
        z = plane + ((seed << 40) + i * n * n) + i64(0x9E3779B97F4A7C15)
        z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
        z = z ^ shr(z, 31)
        out[i] = shr(z, 40).double() * 2.0 ** -24
    return out if mask is None else out.mul_(mask)


_C32 = float(np.float32(COEF))


def _shift_add(y, x, alpha=1.0):
    """y += alpha * (x at both neighbours along each axis)."""
    for a in range(3):
        n = x.shape[a]
        y.narrow(a, 1, n - 1).add_(x.narrow(a, 0, n - 1), alpha=alpha)
        y.narrow(a, 0, n - 1).add_(x.narrow(a, 1, n - 1), alpha=alpha)
    return y


def _diffuse(x, mask):
    return _shift_add(x * (1.0 - 6.0 * _C32), x, _C32).mul_(mask)


def _box(x, mask):
    for a in range(3):
        n = x.shape[a]
        y = x.clone()
        y.narrow(a, 1, n - 1).add_(x.narrow(a, 0, n - 1))
        y.narrow(a, 0, n - 1).add_(x.narrow(a, 1, n - 1))
        x = y
    return x.mul_(1.0 / 27.0).mul_(mask)


def _diffusion(n, bounds, seed, steps):
    mask = _mask(n, *bounds)
    x, sums = _hash_values(seed, n, mask), []
    for _ in range(steps):
        x = _box(_diffuse(x, mask), mask)
        sums.append(x.sum())
    return x, mask, sums


def _weights(X):
    base = torch.floor(X - 0.5)
    f = X - base
    return base.long(), f, torch.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2], 0)


def _stencil(x, n):
    """The 27 (node index, in-domain, weight, offset in cells) of every particle."""
    base, f, w = _weights(x * n)
    for a in range(3):
        for b in range(3):
            for c in range(3):
                o = torch.tensor([a, b, c], device=DEV)
                node = base + o
                inside = ((node >= 0) & (node < n)).all(1)
                node = node.clamp(0, n - 1)
                yield (node[:, 0] * n + node[:, 1]) * n + node[:, 2], inside, w[a, :, 0] * w[b, :, 1] * w[c, :, 2], o - f


def _p2g(x, v, C, n):
    grid = torch.zeros(n ** 3, 4, dtype=torch.float64, device=DEV)
    for idx, inside, w, d in _stencil(x, n):
        u = v if C is None else v + torch.bmm(C.view(-1, 3, 3), (d / n)[:, :, None])[:, :, 0]
        wm = w * inside
        grid.index_add_(0, idx, torch.cat([wm[:, None], wm[:, None] * u], 1))
    m = grid[:, :1]
    u = torch.where(m > 0, grid[:, 1:] / m.clamp_min(1e-300), 0.0)
    u[:, 2] -= torch.where(m[:, 0] > 0, DT * GRAVITY, 0.0)
    u = u.view(n, n, n, 3)
    for a in range(3):
        ua = u[..., a]
        lo, hi = ua.narrow(a, 0, BOUND), ua.narrow(a, n - BOUND + 1, BOUND - 1)
        lo.clamp_(min=0.0)
        hi.clamp_(max=0.0)
    return u.view(-1, 3)


def _g2p(grid, x, n, affine):
    v = torch.zeros_like(x)
    B = torch.zeros(x.shape[0], 3, 3, dtype=torch.float64, device=DEV)
    for idx, inside, w, d in _stencil(x, n):
        u = grid[idx] * (w * inside)[:, None]
        v += u
        if affine:
            B += u[:, :, None] * (d / n)[:, None, :]
    return x + DT * v, v, (4.0 * n * n * B).view(-1, 9) if affine else None


def _trilinear(fields, n, p):
    """Samples of dense padded fields (one cell of zeros outside the domain) at cell positions p, and the corner values' range."""
    X = p - 0.5
    b = torch.floor(X)
    f = X - b
    b = b.long()
    m = n + 2
    s = [0.0] * len(fields)
    lo, hi = [None] * len(fields), [None] * len(fields)
    for a in range(2):
        for c in range(2):
            for d in range(2):
                q = [(b[:, e] + o + 1).clamp_(0, m - 1) for e, o in enumerate((a, c, d))]
                idx = (q[0] * m + q[1]) * m + q[2]
                w = (f[:, 0] if a else 1 - f[:, 0]) * (f[:, 1] if c else 1 - f[:, 1]) * (f[:, 2] if d else 1 - f[:, 2])
                for e, fld in enumerate(fields):
                    val = fld.view(-1)[idx]
                    s[e] = s[e] + w * val
                    lo[e] = val if lo[e] is None else torch.minimum(lo[e], val)
                    hi[e] = val if hi[e] is None else torch.maximum(hi[e], val)
    return s, lo, hi


def _pad(a):
    return torch.nn.functional.pad(a, (1, 1, 1, 1, 1, 1))


def _exact_tube(case, seed):
    n, m = case["n"], case["channels"]
    lo2, hi2 = _tube(n)
    d = (2 * torch.arange(n, device=DEV) + 1 - n) ** 2
    D = d[:, None] + d[None, :]
    mask = ((D >= lo2) & (D < hi2))[:, :, None].expand(n, n, n).contiguous()
    i = torch.arange(n, device=DEV)
    cells = torch.stack(torch.meshgrid(i, i, i, indexing="ij"), -1)
    vel, ch = _tube_fields(n, cells, seed, m)
    at = mask.nonzero()
    del cells
    vel = [_pad(v.double() * mask) for v in vel]
    qs = [c.double() * mask for c in ch]
    x = at.double() + 0.5
    back = {}
    for sign in (1.0, -1.0):
        h = float(np.float32(sign / n)) * n
        k1 = torch.stack(_trilinear(vel, n, x)[0], 1)
        k2 = torch.stack(_trilinear(vel, n, x - 0.5 * h * k1)[0], 1)
        k3 = torch.stack(_trilinear(vel, n, x - 0.75 * h * k2)[0], 1)
        back[sign] = x - h * (2.0 * k1 + 3.0 * k2 + 4.0 * k3) / 9.0

    def dense(vals):
        o = torch.zeros(n, n, n, dtype=torch.float64, device=DEV)
        o[mask] = vals
        return o

    for _ in range(case["steps"]):
        for c in range(m):
            (qh,), (lo,), (hi,) = _trilinear([_pad(qs[c])], n, back[1.0])
            (qt,), _, _ = _trilinear([_pad(dense(qh))], n, back[-1.0])
            qs[c] = dense(torch.minimum(torch.maximum(qh + 0.5 * (qs[c][mask] - qt), lo), hi))
    return [_packed(q, mask) for q in qs]


def _exact_vcycle(case, seed):
    masks = [_mask(case["n"], *_bounds(case["r"], case["h"]))]
    for _ in range(3):
        masks.append(torch.nn.functional.max_pool3d(masks[-1][None, None].half(), 2)[0, 0] > 0)
    x = [_hash_values(seed, case["n"], masks[0])] + [None] * 3
    for _ in range(case["steps"]):
        for l in range(3):
            n = x[l].shape[0] // 2
            b = 0.125 * x[l].view(n, 2, n, 2, n, 2).sum((1, 3, 5))
            x[l + 1] = _diffuse(b, masks[l + 1])
        for l in (2, 1, 0):
            n = x[l + 1].shape[0]
            up = x[l + 1][:, None, :, None, :, None].expand(n, 2, n, 2, n, 2).reshape(2 * n, 2 * n, 2 * n)
            x[l] = _diffuse((x[l] + 0.5 * up).mul_(masks[l]), masks[l])
    return {"x": _packed(x[0], masks[0])}


def exact(case, seed):
    k, s24 = case["kind"], seed % (1 << 24)
    if k in ("shell", "band"):
        b = _bounds(case["r"], case["h"])
        if k == "band":
            x, mask, sums = _diffusion(case["n"], b, s24, case["steps"])
            return {"sums": torch.stack(sums).cpu(), "x": _packed(x, mask)}
        mask = _mask(case["n"], *b)
        x = _hash_values(s24, case["n"], mask)
        for _ in range(case["steps"]):
            x = _diffuse(x, mask)
        return {"x": _packed(x, mask)}
    if k == "rebuild":
        sums = []
        for i in range(case["steps"]):
            x, mask, one = _diffusion(case["n"], _bounds(case["r"] + i % 2, case["h"]), (s24 + i) % (1 << 24), 1)
            sums += one
        return {"sums": torch.stack(sums).cpu(), "x": _packed(x, mask)}
    if k == "ew":
        mask = _mask(case["n"], *_bounds(case["r"], case["h"]))
        x, y = _packed(_hash_values(s24, case["n"]), mask), _packed(_hash_values((s24 + 1) % (1 << 24), case["n"]), mask)
        z, grad, sums = None, torch.zeros_like(x), []
        for _ in range(case["steps"]):
            if case["program"] == "saxpy":
                z = 2.0 * x + y
                y = 0.25 * z + x
                z = z + y
            elif case["program"] == "copies":
                y = x + 1.0
                z = y + 4.0
                x = 0.5 * x + 0.25 * z
            else:
                sums.append((x * x).sum())
                grad = grad + 2.0 * x
                z = 0.5 * grad + 1.0
        return {"z": z, "sums": torch.stack(sums).cpu()} if sums else {"z": z}
    if k in ("batch", "serve"):
        specs, steps, seeds = _mix(case, seed)
        sums, parts, at = [], [], 0
        for (n, lo2, hi2, strict), m, v in zip(specs, steps, seeds):
            x, mask, one = _diffusion(n, (lo2, hi2, strict), v, case["steps"] if k == "batch" else m)
            sums.append(one[-1])
            p = _packed(x, mask)
            pad = (-p.numel()) % 4
            parts.append(torch.nn.functional.pad(p, (0, pad)))
        return {"sums": torch.stack(sums).cpu(), "x": torch.cat(parts)}
    if k in ("pic", "mpm"):
        n = case["n"]
        x, v, C = _spheres(case, seed)
        x, v, C = x.double(), v.double(), None if C is None else C.double()
        affine = C is not None
        if k == "mpm":
            u = _p2g(x, v, C, n)
        for _ in range(case["steps"]):
            if k == "pic":
                u = _p2g(x, v, C, n)
            x, v, C = _g2p(u, x, n, affine)
            if k == "mpm":
                u = _p2g(x, v, C, n)
        out = {"x": x, "v": v}
        return dict(out, C=C) if k == "pic" and affine else out
    if k == "tube":
        return _exact_tube(case, seed)
    return _exact_vcycle(case, seed)
