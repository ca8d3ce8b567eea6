"""The work that users of the free-surface LBM library have it do, as cases that can be timed.

Each case is one pass of a user's program through the public entry points
(``fslbm.Context``, ``fslbm.Batch``, ``fslbm.Server`` and the C calls they
wrap): a live simulation advanced to its next output, a whole run from host
arrays to host results, a batch of uneven domains, a served request stream,
or the monitoring of a large state.  The flows are those of the package's
workloads; the inputs are made here on the GPU so that they are quick to make,
and the seed moves every surface by a fraction of a cell.

``exact`` advances the same inputs with a plain FP64 torch implementation of
the method (arXiv 2207.13962, Sec. 2 and 3) that shares nothing with the
package.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2207_13962_gb300 import fslbm

GAS, IFACE, LIQ, OBST = 0, 1, 2, 3
ELEM = {"FP64": 8, "FP32": 4, "FP16S": 2, "BF16S": 2, "FP32MC": 4, "FP16SMC": 2}
REST = {"FP32MC": 4, "FP16SMC": 4}
NO_SLIP, PERIODIC, FREE_SLIP = 0, 1, 2

# Directions in the library's PDF order (include/fslbm.h).
DIRS = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
        (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
        (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 1, 1), (-1, -1, -1), (1, 1, -1),
        (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]


# ------------------------------------------------------------------ cases

def listed():
    return [
        # a small quasi-2-D wave tank in the parity precision: many short steps, all state read back
        dict(name="wave_fp64", kind="wave", nx=32, ny=64, nz=1, q=19, collision="TRT", variant="OM",
             precision="FP64", steps=100),
        # a small ragged tank with obstacles, 27 directions, SRT, the normal-based variant: odd sizes, every branch
        dict(name="ragged_fp32", kind="ragged", nx=37, ny=21, nz=11, q=27, collision="SRT", variant="NBRC",
             precision="FP32", steps=50),
        # the rectangular dam break run from host arrays to host results
        dict(name="dam_fp32", kind="dam", nx=256, ny=128, nz=64, q=19, collision="TRT", variant="OM",
             precision="FP32", steps=200, les=False),
        # the paper's own dam-break setup (free-slip walls, SRT, Smagorinsky model) in FP64, odd sizes
        dict(name="dam_les_fp64", kind="dam", nx=131, ny=67, nz=33, q=19, collision="SRT", variant="OM3",
             precision="FP64", steps=40, les=True),
        # the rising Taylor bubble, the benchmark's domain, advanced to its next output
        dict(name="taylor_fp32", kind="taylor", nx=160, ny=160, nz=1024, q=19, collision="TRT", variant="OM",
             precision="FP32", steps=50),
        # a smaller tube in the mass-conserving 16-bit storage
        dict(name="taylor_fp16smc", kind="taylor", nx=96, ny=96, nz=384, q=19, collision="TRT", variant="OM",
             precision="FP16SMC", steps=50),
        # uneven cylindrical dam breaks advanced together
        dict(name="cylinders_fp32", kind="batch", members=20, lo=64, hi=160, sizes=2207, q=27, collision="TRT",
             variant="OM", precision="FP32", steps=50),
        # a few small ones in the mass-conserving 16-bit storage
        dict(name="cylinders_fp16smc", kind="batch", members=8, lo=64, hi=96, sizes=13962, q=27, collision="TRT",
             variant="OM", precision="FP16SMC", steps=50),
        # a drop falling into a pool, run from host arrays to host results (velocity field uploaded)
        dict(name="drop_fp32", kind="drop", nx=192, ny=192, nz=192, q=19, collision="TRT", variant="OM",
             precision="FP32", steps=100),
        # a few drop requests through the continuous-batching server, fewer slots than requests
        dict(name="served_fp32", kind="serve", members=4, lo=96, hi=128, sizes=7, q=19, collision="TRT",
             variant="OM", precision="FP32", steps=250),
        # the monitoring of a large live state: observables and bubble pressures
        dict(name="monitor_fp32", kind="monitor", nx=160, ny=160, nz=512, q=19, collision="TRT", variant="OM",
             precision="FP32", steps=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: every kind, sizes spread over their logarithm, all formats."""
    kind = rng.choice(["wave", "ragged", "dam", "dam", "taylor", "taylor", "batch", "drop", "serve", "monitor"])
    variant = rng.choice(["OM", "OM", "OM3", "NBRC", "NBKC"])
    c = dict(kind=kind, q=rng.choice([19, 19, 27]), collision=rng.choice(["TRT", "TRT", "SRT"]), variant=variant,
             precision=rng.choice(["FP32", "FP32", "FP64", "FP32MC", "FP16SMC", "FP16S", "BF16S"]))
    if kind == "wave":
        c.update(nx=_log_int(rng, 32, 256), ny=_log_int(rng, 64, 256), nz=rng.choice([1, 1, 2, 5]),
                 steps=_log_int(rng, 20, 100))
    elif kind == "ragged":
        c.update(nx=_log_int(rng, 20, 90), ny=_log_int(rng, 18, 60), nz=_log_int(rng, 8, 40),
                 steps=_log_int(rng, 20, 60))
    elif kind == "dam":
        c.update(nx=_log_int(rng, 96, 256), ny=_log_int(rng, 48, 128), nz=_log_int(rng, 24, 64),
                 steps=_log_int(rng, 20, 100), les=rng.random() < 0.3)
    elif kind in ("taylor", "monitor"):
        n = _log_int(rng, 48, 144)
        c.update(nx=n, ny=n, nz=_log_int(rng, 128, 640), steps=0 if kind == "monitor" else _log_int(rng, 10, 40),
                 precision=rng.choice(["FP32", "FP32", "FP32MC", "FP16SMC", "FP16S", "BF16S"]))
    elif kind == "batch":
        c.update(members=rng.randint(3, 16), lo=64, hi=_log_int(rng, 80, 140), sizes=rng.randrange(1 << 20), q=27,
                 steps=_log_int(rng, 10, 40))
    elif kind == "drop":
        n = _log_int(rng, 96, 176)
        c.update(nx=n, ny=n, nz=n, steps=_log_int(rng, 20, 80))
    else:
        c.update(members=rng.randint(2, 4), lo=64, hi=_log_int(rng, 72, 110), sizes=rng.randrange(1 << 20),
                 steps=_log_int(rng, 60, 200))
    return c


# ----------------------------------------------------------------- inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _coords(shape):
    """Cell centres x, y, z as broadcastable FP64 tensors indexed [z, y, x]."""
    nx, ny, nz = shape
    dev = _device()
    x = torch.arange(nx, device=dev, dtype=torch.float64).add_(0.5).view(1, 1, nx)
    y = torch.arange(ny, device=dev, dtype=torch.float64).add_(0.5).view(1, ny, 1)
    z = torch.arange(nz, device=dev, dtype=torch.float64).add_(0.5).view(nz, 1, 1)
    return x, y, z


def _classify(fill, obstacle, boundary, q):
    """Cell types of fill levels in [0, 1], with a closed interface layer: a liquid cell with a gas cell
    in its lattice neighbourhood becomes an interface cell."""
    fill = fill.clamp(0.0, 1.0)
    t = torch.full(fill.shape, IFACE, dtype=torch.uint8, device=fill.device)
    t[fill >= 1.0] = LIQ
    t[fill <= 0.0] = GAS
    if obstacle is not None:
        t[obstacle] = OBST
    g = (t == GAS)
    for axis, a in ((0, 2), (1, 1), (2, 0)):  # one layer around the cells, wrapped across periodic faces
        lo, hi = g.narrow(axis, 0, 1), g.narrow(axis, g.shape[axis] - 1, 1)
        none = torch.zeros_like(lo)
        per = boundary[a] == PERIODIC
        g = torch.cat([hi if per else none, g, lo if per else none], dim=axis)
    near = torch.zeros_like(t, dtype=torch.bool)
    nz, ny, nx = t.shape
    for cx, cy, cz in DIRS[1:q]:
        near |= g[1 + cz:1 + cz + nz, 1 + cy:1 + cy + ny, 1 + cx:1 + cx + nx]
    t[(t == LIQ) & near] = IFACE
    fill = torch.where(t == LIQ, 1.0, torch.where(t == IFACE, fill, 0.0))
    return fill, t


def _flow(kind, shape, q, rng, les=False, drop=None):
    """One domain's initial state and parameters.  ``rng`` moves its surfaces by fractions of a cell."""
    nx, ny, nz = shape
    x, y, z = _coords(shape)
    obstacle = vel = rho = None
    sigma, bubble, cs, omega = 0.0, False, 0.0, None
    if kind == "wave":  # standing gravity wave, periodic x and z
        boundary, g, nu = (PERIODIC, NO_SLIP, PERIODIC), (0.0, -1e-5, 0.0), 0.01
        level = ny / 2 + 0.01 * nx * torch.cos(2 * math.pi * (x - 0.5) / nx + rng.uniform(0, 2 * math.pi))
        fill = (level - (y - 0.5)).expand(nz, ny, nx)
        up, h_ref = y, ny / 2
    elif kind == "ragged":  # rough surface with droplets of liquid and obstacle blocks, periodic x and z
        boundary, g, nu, sigma = (PERIODIC, NO_SLIP, PERIODIC), (0.0, -1e-4, 0.0), 0.05, 1e-3
        gen = torch.Generator(device="cpu").manual_seed(rng.randrange(1 << 30))
        level = ny / 2 + 2.0 * torch.sin(2 * math.pi * x / nx + rng.uniform(0, 6)) * torch.cos(2 * math.pi * z / nz)
        noise = torch.rand((nz, 1, nx), generator=gen, dtype=torch.float64).to(level.device)
        level = level + 0.8 * (noise - 0.5)
        fill = level - (y - 0.5)
        r = torch.sqrt((x - 0.3 * nx) ** 2 + (y - 0.8 * ny) ** 2 + (z - 0.5 * nz) ** 2)
        fill = torch.maximum(fill.clamp(0, 1), (2.8 - r).clamp(0, 1))
        obstacle = (((y < max(2, ny // 6)) & (x > nx // 2) & (x < nx // 2 + 3))
                    | ((y > ny // 3) & (y < ny // 3 + 2) & (x < 3))).expand(nz, ny, nx)
        up, h_ref = y, ny / 2
        v = torch.rand((3, nz, ny, nx), generator=gen, dtype=torch.float64).to(level.device)
        vel = 0.02 * (2 * v - 1)
    elif kind == "dam":  # rectangular column of liquid in one corner of a closed box
        boundary = (FREE_SLIP,) * 3 if les else (NO_SLIP,) * 3
        g, nu = (0.0, -1e-5, 0.0), 1e-3
        w, h = nx / 4 + rng.uniform(-0.5, 0.5), ny / 2 + rng.uniform(-0.5, 0.5)
        fill = ((w - (x - 0.5)).clamp(0, 1) * (h - (y - 0.5)).clamp(0, 1)).expand(nz, ny, nx)
        up, h_ref = y, h
        if les:
            cs, omega = 0.1, 1.9995
    elif kind == "taylor":  # long gas bubble rising in a tube of obstacle cells
        boundary, g, nu, sigma, bubble = (NO_SLIP,) * 3, (0.0, 0.0, -1e-6), 5e-3, 1e-4, True
        obstacle = (((x - nx / 2) ** 2 + (y - ny / 2) ** 2) >= (0.4 * nx) ** 2).expand(nz, ny, nx)
        dx, dy, dz = (rng.uniform(-0.5, 0.5) for _ in range(3))
        r = torch.sqrt((x - nx / 2 - dx) ** 2 + (y - ny / 2 - dy) ** 2) - 0.3 * nx
        zc, hl = nz / 8 + nz / 8 + dz, nz / 8
        fill = 0.5 + torch.maximum(r, (z - zc).abs() - hl)
        up, h_ref = z, nz / 2
    elif kind == "cylinder":  # cylindrical dam break in a closed box
        boundary, g, nu = (NO_SLIP,) * 3, (0.0, 0.0, -1e-5), 1e-3
        rf, hf = drop
        r = torch.sqrt((x - nx / 2 - rng.uniform(-0.5, 0.5)) ** 2 + (y - ny / 2 - rng.uniform(-0.5, 0.5)) ** 2)
        h = hf * nz + rng.uniform(-0.5, 0.5)
        fill = 0.5 - torch.maximum(r - rf * nx, z - h)
        up, h_ref = z, h
    else:  # drop above a thin pool, periodic x and y
        boundary, g, nu, sigma = (PERIODIC, PERIODIC, NO_SLIP), (0.0, 0.0, -1e-5), 1e-3, 1e-4
        rf, u = drop
        depth, rad = 0.1 * nz, rf * nx
        zc = depth + rad + 1.0
        dx, dy = rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5)
        r = torch.sqrt((x - nx / 2 - dx) ** 2 + (y - ny / 2 - dy) ** 2 + (z - zc) ** 2)
        pool = depth + rng.uniform(-0.2, 0.2) - (z - 0.5)
        fill = torch.maximum((0.5 - (r - rad)).clamp(0, 1), pool.clamp(0, 1).expand(nz, ny, nx))
        up, h_ref = z, depth
    fill, t = _classify(fill, obstacle, boundary, q)
    fluid = (t == LIQ) | (t == IFACE)
    rho = 1.0 + 3.0 * math.sqrt(sum(a * a for a in g)) * (h_ref - up)
    rho = torch.where(fluid, rho, 1.0)
    if kind == "drop":
        above = (z > depth + 1.0) & fluid
        rho = torch.where(above, 1.0, rho)
        vel = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device=fill.device)
        vel[2][above] = -u
    elif vel is not None:
        vel = torch.where(fluid, vel, 0.0)
    return dict(shape=shape, boundary=boundary, q=q, g=g, sigma=sigma, bubble=bubble, cs=cs,
                omega=omega if omega else 1.0 / (3.0 * nu + 0.5), fill=fill.reshape(-1), flags=t.reshape(-1),
                density=rho.reshape(-1), velocity=None if vel is None else vel.reshape(-1))


def _flows(case, seed):
    """The domains of a case: one, or the members of a batch or request stream."""
    rng = random.Random(int(seed) * 2 + 1)
    kind, q = case["kind"], case["q"]
    if kind in ("batch", "serve"):
        sizes = random.Random(case["sizes"])
        out = []
        for _ in range(case["members"]):
            n = sizes.randint(case["lo"], case["hi"])
            if kind == "batch":
                par = (sizes.uniform(0.2, 0.4), sizes.uniform(0.2, 0.4))
                out.append(_flow("cylinder", (n, n, n), q, rng, drop=par))
            else:
                par = (sizes.uniform(0.08, 0.15), sizes.uniform(0.02, 0.05))
                out.append(_flow("drop", (n, n, n), q, rng, drop=par))
        return out
    name = "taylor" if kind == "monitor" else kind
    par = (0.12, 0.03) if kind == "drop" else None
    return [_flow(name, (case["nx"], case["ny"], case["nz"]), q, rng, les=case.get("les", False), drop=par)]


def _request_steps(case):
    """Steps of each request of a served stream (uneven, so that runs retire at different times)."""
    r = random.Random(case["sizes"] + 1)
    return [max(1, int(case["steps"] * r.uniform(0.6, 1.0))) for _ in range(case["members"])]


def _pinned(t):
    """Host copy of a tensor in pinned memory."""
    if t is None:
        return None
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=torch.cuda.is_available())
    h.copy_(t)
    return h


def _host(flow):
    return {k: _pinned(flow[k]) for k in ("fill", "flags", "density", "velocity")}


def _context(case, flow):
    return fslbm.Context(flow["shape"], periodic=flow["boundary"], q=case["q"], collision=case["collision"],
                         variant=case["variant"], precision=case["precision"], omega=flow["omega"], g=flow["g"],
                         sigma=flow["sigma"], bubble_model=flow["bubble"], smagorinsky_cs=flow["cs"])


def _init(ctx, host):
    vel, den = host["velocity"], host["density"]
    st = ctx.init_raw(host["fill"].data_ptr(), host["flags"].data_ptr(), None if vel is None else vel.data_ptr(),
                      None if den is None else den.data_ptr())
    if st != fslbm.OK:
        raise fslbm.FslbmError(st, ctx.lib.fslbm_last_error(ctx.h).decode())


def _out_buffers(ctx, pdf):
    pin = torch.cuda.is_available()
    out = {"fill": torch.empty(ctx.N, dtype=torch.float64, pin_memory=pin),
           "flags": torch.empty(ctx.N, dtype=torch.uint8, pin_memory=pin),
           "mass": torch.empty(ctx.N, dtype=torch.float64, pin_memory=pin)}
    if pdf:
        out["pdf"] = torch.empty((ctx.q, ctx.N), dtype=torch.float64, pin_memory=pin)
    return out


def _read(ctx, out):
    ptr = {k: fslbm.C.c_void_p(v.data_ptr()) for k, v in out.items()}
    st = ctx.lib.fslbm_read_fields(ctx.h, ptr.get("pdf"), ptr["fill"], ptr["flags"], ptr["mass"])
    if st != fslbm.OK:
        raise fslbm.FslbmError(st, ctx.lib.fslbm_last_error(ctx.h).decode())
    return out


WHOLE_RUN = ("dam", "drop")      # a pass is a run from host arrays to host results
WITH_PDF = ("wave", "ragged")    # small states are read back whole, PDFs too


def _reads_pdf(case):
    return case["kind"] in WITH_PDF or (case["kind"] == "dam" and case["precision"] == "FP64")


def prepare(case, seed):
    flows = _flows(case, seed)
    kind = case["kind"]
    if kind == "serve":
        reqs = []
        for f, n in zip(flows, _request_steps(case)):
            host = {k: None if f[k] is None else f[k].cpu().numpy() for k in ("fill", "flags", "density", "velocity")}
            reqs.append((_Request(f, case, host), n))
        return {"case": case, "requests": reqs}
    if kind == "batch":
        ctxs, outs = [], []
        for f in flows:
            c = _context(case, f)
            _init(c, _host(f))
            ctxs.append(c)
            outs.append(_out_buffers(c, False))
        return {"case": case, "batch": fslbm.Batch(ctxs), "ctxs": ctxs, "outs": outs}
    ctx, host = _context(case, flows[0]), _host(flows[0])
    state = {"case": case, "ctx": ctx}
    if kind in WHOLE_RUN:
        state["host"] = host
    else:
        _init(ctx, host)
    if kind != "monitor":
        state["out"] = _out_buffers(ctx, _reads_pdf(case))
    return state


class _Request:
    """What ``fslbm.Server.submit`` takes for a request: a state on the host and its parameters."""

    def __init__(self, flow, case, host):
        self.shape, self.periodic, self.variant = flow["shape"], flow["boundary"], case["variant"]
        self.N = int(np.prod(self.shape))
        self.omega, self.g, self.sigma, self.bubble_model = flow["omega"], flow["g"], flow["sigma"], False
        self.fill, self.flags, self.density, self.velocity = (host[k] for k in ("fill", "flags", "density",
                                                                                "velocity"))


OBS_COUNTS = ("n_liquid", "n_interface", "n_gas", "n_obstacle", "n_bubbles")
OBS_VALUES = ("total_mass", "liquid_volume", "max_u")


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        srv = fslbm.Server(q=case["q"], collision=case["collision"], precision=case["precision"], max_active=3,
                           chunk_steps=50)
        ids = [srv.submit(rq, n) for rq, n in state["requests"]]
        while srv.stats()["completed"] < len(ids):
            srv.poll()
        res = [srv.result(i) for i in ids]
        srv.close()
        return [{"fill": r["fill"], "flags": r["flags"], "steps": r["steps"]} for r in res]
    if kind == "batch":
        state["batch"].step(case["steps"])
        return [_read(c, o) for c, o in zip(state["ctxs"], state["outs"])]
    ctx = state["ctx"]
    if kind == "monitor":
        obs = ctx.observables()
        volume, pressure = ctx.bubbles(16)
        return {"counts": [obs[k] for k in OBS_COUNTS], "values": [obs[k] for k in OBS_VALUES],
                "volume": volume, "pressure": pressure}
    if kind in WHOLE_RUN:
        _init(ctx, state["host"])
    ctx.step(case["steps"])
    return _read(ctx, state["out"])


def work(case):
    """Each step reads and writes the PDFs of the liquid and interface cells once; a whole run also takes its
    inputs in, and every pass gives its outputs out."""
    s = ELEM[case["precision"]]
    q = case["q"]
    per_cell = 2 * ((q - 1) * s + REST.get(case["precision"], s))
    nbytes = flops = 0.0
    flows = _flows(case, 1)
    steps = _request_steps(case) if case["kind"] == "serve" else [case["steps"]] * len(flows)
    for f, n in zip(flows, steps):
        cells = f["flags"].numel()
        fluid = int(((f["flags"] == LIQ) | (f["flags"] == IFACE)).sum())
        iface = int((f["flags"] == IFACE).sum())
        if case["kind"] == "monitor":
            nbytes += fluid * per_cell / 2 + cells + fluid * 8 + iface * 8
            flops += fluid * (5.0 * q + 10)
            continue
        nbytes += n * (fluid * (per_cell + 1) + iface * 64)
        flops += n * (fluid * 12.0 * q + iface * 400.0)
        nbytes += cells * (9 if case["kind"] == "serve" else 17)
        if case["kind"] in WHOLE_RUN + ("serve",):
            nbytes += cells * (17 + (24 if f["velocity"] is not None else 0))
        if _reads_pdf(case):
            nbytes += cells * q * 8
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ exact

class _Plain:
    """The method in plain FP64 torch: whole-array geometry, gathers over the list of fluid cells."""

    def __init__(self, flow, case):
        self.q, self.case, self.flow = flow["q"], case, flow
        self.n = flow["shape"]
        self.N = flow["flags"].numel()
        dev = flow["fill"].device
        self.dev = dev
        self.c = torch.tensor(DIRS[: self.q], device=dev, dtype=torch.float64)
        n2 = (self.c ** 2).sum(1).long().tolist()
        w = {19: [1 / 3, 1 / 18, 1 / 36], 27: [8 / 27, 2 / 27, 1 / 54, 1 / 216]}[self.q]
        self.w = [w[k] for k in n2]
        self.opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, self.q)]
        self.reflect = [[DIRS.index(tuple(-a if (m >> k) & 1 else a for k, a in enumerate(d))) for m in range(8)]
                        for d in DIRS[: self.q]]
        # one more entry than cells: whatever lies outside the domain is an obstacle
        self.t = torch.cat([flow["flags"], torch.tensor([OBST], dtype=torch.uint8, device=dev)])
        t = flow["flags"]
        self.phi, rho = flow["fill"].clone(), flow["density"]
        self.mass = torch.where(t == LIQ, rho, torch.where(t == IFACE, self.phi * rho, 0.0))
        vel = flow["velocity"]
        u = vel.view(3, -1) if vel is not None else torch.zeros((3, 1), dtype=torch.float64, device=dev)
        fluid = ((t == LIQ) | (t == IFACE)).double()
        self.f = torch.stack([self.feq(i, rho, u) * fluid for i in range(self.q)])
        self.bid = torch.full((self.N,), -1, dtype=torch.int64, device=dev)
        if flow["bubble"]:  # one gas region
            cells = torch.arange(self.N, device=dev)
            near = torch.zeros(self.N, dtype=torch.bool, device=dev)
            for i in range(1, self.q):
                near |= self.t[self.neighbour(cells, i)] == GAS
            self.bid[(t == GAS) | ((t == IFACE) & near)] = 0
        self.pv0 = self.pv = 1.0 / 3.0
        self.V0 = self.V = self.volume()

    def feq(self, i, rho, u):
        cx, cy, cz = DIRS[i]
        cu = cx * u[0] + cy * u[1] + cz * u[2]
        return self.w[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))

    def volume(self):
        t, mine = self.t[:-1], self.bid >= 0
        return float((mine & (t == GAS)).sum() + torch.where(mine & (t == IFACE), 1.0 - self.phi, 0.0).sum())

    def xyz(self, cells):
        nx, ny, _ = self.n
        return [cells % nx, (cells // nx) % ny, cells // (nx * ny)]

    def neighbour(self, cells, i, pos=None):
        """Index of x + c_i, N outside a wall."""
        pos = self.xyz(cells) if pos is None else pos
        out, idx, stride = None, 0, 1
        for a in range(3):
            v = pos[a] + DIRS[i][a]
            if DIRS[i][a]:
                if self.flow["boundary"][a] == PERIODIC:
                    v = v % self.n[a]
                else:
                    bad = (v < 0) | (v >= self.n[a])
                    out = bad if out is None else out | bad
                    v = v.clamp(0, self.n[a] - 1)
            idx = idx + v * stride
            stride *= self.n[a]
        return idx if out is None else torch.where(out, self.N, idx)

    def source(self, i, pos):
        """Cell x - c_i (mirrored at free-slip walls, N outside a wall) and the PDF that arrives from it."""
        out, idx, stride, mirror = None, 0, 1, None
        for a in range(3):
            v = pos[a] - DIRS[i][a]
            if DIRS[i][a]:
                kind = self.flow["boundary"][a]
                bad = (v < 0) | (v >= self.n[a])
                if kind == PERIODIC:
                    v = v % self.n[a]
                elif kind == FREE_SLIP:
                    v = torch.where(bad, pos[a], v)
                    m = bad.long() << a
                    mirror = m if mirror is None else mirror + m
                else:
                    out = bad if out is None else out | bad
                    v = v.clamp(0, self.n[a] - 1)
            idx = idx + v * stride
            stride *= self.n[a]
        idx = idx if out is None else torch.where(out, self.N, idx)
        if mirror is None:
            return idx, i
        return idx, torch.tensor(self.reflect[i], device=self.dev)[mirror]

    # K8 smoothing, Parker-Youngs normal, finite-difference curvature; solid points take the centre's value
    def _padded(self, a):
        for axis, ax in ((0, 2), (1, 1), (2, 0)):
            per = self.flow["boundary"][ax] == PERIODIC
            lo, hi = a.narrow(axis, 0, 1), a.narrow(axis, a.shape[axis] - 1, 1)
            nan = torch.full_like(lo, math.nan)
            a = torch.cat([hi if per else nan, a, lo if per else nan], dim=axis)
        return a

    def geometry(self, cells):
        nx, ny, nz = self.n
        solid = (self.t[:-1] == OBST).view(nz, ny, nx)
        raw = torch.where(solid, math.nan, self.phi.view(nz, ny, nx))

        def at(p, d, centre):
            v = p[1 + d[2]:1 + d[2] + nz, 1 + d[1]:1 + d[1] + ny, 1 + d[0]:1 + d[0] + nx]
            return torch.where(torch.isnan(v), centre, v)

        k8 = [1.0, 0.31640625, 0.0625, 0.00390625]
        p = self._padded(raw)
        sm = torch.zeros_like(raw)
        for d in ((a, b, c) for c in (-1, 0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1)):
            sm += k8[d[0] ** 2 + d[1] ** 2 + d[2] ** 2] * at(p, d, raw)
        sm /= 3.6796875
        p = self._padded(sm)
        n = []
        for a in range(3):
            acc = torch.zeros_like(sm)
            for b in (-1, 0, 1):
                for c in (-1, 0, 1):
                    d = [b, c]
                    d.insert(a, 1)
                    wt = 4.0 / (1 << (abs(b) + abs(c)))
                    hi = at(p, d, sm)
                    d[a] = -1
                    acc += wt * (hi - at(p, d, sm))
            n.append(acc)
        ln = torch.sqrt(n[0] ** 2 + n[1] ** 2 + n[2] ** 2)
        n = [torch.where(solid, math.nan, torch.where(ln > 0, v / ln, 0.0)) for v in n]
        kappa = torch.zeros_like(sm)
        for a in range(3):
            p = self._padded(n[a])
            d = [0, 0, 0]
            d[a] = 1
            hi = at(p, d, n[a])
            d[a] = -1
            kappa -= 0.5 * (hi - at(p, d, n[a]))
        return [v.reshape(-1)[cells] for v in n], kappa.reshape(-1)[cells]

    def collide(self, f):
        fl, q = self.flow, self.q
        g, om = fl["g"], fl["omega"]
        rho = f.sum(0)
        u = [(self.c[:, a] @ f) / rho + 0.5 * g[a] for a in range(3)]
        F = [rho * g[a] for a in range(3)]
        fe = torch.stack([self.feq(i, rho, u) for i in range(q)])
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        s = []
        for i in range(q):
            cx, cy, cz = DIRS[i]
            cu = cx * u[0] + cy * u[1] + cz * u[2]
            cF = cx * F[0] + cy * F[1] + cz * F[2]
            s.append(self.w[i] * (3 * (cF - uF) + 9 * cu * cF))
        s = torch.stack(s)
        if fl["cs"] > 0:
            dn = f - fe
            q2 = torch.zeros_like(rho)
            for a in range(3):
                for b in range(3):
                    q2 += ((self.c[:, a] * self.c[:, b]) @ dn) ** 2
            tau0 = 1 / om
            om = 2 / (tau0 + torch.sqrt(tau0 ** 2 + 18 * math.sqrt(2) * fl["cs"] ** 2 * torch.sqrt(2 * q2) / rho))
        if self.case["collision"] == "SRT":
            return f - om * (f - fe) + (1 - 0.5 * om) * s, rho
        omm = 1 / (0.5 + (3 / 16) / (1 / om - 0.5))
        dn, dno, so = f - fe, (f - fe)[self.opp], s[self.opp]
        return (f - om * 0.5 * (dn + dno) - omm * 0.5 * (dn - dno) + (1 - 0.5 * om) * 0.5 * (s + so)
                + (1 - 0.5 * omm) * 0.5 * (s - so)), rho

    def moments(self, f):
        rho = f.sum(0)
        return rho, [(self.c[:, a] @ f) / rho - 0.5 * self.flow["g"][a] for a in range(3)]

    def step(self):
        q, N, t, A, opp = self.q, self.N, self.t, self.f, self.opp
        g = self.flow["g"]
        cells = torch.nonzero((t[:-1] == LIQ) | (t[:-1] == IFACE)).view(-1)
        isI = t[cells] == IFACE
        band = cells[isI]
        normal, kappa = self.geometry(band)
        pv = self.pv0 + (self.bid[band] >= 0).double() * (self.pv - self.pv0)
        rg = 3 * (pv + self.flow["sigma"] * kappa)
        pos = self.xyz(cells)
        pulled = torch.empty((q, cells.numel()), dtype=torch.float64, device=self.dev)
        flat = A.reshape(-1)
        src_b, typ_b = [None] * q, [None] * q  # of the interface cells
        for i in range(q):
            src, j = self.source(i, pos)
            ts = t[src]
            fluid = (ts == LIQ) | (ts == IFACE)
            pulled[i] = flat[torch.where(fluid, j * N + src, opp[i] * N + cells)]
            src_b[i], typ_b[i] = src[isI], ts[isI]
        fI, own = pulled[:, isI], A[:, band]
        # Thuerey classes
        pos_b = [p[isI] for p in pos]
        nid = [self.neighbour(band, i, pos_b) for i in range(q)]
        nt = [t[n] for n in nid]
        hl = torch.zeros(band.numel(), dtype=torch.bool, device=self.dev)
        hg = hl.clone()
        for i in range(1, q):
            hl |= nt[i] == LIQ
            hg |= nt[i] == GAS
        cls = torch.where(~hl & hg, 1, torch.where(hl & ~hg, 2, 0))  # 1: no liquid, 2: no gas neighbour
        cls_all = torch.zeros(N + 1, dtype=torch.int64, device=self.dev)
        cls_all[band] = cls
        phi1 = torch.cat([self.phi, self.phi.new_zeros(1)])
        dm = torch.zeros(band.numel(), dtype=torch.float64, device=self.dev)
        for i in range(1, q):
            n, ty = src_b[opp[i]], typ_b[opp[i]]
            fa, fb, cn = fI[opp[i]], own[i], cls_all[n]
            v = torch.where(cls == cn, fa - fb,
                            torch.where(cls == 0, torch.where(cn == 1, fa, -fb), torch.where(cls == 1, -fb, fa)))
            dm += torch.where(ty == LIQ, fa - fb,
                              torch.where(ty == IFACE, 0.5 * (self.phi[band] + phi1[n]) * v, 0.0))
        m_next = self.mass[band] + dm
        # free-surface boundary condition
        rc, u = self.moments(own)
        miss = torch.stack([ty == GAS for ty in typ_b])
        miss[0] = False
        var = self.case["variant"]
        om_set = torch.ones_like(isI[isI])
        if var == "OM3":
            om_set = miss.sum(0) >= 3
        elif var != "OM":
            om_set = torch.zeros_like(om_set)
        for i in range(q):
            dot = DIRS[i][0] * normal[0] + DIRS[i][1] * normal[1] + DIRS[i][2] * normal[2]
            rec = (dot >= -2.0 ** -20) if var == "NBRC" else (dot > 2.0 ** -20)
            rec = miss[i] | (rec & ~om_set)
            new = self.feq(i, rg, u) + self.feq(opp[i], rg, u) - own[opp[i]]
            fI[i] = torch.where(rec, new, fI[i])
        pulled[:, isI] = fI
        del fI, own
        fs, rho = self.collide(pulled)
        del pulled
        B = torch.zeros_like(A)
        B[:, cells] = fs
        rho_b = rho[isI]
        mr, mu = self.moments(fs[:, isI])
        del fs
        phi_next = m_next / rho_b
        eps = 1e-2
        # conversion: marks, conflict rule, claims
        full = torch.zeros(N + 1, dtype=torch.int64, device=self.dev)
        mark = torch.where(phi_next > 1 + eps, 1, torch.where(phi_next < -eps, 2, 0))
        full[band] = mark
        near_tol = torch.zeros_like(hl)
        for i in range(1, q):
            near_tol |= (nt[i] == IFACE) & (full[nid[i]] == 1)
        conv = torch.where((mark == 2) & near_tol, 0, mark)
        full[band] = conv
        claim = torch.zeros(N + 1, dtype=torch.bool, device=self.dev)
        for i in range(1, q):
            claim[nid[i][((conv == 1) & (nt[i] == GAS)) | ((conv == 2) & (nt[i] == LIQ))]] = True
        nrecv = torch.zeros_like(conv)
        for i in range(1, q):
            nrecv += torch.where(nt[i] == IFACE, full[nid[i]] == 0, (nt[i] != OBST) & claim[nid[i]]).long()
        fin = torch.where((conv > 0) & (nrecv == 0), 3, conv)
        fin_all = torch.zeros(N + 1, dtype=torch.int64, device=self.dev)
        fin_all[band] = fin
        gone = (fin == 1) | (fin == 2)
        share = torch.zeros(N + 1, dtype=torch.float64, device=self.dev)
        excess = torch.where(conv == 1, m_next - rho_b, m_next) / nrecv.clamp(min=1)
        share[band] = torch.where(gone, excess, 0.0)
        got = torch.zeros_like(m_next)
        for i in range(1, q):
            got += torch.where(nt[i] == IFACE, share[nid[i]], 0.0)
        plain = fin == 0
        m_next = torch.where(plain, m_next + got, m_next)
        phi_next = torch.where(plain, m_next / rho_b, phi_next)
        self.mass[band] = torch.where(fin == 1, rho_b, torch.where(fin == 2, 0.0, m_next))
        self.phi[band] = torch.where(fin == 1, 1.0, torch.where(fin == 2, 0.0, phi_next))
        # new interface cells
        new = torch.nonzero(claim[:-1]).view(-1)
        if new.numel():
            was_gas = t[new] == GAS
            nn = [self.neighbour(new, i) for i in range(q)]
            tn = [t[n] for n in nn]
            s = torch.zeros(new.numel(), dtype=torch.float64, device=self.dev)
            acc = torch.zeros((4, new.numel()), dtype=torch.float64, device=self.dev)
            cnt = torch.zeros_like(s)
            best = torch.full_like(new, 1 << 40)
            mom = torch.zeros((4, N + 1), dtype=torch.float64, device=self.dev)
            mom[0, band], mom[1, band], mom[2, band], mom[3, band] = mr, mu[0], mu[1], mu[2]
            for i in range(1, q):
                n, ty, fn = nn[i], tn[i], fin_all[nn[i]]
                s += torch.where(ty == IFACE, share[n], 0.0)
                use = ((ty == IFACE) & (fn != 2)) | ((ty == LIQ) & ~claim[n])
                v = mom[:, n]
                liq = torch.nonzero(use & (ty == LIQ) & was_gas).view(-1)
                if liq.numel():
                    r1, u1 = self.moments(B[:, n[liq]])
                    v[:, liq] = torch.stack([r1, *u1])
                acc += torch.where(use, v, 0.0)
                cnt += use
                gas_after = ((ty == GAS) & ~claim[n]) | ((ty == IFACE) & (fn == 2))
                b = self.bid[n.clamp(max=N - 1)]
                best = torch.where(gas_after & (b >= 0), torch.minimum(best, b), best)
            r, *un = torch.where(cnt > 0, acc / cnt.clamp(min=1), torch.tensor([[1.0], [0], [0], [0]],
                                                                                 dtype=torch.float64, device=self.dev))
            rl, _ = self.moments(B[:, new])
            r = torch.where(was_gas, r, rl)
            feq = torch.stack([self.feq(i, r, un) for i in range(q)])
            B[:, new] = torch.where(was_gas, feq, B[:, new])
            m = torch.where(was_gas, s, rl + s)
            self.mass[new], self.phi[new] = m, m / r
            self.bid[new] = torch.where(was_gas, self.bid[new], torch.where(best < (1 << 40), best, -1))
        self.t[band] = torch.where(fin == 1, LIQ, torch.where(fin == 2, GAS, IFACE)).to(torch.uint8)
        self.bid[band[fin == 1]] = -1
        self.t[new] = IFACE
        self.f = B
        if self.flow["bubble"]:
            self.V = self.volume()
            self.pv = self.pv0 * self.V0 / self.V if self.V > 0 else self.pv0

    def read(self, pdf):
        t = self.t[:-1]
        out = {"fill": self.phi, "flags": t, "mass": self.mass}
        if pdf:
            out["pdf"] = torch.where((t == LIQ) | (t == IFACE), self.f, 0.0)
        return out


def exact(case, seed):
    flows = _flows(case, seed)
    kind = case["kind"]
    if kind == "monitor":
        s = _Plain(flows[0], case)
        t = s.t[:-1]
        cells = torch.nonzero((t == LIQ) | (t == IFACE)).view(-1)
        rho, u = s.moments(s.f[:, cells])
        mass = torch.where(t[cells] == LIQ, rho, s.mass[cells]).sum()
        speed = torch.sqrt(u[0] ** 2 + u[1] ** 2 + u[2] ** 2).max()
        counts = [int((t == k).sum()) for k in (LIQ, IFACE, GAS, OBST)] + [1]
        return {"counts": counts, "values": [float(mass), float(s.phi[cells].sum()), float(speed)],
                "volume": np.array([s.V0]), "pressure": np.array([s.pv0])}
    steps = _request_steps(case) if kind == "serve" else [case["steps"]] * len(flows)
    # seconds: launches, then the arrays of each step
    if sum(n * (0.02 + f["flags"].numel() * 3e-9 * case["q"] / 19) for f, n in zip(flows, steps)) > 20:
        return None
    out = []
    for f, n in zip(flows, steps):
        s = _Plain(f, case)
        for _ in range(n):
            s.step()
        r = s.read(_reads_pdf(case))
        if kind == "serve":
            r = {"fill": r["fill"], "flags": r["flags"], "steps": n}
        out.append(r)
        del s
    return out if kind in ("serve", "batch") else out[0]
