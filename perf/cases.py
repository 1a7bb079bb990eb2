"""Performance cases: what users of this solver have it do, over the range of sizes in which they do it.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (an initial field on the
GPU, the solver's handle), ``run`` is one pass through the public entry points, ``work`` the bytes and operations
that a pass cannot do without, and ``exact`` the same outputs in plain 64-bit torch.

Families ("kind"):
  step2d  restart from a field, advance explicit SSP-RK3 steps, read the field and the body force.  The production
          form is FP32-bulk; FP64 is the form that a new configuration is validated in.
  dual2d  the same with one dual-time physical step (low Mach numbers).
  step3d  the same around a triangulated body.
  body3d  3-D pre-processing: classification, tags, ordered lists, closest features of a triangulated body.
  serve   a burst of requests through the request loop until all are done.

Fields and forces of the FP32-bulk form are returned in 32 bits, the precision that the form carries.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1912_11908_gb300 import ibm
from paper_1912_11908_gb300 import workloads as W

F64 = torch.float64
STAGE_FLOPS_2D, STAGE_FLOPS_3D, DUAL_FLOPS = 1073, 2780, 126  # per cell and stage, counted from the formulas


def listed():
    step2d = dict(kind="step2d", motion="static", ib="rebuild", scheme="weno5", interp="linear", bits=32)
    return [
        # the smallest interactive call: one step of a coarse cylinder, launches and latency
        dict(step2d, name="cylinder_160x80_1step", body="cylinder", nx=160, ny=80, mach=0.2, re=40.0, steps=1),
        # the headline workload: a supersonic wedge on an ordinary grid
        dict(step2d, name="wedge_768x384", body="wedge", nx=768, ny=384, mach=2.0, re=1.0e4, ib="advance", steps=10),
        # the same flow resolved for production: larger than the L2 cache
        dict(step2d, name="wedge_3072x1536", body="wedge", nx=3072, ny=1536, mach=2.0, re=1.0e4, ib="advance",
             steps=4),
        # a moving body: re-classified, re-tagged and given new stencils at every step
        dict(step2d, name="oscillating_cylinder_1024x512", body="cylinder", nx=1024, ny=512, mach=0.2, re=185.0,
             motion="sin", steps=10),
        # validation of the same method in 64 bits
        dict(step2d, name="wedge_768x384_fp64", body="wedge", nx=768, ny=384, mach=2.0, re=1.0e4, ib="advance",
             steps=2, bits=64),
        # low Mach number: one physical step of 30 sub-iterations
        dict(kind="dual2d", name="naca0012_2048x1024_dual", body="naca", nx=2048, ny=1024, mach=0.001, re=1000.0,
             subiters=30, bits=32),
        # ... and its validation in 64 bits on a coarser grid, an odd size
        dict(kind="dual2d", name="naca0012_257x131_dual_fp64", body="naca", nx=257, ny=131, mach=0.01, re=1000.0,
             subiters=30, bits=64),
        # 3-D flow past a sphere, production form
        dict(kind="step3d", name="sphere_192x96x96", nx=192, ny=96, nz=96, nlat=21, nlon=30, mach=0.3, re=100.0,
             steps=4, bits=32),
        # 3-D in 64 bits on a coarser grid
        dict(kind="step3d", name="sphere_96x48x48_fp64", nx=96, ny=48, nz=48, nlat=21, nlon=30, mach=0.3, re=100.0,
             steps=2, bits=64),
        # 3-D pre-processing of a sphere in a cube, small and large
        dict(kind="body3d", name="sphere_in_cube_40", nx=40, ny=40, nz=40, nlat=21, nlon=30),
        dict(kind="body3d", name="sphere_in_cube_256", nx=256, ny=256, nz=256, nlat=21, nlon=30),
        # a burst of mixed requests (bodies, motions, Mach numbers, grids) through the request loop
        dict(kind="serve", name="serve_16_requests", requests=16, mix=1, steps=20, subiters=10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step2d", "step2d", "step2d", "dual2d", "step3d", "body3d", "serve"])
    bits = rng.choice([32, 32, 64])
    if kind == "step2d":
        body = rng.choice(["cylinder", "naca", "wedge"])
        nx = int(_log(rng, 96, 3072 if bits == 32 else 768))
        ny = max(64, int(nx * rng.uniform(0.4, 0.6)))
        mach = rng.uniform(1.3, 2.0) if body == "wedge" else _log(rng, 0.1, 0.6)
        return dict(kind=kind, body=body, nx=nx, ny=ny, mach=mach, re=_log(rng, 40.0, 1.0e4),
                    motion=rng.choice(["static", "static", "sin"]) if body != "wedge" else "static",
                    ib="advance" if body == "wedge" else "rebuild",
                    scheme=rng.choice(["weno5", "weno5", "weno5", "tvd2"]),
                    interp=rng.choice(["linear", "linear", "linear", "quadratic"]) if mach < 0.4 else "linear",
                    steps=rng.randint(1, 10 if nx < 1500 else 4) if bits == 32 else rng.randint(1, 2), bits=bits)
    if kind == "dual2d":
        nx = int(_log(rng, 128, 2048 if bits == 32 else 320))
        return dict(kind=kind, body=rng.choice(["cylinder", "naca"]), nx=nx, ny=max(64, int(nx * rng.uniform(0.4, 0.5))),
                    mach=_log(rng, 0.001, 0.1), re=_log(rng, 40.0, 3000.0), subiters=rng.randint(5, 30), bits=bits)
    if kind == "step3d":
        ny, nz = (int(_log(rng, 24, 96 if bits == 32 else 48)) for _ in range(2))
        return dict(kind=kind, nx=int(rng.uniform(1.0, 2.0) * max(ny, nz)), ny=ny, nz=nz, nlat=rng.randint(9, 31),
                    nlon=rng.randint(12, 45), mach=_log(rng, 0.2, 0.6), re=_log(rng, 40.0, 1000.0),
                    steps=rng.randint(1, 4) if bits == 32 else rng.randint(1, 2), bits=bits)
    if kind == "body3d":
        nx, ny, nz = (int(_log(rng, 20, 256)) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, nlat=rng.randint(9, 31), nlon=rng.randint(12, 45))
    return dict(kind=kind, requests=rng.randint(2, 16), mix=rng.randint(2, 1 << 20), steps=rng.randint(5, 20),
                subiters=rng.randint(3, 10))


# ---- inputs -------------------------------------------------------------------------------------------------------

DOMAIN = {"cylinder": (-8.0, 24.0, -8.0, 8.0), "naca": (-4.0, 8.0, -3.0, 3.0), "wedge": (-1.0, 3.0, -1.0, 1.0)}
MOVING_DOMAIN = (-10.0, 30.0, -10.0, 10.0)


def _refined(verts, pieces):
    """Every segment in equal pieces: the surface integral of the force has one probe per segment."""
    nxt = np.roll(verts, -1, axis=0)
    return np.concatenate([verts[k] + np.arange(pieces)[:, None] / pieces * (nxt[k] - verts[k])
                           for k in range(len(verts))])


def _spec2d(case, seed):
    """The 2-D case: the configuration's body, shifted within a cell by the seed."""
    rng = np.random.default_rng(seed)
    moving = case.get("motion") == "sin"
    dom = MOVING_DOMAIN if moving and case["body"] == "cylinder" else DOMAIN[case["body"]]
    verts = {"cylinder": lambda: W.cylinder(256), "naca": lambda: W.naca00xx(0.12, 400, 5.0),
             "wedge": lambda: _refined(W.wedge(15.0), 64)}[case["body"]]()
    dx, dy = (dom[1] - dom[0]) / case["nx"], (dom[3] - dom[2]) / case["ny"]
    verts = verts + rng.uniform(-0.4, 0.4, 2) * [dx, dy]
    kw = dict(precision=W.PREC_FP32_BULK if case["bits"] == 32 else W.PREC_FP64)
    if case["kind"] == "dual2d":
        kw.update(time_scheme=W.TIME_DUAL, dt_phys=0.5 * dx, subiters=case["subiters"])
    else:
        kw.update(ib_mode=W.IB_ADVANCE if case["ib"] == "advance" else W.IB_REBUILD,
                  scheme=W.SCHEME_TVD2 if case["scheme"] == "tvd2" else W.SCHEME_WENO5,
                  ib_interp=W.INTERP_QUADRATIC if case["interp"] == "quadratic" else W.INTERP_LINEAR)
    if moving:
        kw.update(motion=W.MOTION_SIN, amp=(0.0, 0.2), freq=0.16)
    return W.case_spec(verts, case["nx"], case["ny"], dom, case["mach"], case["re"],
                       W.SUPERSONIC if case["mach"] > 1.0 else W.FAR, **kw)


def _mesh(case, seed, radius):
    """A closed sphere mesh with seeded radial bumps, off the lattice's symmetry planes."""
    rng = np.random.default_rng(seed)
    verts, tris = W.uv_sphere(case["nlat"], case["nlon"], 1.0)
    k = rng.uniform(1.0, 3.0, (3, 3))
    ph = rng.uniform(0.0, 2.0 * math.pi, 3)
    bump = 1.0 + 0.02 * np.sin(verts @ k.T + ph).sum(axis=1, keepdims=True)
    return radius * verts * bump + rng.uniform(-0.02, 0.02, 3), tris


def _spec3d(case, seed):
    verts, tris = _mesh(case, seed, 0.5)
    n = (case["nx"], case["ny"], case["nz"])
    lo, hi = (-3.0, -3.0, -3.0), (-3.0 + 6.0 * case["nx"] / max(case["ny"], case["nz"]), 3.0, 3.0)
    return W.case3d_spec(verts, tris, n, lo, hi, case["mach"], case["re"], W.FAR3D, ref_area=math.pi * 0.25,
                         precision=W.PREC_FP32_BULK if case["bits"] == 32 else W.PREC_FP64)


def _specs_serve(case, seed):
    """The mix's requests (low Mach numbers by dual time); the seed moves their Mach and Reynolds numbers by a few
    per cent."""
    rng = np.random.default_rng(seed)
    out = []
    for r in W.serving_mix(case["requests"], 1000 + case["mix"], nsteps=case["steps"], dual_steps=1,
                           dual_mach=0.1, subiters=case["subiters"]):
        f, spec = rng.uniform(0.97, 1.0, 2), r["spec"]
        verts = _refined(spec["verts"], 64) if len(spec["verts"]) == 3 else spec["verts"]
        out.append((dict(spec, verts=verts, mach=spec["mach"] * f[0], re=spec["re"] * f[1]), r["nsteps"]))
    return out


def _field(n, lo, hi, verts, mach, gamma, uinf, seed):
    """A flow in progress, conserved [1 + d + 1][..., ny, nx] on the GPU: the free stream brought to rest around the
    body, with smooth velocity (5 %), pressure and temperature fluctuations of a few seeded wavelengths."""
    d = len(n)
    rng = np.random.default_rng(seed + 7)
    ax = [lo[a] + (torch.arange(n[a], dtype=F64, device="cuda") + 0.5) * ((hi[a] - lo[a]) / n[a]) for a in range(d)]
    x = [ax[a].reshape([-1 if d - 1 - b == a else 1 for b in range(d)]) for a in range(d)]

    def waves(amp):
        s = 0.0
        for _ in range(3):
            w, t = 1.0, rng.uniform(0.0, 2.0 * math.pi, d)
            for a in range(d):
                w = w * torch.sin(rng.integers(1, 5) * 2.0 * math.pi / (hi[a] - lo[a]) * x[a] + t[a])
            s = s + amp / 3.0 * w
        return s

    c, e = 0.5 * (verts.max(0) + verts.min(0)), 0.5 * (verts.max(0) - verts.min(0))
    r = sum(((x[a] - c[a]) / e[a]) ** 2 for a in range(d)) ** 0.5
    wall = 1.0 - torch.exp(-torch.clamp(r - 1.0, min=0.0) / 0.4)
    pinf = 1.0 / (gamma * mach * mach)
    load = min(0.4, 0.4 * pinf) * (1.0 - wall * wall) / torch.clamp(r, min=1.0)  # high in front, low behind
    p = pinf + waves(0.03) - load * (x[0] - c[0]) / e[0]
    T = 1.0 + waves(0.02) * min(1.0, mach)
    rho = p / (pinf * T)
    vel = [(uinf[a] + waves(0.05)) * wall for a in range(d)]
    rE = p / (gamma - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [rE]).contiguous()


def _field_of(case, spec, seed):
    if case["kind"] == "step3d":
        return _field(spec["n"], spec["lo"], spec["hi"], spec["verts"], spec["mach"], spec["gamma"], spec["uinf"], seed)
    x0, x1, y0, y1 = spec["domain"]
    return _field((spec["nx"], spec["ny"]), (x0, y0), (x1, y1), spec["verts"], spec["mach"], spec["gamma"],
                  spec["uinf"], seed)


def _lattice(case):
    return (case["nx"], case["ny"], case["nz"]), (-2.0, -2.0, -2.0), (2.0, 2.0, 2.0)


def _listed_nodes(case):
    """About how many nodes lie in the four layers (IB and three ghost) at the unit sphere."""
    n, lo, hi = _lattice(case)
    h = [(hi[a] - lo[a]) / n[a] for a in range(3)]
    return 4.0 * math.pi * 4.0 / (h[0] * h[1] * h[2]) * (h[0] + h[1] + h[2]) / 3.0


def _records(case):
    """Entries of the caller's record buffer: room for every seed's list (unused ones stay zero)."""
    return int(2.0 * _listed_nodes(case)) + 4096


def _pinned(shape, dtype):
    n = int(np.prod(shape)) * np.dtype(dtype).itemsize
    return torch.zeros(n, dtype=torch.uint8, pin_memory=True).numpy().view(dtype).reshape(shape)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "body3d":
        # the program's own page-locked result buffers
        return dict(kind=kind, body=ibm.Body3D(*_mesh(case, seed, 1.0)), lattice=_lattice(case),
                    tags=_pinned((case["nz"], case["ny"], case["nx"]), np.uint8), counts=_pinned(4, np.int32),
                    rec=_pinned(_records(case), ibm.CLOSEST3D_DTYPE))
    if kind == "serve":
        return dict(kind=kind, specs=_specs_serve(case, seed), server=ibm.Server(max_active=32, steps_per_chunk=10))
    spec = _spec3d(case, seed) if kind == "step3d" else _spec2d(case, seed)
    u0 = _field_of(case, spec, seed)
    solver = ibm.Case3D(spec) if kind == "step3d" else ibm.Case(spec)
    return dict(kind=kind, case=solver, u0=u0, u=torch.empty_like(u0), steps=case.get("steps", 1), bits=case["bits"])


# ---- one pass -----------------------------------------------------------------------------------------------------


def _ok(status):
    if status != ibm.IBM_OK:
        raise ibm.IbmError(status, ibm.lib().ibm_last_error().decode())


def run(state):
    kind = state["kind"]
    if kind == "body3d":
        b = state["body"]
        b.classify(*state["lattice"])
        for what, dst in ((ibm.IBM_3D_TAGS, "tags"), (ibm.IBM_3D_COUNTS, "counts"), (ibm.IBM_3D_CLOSEST, "rec")):
            a = state[dst]
            _ok(ibm.lib().ibm_body3d_get(b.h, what, a.ctypes.data_as(ctypes.c_void_p), a.nbytes))
        rec = state["rec"]
        return dict(tags=state["tags"], counts=state["counts"], node=rec["node"], tri=rec["tri"], feature=rec["kind"],
                    cp=rec["cp"], n=rec["n"])
    if kind == "serve":
        s = state["server"]
        ids = [s.submit(spec, n) for spec, n in state["specs"]]
        s.drain()
        res = [s.poll(i) for i in ids]
        return dict(forces=np.stack([r["forces"] for r in res]).astype(np.float32),
                    t=np.array([r["t"] for r in res], np.float32), steps=np.array([r["steps_done"] for r in res]),
                    status=np.array([r["status"] for r in res]))
    c, u0, u = state["case"], state["u0"], state["u"]
    nbytes = u0.numel() * 8
    if kind == "step3d":
        L = ibm.lib()
        _ok(L.ibm_case3d_set_state(c.h, ctypes.c_void_p(u0.data_ptr()), nbytes, 1))
        _ok(L.ibm_case3d_step(c.h, state["steps"]))
        _ok(L.ibm_case3d_get(c.h, ibm.IBM_3D_STATE, ctypes.c_void_p(u.data_ptr()), nbytes, 1))
    else:
        c.set_state_from_ptr(u0.data_ptr(), nbytes, True, wait=False)
        c.step(state["steps"])
        c.state_to_device(u)
    f = c.forces()
    if state["bits"] == 32:
        return dict(field=u.float(), forces=f.astype(np.float32))
    return dict(field=u, forces=f)


def work(case):
    kind = case["kind"]
    if kind == "body3d":
        n = _lattice(case)[0]
        # one tag per node, one record and one face test per listed node, three axis rays per line
        lines = n[0] * n[1] + n[1] * n[2] + n[2] * n[0]
        return dict(bytes=n[0] * n[1] * n[2] + 64.0 * _listed_nodes(case),
                    flops=100.0 * _listed_nodes(case) + 60.0 * lines)
    if kind == "serve":
        b = f = 0.0
        for spec, n in _specs_serve(case, 0):
            cells = spec["nx"] * spec["ny"]
            dual = spec["time_scheme"] == W.TIME_DUAL
            b += 2 * 4 * 4.0 * cells * n
            f += (STAGE_FLOPS_2D + DUAL_FLOPS * dual) * 3.0 * cells * n * (spec["subiters"] if dual else 1)
        return dict(bytes=b, flops=f)
    per = 4.0 if case["bits"] == 32 else 8.0
    if kind == "step3d":
        cells = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=2 * 5 * 8.0 * cells + 2 * 5 * per * cells * case["steps"],
                    flops=STAGE_FLOPS_3D * 3.0 * cells * case["steps"])
    cells = case["nx"] * case["ny"]
    steps = case.get("steps", 1) * (case["subiters"] if kind == "dual2d" else 1)
    return dict(bytes=2 * 4 * 8.0 * cells + 2 * 4 * per * cells * steps,
                flops=(STAGE_FLOPS_2D + (DUAL_FLOPS if kind == "dual2d" else 0)) * 3.0 * cells * steps)


# ---- the same in plain 64-bit torch -------------------------------------------------------------------------------

FLUID, SOLID, IB, G1 = 0, 1, 2, 3


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _shift(t, d, s, fill):
    """t moved so that entry i holds t[i + s] along dimension d."""
    r, n = torch.full_like(t, fill), t.shape[d]
    if abs(s) < n:
        r.narrow(d, max(0, -s), n - abs(s)).copy_(t.narrow(d, max(0, s), n - abs(s)))
    return r


def _tags(solid):
    tag = torch.where(solid, SOLID, FLUID)
    level = torch.zeros_like(tag)
    for s in (3, 2, 1):
        for d in range(solid.ndim):
            for sg in (s, -s):
                level = torch.where(~_shift(solid, d, sg, True), s, level)
                if s == 1:
                    tag = torch.where(~solid & _shift(solid, d, sg, False), IB, tag)
    return torch.where(solid & (level > 0), G1 - 1 + level, tag)


class _Exact:
    """A flow on a uniform block in 64 bits, in `d` dimensions; subclasses bring the body."""

    def __init__(self, n, lo, hi, bc, spec):
        self.n, self.d, self.lo, self.bc, self.spec = n, len(n), lo, bc, spec
        self.h = [(hi[a] - lo[a]) / n[a] for a in range(self.d)]
        self.diag, self.dmin = math.sqrt(sum(h * h for h in self.h)), min(self.h)
        self.g = spec["gamma"]
        self.R = self.pinf = 1.0 / (self.g * spec["mach"] ** 2)
        self.cp = self.g * self.R / (self.g - 1.0)
        self.mu = 1.0 / spec["re"] if spec["re"] > 0.0 else 0.0
        self.kap = self.mu * self.cp / spec["prandtl"]
        u = spec["uinf"]
        self.Uinf = [1.0] + list(u) + [self.pinf / (self.g - 1.0) + 0.5 * sum(v * v for v in u)]
        self.t, self.dual = 0.0, spec.get("time_scheme", W.TIME_RK3) == W.TIME_DUAL
        self.advance, self.quad = spec.get("ib_mode") == W.IB_ADVANCE, spec.get("ib_interp") == W.INTERP_QUADRATIC
        self.tvd = spec.get("scheme") == W.SCHEME_TVD2
        self.bits = [[b >> a & 1 for a in range(self.d)] for b in range(1 << self.d)]

    # cell index [M, d] (x first) of flat node numbers, and centres
    def cells(self, node):
        out = []
        for a in range(self.d):
            out.append(node % self.n[a])
            node = torch.div(node, self.n[a], rounding_mode="floor")
        return torch.stack(out, 1)

    def flat(self, ijk):
        f = ijk[:, self.d - 1]
        for a in range(self.d - 2, -1, -1):
            f = f * self.n[a] + ijk[:, a]
        return f

    def centre(self, ijk):
        return torch.stack([self.lo[a] + (ijk[:, a].to(F64) + 0.5) * self.h[a] for a in range(self.d)], 1)

    def weights(self, X, ok):
        """Corner nodes [M, 2^d] and weights around X; ok: flat mask of usable nodes."""
        base = torch.stack([torch.floor((X[:, a] - self.lo[a]) / self.h[a] - 0.5).long() for a in range(self.d)], 1)
        f = (X - self.centre(base)) / torch.tensor(self.h, dtype=F64, device="cuda")
        node, use, lin, inv = [], [], [], []
        for b in self.bits:
            c = base + torch.tensor(b, device="cuda")
            inside = torch.ones_like(c[:, 0], dtype=torch.bool)
            for a in range(self.d):
                inside &= (c[:, a] >= 0) & (c[:, a] < self.n[a])
            fl = torch.where(inside, self.flat(c), torch.zeros_like(c[:, 0]))
            w = 1.0
            for a in range(self.d):
                w = w * (f[:, a] if b[a] else 1.0 - f[:, a])
            node.append(fl)
            use.append(inside & ok[fl])
            lin.append(w)
            inv.append(1.0 / ((X - self.centre(c)) ** 2).sum(1))
        node, use, lin, inv = (torch.stack(v, 1) for v in (node, use, lin, inv))
        hit = torch.isinf(inv) & use
        inv = torch.where(hit.any(1, keepdim=True), hit.to(F64), torch.where(use, inv, torch.zeros_like(inv)))
        inv = inv / inv.sum(1, keepdim=True)
        w = torch.where(use.all(1, keepdim=True), lin, inv)
        return node, torch.where(use, w, torch.zeros_like(w)), use.any(1)

    def probe(self, b, nrm, xi, ok):
        """weights() at b + xi n, pushed out by dmin up to three times while no corner is usable."""
        node, w, found = self.weights(b + xi[:, None] * nrm, ok)
        for _ in range(3):
            if bool(found.all()):
                break
            xi = torch.where(found, xi, xi + self.dmin)
            node, w, found = self.weights(b + xi[:, None] * nrm, ok)
        return node, w, xi, found

    def build_stencils(self, tag, geometry):
        """geometry(nodes, ghost) -> boundary point, normal, xi_node, curvature."""
        self.tag = tag
        ft = tag.reshape(-1)
        self.sets = []
        for ghost in (False, True):
            nodes = torch.nonzero(ft >= G1 if ghost else ft == IB).reshape(-1)
            if nodes.numel() == 0:
                continue
            b, nrm, xi, curv = geometry(nodes, ghost)
            xp = torch.clamp(-xi, min=0.5 * self.dmin) if ghost else xi + self.diag
            ok = (ft == FLUID) | (ft == IB) if ghost else ft == FLUID
            node, w, xp, _ = self.probe(b, nrm, xp, ok)
            s = dict(ghost=ghost, nodes=nodes, b=b, n=nrm, xi=xi, curv=curv, node=node, w=w, xp=xp)
            if self.quad:
                s["node2"], s["w2"], s["xp2"], s["found2"] = self.probe(b, nrm, xp + self.diag, ok)
            self.sets.append(s)

    def prims(self, U):
        """rho, velocities, p of conserved U[1 + d + 1, ...]."""
        vel = U[1:-1] / U[:1]
        p = (self.g - 1.0) * (U[-1:] - 0.5 * U[:1] * (vel * vel).sum(0, keepdim=True))
        return torch.cat([U[:1], vel, p])

    def motion(self, t):
        z = torch.zeros(self.d, dtype=F64, device="cuda")
        if self.spec.get("motion", W.MOTION_STATIC) != W.MOTION_SIN:
            return z, z, z
        w, amp = 2.0 * math.pi * self.spec["freq"], _dev(np.array(self.spec["amp"]))
        return amp * math.sin(w * t), amp * w * math.cos(w * t), -amp * w * w * math.sin(w * t)

    def supersonic(self, V):
        return (self.spec.get("motion", W.MOTION_STATIC) != W.MOTION_STATIC and
                float(((V - _dev(np.array(self.spec["uinf"]))) ** 2).sum()) > self.g * self.R)

    def at(self, Uf, node, w):
        """(p, velocities, T) [d + 2, M] interpolated on corners."""
        q = self.prims(Uf[:, node])
        q = torch.cat([q[-1:], q[1:-1], q[-1:] / (q[:1] * self.R)])
        return (q * w).sum(-1)

    def reconstruct(self, U, t):
        Uf = U.view(U.shape[0], -1)
        _, V, A = self.motion(t)
        sup = self.supersonic(V)
        for s in self.sets:
            if self.advance and not s["ghost"]:
                continue
            q = self.at(Uf, s["node"], s["w"])
            G = -(s["n"] @ A)
            if sup:
                ut = -(q[1] - V[0]) * s["n"][:, 1] + (q[2] - V[1]) * s["n"][:, 0]
                G = G + ut * ut * s["curv"]
            Vw, s1, sn = V[:, None], s["xp"], s["xi"]
            p = q[0] * torch.exp(-(s1 - sn) * G / (self.R * q[-1]))
            vel, T = Vw + (q[1:-1] - Vw) * (sn / s1), q[-1]
            if self.quad:
                r, s2 = self.at(Uf, s["node2"], s["w2"]), s["xp2"]
                m = (sn * sn - s1 * s1) / (s2 * s2 - s1 * s1)
                L1, L2 = sn * (sn - s2) / (s1 * (s1 - s2)), sn * (sn - s1) / (s2 * (s2 - s1))
                p2 = q[0] + (r[0] - q[0]) * m + q[0] / (self.R * q[-1]) * G * ((sn - s1) - (s2 - s1) * m)
                vel2 = Vw + (q[1:-1] - Vw) * L1 + (r[1:-1] - Vw) * L2
                T2, f = q[-1] + (r[-1] - q[-1]) * m, s["found2"]
                p, vel, T = torch.where(f, p2, p), torch.where(f, vel2, vel), torch.where(f, T2, T)
            rho = p / (self.R * T)
            Uf[:, s["nodes"]] = torch.cat([rho[None], rho * vel,
                                           (p / (self.g - 1.0) + 0.5 * rho * (vel * vel).sum(0))[None]])

    def padded(self, U):
        """Three halo layers; the axes from the last to x."""
        for a in range(self.d - 1, -1, -1):
            dim, parts = U.ndim - 1 - a, []
            for side in (0, 1):
                bc = self.bc[2 * a + side]
                if bc == W.BC_PERIODIC:
                    h = U.narrow(dim, U.shape[dim] - 3 if side == 0 else 0, 3)
                else:
                    h = U.narrow(dim, 0 if side == 0 else U.shape[dim] - 1, 1).repeat_interleave(3, dim)
                    if bc == W.BC_FREESTREAM:
                        h = torch.tensor(self.Uinf, dtype=F64, device="cuda").reshape([-1] + [1] * self.d).expand(
                            h.shape)
                parts.append(h)
            U = torch.cat([parts[0], U, parts[1]], dim)
        return U

    def box(self, q, starts, sizes):
        """The part of padded q[..., z, y, x] that begins at starts (x first)."""
        for a in range(self.d):
            q = q.narrow(q.ndim - 1 - a, starts[a], sizes[a])
        return q

    @staticmethod
    def weno(f0, f1, f2, f3, f4):
        a0, a1, a2 = f0 - 2.0 * f1 + f2, f1 - 2.0 * f2 + f3, f2 - 2.0 * f3 + f4
        c = 13.0 / 12.0
        b0 = c * a0 * a0 + 0.25 * (f0 - 4.0 * f1 + 3.0 * f2) ** 2
        b1 = c * a1 * a1 + 0.25 * (f1 - f3) ** 2
        b2 = c * a2 * a2 + 0.25 * (3.0 * f2 - 4.0 * f3 + f4) ** 2
        w0, w1, w2 = 0.1 / (1e-6 + b0) ** 2, 0.6 / (1e-6 + b1) ** 2, 0.3 / (1e-6 + b2) ** 2
        s = w0 * (2.0 * f0 - 7.0 * f1 + 11.0 * f2) + w1 * (-f1 + 5.0 * f2 + 2.0 * f3) + w2 * (2.0 * f2 + 5.0 * f3 - f4)
        return s / (6.0 * (w0 + w1 + w2))

    @staticmethod
    def minmod(f0, f1, f2):
        a, b = f1 - f0, f2 - f1
        m = torch.where(a.abs() < b.abs(), a, b)
        return f1 + 0.5 * torch.where(a * b > 0.0, m, torch.zeros_like(m))

    def ldfss(self, L, R, a):
        """Face flux of states (rho, velocities, p) along axis a; low-Mach scaled in dual time."""
        g = self.g
        rL, rR, pL, pR, uL, uR = L[0], R[0], L[-1], R[-1], L[1:-1], R[1:-1]
        cL, cR = torch.sqrt(g * pL / rL), torch.sqrt(g * pR / rR)
        HL = g / (g - 1.0) * pL / rL + 0.5 * (uL * uL).sum(0)
        HR = g / (g - 1.0) * pR / rR + 0.5 * (uR * uR).sum(0)
        cb, ub = 0.5 * (cL + cR), 0.5 * (uL[a] + uR[a])
        cs, mr2 = cb, torch.ones_like(cb)
        if self.dual:
            Vm = torch.sqrt(((0.5 * (uL + uR)) ** 2).sum(0))
            Ur = torch.maximum(torch.clamp(Vm, min=1.0), self.mu / (0.5 * (rL + rR)) / self.h[a])
            mr2 = torch.clamp((torch.minimum(Ur, cb) / cb) ** 2, max=1.0)
            cs = 0.5 * torch.sqrt((1.0 - mr2) ** 2 * ub * ub + 4.0 * mr2 * cb * cb)

        def split(m, sg):  # supersonic switch and subsonic flag of one side
            return (sg * m >= 0.0 if sg > 0 else m < 0.0).to(F64), (m.abs() < 1.0).to(F64)

        ML, MR = uL[a] / cs, uR[a] / cs
        (aL, bL), (aR, bR) = split(ML, 1), split(MR, -1)
        CL = aL * (1.0 - bL) * ML + bL * 0.25 * (ML + 1.0) ** 2
        CR = aR * (1.0 - bR) * MR - bR * 0.25 * (MR - 1.0) ** 2
        Mh = 0.25 * bL * bR * (torch.sqrt(0.5 * (ML * ML + MR * MR)) - 1.0) ** 2
        dp = pL - pR
        Cp = CL - Mh * (1.0 - (dp + dp.abs()) / (2.0 * rL * cs * cs))
        Cm = CR + Mh * (1.0 - (dp.abs() - dp) / (2.0 * rR * cs * cs))
        m1, m2 = (torch.where(mr2 < 1.0, u[a] / cb, u[a] / cs) for u in (uL, uR))
        (aL, bL), (aR, bR) = split(m1, 1), split(m2, -1)
        DL = aL * (1.0 - bL) + bL * 0.25 * (m1 + 1.0) ** 2 * (2.0 - m1)
        DR = aR * (1.0 - bR) + bR * 0.25 * (m2 - 1.0) ** 2 * (2.0 + m2)
        ph = torch.where(mr2 < 1.0, 0.5 * (pL + pR) + cs / cb * ((DL - 0.5) * pL + (DR - 0.5) * pR),
                         DL * pL + DR * pR)
        mL, mR = rL * cs * Cp, rR * cs * Cm
        F = [mL + mR] + [mL * uL[c] + mR * uR[c] for c in range(self.d)] + [mL * HL + mR * HR]
        F[1 + a] = F[1 + a] + ph
        return torch.stack(F)

    def residual(self, U):
        """-(sum of flux differences) over the interior."""
        d, n = self.d, list(self.n)
        Q = self.prims(self.padded(U))
        T = Q[-1] / (Q[0] * self.R)
        out = 0.0
        for a in range(d):
            size = [n[c] + (c == a) for c in range(d)]

            def part(q, off, b=None, o=0):  # q at the face's lower cell moved by off along a and o along b
                st = [3 - (c == a) + off * (c == a) + (o if c == b else 0) for c in range(d)]
                return self.box(q, st, size)

            f = [part(Q, k - 2) for k in range(6)]
            if self.tvd:
                L, R = self.minmod(f[1], f[2], f[3]), self.minmod(f[4], f[3], f[2])
            else:
                L, R = self.weno(*f[:5]), self.weno(*f[:0:-1])
            bad = ~((L[0] > 0.0) & (L[-1] > 0.0) & (R[0] > 0.0) & (R[-1] > 0.0))
            L, R = torch.where(bad, f[2], L), torch.where(bad, f[3], R)
            F = self.ldfss(L, R, a)
            if self.mu > 0.0:
                V, lo, hi = Q[1:-1], f[2][1:-1], f[3][1:-1]
                G = [None] * d  # G[b][c] = d u_c / d x_b
                G[a] = (hi - lo) / self.h[a]
                for b in range(d):
                    if b != a:
                        G[b] = (part(V, 0, b, 1) - part(V, 0, b, -1) + part(V, 1, b, 1) - part(V, 1, b, -1)) / (
                            4.0 * self.h[b])
                div = sum(G[b][b] for b in range(d))
                tau = torch.stack([self.mu * (G[a][c] + G[c][a] - (2.0 / 3.0 * div if c == a else 0.0))
                                   for c in range(d)])
                F[1:-1] -= tau
                F[-1] -= (0.5 * (lo + hi) * tau).sum(0) + self.kap * (part(T, 1) - part(T, 0)) / self.h[a]
            dim = F.ndim - 1 - a
            out = out - (F.narrow(dim, 1, n[a]) - F.narrow(dim, 0, n[a])) / self.h[a]
        return out

    def live(self):
        return (self.tag == FLUID) | (self.tag == IB) if self.advance else self.tag == FLUID

    def diffusion(self):
        return 2.0 * self.g * self.mu / self.spec["prandtl"] * sum(1.0 / (h * h) for h in self.h)

    def explicit_step(self, A):
        live = self.live()
        Q = self.prims(A)
        c = torch.sqrt(self.g * Q[-1] / Q[0])
        lam = sum((Q[1 + a].abs() + c) / self.h[a] for a in range(self.d)) + self.diffusion() / Q[0]
        dt = self.spec["dt_fixed"] or self.spec["cfl"] / float(lam[live].max())
        B, C = (torch.tensor(self.Uinf, dtype=F64, device="cuda").reshape([-1] + [1] * self.d).repeat(1, *A.shape[1:])
                for _ in range(2))
        sets, out = [A, B, C], [B, C, A]
        for k, (ca, cb, ts) in enumerate(((0.0, 1.0, 0.0), (0.75, 0.25, dt), (1.0 / 3.0, 2.0 / 3.0, 0.5 * dt))):
            self.reconstruct(sets[k], self.t + ts)
            new = ca * A + cb * (sets[k] + dt * self.residual(sets[k]))
            out[k].copy_(torch.where(live, new, out[k]))
        self.t += dt

    def dual_step(self, A):
        """The first physical step (BDF1) of dual time."""
        s, live, Wn, dt, g = self.spec, self.live(), A.clone(), self.spec["dt_phys"], self.g
        B, C = A.clone(), A.clone()
        sets, out = [A, B, C], [B, C, A]
        for _ in range(s["subiters"]):
            Q0 = None
            for k, (ca, cb) in enumerate(((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))):
                X = sets[k]
                self.reconstruct(X, self.t + dt)
                S = self.residual(X) - (X - Wn) / dt
                q = self.prims(X)
                r, vel, p = q[0], q[1:-1], q[-1]
                T = p / (r * self.R)
                c, Vm = torch.sqrt(g * p / r), torch.sqrt((vel * vel).sum(0))
                Ur = torch.minimum(torch.maximum(torch.clamp(Vm, min=1.0), self.mu / r / self.dmin), c)
                mr2 = (Ur / c) ** 2
                lam = (0.5 * Vm * (1.0 + mr2) + 0.5 * torch.sqrt((1.0 - mr2) ** 2 * Vm * Vm + 4.0 * Ur * Ur)) * sum(
                    1.0 / h for h in self.h) + self.diffusion() / r
                idt, a, rT = lam / s["cfl_tau"], 1.0 / dt, -r / T
                th = idt * (1.0 / (Ur * Ur) + 1.0 / (T * self.cp)) + a / (self.R * T)
                sc, H = idt + a, self.cp * T + 0.5 * (vel * vel).sum(0)
                du = (S[1:-1] - vel * S[0]) / (sc * r)
                Y = (S[-1] - H * S[0]) / sc - r * (vel * du).sum(0)  # r cp dT - dp
                dT = (S[0] + th * Y) / (th * r * self.cp + sc * rT)
                dp = r * self.cp * dT - Y
                q = torch.cat([p[None], vel, T[None]])
                Q0 = q if Q0 is None else Q0
                q = ca * Q0 + cb * (q + torch.cat([dp[None], du, dT[None]]))
                rn = q[0] / (self.R * q[-1])
                new = torch.cat([rn[None], rn * q[1:-1], (q[0] / (g - 1.0) + 0.5 * rn * (q[1:-1] ** 2).sum(0))[None]])
                out[k].copy_(torch.where(live, new, out[k]))
        self.t += dt

    def force_on(self, A, mid, nrm, tang, area, curv):
        """The summed force of the surface elements; tang: unit tangents (2-D), None: the projected velocity."""
        _, V, Acc = self.motion(self.t)
        ok = self.tag.reshape(-1) == FLUID
        node, w, xi, found = self.probe(mid, nrm, torch.full_like(area, self.diag), ok)
        q = self.at(A.view(A.shape[0], -1), node, w)
        G = -(nrm @ Acc)
        rel = (q[1:-1] - V[:, None]).T
        along = (rel * tang).sum(1, keepdim=True) * tang if tang is not None else rel - (rel * nrm).sum(
            1, keepdim=True) * nrm
        if self.supersonic(V):
            G = G + (along ** 2).sum(1) * curv
        ps = q[0] * torch.exp(-xi * G / (self.R * q[-1]))
        F = (-(ps - self.pinf)[:, None] * nrm + self.mu * along / xi[:, None]) * area[:, None]
        return torch.where(found[:, None], F, torch.zeros_like(F)).sum(0)


class _Exact2D(_Exact):
    def __init__(self, spec):
        x0, x1, y0, y1 = spec["domain"]
        super().__init__((spec["nx"], spec["ny"]), (x0, y0), (x1, y1), spec["bc"], spec)
        self.ref = _dev(np.asarray(spec["verts"], np.float64))
        e2 = torch.roll(self.ref, -1, 0) - self.ref
        self.sn = torch.stack([e2[:, 1], -e2[:, 0]], 1) / e2.norm(dim=1, keepdim=True)
        s = torch.roll(self.sn, 1, 0) + self.sn
        self.vn = s / s.norm(dim=1, keepdim=True)
        e1 = torch.roll(e2, 1, 0)
        self.vk = 2.0 * (e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0]) / (
            e1.norm(dim=1) * e2.norm(dim=1) * (e1 + e2).norm(dim=1))

    def classify(self):
        v = self.v = self.ref + self.motion(self.t)[0]
        nv, (nx, ny) = v.shape[0], self.n
        b = torch.roll(v, -1, 0)
        X, Y = (self.lo[a] + (torch.arange(self.n[a], dtype=F64, device="cuda") + 0.5) * self.h[a] for a in (0, 1))
        solid = torch.zeros((ny, nx), dtype=torch.bool, device="cuda")
        rows = torch.nonzero((Y >= v[:, 1].min()) & (Y <= v[:, 1].max())).reshape(-1)
        cols = (X >= v[:, 0].min()) & (X <= v[:, 0].max())
        for r in rows.split(64):
            y = Y[r][:, None]
            cross = (v[:, 1] > y) != (b[:, 1] > y)
            at = torch.where(cross, v[:, 0] + (y - v[:, 1]) * (b[:, 0] - v[:, 0]) / (b[:, 1] - v[:, 1]), -math.inf)
            odd = torch.zeros((r.numel(), nx), dtype=torch.long, device="cuda")
            for k in range(0, nv, 64):
                odd += (at[:, None, k:k + 64] > X[None, :, None]).sum(2)
            solid[r] = (odd % 2 == 1) & cols
        self.build_stencils(_tags(solid), self.geometry)

    def geometry(self, nodes, ghost):
        P = self.centre(self.cells(nodes))
        a, e = self.v, torch.roll(self.v, -1, 0) - self.v
        nv, inf = a.shape[0], math.inf
        b, nrm, xi, curv = [], [], [], []
        for p in P.split(4096):
            w = p[:, None] - a
            u = ((w * e).sum(2) / (e * e).sum(1)).clamp(0.0, 1.0)
            c = a + u[..., None] * e
            c = torch.where((u >= 1.0)[..., None], torch.roll(a, -1, 0).expand_as(c), c)
            d2 = ((p[:, None] - c) ** 2).sum(2)
            k = d2.argmin(1)
            m = torch.arange(p.shape[0], device="cuda")
            uk, ck = u[m, k], c[m, k]
            vert = (uk <= 0.0) | (uk >= 1.0)
            feat = torch.where(uk >= 1.0, (k + 1) % nv, k)
            n = torch.where(vert[:, None], self.vn[feat], self.sn[feat])
            # the crossing of the line along n with the polyline nearest the node, on the surface's side
            den = e[:, 0] * n[:, 1:] - e[:, 1] * n[:, :1]
            uu = (w[..., 0] * n[:, 1:] - w[..., 1] * n[:, :1]) / den
            s = (w[..., 0] * e[:, 1] - w[..., 1] * e[:, 0]) / den
            okc = (den != 0.0) & (uu >= 0.0) & (uu <= 1.0) & ((s >= 0.0) if ghost else (s <= 0.0))
            dist = torch.where(okc, s.abs(), inf)
            j = dist.argmin(1)
            fb = torch.isinf(dist[m, j])
            sj, dk = s[m, j], d2[m, k].sqrt()
            b.append(torch.where(fb[:, None], ck, p + sj[:, None] * n))
            xi.append(torch.where(fb, -dk if ghost else dk, -sj))
            seg, us = torch.where(fb, feat, j), torch.where(fb, uk, uu[m, j])
            cv = (1.0 - us) * self.vk[seg] + us * self.vk[(seg + 1) % nv]
            curv.append(torch.where(fb & vert, self.vk[feat], cv))
            nrm.append(n)
        return torch.cat(b), torch.cat(nrm), torch.cat(xi), torch.cat(curv)

    def advance_steps(self, A, steps):
        for k in range(steps):
            if k == 0 or self.spec["motion"] != W.MOTION_STATIC:
                self.classify()
            self.dual_step(A) if self.dual else self.explicit_step(A)

    def forces(self, A):
        e = torch.roll(self.v, -1, 0) - self.v
        L = e.norm(dim=1)
        tang = e / L[:, None]
        F = self.force_on(A, self.v + 0.5 * e, torch.stack([tang[:, 1], -tang[:, 0]], 1), tang, L,
                          0.5 * (self.vk + torch.roll(self.vk, -1, 0)))
        return torch.cat([F / (0.5 * self.spec["ref_len"]), F])


def _solid3(verts, tris, n, lo, h):
    """Ray parity along x of the lattice nodes [nz, ny, nx]."""
    V = _dev(verts)[_dev(tris).long()]
    X, Y, Z = (lo[a] + (torch.arange(n[a], dtype=F64, device="cuda") + 0.5) * h[a] for a in range(3))
    odd = torch.zeros((n[2], n[1], n[0]), dtype=torch.bool, device="cuda")
    yz = torch.stack(torch.meshgrid(Z, Y, indexing="ij"), -1).reshape(-1, 2)
    flat = odd.view(-1, n[0])
    for first in range(0, yz.shape[0], 4096):
        z, y = yz[first:first + 4096, :1], yz[first:first + 4096, 1:]
        E = []
        for k in range(3):
            a, b = V[:, k], V[:, (k + 1) % 3]
            E.append((b[:, 1] - a[:, 1]) * (z - a[:, 2]) - (b[:, 2] - a[:, 2]) * (y - a[:, 1]))
        hit = ((E[0] > 0) & (E[1] > 0) & (E[2] > 0)) | ((E[0] < 0) & (E[1] < 0) & (E[2] < 0))
        line, f = torch.nonzero(hit, as_tuple=True)
        s = E[0][line, f] + E[1][line, f] + E[2][line, f]
        # the barycentric weight of a vertex is the edge function of the opposite edge
        x = (E[1][line, f] * V[f, 0, 0] + E[2][line, f] * V[f, 1, 0] + E[0][line, f] * V[f, 2, 0]) / s
        par = torch.zeros((yz[first:first + 4096].shape[0], n[0]), dtype=torch.int32, device="cuda")
        par.index_add_(0, line, (x[:, None] > X).to(torch.int32))
        flat[first:first + 4096] = par % 2 == 1
    return odd


def _closest3(verts, tris, P):
    """Closest surface point of every P and the pseudo-normal of its feature (face, edge or vertex)."""
    V, t = _dev(verts), _dev(tris).long()
    A, B, C = V[t[:, 0]], V[t[:, 1]], V[t[:, 2]]
    fn = torch.linalg.cross(B - A, C - A)
    fn = fn / fn.norm(dim=1, keepdim=True)
    vn = torch.zeros_like(V)
    for k in range(3):
        a, b = V[t[:, (k + 1) % 3]] - V[t[:, k]], V[t[:, (k + 2) % 3]] - V[t[:, k]]
        ang = torch.acos(((a * b).sum(1) / (a.norm(dim=1) * b.norm(dim=1))).clamp(-1.0, 1.0))
        vn.index_add_(0, t[:, k], ang[:, None] * fn)
    vn = vn / vn.norm(dim=1, keepdim=True)
    key = {}
    for f, tri in enumerate(tris.tolist()):
        for k in range(3):
            key.setdefault((tri[k], tri[(k + 1) % 3]), f)
    nb = _dev(np.array([[key[(tri[(k + 1) % 3], tri[k])] for k in range(3)] for tri in tris.tolist()]))
    en = fn[:, None] + fn[nb]
    en = en / en.norm(dim=2, keepdim=True)
    e1, e2 = B - A, C - A
    a11, a12, a22 = (e1 * e1).sum(1), (e1 * e2).sum(1), (e2 * e2).sum(1)
    det = a11 * a22 - a12 * a12
    cps, ns = [], []
    for p in P.split(max(1, 12_000_000 // t.shape[0])):
        # p.e = p @ e - A.e keeps the pairs [M, faces] two-dimensional
        w1, w2 = p @ e1.T - (A * e1).sum(1), p @ e2.T - (A * e2).sum(1)
        s, r = (w1 * a22 - w2 * a12) / det, (a11 * w2 - a12 * w1) / det
        inside = (s >= 0.0) & (r >= 0.0) & (s + r <= 1.0)
        plane = (p @ fn.T - (A * fn).sum(1)) ** 2
        best = torch.where(inside, plane, math.inf)
        for k in range(3):
            E0, ed = V[t[:, k]], V[t[:, (k + 1) % 3]] - V[t[:, k]]
            u = ((p @ ed.T - (E0 * ed).sum(1)) / (ed * ed).sum(1)).clamp(0.0, 1.0)
            d2 = sum((p[:, c:c + 1] - E0[:, c] - u * ed[:, c]) ** 2 for c in range(3))
            best = torch.where(inside, best, torch.minimum(best, d2))
        f = best.argmin(1)
        m = torch.arange(p.shape[0], device="cuda")
        # the winning face once more, by differences
        w = p - A[f]
        w1, w2 = (w * e1[f]).sum(1), (w * e2[f]).sum(1)
        s, r = (w1 * a22[f] - w2 * a12[f]) / det[f], (a11[f] * w2 - a12[f] * w1) / det[f]
        inside = (s >= 0.0) & (r >= 0.0) & (s + r <= 1.0)
        c0, n0 = A[f] + s[:, None] * e1[f] + r[:, None] * e2[f], fn[f]
        d0 = torch.where(inside, -1.0, torch.full_like(s, math.inf))
        for k in range(3):
            E0, E1 = V[t[f, k]], V[t[f, (k + 1) % 3]]
            u = (((p - E0) * (E1 - E0)).sum(1) / ((E1 - E0) ** 2).sum(1))
            c = torch.where((u <= 0.0)[:, None], E0, torch.where((u >= 1.0)[:, None], E1,
                                                                 E0 + u[:, None] * (E1 - E0)))
            n = torch.where((u <= 0.0)[:, None], vn[t[f, k]],
                            torch.where((u >= 1.0)[:, None], vn[t[f, (k + 1) % 3]], en[f, k]))
            d = ((p - c) ** 2).sum(1)
            nearer = (d < d0)[:, None]
            c0, n0, d0 = torch.where(nearer, c, c0), torch.where(nearer, n, n0), torch.minimum(d, d0)
        cps.append(c0)
        ns.append(n0)
    return torch.cat(cps), torch.cat(ns)


class _Exact3D(_Exact):
    def __init__(self, spec):
        super().__init__(spec["n"], spec["lo"], spec["hi"], spec["bc"], spec)
        self.verts, self.tris = spec["verts"], spec["tris"]
        self.build_stencils(_tags(_solid3(self.verts, self.tris, self.n, self.lo, self.h)), self.geometry)

    def geometry(self, nodes, ghost):
        X = self.centre(self.cells(nodes))
        c, n = _closest3(self.verts, self.tris, X)
        xi = ((X - c) * n).sum(1)
        return X - xi[:, None] * n, n, xi, None

    def advance_steps(self, A, steps):
        for _ in range(steps):
            self.explicit_step(A)

    def forces(self, A):
        v = _dev(self.verts)[_dev(self.tris).long()]
        cr = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
        L = cr.norm(dim=1)
        F = self.force_on(A, v.sum(1) / 3.0, cr / L[:, None], None, 0.5 * L, None)
        return torch.cat([F / (0.5 * self.spec["ref_area"]), F])


def exact(case, seed):
    kind = case["kind"]
    if kind == "body3d":
        verts, tris = _mesh(case, seed, 1.0)
        n, lo, hi = _lattice(case)
        h = [(hi[a] - lo[a]) / n[a] for a in range(3)]
        tag = _tags(_solid3(verts, tris, n, lo, h)).reshape(-1)
        nodes = torch.cat([torch.nonzero(tag == k).reshape(-1) for k in (IB, G1, G1 + 1, G1 + 2)])
        ijk = torch.stack([nodes % n[0], nodes // n[0] % n[1], nodes // (n[0] * n[1])], 1).to(F64)
        P = torch.stack([lo[a] + (ijk[:, a] + 0.5) * h[a] for a in range(3)], 1)
        cp, nrm = (torch.cat([v, torch.zeros(_records(case) - v.shape[0], 3, dtype=F64, device="cuda")])
                   for v in _closest3(verts, tris, P))
        return dict(tags=None, counts=None, node=None, tri=None, feature=None, cp=cp, n=nrm)
    if kind == "serve":
        forces, t = [], []
        for spec, steps in _specs_serve(case, seed):
            e = _Exact2D(spec)
            A = torch.tensor(e.Uinf, dtype=F64, device="cuda").reshape(4, 1, 1).repeat(1, spec["ny"], spec["nx"])
            e.advance_steps(A, steps)
            forces.append(e.forces(A))
            t.append(e.t)
        return dict(forces=torch.stack(forces), t=torch.tensor(t, dtype=F64), steps=None, status=None)
    spec = _spec3d(case, seed) if kind == "step3d" else _spec2d(case, seed)
    A = _field_of(case, spec, seed)
    e = _Exact3D(spec) if kind == "step3d" else _Exact2D(spec)
    e.advance_steps(A, case.get("steps", 1))
    return dict(field=A, forces=e.forces(A))
