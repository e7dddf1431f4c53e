"""The workloads this library's speed is measured on.

Each case is one pass of a user's program through the public entry points:
a step of a periodic patch (`runner.PeriodicRunner`), a batch of the serving
stream (`serve.GpuBackend`), a coarse step of an AMR hierarchy as one CUDA
graph (`amr.Hierarchy.capture_graph` / `replay`) or through the level-step
server (`serve.AmrLevelServer`), and the reductions and scans a program runs
between coarse steps (`capi.mhd_conservation_sums`, `mhd_cfl_dt`,
`mhd_flag_cells`).  Sizes are those of the library's own configurations: the
128^2 Orszag-Tang vortex, the 128^3 blast, serving cubes of edge 16-128, AMR
patches of edge 8-64 on a base of 32^3 or 64^3.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1112_1710_gb300 import capi
from paper_1112_1710_gb300.amr import Hierarchy
from paper_1112_1710_gb300.patch import Patch, patch_shape
from paper_1112_1710_gb300.runner import PeriodicRunner
from paper_1112_1710_gb300.serve import AmrLevelServer, GpuBackend, Request

GAMMA = 5.0 / 3.0
DT = {"f32": torch.float32, "f64": torch.float64}
# flops of one cell update and of its share of the CFL reduction (each add,
# multiply, division and square root counted once)
FLOPS, FLOPS_CFL = 2200, 92


def listed():
    return [
        # the 2D Orszag-Tang vortex, one eager launch sequence per step: a small
        # call in the default build (FP64 parity, upwinded EMF)
        dict(name="ot2d_128_f64", kind="step", problem="vortex", nx=128, ny=128, nz=1, g=2, dtype="f64",
             contract=0, emf=0, limiter=0, graph=False),
        # a small odd 3D patch stepped eagerly in FP32: launches and host time
        dict(name="box_21x18x25_f32", kind="step", problem="vortex", nx=21, ny=18, nz=25, g=4, dtype="f32",
             contract=0, emf=0, limiter=1, graph=False),
        # the 128^3 blast, one step as a CUDA graph: the headline configuration,
        # in FP32 and in the contracted FP64 build
        dict(name="blast_128_f32", kind="step", problem="blast", nx=128, ny=128, nz=128, g=2, dtype="f32",
             contract=0, emf=1, limiter=0, graph=True),
        dict(name="blast_128_f64c", kind="step", problem="blast", nx=128, ny=128, nz=128, g=2, dtype="f64",
             contract=1, emf=1, limiter=0, graph=True),
        # ragged 3D boxes with the default upwinded EMF: the FP64 parity build,
        # and FP32 with the monotonised-central limiter
        dict(name="box_90x75x66_f64", kind="step", problem="vortex", nx=90, ny=75, nz=66, g=2, dtype="f64",
             contract=0, emf=0, limiter=0, graph=True),
        dict(name="box_149x101x83_f32", kind="step", problem="vortex", nx=149, ny=101, nz=83, g=4, dtype="f32",
             contract=0, emf=0, limiter=2, graph=True),
        # one batch of the serving stream (mixed cube edges, each request with
        # its own dt), in the stream's two precisions
        dict(name="serve_4M_f32", kind="batch", cells=4 << 20, mix=11, dtype="f32", contract=0),
        dict(name="serve_1M_f64c", kind="batch", cells=1 << 20, mix=12, dtype="f64", contract=1),
        # a whole subcycled coarse step of an AMR hierarchy as one CUDA graph:
        # the large FP32 configuration, and a smaller one in the parity build
        dict(name="amr_64_l4_f32", kind="amr", base=64, levels=4, boxes=42, size_max=64, dtype="f32"),
        dict(name="amr_32_l3_f64", kind="amr", base=32, levels=3, boxes=43, size_max=24, dtype="f64"),
        # a deep turbulent hierarchy through the level-step server, each level
        # with children on a stream of its own, density and pressure floors on
        dict(name="deep_32_l5_f32", kind="deep", base=32, levels=5, boxes=5, size_max=64, dtype="f32"),
        # what a program runs over a level between coarse steps: FP64 totals,
        # the CFL dt and the refinement flags
        dict(name="scan_200_f32", kind="scan", patches=200, mix=7, dtype="f32"),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["step", "step", "step", "batch", "amr", "deep", "scan"])
    dtype = rng.choice(["f32", "f64"])
    if kind == "step":
        flat = rng.random() < 0.2
        n = [log_int(16, 160) for _ in range(3)]
        if flat:
            n = [log_int(48, 256), log_int(48, 256), 1]
        problem = "vortex" if flat else rng.choice(["vortex", "blast"])
        if problem == "blast":
            n = [n[0]] * 3
        while n[0] * n[1] * n[2] > 128 ** 3:
            n[n.index(max(n))] //= 2
            if problem == "blast":
                n = [min(n)] * 3
        return dict(kind="step", problem=problem, nx=n[0], ny=n[1], nz=n[2], g=rng.choice([2, 3, 4]), dtype=dtype,
                    contract=rng.choice([0, 1]) if dtype == "f64" else 0, emf=1 if problem == "blast" else rng.choice([0, 1]),
                    limiter=rng.choice([0, 1, 2]), graph=rng.random() < 0.6)
    if kind == "batch":
        return dict(kind="batch", cells=log_int(1 << 15, 4 << 20 if dtype == "f32" else 1 << 20), mix=rng.randrange(1000),
                    dtype=dtype, contract=rng.choice([0, 1]) if dtype == "f64" else 0)
    if kind == "amr":
        levels = rng.choice([2, 3, 4]) if dtype == "f32" else rng.choice([2, 3])
        return dict(kind="amr", base=rng.choice([32, 40, 48]), levels=levels, boxes=rng.randrange(1000),
                    size_max=rng.choice([16, 24, 40, 64]), dtype=dtype)
    if kind == "deep":
        return dict(kind="deep", base=32, levels=rng.choice([3, 4, 5]), boxes=rng.randrange(1000),
                    size_max=rng.choice([24, 40, 64]), dtype="f32")
    return dict(kind="scan", patches=log_int(10, 400), mix=rng.randrange(1000), dtype=dtype)


# ------------------------------------------------------------------ initial data
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _coords(lo, n, dx):
    """Cell-centre coordinates on [-1/2, 1/2] as broadcastable z, y, x arrays."""
    c = [-0.5 + (torch.arange(lo[d], lo[d] + n[d], dtype=torch.float64, device="cuda") + 0.5) * dx[d] for d in range(3)]
    return c[0][None, None, :], c[1][None, :, None], c[2][:, None, None]


def _pack(n, g, prim, B):
    """State array (8, NZ+1, NY+1, PX) of interior primitives (rho, vx, vy, vz,
    p) and interior faces B (each with its extra upper face); ghosts zero."""
    nx, ny, nz = n
    st = torch.zeros(patch_shape(n, g), dtype=torch.float64, device="cuda")
    st[5, g:g + nz, g:g + ny, g:g + nx + 1] = B[0]
    st[6, g:g + nz, g:g + ny + 1, g:g + nx] = B[1]
    st[7, g:g + nz + 1, g:g + ny, g:g + nx] = B[2]
    bx = 0.5 * (B[0][:, :, 1:] + B[0][:, :, :-1])
    by = 0.5 * (B[1][:, 1:] + B[1][:, :-1])
    bz = 0.5 * (B[2][1:] + B[2][:-1])
    rho, vx, vy, vz, p = prim
    c = (slice(g, g + nz), slice(g, g + ny), slice(g, g + nx))
    st[(0,) + c], st[(1,) + c], st[(2,) + c], st[(3,) + c] = rho, rho * vx, rho * vy, rho * vz
    st[(4,) + c] = p / (GAMMA - 1.0) + 0.5 * rho * (vx * vx + vy * vy + vz * vz) + 0.5 * (bx * bx + by * by + bz * bz)
    return st


def _uniform_faces(n, b):
    nx, ny, nz = n
    f = dict(dtype=torch.float64, device="cuda")
    return [torch.full((nz, ny, nx + 1), b[0], **f), torch.full((nz, ny + 1, nx), b[1], **f),
            torch.full((nz + 1, ny, nx), b[2], **f)]


def blast_state(lo, n, g, dx, seed, r0=0.1):
    """Blast wave on [-1/2, 1/2]^3: rho = 1 +- 1% noise, p = 10 inside r < r0
    and 0.1 outside, v = 0, B = (1, 1, 0)/sqrt 2."""
    X, Y, Z = _coords(lo, n, dx)
    p = torch.where(X * X + Y * Y + Z * Z < r0 * r0, 10.0, 0.1).to(torch.float64)
    rho = 1.0 + 0.01 * (2.0 * torch.rand(n[2], n[1], n[0], generator=_gen(seed), dtype=torch.float64, device="cuda") - 1.0)
    v = torch.zeros_like(rho)
    b = 1.0 / math.sqrt(2.0)
    return _pack(n, g, (rho, v, v, v, p), _uniform_faces(n, (b, b, 0.0)))


def vortex_state(n, g, dx, seed):
    """Smooth periodic vortices: the Orszag-Tang vortex with seeded phases, and
    in 3D its field and flow along all three axes.  Face B is the discrete curl
    of an edge-sampled potential, so it is divergence-free to rounding."""
    rng = np.random.default_rng(int(seed) + 31)
    ph = rng.uniform(-0.3, 0.3, 8)
    flat = n[2] == 1
    X, Y, Z = (c + 0.5 for c in _coords((0, 0, 0), n, dx))
    L = [n[d] * dx[d] for d in range(3)]
    k = [2.0 * math.pi / v for v in L]
    one = torch.ones(n[2], n[1], n[0], dtype=torch.float64, device="cuda")
    vx = -torch.sin(k[1] * Y + ph[0]) * one
    vy = torch.sin(k[0] * X + ph[1]) * one
    vz = 0.0 * one if flat else 0.5 * torch.sin(k[0] * X + k[1] * Y + ph[2]) * one
    rho = 25.0 / (36.0 * math.pi) * one
    p = (5.0 / (12.0 * math.pi) if flat else 0.6) * one
    b0 = 1.0 / math.sqrt(4.0 * math.pi)

    def edge(axis, f):
        """f sampled on the edges along `axis` (lower corners elsewhere), with
        one extra entry along the other two axes."""
        c = []
        for d in range(3):
            m = n[d] if d == axis else n[d] + 1
            c.append((torch.arange(m, dtype=torch.float64, device="cuda") + (0.5 if d == axis else 0.0)) * dx[d])
        return f(c[0][None, None, :], c[1][None, :, None], c[2][:, None, None])

    az = edge(2, lambda x, y, z: b0 * (torch.cos(2 * k[0] * x + ph[3]) / (2 * k[0]) + torch.cos(k[1] * y + ph[4]) / k[1]) + 0.0 * z)
    if flat:
        ax, ay = edge(0, lambda x, y, z: 0.0 * (x + y + z)), edge(1, lambda x, y, z: 0.0 * (x + y + z))
    else:
        ax = edge(0, lambda x, y, z: 0.5 * b0 * torch.cos(k[1] * y + k[2] * z + ph[5]) / k[1] + 0.0 * x)
        ay = edge(1, lambda x, y, z: 0.5 * b0 * torch.cos(k[2] * z + ph[6]) / k[2] + 0.0 * (x + y))
    B = [(az[:, 1:] - az[:, :-1]) / dx[1] - (ay[1:] - ay[:-1]) / dx[2],
         (ax[1:] - ax[:-1]) / dx[2] - (az[:, :, 1:] - az[:, :, :-1]) / dx[0],
         (ay[:, :, 1:] - ay[:, :, :-1]) / dx[0] - (ax[:, 1:] - ax[:, :-1]) / dx[1]]
    return _pack(n, g, (rho, vx, vy, vz, p), B)


def _step_state(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    dx = (1.0 / max(n),) * 3 if case["problem"] == "vortex" else (1.0 / n[0],) * 3
    st = (vortex_state(n, case["g"], dx, seed) if case["problem"] == "vortex"
          else blast_state((0, 0, 0), n, case["g"], dx, seed))
    return st.to(DT[case["dtype"]]), n, dx


# ------------------------------------------------------------------ serving batch
def _edges(case):
    """Cube edges of one serving batch: log-uniform in [16, 128], even, until
    the batch holds about case["cells"] cells (at most 48 requests)."""
    rng = np.random.default_rng(case["mix"])
    out, left = [], case["cells"]
    while left > 0 and len(out) < 48:
        n = int(2 * round(math.exp(rng.uniform(math.log(16), math.log(128))) / 2))
        n = max(16, min(n, 2 * int(max(left, 4096) ** (1 / 3) / 2)))
        out.append(n)
        left -= n ** 3
        if left < 4096:
            break
    return out


def _serve_templates(case, seed):
    """{(edge, dtype): (ghost-celled blast cube, its CFL dt)}."""
    out = {}
    for n in sorted(set(_edges(case))):
        dx = (1.0 / n,) * 3
        st = blast_state((0, 0, 0), (n, n, n), 4, dx, seed * 131 + n).to(DT[case["dtype"]])
        # fastest signal of the blast's two states bounds the CFL step
        dt = 0.4 * dx[0] / math.sqrt((GAMMA * 10.0 + 1.0) / 0.99)
        out[(n, case["dtype"])] = (Patch(st, (0, 0, 0), (n, n, n), 4, dx), dt)
    return out


# ------------------------------------------------------------------ AMR boxes
def _cut(rng, a, end, smin, smax):
    """[a, end) cut into consecutive even-length pieces of log-uniform length."""
    out = []
    while a < end:
        s = max(smin, 2 * int(round(math.exp(rng.uniform(math.log(smin), math.log(smax))) / 2)))
        b = end if end - (a + s) < smin else a + s
        out.append((a, b))
        a = b
    return out


def _nested(boxes, n, margin):
    """Summed-area table of the cells of a level (n a side) at least `margin`
    cells inside the union of its boxes and the domain."""
    m = torch.zeros((1, 1, n, n, n), device="cuda")
    for lo, hi in boxes:
        m[0, 0, lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1] = 1.0
    m = torch.nn.functional.pad(m, (margin,) * 6)
    m = (1.0 - torch.nn.functional.max_pool3d(1.0 - m, 2 * margin + 1, stride=1))[0, 0]
    s = np.zeros((n + 1,) * 3, dtype=np.int64)
    s[1:, 1:, 1:] = m.to(torch.int64).cumsum(0).cumsum(1).cumsum(2).cpu().numpy()
    return s


def _count(s, a, b):
    return int(s[b[2], b[1], b[0]] - s[a[2], b[1], b[0]] - s[b[2], a[1], b[0]] - s[b[2], b[1], a[0]]
               + s[a[2], a[1], b[0]] + s[a[2], b[1], a[0]] + s[b[2], a[1], a[0]] - s[a[2], a[1], a[0]])


def _refine(parents, n, rng, size_max, wanted, margin=3, size_min=8):
    """Uneven even-aligned boxes of the level with n cells a side that lie
    `margin` parent cells inside the parent level and that `wanted` keeps;
    a box that sticks out is halved."""
    s = _nested(parents, n // 2, margin)
    cuts = [_cut(rng, 2 * margin, n - 2 * margin, size_min, size_max) for _ in range(3)]
    stack = [tuple(zip(cx, cy, cz)) for cz in cuts[2] for cy in cuts[1] for cx in cuts[0]]
    out = []
    while stack:
        a, b = stack.pop()
        if not wanted(a, b):
            continue
        inside = _count(s, [v // 2 for v in a], [v // 2 for v in b])
        vol = (b[0] - a[0]) * (b[1] - a[1]) * (b[2] - a[2]) // 8
        if inside == vol:
            out.append((a, tuple(v - 1 for v in b)))
        elif inside:
            ext = [b[d] - a[d] for d in range(3)]
            d = ext.index(max(ext))
            if ext[d] < 2 * size_min:
                continue
            mid = a[d] + ext[d] // 4 * 2
            stack.append((a, tuple(mid if e == d else b[e] for e in range(3))))
            stack.append((tuple(mid if e == d else a[e] for e in range(3)), b))
    return sorted(out, key=lambda q: (q[0][2], q[0][1], q[0][0]))


_BOXES = {}


def _boxes(case):
    """Boxes per level: a spherical shell around the blast front (amr), or the
    blocks of seeded strong-gradient centres (deep).  A pure function of the
    case; kept, as a program keeps its grid list."""
    key = (case["kind"], case["base"], case["levels"], case["boxes"], case["size_max"])
    if key in _BOXES:
        return _BOXES[key]
    rng = np.random.default_rng(case["boxes"])
    n0 = case["base"]
    H = [[((0, 0, 0), (n0 - 1,) * 3)]]
    centres = rng.uniform(0.25, 0.75, (4, 3))
    for lev in range(1, case["levels"]):
        n = n0 * 2 ** lev
        if case["kind"] == "amr":
            r1, r2 = 0.25 * (1 + 0.1 * rng.uniform(-1, 1)), 0.35 * (1 + 0.1 * rng.uniform(-1, 1))

            def wanted(a, b):
                near = far = 0.0
                for d in range(3):
                    p, q = a[d] / n - 0.5, b[d] / n - 0.5
                    near += 0.0 if p <= 0.0 <= q else min(p * p, q * q)
                    far += max(p * p, q * q)
                return near <= r2 * r2 and far >= r1 * r1
        else:
            r = 0.22 * 0.72 ** lev

            def wanted(a, b):
                return any(sum(max(a[d] / n - c[d], c[d] - b[d] / n, 0.0) ** 2 for d in range(3)) <= r * r for c in centres)
        bl = _refine(H[-1], n, rng, case["size_max"], wanted)
        if not bl:
            break
        H.append(bl)
    if len(_BOXES) > 32:
        _BOXES.clear()
    _BOXES[key] = H
    return H


def _velocity(seed, m=64, kmax=8, mach=5.0):
    """k^-4 random velocity field (3, m, m, m) of rms speed `mach` on the unit
    periodic cube."""
    gen = _gen(seed)
    k = torch.fft.fftfreq(m, 1.0 / m, device="cuda", dtype=torch.float64)
    kk = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :m // 2 + 1] ** 2).sqrt()
    kk[-1] = kk[-1]
    amp = torch.where((kk >= 1.0) & (kk <= kmax), kk.clamp(min=1.0) ** -2.0, torch.zeros_like(kk))
    v = torch.stack([torch.fft.irfftn(amp * torch.complex(torch.randn(amp.shape, generator=gen, dtype=torch.float64, device="cuda"),
                                                          torch.randn(amp.shape, generator=gen, dtype=torch.float64, device="cuda")),
                                      s=(m, m, m)) for _ in range(3)])
    return v * (mach / float((v * v).sum(0).mean().sqrt()))


def _turb_state(lo, n, g, res, v):
    """Patch of a turbulent level with res cells a side: rho = 1, p = 1/gamma, v
    the field interpolated to the cell centres, uniform B along x at beta 1."""
    m = v.shape[1]
    idx, w = [], []
    for d in range(3):
        u = (torch.arange(lo[d], lo[d] + n[d], dtype=torch.float64, device="cuda") + 0.5) / res * m - 0.5
        i = torch.floor(u)
        idx.append((i.long() % m, (i.long() + 1) % m))
        w.append((1.0 - (u - i), u - i))
    out = 0.0
    for c in (0, 1):
        for b in (0, 1):
            for a in (0, 1):
                wt = w[2][c][:, None, None] * w[1][b][None, :, None] * w[0][a][None, None, :]
                out = out + wt * v[:, idx[2][c][:, None, None], idx[1][b][None, :, None], idx[0][a][None, None, :]]
    p = 1.0 / GAMMA
    one = torch.ones(n[2], n[1], n[0], dtype=torch.float64, device="cuda")
    return _pack(n, g, (one, out[0], out[1], out[2], p * one), _uniform_faces(n, (math.sqrt(2.0 * p), 0.0, 0.0)))


def _hierarchy(case, seed):
    H, n0 = _boxes(case), case["base"]
    deep = case["kind"] == "deep"
    v = _velocity(seed) if deep else None
    states, pools = [], []
    for l, bl in enumerate(H):
        res = n0 * 2 ** l
        size = [tuple(hi[d] - lo[d] + 1 for d in range(3)) for lo, hi in bl]
        shape = [patch_shape(n, 4) for n in size]
        at = np.concatenate([[0], np.cumsum([math.prod(q) for q in shape])])
        pool = torch.empty(int(at[-1]), dtype=DT[case["dtype"]], device="cuda")
        row = []
        for i, ((lo, hi), n, q) in enumerate(zip(bl, size, shape)):
            st = pool[at[i]:at[i + 1]].view(q)
            st.copy_(_turb_state(lo, n, 4, res, v) if deep
                     else blast_state(lo, n, 4, (1.0 / res,) * 3, seed * 10007 + l * 4001 + i))
            row.append(st)
        states.append(row)
        pools.append(pool)
    floors = dict(p_floor=1e-3 / GAMMA, rho_floor=1e-3) if deep else {}
    ctx = capi.mhd_ctx_create(gamma=GAMMA, emf=1, **floors)
    torch.cuda.synchronize()
    h = Hierarchy(H, n0, states, (1.0 / n0,) * 3, g=4, dtype=case["dtype"], ctx=ctx, stream=torch.cuda.Stream(),
                  concurrent=deep, floors=deep)
    h.initialise()
    torch.cuda.synchronize()
    h.own_ctx = True
    return h, pools


class _Hier:
    """A hierarchy with its captured coarse step (amr) or its level-step server
    (deep); freed with the state."""

    def __init__(self, case, seed):
        self.h, self.pools = _hierarchy(case, seed)
        self.server = AmrLevelServer(self.h) if case["kind"] == "deep" else None
        if self.server is None:
            self.h.capture_graph()
        torch.cuda.synchronize()

    def __del__(self):
        torch.cuda.synchronize()
        self.h.close()


class _Step:
    """A periodic patch with its context, stepped eagerly or as a graph."""

    def __init__(self, case, seed):
        st, n, dx = _step_state(case, seed)
        self.ctx = capi.mhd_ctx_create(gamma=GAMMA, emf=case["emf"], limiter=case["limiter"], fp64_contract=case["contract"])
        p = Patch(st, (0, 0, 0), n, case["g"], dx)
        self.graph = case["graph"]
        self.runner = PeriodicRunner(p, self.ctx, torch.cuda.Stream() if self.graph else None)
        if self.graph:
            first = st.clone()
            torch.cuda.synchronize()
            self.runner.capture_graph()
            torch.cuda.synchronize()
            st.copy_(first)
            torch.cuda.synchronize()

    def __del__(self):
        torch.cuda.synchronize()
        capi.mhd_ctx_destroy(self.ctx)


class _Batch:
    def __init__(self, case, seed):
        self.backend = GpuBackend(_serve_templates(case, seed), n_slots=1, g=4, keep=True,
                                  solver=dict(gamma=GAMMA, emf=1, fp64_contract=case["contract"]))
        self.requests = [Request(i, 0.0, n, i % 8, case["dtype"]) for i, n in enumerate(_edges(case))]
        torch.cuda.synchronize()

    def __del__(self):
        torch.cuda.synchronize()
        self.backend.close()


def _scan_sizes(case):
    rng = np.random.default_rng(case["mix"])
    e = np.exp(rng.uniform(math.log(8), math.log(64), (case["patches"], 3)))
    return [tuple(int(v) for v in row) for row in np.clip(2 * np.rint(e / 2), 8, 64)]


def _scan_states(case, seed):
    return [blast_state((-n[0] // 2 + 128, -n[1] // 2 + 128, -n[2] // 2 + 128), tuple(v + 2 for v in n), 3, (1.0 / 256,) * 3,
                        seed * 10007 + i).to(DT[case["dtype"]]) for i, n in enumerate(_scan_sizes(case))]


class _Scan:
    """A level's patches (one valid ghost layer around each interior) and the
    outputs of the scans over them."""

    def __init__(self, case, seed):
        # generated one cell wider on every side: the rim is the ghost layer
        self.patches = [Patch(st, (0, 0, 0), n, 4, (1.0 / 256,) * 3, 2, i)
                        for i, (st, n) in enumerate(zip(_scan_states(case, seed), _scan_sizes(case)))]
        self.descs = [p.desc() for p in self.patches]
        self.ctx = capi.mhd_ctx_create(gamma=GAMMA)
        self.scale = [4.0] * len(self.patches)
        self.sums = torch.zeros(8, dtype=torch.float64, device="cuda")
        self.dt = torch.zeros(1, dtype=torch.float64, device="cuda")
        self.flags = torch.zeros(sum(p.cells for p in self.patches), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()

    def __del__(self):
        torch.cuda.synchronize()
        capi.mhd_ctx_destroy(self.ctx)


def prepare(case, seed):
    return {"step": _Step, "batch": _Batch, "amr": _Hier, "deep": _Hier, "scan": _Scan}[case["kind"]](case, seed)


def run(state):
    if isinstance(state, _Step):
        state.runner.replay() if state.graph else state.runner.step()
        return {"state": state.runner.patch.state, "dt": state.runner.d_dt}
    if isinstance(state, _Batch):
        return state.backend.finish(state.backend.launch(0, state.requests))
    if isinstance(state, _Hier):
        if state.server is not None:
            state.server.run(1, timing=False)
        else:
            state.h.replay()
        return {"dt": state.h.d_dt, "levels": state.pools}  # every patch, one allocation per level
    s = torch.cuda.current_stream().cuda_stream
    capi.mhd_conservation_sums(state.ctx, state.descs, state.sums.data_ptr(), s)
    capi.mhd_cfl_dt(state.ctx, state.descs, state.dt.data_ptr(), s, scale=state.scale)
    capi.mhd_flag_cells(state.ctx, state.descs, 0.02, state.flags.data_ptr(), s)
    return {"sums": state.sums, "dt": state.dt, "flags": state.flags}


def work(case):
    s = 4 if case["dtype"] == "f32" else 8
    if case["kind"] == "step":
        n = (case["nx"], case["ny"], case["nz"])
        cells = n[0] * n[1] * n[2]
        ext = math.prod(v + 2 * case["g"] for v in n)
        return {"bytes": 8 * s * (cells + ext), "flops": (FLOPS + FLOPS_CFL) * cells}
    if case["kind"] == "batch":
        e = _edges(case)
        return {"bytes": 8 * s * sum(n ** 3 + (n + 8) ** 3 for n in e), "flops": FLOPS * sum(n ** 3 for n in e)}
    if case["kind"] == "scan":
        cells = sum(math.prod(n) for n in _scan_sizes(case))
        return {"bytes": (8 * s + 1) * cells, "flops": 150 * cells}
    updates = sum(2 ** l * math.prod(hi[d] - lo[d] + 1 for d in range(3)) for l, bl in enumerate(_boxes(case)) for lo, hi in bl)
    return {"bytes": 16 * s * updates, "flops": FLOPS * updates}


# ------------------------------------------------------------------ 64-bit values
def _sh(a, d, k):
    """a at index + k along axis d (x, y, z = 0, 1, 2) of a periodic array."""
    return torch.roll(a, -k, 2 - d)


def _limit(kind, a, b):
    ab = a * b
    if kind == 1:
        s = torch.where(a.abs() < b.abs(), a, b)
    elif kind == 2:
        s = torch.sign(a) * torch.minimum(torch.minimum(2 * a.abs(), 2 * b.abs()), 0.5 * (a + b).abs())
    else:
        s = 2 * ab / torch.where(ab > 0, a + b, torch.ones_like(a))
    return torch.where(ab > 0, s, torch.zeros_like(s))


def _prim(u):
    v = [u[1] / u[0], u[2] / u[0], u[3] / u[0]]
    p = (GAMMA - 1) * (u[4] - 0.5 * u[0] * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) - 0.5 * (u[5] ** 2 + u[6] ** 2 + u[7] ** 2))
    return [u[0], *v, p, u[5], u[6], u[7]]


def _cons(w):
    e = w[4] / (GAMMA - 1) + 0.5 * w[0] * (w[1] ** 2 + w[2] ** 2 + w[3] ** 2) + 0.5 * (w[5] ** 2 + w[6] ** 2 + w[7] ** 2)
    return [w[0], w[0] * w[1], w[0] * w[2], w[0] * w[3], e, w[5], w[6], w[7]]


def _fast(rho, p, bn, b2):
    a2, c2 = GAMMA * p / rho, (bn * bn + b2) / rho
    s = a2 + c2
    return torch.sqrt(0.5 * (s + torch.sqrt(torch.clamp(s * s - 4 * a2 * bn * bn / rho, min=0.0))))


def _flux(d, w):
    """Physical flux along axis d of a primitive state (own normal field)."""
    v, b = w[1:4], w[5:8]
    pt = w[4] + 0.5 * (b[0] ** 2 + b[1] ** 2 + b[2] ** 2)
    vb = v[0] * b[0] + v[1] * b[1] + v[2] * b[2]
    f = [w[0] * v[d]] + [w[0] * v[d] * v[c] - b[d] * b[c] for c in range(3)]
    f[1 + d] = f[1 + d] + pt
    f.append((_cons(w)[4] + pt) * v[d] - b[d] * vb)
    return f + [b[c] * v[d] - b[d] * v[c] for c in range(3)]


def _hlld(d, wl, wr, bn, eps, degen):
    """HLLD flux (Miyoshi & Kusano 2005) and the upwind side of the contact."""
    wl, wr = list(wl), list(wr)
    wl[5 + d] = wr[5 + d] = bn
    t = [(d + 1) % 3, (d + 2) % 3]
    W = (wl, wr)
    u = [w[1 + d] for w in W]
    pt = [w[4] + 0.5 * (w[5] ** 2 + w[6] ** 2 + w[7] ** 2) for w in W]
    c = torch.maximum(*[_fast(w[0], w[4], bn, w[5 + t[0]] ** 2 + w[5 + t[1]] ** 2) for w in W])
    S = [torch.minimum(*u) - c, torch.maximum(*u) + c]
    rs = [(S[k] - u[k]) * W[k][0] for k in (0, 1)]
    sm = (rs[1] * u[1] - rs[0] * u[0] - pt[1] + pt[0]) / (rs[1] - rs[0])
    pts = (rs[1] * pt[0] - rs[0] * pt[1] + rs[0] * rs[1] * (u[1] - u[0])) / (rs[1] - rs[0])
    F, U, US, star = [], [], [], []
    for k in (0, 1):
        w = W[k]
        cons = _cons(w)
        den = rs[k] * (S[k] - sm) - bn * bn
        deg = den.abs() <= degen * torch.maximum(rs[k] * (S[k] - u[k]), bn * bn)
        den = torch.where(deg, torch.ones_like(den), den)
        fv = torch.where(deg, torch.zeros_like(den), bn * (sm - u[k]) / den)
        fb = torch.where(deg, torch.ones_like(den), 1 + rs[k] * (sm - u[k]) / den)
        rho = rs[k] / (S[k] - sm)
        ws = [rho, None, None, None, None, None, None, None]
        ws[1 + d], ws[5 + d] = sm, bn
        for q in t:
            ws[1 + q], ws[5 + q] = w[1 + q] - w[5 + q] * fv, w[5 + q] * fb
        vb = sum(w[1 + q] * w[5 + q] for q in range(3))
        vbs = sum(ws[1 + q] * ws[5 + q] for q in range(3))
        e = ((S[k] - u[k]) * cons[4] - pt[k] * u[k] + pts * sm + bn * (vb - vbs)) / (S[k] - sm)
        F.append(_flux(d, w))
        U.append(cons)
        US.append([rho, rho * ws[1], rho * ws[2], rho * ws[3], e, ws[5], ws[6], ws[7]])
        star.append((ws, vbs))
    sq = [torch.sqrt(US[k][0]) for k in (0, 1)]
    Ss = [sm - bn.abs() / sq[0], sm + bn.abs() / sq[1]]
    sg = torch.where(bn >= 0, 1.0, -1.0)
    (a, vba), (b, vbb) = star
    dd = [None] * 8
    dd[1 + d], dd[5 + d] = sm, bn
    for q in t:
        dd[1 + q] = (sq[0] * a[1 + q] + sq[1] * b[1 + q] + sg * (b[5 + q] - a[5 + q])) / (sq[0] + sq[1])
        dd[5 + q] = (sq[0] * b[5 + q] + sq[1] * a[5 + q] + sg * sq[0] * sq[1] * (b[1 + q] - a[1 + q])) / (sq[0] + sq[1])
    vbd = sum(dd[1 + q] * dd[5 + q] for q in range(3))
    edd = [US[0][4] - sq[0] * (vba - vbd) * sg, US[1][4] + sq[1] * (vbb - vbd) * sg]
    left = sm >= 0
    out = []
    for q in range(8):
        g = []
        for k in (0, 1):
            fs = F[k][q] + S[k] * (US[k][q] - U[k][q])
            x = dd[q] if q > 4 else US[k][0] * dd[q] if q in (1, 2, 3) else US[k][0] if q == 0 else edd[k]
            inner = Ss[0] < 0 if k == 0 else Ss[1] >= 0
            g.append(torch.where(inner, fs + Ss[k] * (x - US[k][q]), fs))
        f = torch.where(left, g[0], g[1])
        out.append(torch.where(S[0] >= 0, F[0][q], torch.where(S[1] < 0, F[1][q], f)))
    tie = eps * (S[1] - S[0])
    up = torch.where((S[0] >= 0) | (sm > tie), 1, torch.where((S[1] < 0) | (sm < -tie), -1, 0))
    return out, up


def _advance64(U, B, dx, dt, limiter, emf, f32):
    """One step of a periodic box in 64 bits: cells U (5), lower faces B (3),
    each (nz, ny, nx); dt None: the CFL step.  Returns (U, B, dt)."""
    eps, degen = (1e-5, 1e-5) if f32 else (1e-10, 1e-12)
    bc = [0.5 * (B[d] + _sh(B[d], d, 1)) for d in range(3)]
    w = _prim([*U, *bc])
    if dt is None:
        b2 = sum(x * x for x in bc)
        dt = 0.4 * min(float((dx[d] / (w[1 + d].abs() + _fast(w[0], w[4], bc[d], b2 - bc[d] ** 2))).min()) for d in range(3))
    E = [w[1 + (a + 2) % 3] * w[5 + (a + 1) % 3] - w[1 + (a + 1) % 3] * w[5 + (a + 2) % 3] for a in range(3)]
    dw = [[_limit(limiter, x - _sh(x, d, -1), _sh(x, d, 1) - x) for x in w] for d in range(3)]
    bad = torch.zeros_like(w[0], dtype=torch.bool)
    for d in range(3):
        for q in (0, 4):
            bad |= ~(w[q] - 0.5 * dw[d][q].abs() > 0)
    dw = [[torch.where(bad, torch.zeros_like(s), s) for s in dw[d]] for d in range(3)]
    fw = [[[x + sg * 0.5 * s for x, s in zip(w, dw[d])] for sg in (-1, 1)] for d in range(3)]
    du = [torch.zeros_like(w[0]) for _ in range(8)]
    for d in range(3):
        fm, fp = _flux(d, fw[d][0]), _flux(d, fw[d][1])
        du = [du[q] - 0.5 * dt / dx[d] * (fp[q] - fm[q]) for q in range(8)]
    fs = [[_prim([x + y for x, y in zip(_cons(fw[d][k]), du)]) for k in (0, 1)] for d in range(3)]
    bad = torch.zeros_like(bad)
    for d in range(3):
        for k in (0, 1):
            bad |= ~(fs[d][k][0] > 0) | ~(fs[d][k][4] > 0)
    fs = [[[torch.where(bad, x, y) for x, y in zip(w, fs[d][k])] for k in (0, 1)] for d in range(3)]
    du = [torch.where(bad, torch.zeros_like(x), x) for x in du]
    edge = []
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        e = E[a] + _sh(E[a], b, -1)
        edge.append(0.25 * (e + _sh(e, c, -1)))
    F, up = [], []
    for d in range(3):
        b, c = (d + 1) % 3, (d + 2) % 3
        bn = B[d] - 0.5 * dt * ((_sh(edge[c], b, 1) - edge[c]) / dx[b] - (_sh(edge[b], c, 1) - edge[b]) / dx[c])
        f, s = _hlld(d, [_sh(x, d, -1) for x in fs[d][1]], fs[d][0], bn, eps, degen)
        F.append(f)
        up.append(s)
    em = []
    uh = [x + y for x, y in zip(_cons(w), du)]
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        ebh, ech = -F[b][5 + c], F[c][5 + b]
        ebl, ecl = _sh(ebh, c, -1), _sh(ech, b, -1)
        avg = 0.25 * (ebl + ebh + ecl + ech)
        if emf == 0:
            r11 = (uh[1 + c] * uh[5 + b] - uh[1 + b] * uh[5 + c]) / uh[0]
            r01, r10 = _sh(r11, b, -1), _sh(r11, c, -1)
            r00 = _sh(r10, b, -1)
            mb, mc = up[b], up[c]

            def side(m, lo, hi):
                return torch.where(m > 0, lo, torch.where(m < 0, hi, 0.5 * (lo + hi)))

            avg = avg + 0.25 * (side(_sh(mb, c, -1), ecl - r00, ech - r10) - side(mb, r01 - ecl, r11 - ech)
                                + side(_sh(mc, b, -1), ebl - r00, ebh - r01) - side(mc, r10 - ebl, r11 - ebh))
        em.append(avg)
    Un = [U[q] - dt * sum((_sh(F[d][q], d, 1) - F[d][q]) / dx[d] for d in range(3)) for q in range(5)]
    Bn = []
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        Bn.append(B[a] - dt * ((_sh(em[c], b, 1) - em[c]) / dx[b] - (_sh(em[b], c, 1) - em[b]) / dx[c]))
    return Un, Bn, dt


def _stepped(st, n, g, dx, dt, limiter, emf):
    """The state array after a ghost fill and one step: periodic images of the
    old state in the ghosts, the new state in the interior."""
    f32 = st.dtype == torch.float32
    st = st.double()
    c = tuple(slice(g, g + n[d]) for d in (2, 1, 0))
    old = [st[(q,) + c] for q in range(8)]
    U, B, dt = _advance64(old[:5], old[5:], dx, dt, limiter, emf, f32)
    out = torch.zeros_like(st)
    at = [(torch.arange(n[d] + 2 * g + 1, device=st.device) - g) % n[d] for d in range(3)]
    for q in range(8):
        top = [n[d] + 2 * g + (1 if q == 5 + d else 0) for d in range(3)]
        out[q, :top[2], :top[1], :top[0]] = old[q][at[2][:top[2], None, None], at[1][None, :top[1], None], at[0][None, None, :top[0]]]
        new = U[q] if q < 5 else B[q - 5]
        m = [n[d] + (1 if q == 5 + d else 0) for d in range(3)]
        i = [torch.arange(m[d], device=st.device) % n[d] for d in range(3)]
        out[q, g:g + m[2], g:g + m[1], g:g + m[0]] = new[i[2][:, None, None], i[1][None, :, None], i[0][None, None, :]]
    return out, dt


def exact(case, seed):
    """run()'s outputs in 64 bits from the same inputs.  None for the
    hierarchies: their step is hundreds of batched calls over patches of every
    level, which takes minutes without the library."""
    if case["kind"] == "step":
        st, n, dx = _step_state(case, seed)
        out, dt = _stepped(st, n, case["g"], dx, None, case["limiter"], case["emf"])
        return {"state": out, "dt": torch.tensor([dt], dtype=torch.float64)}
    if case["kind"] == "batch":
        tpl = _serve_templates(case, seed)
        done = {k: _stepped(p.state, p.n, p.g, p.dx, dt, 0, 1)[0] for k, (p, dt) in tpl.items()}
        return [done[(n, case["dtype"])] for n in _edges(case)]
    if case["kind"] == "scan":
        sums, dt = torch.zeros(8, dtype=torch.float64, device="cuda"), math.inf
        for st, n in zip(_scan_states(case, seed), _scan_sizes(case)):
            st = st.double()
            c = tuple(slice(4, 4 + n[d]) for d in (2, 1, 0))
            sums += torch.stack([st[(q,) + c].sum() for q in range(8)]) / 256.0 ** 3
            bc = [0.5 * (st[5 + d] + torch.roll(st[5 + d], -1, 2 - d))[c] for d in range(3)]
            w = _prim([st[(q,) + c] for q in range(5)] + bc)
            b2 = sum(x * x for x in bc)
            dt = min([dt] + [0.4 * 4.0 / 256 / float((w[1 + d].abs() + _fast(w[0], w[4], bc[d], b2 - bc[d] ** 2)).max()) for d in range(3)])
        return {"sums": sums, "dt": torch.tensor([dt], dtype=torch.float64), "flags": None}
    return None
