"""Timed cases of the library: the calls its users make, over the sizes they make them at.

Each case is one call sequence of the public C ABI (through the ctypes binding): advancing a
flow by a few time steps from a given state, one coarse Poisson solve, one prolongation, one
allocation-free solve, a batched step, or a few training steps of the learned guess.  Sizes
and parameters are those of the repository's workloads, tests and benchmark.  Solver
tolerances: the library's defaults for single solves; for time steps those of the
manufactured-flow tests (momentum 1e-12, Poisson 1e-11, mass: the default), since the
pressure takes up the momentum residual times 1.5 / dt.  ``exact`` computes the same
quantities from the same inputs in 64-bit torch arithmetic, with none of the library's code.
"""

import ctypes
import functools
import math

import numpy as np
import torch

from paper_1812_00185_gb300 import binding as cg
from workloads import batch_instances, channel_cylinder_mesh, square_mesh

DEV = "cuda"
F64 = torch.float64
VEL_DIR, PHI_ZERO = 1, 2
CAVITY, CHANNEL, TG_PERIODIC = cg.CGP_BC_CAVITY, cg.CGP_BC_CHANNEL, cg.CGP_BC_TG_PERIODIC
CHANNEL_L, CHANNEL_H, UMAX = 2.2, 0.41, 0.3


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest workload: 64x64 lid-driven cavity, standard form, all FP64.  Kernels of a
        # few microseconds: launches and loop control count
        {"name": "step_cavity64_fp64", "kind": "step", "flow": "cavity", "base": 32, "levels": 1, "k": 1,
         "form": "fp64", "chi": 0, "Re": 100.0, "dt": 0.01, "steps": 4},
        # an ordinary run: forced Taylor-Green on 512x512 squares, rotational form, pressure two
        # levels coarser, FP32 inner / FP64 outer solves
        {"name": "step_tgp512_k2_mixed", "kind": "step", "flow": "tgp", "base": 64, "levels": 3, "k": 2,
         "form": "mixed", "chi": 1, "Re": 100.0, "dt": 0.002, "steps": 2},
        # the 512x512 cavity with the pressure one level coarser: its coarse system is too large
        # for one cluster, so the grid-wide solve runs
        {"name": "step_cavity512_k1_mixed", "kind": "step", "flow": "cavity", "base": 64, "levels": 3, "k": 1,
         "form": "mixed", "chi": 1, "Re": 400.0, "dt": 0.002, "steps": 2},
        # the headline mesh (unstructured channel with a cylinder, 1M triangles), mixed form
        {"name": "step_channel1m_k2_mixed", "kind": "step", "flow": "channel", "h": 0.0084, "levels": 3, "k": 2,
         "form": "mixed", "chi": 1, "Re": 1000.0, "dt": 0.002, "steps": 2},
        # the same step with every solve in FP64, the form the others are compared with
        {"name": "step_channel1m_k2_fp64", "kind": "step", "flow": "channel", "h": 0.0084, "levels": 3, "k": 2,
         "form": "fp64", "chi": 1, "Re": 1000.0, "dt": 0.002, "steps": 1},
        # the coarse Poisson problem alone (Eq. 23), FP64, pure Neumann: 129^2 unknowns
        {"name": "poisson_sq128_fp64", "kind": "poisson", "flow": "cavity", "base": 32, "levels": 2, "k": 0,
         "form": "fp64"},
        # the same problem of the channel's pressure mesh (32k unknowns), mixed form
        {"name": "poisson_channel_mixed", "kind": "poisson", "flow": "channel", "h": 0.0084, "levels": 1, "k": 0,
         "form": "mixed"},
        # the largest Poisson problem in use (plain scheme on 1024x1024 squares: k = 0)
        {"name": "poisson_sq1024_fp64", "kind": "poisson", "flow": "cavity", "base": 128, "levels": 3, "k": 0,
         "form": "fp64"},
        # a host program without an allocator of its own: a small solve in fixed memory
        {"name": "noalloc_channel", "kind": "noalloc", "h": 0.05, "levels": 2},
        # the transfer of Eq. 24 alone onto a 2048x2048 mesh, two levels
        {"name": "prolong_sq2048_k2", "kind": "prolong", "base": 256, "levels": 3, "k": 2},
        # many uneven cavities at once, one persistent launch a step
        {"name": "batch32_mixed", "kind": "batch", "n": 32, "draw": 20181203, "steps": 2},
        # training the learned guess on the channel's pressure mesh, batches of 8
        {"name": "train_channel_b8", "kind": "train", "flow": "channel", "h": 0.0084, "levels": 1, "batch": 8,
         "iters": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "poisson", "poisson", "noalloc", "prolong", "batch", "train"])
    h = round(0.0084 * math.exp(rng.uniform(0.0, math.log(4.0))), 4)
    form = rng.choice(["fp64", "mixed"])
    if kind == "step":
        levels = rng.randint(1, 3)
        c = {"kind": kind, "levels": levels, "k": rng.randint(1, levels), "form": form, "chi": rng.randint(0, 1),
             "steps": rng.randint(1, 3)}
        flow = rng.choice(["cavity", "tgp", "channel"])
        if flow == "channel":
            return dict(c, flow=flow, h=h, Re=1000.0, dt=0.002)
        side = _log(rng, 32, 512)
        return dict(c, flow=flow, base=max(4, side >> levels), Re=rng.choice([100.0, 400.0]),
                    dt=rng.choice([0.01, 0.005, 0.002]))
    if kind == "poisson":
        if rng.random() < 0.3:
            return {"kind": kind, "flow": "channel", "h": h, "levels": rng.randint(0, 2), "k": 0, "form": form}
        levels = rng.randint(0, 2)
        return {"kind": kind, "flow": "cavity", "base": max(8, _log(rng, 16, 700) >> levels), "levels": levels, "k": 0,
                "form": form}
    if kind == "noalloc":
        return {"kind": kind, "h": max(h, 0.013), "levels": rng.randint(0, 2)}
    if kind == "prolong":
        levels = rng.randint(1, 3)
        return {"kind": kind, "base": max(4, _log(rng, 64, 1600) >> levels), "levels": levels,
                "k": rng.randint(1, levels)}
    if kind == "batch":
        return {"kind": kind, "n": rng.randint(3, 32), "draw": rng.randint(1, 10 ** 6), "steps": rng.randint(1, 2)}
    if rng.random() < 0.3:
        return {"kind": "train", "flow": "channel", "h": max(h, 0.012), "levels": 1, "batch": rng.randint(1, 8),
                "iters": rng.randint(1, 3)}
    return {"kind": "train", "flow": "cavity", "base": _log(rng, 16, 180), "levels": 0, "batch": rng.randint(1, 8),
            "iters": rng.randint(1, 3)}


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=16)
def _base(flow, size):
    if flow == "channel":
        return channel_cylinder_mesh(seed=0, h=size)
    return square_mesh(size, boundary_flags=VEL_DIR)


def _base_of(case):
    flow = "channel" if case["kind"] == "noalloc" else case.get("flow", "cavity")
    return _base(flow, case["h"] if flow == "channel" else case["base"])


def _bc(case):
    return {"cavity": CAVITY, "tgp": TG_PERIODIC, "channel": CHANNEL}[case.get("flow", "cavity")]


def _bc_param(bc):
    return (UMAX, CHANNEL_H, 0.0, 0.0) if bc == CHANNEL else (1.0, 0.0, 0.0, 0.0)


def _gen(seed):
    return torch.Generator().manual_seed(int(seed) * 7919 + 17)


def _modes(x, y, g, n=6, top=3.0):
    """A smooth random field: n cosine waves of wave numbers up to `top`, unit size."""
    s = torch.zeros_like(x)
    for a, kx, ky, p in torch.rand(n, 4, generator=g, dtype=F64).tolist():
        s += (a - 0.5) * torch.cos(math.pi * top * (kx * x + ky * y) + 2 * math.pi * p)
    return s


def _tg(x, y, a):
    tp = 2 * math.pi
    return (torch.stack([-torch.cos(tp * x) * torch.sin(tp * y), torch.sin(tp * x) * torch.cos(tp * y)], 1) * a,
            -(torch.cos(2 * tp * x) + torch.cos(2 * tp * y)) / 4 * a * a)


def _curl(psi, x, y):
    """(psi_y, -psi_x): a divergence-free velocity from its stream function."""
    x, y = x.clone().requires_grad_(), y.clone().requires_grad_()
    gx, gy = torch.autograd.grad(psi(x, y).sum(), (x, y))
    return torch.stack([gy, -gx], 1)


def _flow_state(flow, xy, dt, seed):
    """(U, Uprev, P, t) of a flow under way: the closed form with a small disturbance
    (Taylor-Green), a recirculating cavity, a channel stream around the cylinder."""
    g = _gen(seed)
    x, y = xy[:, 0].contiguous(), xy[:, 1].contiguous()
    t = 0.05 + 0.1 * float(torch.rand(1, generator=g, dtype=F64))
    waves = torch.rand(6, 4, generator=g, dtype=F64).tolist()

    def rough(x, y):
        return sum((a - 0.5) * torch.cos(3 * math.pi * (kx * x + ky * y) + 2 * math.pi * p) for a, kx, ky, p in waves)

    def bubble(x, y):
        return 16 * (x * (1 - x) * y * (1 - y)) ** 2

    if flow == "tgp":
        U, P = _tg(x, y, math.cos(2 * math.pi * t))
        Up, _ = _tg(x, y, math.cos(2 * math.pi * (t - dt)))
        d = _curl(lambda x, y: 0.1 * bubble(x, y) * rough(x, y), x, y)
        return U + d, Up + d, P, t
    if flow == "channel":
        def psi(x, y):
            d2 = ((x - 0.2) ** 2 + (y - 0.2) ** 2 - 0.05 ** 2).clamp(min=0.0)
            f = (1 - torch.exp(-d2 / 0.002)) ** 2
            flux = 4 * UMAX / CHANNEL_H ** 2 * (CHANNEL_H * y ** 2 / 2 - y ** 3 / 3 - CHANNEL_H * 0.02 + 0.008 / 3)
            wall = (y * (CHANNEL_H - y)) ** 2 / CHANNEL_H ** 4 * (x / CHANNEL_L) ** 2
            return flux * f + 0.02 * wall * f * rough(x, y)
        U = _curl(psi, x, y)
        return U, U * (1 - 0.2 * dt), (CHANNEL_L - x) * (0.05 + 0.01 * rough(x, y)), t
    U = _curl(lambda x, y: 16 * (x * (1 - x)) ** 2 * (y ** 3 - y ** 2) + 0.5 * bubble(x, y) * rough(x, y), x, y)
    return U, U * (1 - 0.5 * dt), 0.1 * rough(x, y), t


def _vertices(mesh, level, case):
    """Vertex coordinates of one level, from the mesh handle."""
    return torch.from_numpy(mesh.level(level)["xy"]).to(DEV)


def _params(case, **kw):
    bc = _bc(case)
    if "Re" in case:
        kw = dict(tol_mom=1e-12, tol_poisson=1e-11, **kw)
    return cg.make_params(case.get("Re", 100.0), case.get("dt", 0.01), chi=case.get("chi", 0), k=case["k"],
                          max_it_poisson=50000, precision=cg.CGP_MIXED if case.get("form") == "mixed" else cg.CGP_FP64,
                          bc_kind=bc, bc_param=_bc_param(bc), **kw)


def _source(xy, fixed, seed):
    """Right-hand side of a Poisson problem: a smooth load with a rough part, scaled to a
    vertex's share of the domain, zero where phi is prescribed."""
    g = _gen(seed)
    x, y = xy[:, 0].contiguous(), xy[:, 1].contiguous()
    f = _modes(x, y, g, n=8, top=6.0) + 0.02 * torch.randn(x.numel(), generator=g, dtype=F64).to(DEV)
    return torch.where(fixed, torch.zeros_like(f), f / x.numel())


def _geometry(xy, tri):
    p = xy[tri]
    d = p.roll(-1, 1) - p.roll(-2, 1)                               # edge opposite to each corner, reversed
    det = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1])
    return 0.5 * det, torch.stack([d[:, :, 1], -d[:, :, 0]], 2) / det[:, None, None]


def _summed(n, at, v):
    """Sums of v over equal targets, in an order that is the same every time."""
    before = torch.are_deterministic_algorithms_enabled()
    torch.use_deterministic_algorithms(True)
    out = torch.zeros(n, dtype=F64, device=DEV).index_add_(0, at, v)
    torch.use_deterministic_algorithms(before)
    return out


def _lumped(xy, tri):
    area = _geometry(xy, tri)[0]
    return _summed(len(xy), tri.reshape(-1), (area / 3).repeat_interleave(3))


def _train_samples(case, xy, n, seed):
    g = _gen(seed)
    x, y = xy[:, 0].contiguous(), xy[:, 1].contiguous()
    r, q, t = [], [], []
    for _ in range(case["batch"]):
        r.append(1e-3 * (_modes(x, y, g, top=6.0) + 0.1 * torch.randn(n, generator=g, dtype=F64).to(DEV)))
        q.append(0.05 * _modes(x, y, g))
        t.append(q[-1] + 0.02 * _modes(x, y, g))
    return torch.stack(r), torch.stack(q), torch.stack(t)


def _train_start(seed):
    """Parameters part of the way through training (dense layers, no zero biases)."""
    g = np.random.default_rng(int(seed) + 5)
    p, o = np.zeros(cg.cgp_mlp_param_count(), np.float32), 0
    for fin, fout, scale in ((4, 64, 1.0), (64, 64, 1.0), (64, 1, 0.3)):
        w = g.standard_normal((fout, 2 * fin)) * math.sqrt(1.0 / fin) * scale
        p[o:o + w.size] = w.ravel()
        o += w.size
        p[o:o + fout] = 0.05 * g.standard_normal(fout)
        o += fout
    return p


def _sell(rowptr, col, val):
    """SELL-32 arrays of a CSR matrix (see cgp_pcg_sell_noalloc)."""
    n = rowptr.numel() - 1
    ns = (n + 31) // 32
    length = rowptr[1:] - rowptr[:-1]
    width = torch.cat([length, length.new_zeros(32 * ns - n)]).view(ns, 32).amax(1)
    ptr = torch.cat([width.new_zeros(1), (32 * width).cumsum(0)])
    row = torch.repeat_interleave(torch.arange(n, device=DEV), length)
    at = ptr[row // 32] + 32 * (torch.arange(col.numel(), device=DEV) - rowptr[row]) + row % 32
    scol = torch.repeat_interleave(32 * torch.arange(ns, device=DEV), 32 * width)
    sval = torch.zeros(scol.numel(), dtype=F64, device=DEV)
    scol[at], sval[at] = col, val
    return ns, ptr.int(), scol.int(), sval


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    if kind == "noalloc":
        lev = _hierarchy(_base_of(case), case["levels"])[-1]
        A, dinv, _, _ = _poisson_system(lev)
        ns, ptr, col, val = _sell(A.crow_indices(), A.col_indices(), A.values())
        b = _source(lev["xy"], lev["tag"] & PHI_ZERO != 0, seed)
        return {"case": case, "n": len(b), "ns": ns, "ptr": ptr, "col": col, "val": val, "dinv": dinv, "b": b,
                "x": torch.empty_like(b), "info": torch.zeros(2, dtype=torch.int32, device=DEV)}
    base = _base_of(case)
    mesh = cg.Mesh(base.xy, base.tri, base.tag, case["levels"])
    s = {"case": case, "mesh": mesh}
    if kind == "train":
        xy = _vertices(mesh, case["levels"], case)
        s["net"] = _Net(mesh, case["levels"], case["batch"])
        s["p0"] = _train_start(seed)
        s["rqt"] = _train_samples(case, xy, len(xy), seed)
        return s
    if kind == "prolong":
        s["solver"] = cg.Solver(mesh, _params(case, guess=cg.CGP_GUESS_ZERO))
        xy = _vertices(mesh, case["levels"] - case["k"], case)
        s["phi"] = _modes(xy[:, 0].contiguous(), xy[:, 1].contiguous(), _gen(seed), top=20.0)
        s["out"] = torch.empty(s["solver"].nf, dtype=F64, device=DEV)
        return s
    if kind == "poisson":
        s["solver"] = cg.Solver(mesh, _params(case, guess=cg.CGP_GUESS_ZERO))
        lev = mesh.level(case["levels"])
        xy = torch.from_numpy(lev["xy"]).to(DEV)
        s["rhs"] = _source(xy, torch.from_numpy(lev["tag"]).to(DEV) & PHI_ZERO != 0, seed)
        s["phi"] = torch.zeros_like(s["rhs"])
        return s
    s["solver"] = cg.Solver(mesh, _params(case))
    s["U"], s["Up"], s["P"], s["t"] = _flow_state(case["flow"], _vertices(mesh, case["levels"], case), case["dt"], seed)
    s["phi"] = torch.zeros(s["solver"].nc, dtype=F64, device=DEV)
    s["Uo"], s["Po"] = torch.empty_like(s["U"]), torch.empty_like(s["P"])
    return s


class _Net:
    """Owns a network handle (freed with the state)."""

    def __init__(self, mesh, level, batch):
        self.handle = cg.cgp_mlp_create(mesh.handle, level, batch)

    def __del__(self):
        cg.cgp_mlp_destroy(self.handle)


class _Batch:
    def __init__(self, solvers):
        self.solvers = solvers
        self.handle = cg.cgp_batch_create(solvers)

    def __del__(self):
        cg.cgp_batch_destroy(self.handle)


def _instances(case):
    """(sub-case of one cavity) for every instance of the batch."""
    return [{"flow": "cavity", "base": i["n_fine"] >> i["k"], "levels": i["k"], "k": i["k"], "Re": i["Re"], "dt": 0.005,
             "chi": 1, "form": "mixed"} for i in batch_instances(256, case["draw"])[:case["n"]]]


def _prepare_batch(case, seed):
    s = {"case": case, "meshes": [], "solvers": [], "states": [], "phis": [], "outs": []}
    for j, c in enumerate(_instances(case)):
        base = _base("cavity", c["base"])
        mesh = cg.Mesh(base.xy, base.tri, base.tag, c["levels"])
        s["meshes"].append(mesh)
        s["solvers"].append(cg.Solver(mesh, _params(c)))
        st = _flow_state("cavity", _vertices(mesh, c["levels"], c), c["dt"], seed * 1000 + j)
        s["states"].append(st)
        s["phis"].append(torch.zeros(s["solvers"][-1].nc, dtype=F64, device=DEV))
        s["outs"].append((torch.empty_like(st[0]), torch.empty_like(st[2])))
    s["batch"] = _Batch(s["solvers"])
    return s


# ---------------------------------------------------------------- one pass
def _ok(rc):
    if rc not in (cg.CGP_OK, cg.CGP_ENOTCONV):
        raise cg.CgpError(rc, cg.cgp_last_error())


def _restart(h, U, Up, P, t, phi):
    """A state with its previous increment (the coarse solve's first guess), as from a checkpoint."""
    cg.cgp_set_fields(h, U, Up, P, t, where=cg.CGP_DEVICE)
    _ok(cg.load().cgp_set_vector(h, cg.CGP_VEC_PHI_C, phi.data_ptr(), cg.CGP_DEVICE,
                                 torch.cuda.current_stream().cuda_stream))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        h = s["solver"].handle
        _restart(h, s["U"], s["Up"], s["P"], s["t"], s["phi"])
        cg.cgp_step(h, case["steps"])
        cg.cgp_get_fields(h, s["Uo"], s["Po"], where=cg.CGP_DEVICE)
        return {"U": s["Uo"], "P": s["Po"]}
    if kind == "poisson":
        it = ctypes.c_int32()
        _ok(cg.load().cgp_poisson_solve(s["solver"].handle, s["rhs"].data_ptr(), s["phi"].data_ptr(), ctypes.byref(it),
                                        cg.CGP_DEVICE, torch.cuda.current_stream().cuda_stream))
        return {"phi": s["phi"]}
    if kind == "noalloc":
        s["x"].zero_()
        cg.cgp_pcg_sell_noalloc(s["n"], s["ns"], s["ptr"], s["col"], s["val"], s["dinv"], s["b"], s["x"], 1e-10, 20000,
                                s["info"])
        return {"x": s["x"]}
    if kind == "prolong":
        _ok(cg.load().cgp_prolong(s["solver"].handle, s["phi"].data_ptr(), s["out"].data_ptr(), cg.CGP_DEVICE,
                                  torch.cuda.current_stream().cuda_stream))
        return {"phi_f": s["out"]}
    if kind == "batch":
        for v, (U, Up, P, t), phi in zip(s["solvers"], s["states"], s["phis"]):
            _restart(v.handle, U, Up, P, t, phi)
        cg.cgp_batch_step(s["batch"].handle, case["steps"])
        for v, (U, P) in zip(s["solvers"], s["outs"]):
            cg.cgp_get_fields(v.handle, U, P, where=cg.CGP_DEVICE)
        return {"U": torch.cat([o[0] for o in s["outs"]]), "P": torch.cat([o[1] for o in s["outs"]])}
    net = s["net"].handle
    cg.cgp_mlp_set_params(net, s["p0"])
    r, q, t = s["rqt"]
    loss = 0.0
    for i in range(case["iters"]):
        loss = cg.cgp_mlp_train_step(net, r, q, t, case["batch"], 1e-3, want_loss=i == case["iters"] - 1)
    return {"loss": loss, "params": cg.cgp_mlp_get_params(net)}


# ---------------------------------------------------------------- what a pass cannot do without
def _sizes(base, levels):
    """(vertices, matrix entries) of every level: each refinement adds the edges' midpoints."""
    v, t = base.n_vert, base.n_tri
    e = len(np.unique(np.sort(np.concatenate([base.tri[:, [0, 1]], base.tri[:, [1, 2]], base.tri[:, [2, 0]]]), 1), axis=0))
    out = []
    for _ in range(levels + 1):
        out.append((v, v + 2 * e))
        v, e, t = v + e, 2 * e + 3 * t, 4 * t
    return out


def _step_work(base, levels, k, steps, fine_it, coarse_it):
    """Operators, pattern and state read once a step, the state written once; about
    `fine_it` products with the fine matrices (two components) and `coarse_it` with the coarse."""
    sz = _sizes(base, levels)
    (nf, zf), (nc, zc) = sz[-1], sz[-1 - k]
    return {"bytes": steps * (zf * (4 + 8 * 6) + nf * 8 * 10 + zc * (4 + 8 * 3) + nc * 8 * 4),
            "flops": steps * (fine_it * (4 * zf + 20 * nf) + coarse_it * (2 * zc + 12 * nc))}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_step_work(_base("cavity", c["base"]), c["levels"], c["k"], case["steps"], 60, 2 * c["base"])
                 for c in _instances(case)]
        return {m: sum(p[m] for p in parts) for m in ("bytes", "flops")}
    sz = _sizes(_base_of(case), case["levels"])
    n, z = sz[-1]
    if kind == "step":
        nc = sz[-1 - case["k"]][0]
        return _step_work(_base_of(case), case["levels"], case["k"], case["steps"], 60, 3 * math.sqrt(nc))
    if kind in ("poisson", "noalloc"):
        return {"bytes": 12 * z + 24 * n, "flops": 3 * math.sqrt(n) * (2 * z + 12 * n)}
    if kind == "prolong":
        nc = sz[-1 - case["k"]][0]
        return {"bytes": 8 * nc + 8 * (n - nc) + 8 * n, "flops": 2 * (n - nc)}
    b = case["batch"]
    return {"bytes": case["iters"] * (b * n * 24 + 4 * z + 16 * n),
            "flops": case["iters"] * 3 * b * (2 * n * (8 * 64 + 128 * 64 + 128) + (z - n) * 132)}


# ---------------------------------------------------------------- the same quantities in 64 bits
def _hierarchy(base, levels):
    """The nested levels: edges ranked by (min, max) vertex, midpoints after the old vertices; a
    midpoint of a boundary edge takes the AND of its ends' flags."""
    xy = torch.from_numpy(base.xy).to(DEV)
    tri = torch.from_numpy(base.tri.astype(np.int64)).to(DEV)
    tag = torch.from_numpy(base.tag).to(DEV)
    out = [{"xy": xy, "tri": tri, "tag": tag}]
    for _ in range(levels):
        n = len(xy)
        e = torch.cat([tri[:, [0, 1]], tri[:, [1, 2]], tri[:, [2, 0]]]).sort(1).values
        key, inv, cnt = torch.unique(e[:, 0] * n + e[:, 1], return_inverse=True, return_counts=True)
        ends = torch.stack([key // n, key % n], 1)
        m01, m12, m20 = (n + inv).view(3, -1)
        a, b, c = tri.unbind(1)
        tri = torch.stack([torch.stack(v, 1) for v in ((a, m01, m20), (m01, b, m12), (m20, m12, c), (m01, m12, m20))],
                          1).reshape(-1, 3)
        tag = torch.cat([tag, torch.where(cnt == 1, tag[ends[:, 0]] & tag[ends[:, 1]], torch.zeros_like(tag[:1]))])
        xy = torch.cat([xy, 0.5 * (xy[ends[:, 0]] + xy[ends[:, 1]])])
        out.append({"xy": xy, "tri": tri, "tag": tag, "ends": ends})
    return out


class _Pattern:
    """Assembly of P1 element matrices on one level into CSR."""

    def __init__(self, lev):
        self.n, tri = len(lev["xy"]), lev["tri"]
        rows, cols = tri.repeat_interleave(3, 1).reshape(-1), tri.repeat(1, 3).reshape(-1)
        key, self.inv = torch.unique(rows * self.n + cols, return_inverse=True)
        self.row, self.col = key // self.n, key % self.n
        self.ptr = torch.zeros(self.n + 1, dtype=torch.int64, device=DEV)
        self.ptr[1:] = torch.bincount(self.row, minlength=self.n).cumsum(0)
        self.area, self.g = _geometry(lev["xy"], tri)
        self.tri = tri

    def values(self, Ke):
        return _summed(len(self.col), self.inv, Ke.reshape(-1))

    def csr(self, v):
        return torch.sparse_csr_tensor(self.ptr, self.col, v, (self.n, self.n))

    def mass(self):
        e = torch.ones(3, 3, dtype=F64, device=DEV) + torch.eye(3, dtype=F64, device=DEV)
        return self.values(self.area[:, None, None] / 12 * e)

    def stiff(self):
        return self.values(self.area[:, None, None] * torch.einsum("tid,tjd->tij", self.g, self.g))

    def deriv(self, d):
        return self.values((self.area[:, None] / 3 * self.g[:, :, d])[:, None, :].expand(-1, 3, -1))

    def convect(self, w):
        wt = w[self.tri]
        c = self.area[:, None, None] / 12 * (wt.sum(1, keepdim=True) + wt)
        return self.values(torch.einsum("tid,tjd->tij", c, self.g))

    def diag(self, v):
        d = torch.ones(self.n, dtype=F64, device=DEV)
        on = self.row == self.col
        d[self.row[on]] = v[on]
        return d

    def eliminated(self, v, fixed, rows_only=False):
        on = fixed[self.row] if rows_only else fixed[self.row] | fixed[self.col]
        return torch.where(on, (self.row == self.col).to(F64), v)


def _poisson_system(lev):
    """(K with phi = 0 rows and columns those of the identity, 1/diagonal, pattern, lumped mass)."""
    p = _Pattern(lev)
    v = p.eliminated(p.stiff(), lev["tag"] & PHI_ZERO != 0)
    return p.csr(v), 1 / p.diag(v), p, _lumped(lev["xy"], lev["tri"])


def _dot(a, b):
    return (a * b).sum(0)


def _cg(A, dinv, b, most=20000, rounds=5, free=False):
    """Jacobi CG on the columns of b, restarted from the true residual until it no longer falls;
    free: constants are A's null space, and residuals are kept out of it."""
    x, D = torch.zeros_like(b), dinv[:, None]
    size, last = _dot(b, b).sqrt().clamp(min=1e-300), math.inf
    best = (math.inf, x)
    for _ in range(rounds):
        r = b - A @ x
        r = r - r.mean(0) if free else r
        now = float((_dot(r, r).sqrt() / size).max())
        if now < best[0]:
            best = (now, x)
        if now < 1e-15 or not now < 0.3 * last:
            break
        last = now
        e, z = torch.zeros_like(b), D * r
        p, rz, on = z.clone(), _dot(r, z), torch.ones_like(size)
        goal = 1e-18 * _dot(r, r)
        for k in range(most):
            q = A @ p
            a = on * rz / _dot(p, q).clamp(min=1e-300)
            e += a * p
            r = r - a * q
            z = D * r
            new = _dot(r, z)
            p = z + new / rz.clamp(min=1e-300) * p
            rz, on = new, on * (_dot(r, r) > goal)      # a column that is done stays as it is
            if k % 50 == 49 and not bool(on.any()):
                break
        x = x + e
    return best[1]


def _bicgstab(A, dinv, b, x, rounds=5):
    D = dinv[:, None]
    size, last = _dot(b, b).sqrt().clamp(min=1e-300), math.inf
    best = (math.inf, x)
    for _ in range(rounds):
        r = b - A @ x
        now = float((_dot(r, r).sqrt() / size).max())
        if now < best[0]:
            best = (now, x)
        if now < 1e-16 or not now < 0.3 * last:
            break
        last = now
        r0, e, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b), torch.zeros_like(b)
        rho = al = om = on = torch.ones_like(size)
        goal = 1e-18 * _dot(r, r)
        for k in range(200):
            new = _dot(r0, r)
            p = torch.where(on > 0, r + new / rho * (al / om) * (p - om * v), p)
            rho, y = new, D * p
            v = A @ y
            al = rho / _dot(r0, v)
            s = r - al * v
            z = D * s
            t = A @ z
            om = _dot(t, s) / _dot(t, t).clamp(min=1e-300)
            e = torch.where(on > 0, e + al * y + om * z, e)
            r = torch.where(on > 0, s - om * t, r)
            on = on * (_dot(r, r) > goal)               # a column that is done stays as it is
            if k % 4 == 3 and not bool(on.any()):
                break
        x = x + e
    return best[1]


def _poisson_exact(lev, rhs, system=None):
    """K phi = rhs; without a prescribed phi the range-projected rhs and sum of m_i phi_i = 0."""
    A, dinv, _, mass = system or _poisson_system(lev)
    free = not bool((lev["tag"] & PHI_ZERO != 0).any())
    b = rhs - rhs.mean() if free else rhs
    phi = _cg(A, dinv, b[:, None], free=free)[:, 0]
    return phi - (mass * phi).sum() / mass.sum() if free else phi


def _prolonged(levels, lc, lf, phi):
    for l in range(lc + 1, lf + 1):
        phi = torch.cat([phi, phi[levels[l]["ends"]].mean(1)])
    return phi


def _step_exact(base, c, steps, state):
    """(U, P) after `steps` steps of Eqs. 21-26 from (U, Uprev, P, t)."""
    levels = _hierarchy(base, c["levels"])
    lf, lc = c["levels"], c["levels"] - c["k"]
    F, C = levels[lf], levels[lc]
    p, pc = _Pattern(F), _Pattern(C)
    M, K = p.mass(), p.stiff()
    Mm, Cx, Cy = p.csr(M), p.csr(p.deriv(0)), p.csr(p.deriv(1))
    # (Cx^T)_ij = |T|/3 g_i,x
    CT = [p.csr(p.values((p.area[:, None] / 3 * p.g[:, :, d])[:, :, None].expand(-1, -1, 3))) for d in (0, 1)]
    Cc = [pc.csr(pc.deriv(d)) for d in (0, 1)]
    system = _poisson_system(C)
    x, y = F["xy"][:, 0].contiguous(), F["xy"][:, 1].contiguous()
    wall = F["tag"] & VEL_DIR != 0
    M0 = p.eliminated(M, wall)
    dt, Re, flow = c["dt"], c["Re"], c["flow"]
    U, Up, P, t = state
    fixed = C["tag"] & PHI_ZERO != 0
    for _ in range(steps):
        t = t + dt
        uD, force = torch.zeros_like(U), torch.zeros_like(U)
        if flow == "cavity":
            uD[:, 0] = ((y == 1) & (x > 0) & (x < 1)).to(F64)
        elif flow == "channel":
            uD[:, 0] = torch.where(x == 0, 4 * UMAX * y * (CHANNEL_H - y) / CHANNEL_H ** 2, torch.zeros_like(x))
        else:
            a, da = math.cos(2 * math.pi * t), -2 * math.pi * math.sin(2 * math.pi * t)
            uD = _tg(x, y, a)[0]
            force = _tg(x, y, 1.0)[0] * (da + 8 * math.pi ** 2 * a / Re)
        w = 2 * U - Up
        A = p.eliminated(1.5 * M + dt * p.convect(w) + dt / Re * K, wall, rows_only=True)
        b = Mm @ (dt * force + 2 * U - 0.5 * Up) + dt * torch.stack([m @ P[:, None] for m in CT], 1)[:, :, 0]
        b = torch.where(wall[:, None], uD, b)
        Ut = _bicgstab(p.csr(A), 1 / p.diag(A), b, torch.where(wall[:, None], uD, w))
        Uc = Ut[:pc.n]
        r = -1.5 / dt * (Cc[0] @ Uc[:, :1] + Cc[1] @ Uc[:, 1:])[:, 0]
        r = torch.where(fixed, torch.zeros_like(r), r)
        phi = _prolonged(levels, lc, lf, _poisson_exact(C, r, system))
        g = -2.0 / 3.0 * dt * torch.cat([Cx @ phi[:, None], Cy @ phi[:, None]], 1)
        g = torch.where(wall[:, None], torch.zeros_like(g), g)
        U, Up = Ut + _cg(p.csr(M0), 1 / p.diag(M0), g), U
        P = P + phi
        if c["chi"]:
            P = P - _cg(Mm, 1 / p.diag(M), Cx @ Ut[:, :1] + Cy @ Ut[:, 1:])[:, 0] / Re
    return U, P


def _train_exact(case, seed):
    """The training steps with the forward and backward pass in 64 bits (weights rounded to
    bfloat16 for the forward pass, as the network is defined; biases and Adam as they are)."""
    lev = _hierarchy(_base_of(case), case["levels"])[-1]
    n = len(lev["xy"])
    r, q, t = _train_samples(case, lev["xy"], n, seed)
    pat = _Pattern(lev)
    off = pat.row != pat.col
    row, col = pat.row[off], pat.col[off]
    deg = torch.bincount(row, minlength=n).to(F64).clamp(min=1)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.bincount(row, minlength=n).cumsum(0)
    mean = torch.sparse_csr_tensor(ptr, col, (1 / deg)[row], (n, n))
    order = torch.argsort(col, stable=True)
    ptr_t = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr_t[1:] = torch.bincount(col, minlength=n).cumsum(0)
    mean_t = torch.sparse_csr_tensor(ptr_t, row[order], (1 / deg)[row][order], (n, n))
    p = torch.from_numpy(_train_start(seed)).to(DEV)
    m, v, loss = torch.zeros_like(p), torch.zeros_like(p), 0.0
    shape, at = [], 0
    for fin, fout in ((4, 64), (64, 64), (64, 1)):
        shape.append((at, at + 2 * fin * fout, fout))
        at += 2 * fin * fout + fout
    for it in range(1, case["iters"] + 1):
        half, p64 = p.bfloat16().to(F64), p.to(F64)
        W = [half[a:b].view(o, -1) for a, b, o in shape]
        bias = [p64[b:b + o] for _, b, o in shape]
        grad, loss = torch.zeros(at, dtype=F64, device=DEV), 0.0
        for s in range(case["batch"]):
            sr, sq = r[s].square().mean().sqrt(), q[s].square().mean().sqrt()
            h = [torch.stack([r[s] / sr, q[s] / sq, lev["xy"][:, 0], lev["xy"][:, 1]], 1)]
            X, acts = [], []
            for l in range(3):
                X.append(torch.cat([h[l], mean @ h[l]], 1))
                acts.append(X[l] @ W[l].T + bias[l])
                h.append(acts[l].clamp(min=0))
            d = acts[2][:, 0] - ((t[s] - q[s]) / sq).clamp(-10, 10)
            loss += float(d.square().mean()) / case["batch"]
            ga = (2 * d / (n * case["batch"]))[:, None]
            for l in (2, 1, 0):
                a, b, o = shape[l]
                grad[a:b] += (ga.T @ X[l]).reshape(-1)
                grad[b:b + o] += ga.sum(0)
                if l:
                    gx = ga @ W[l]
                    f = gx.shape[1] // 2
                    ga = (gx[:, :f] + mean_t @ gx[:, f:].contiguous()) * (acts[l - 1] > 0)
        grad = grad.to(torch.float32)
        m = 0.9 * m + (1 - 0.9) * grad
        v = 0.999 * v + (1 - 0.999) * grad * grad
        p = (p.to(F64) - 1e-3 * m.to(F64) / (1 - 0.9 ** it) / ((v.to(F64) / (1 - 0.999 ** it)).sqrt() + 1e-8)).float()
    return {"loss": loss, "params": p.to(F64)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train_exact(case, seed)
    if kind == "batch":
        got = []
        for j, c in enumerate(_instances(case)):
            base = _base("cavity", c["base"])
            xy = _hierarchy(base, c["levels"])[-1]["xy"]
            got.append(_step_exact(base, c, case["steps"], _flow_state("cavity", xy, c["dt"], seed * 1000 + j)))
        return {"U": torch.cat([g[0] for g in got]), "P": torch.cat([g[1] for g in got])}
    base = _base_of(case)
    levels = _hierarchy(base, case["levels"])
    lev = levels[-1]
    if kind == "step":
        U, P = _step_exact(base, case, case["steps"], _flow_state(case["flow"], lev["xy"], case["dt"], seed))
        return {"U": U, "P": P}
    if kind == "prolong":
        xy = levels[case["levels"] - case["k"]]["xy"]
        phi = _modes(xy[:, 0].contiguous(), xy[:, 1].contiguous(), _gen(seed), top=20.0)
        return {"phi_f": _prolonged(levels, case["levels"] - case["k"], case["levels"], phi)}
    rhs = _source(lev["xy"], lev["tag"] & PHI_ZERO != 0, seed)
    return {"x" if kind == "noalloc" else "phi": _poisson_exact(lev, rhs)}
