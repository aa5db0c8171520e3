"""Performance cases of the solver: whole solves through the public entry points.

A case is a dict of plain values; `prepare` plans it (the plan and the device
inputs a program keeps), `run` sets the unknowns and solves once, `exact`
restates the solve in float64 torch without any code of this repository, over
explicit residual lists.

Every case is a solve, because that is the call a program makes: Gauss-Newton
or Levenberg-Marquardt with a fixed count of PCG iterations, on images (warp,
Poisson), edge lists (mesh, embedded deformation, warp on a graph), voxel grids,
in float32 and in float64, one problem at a time, as a batch, or through the
server.  Sizes are those of the configurations (64^2 .. 4096^2 images,
icospheres of level 4 .. 7, a 128^3 volume), with ragged ones among them.  The
outer iterations are held to few, so that a rounding difference does not grow
along the trajectory: one outer iteration costs what every other one costs.
"""
import functools
import math

import numpy as np
import torch

from paper_1604_06525_gb300 import api, synth

SERVER_BUDGET = 64 << 30
SERVER_TOL = 1e-4


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # an interactive warp of a thumbnail: every call is launches and latency
        {"name": "warp_small", "kind": "warp", "W": 64, "H": 64, "masked": False, "method": "gn", "outer": 4,
         "inner": 10, "form": 0},
        # the 1024^2 warp of the benchmark, with the iteration the benchmark takes
        {"name": "warp_hd", "kind": "warp", "W": 1024, "H": 1024, "masked": False, "method": "gn", "outer": 4,
         "inner": 20, "form": 1},
        # a photo of no round size with parts of it cut out, the default iteration, damped
        {"name": "warp_cutout", "kind": "warp", "W": 1411, "H": 1003, "masked": True, "method": "lm", "outer": 3,
         "inner": 15, "form": 0},
        # the largest image: far beyond the L2 cache
        {"name": "warp_uhd", "kind": "warp", "W": 4096, "H": 4096, "masked": False, "method": "gn", "outer": 2,
         "inner": 15, "form": 1},
        # cloning into 30 % of a photo, four channels
        {"name": "poisson_hd", "kind": "poisson", "W": 1024, "H": 1024, "method": "gn", "outer": 2, "inner": 20,
         "form": 0},
        # the scanned-mesh size (163,842 vertices), planned with vertex tiles
        {"name": "mesh_l7", "kind": "mesh", "level": 7, "nx": 0, "ny": 0, "method": "lm", "outer": 2, "inner": 30,
         "tiled": True},
        # a game or editor mesh (10,242 vertices): what an artist drags, as planned by default
        {"name": "mesh_l5", "kind": "mesh", "level": 5, "nx": 0, "ny": 0, "method": "lm", "outer": 3, "inner": 10,
         "tiled": False},
        # volumetric deformation on a voxel grid
        {"name": "volume_128", "kind": "volume", "W": 128, "H": 128, "D": 128, "method": "lm", "outer": 3,
         "inner": 10},
        # embedded deformation: 12 unknowns a vertex
        {"name": "embedded_l7", "kind": "embedded", "level": 7, "nx": 0, "ny": 0, "method": "lm", "outer": 2,
         "inner": 30},
        # the mesh deformation where float32 cannot follow
        {"name": "mesh_f64_l7", "kind": "mesh64", "level": 7, "nx": 0, "ny": 0, "method": "lm", "outer": 2,
         "inner": 30},
        # a folder of images of uneven sizes in one call
        {"name": "batch_warps", "kind": "batch", "n": 96, "sizes_seed": 1604, "lo": 32, "hi": 512,
         "method": "gn", "outer": 3, "inner": 10, "form": 0},
        # requests of several users: planned, solved together and given back by the server
        {"name": "server_mix", "kind": "server", "n_warps": 10, "sizes_seed": 1610, "lo": 64, "hi": 1024, "n_meshes": 6,
         "level_lo": 4, "level_hi": 6, "outer": 4, "inner": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["warp", "warp", "poisson", "mesh", "volume", "embedded", "warp_graph", "warp64", "poisson64",
                       "mesh64", "batch", "server"])
    method = rng.choice(["gn", "lm"])
    outer = rng.randint(1, 3)
    inner = rng.randint(6, 20)
    if kind in ("warp", "poisson", "warp64", "poisson64"):
        hi = 2048 if kind == "warp" else 1400 if kind == "poisson" else 900
        lo = 48
        W, H = _log_int(rng, lo, hi), _log_int(rng, lo, hi)
        c = {"kind": kind, "W": W, "H": H, "method": method, "outer": outer, "inner": inner}
        if kind in ("warp", "poisson"):
            c["form"] = rng.randint(0, 1)
        if kind in ("warp", "warp64"):
            c["masked"] = rng.random() < 0.4
        return c
    if kind == "warp_graph":
        return {"kind": kind, "W": _log_int(rng, 48, 700), "H": _log_int(rng, 48, 700), "masked": rng.random() < 0.4,
                "method": method, "outer": outer, "inner": inner}
    if kind in ("mesh", "mesh64", "embedded"):
        # an open triangulated sheet of nx x ny vertices (degree 2 .. 6)
        hi = 400 if kind == "mesh" else 250
        c = {"kind": kind, "level": -1, "nx": _log_int(rng, 20, hi), "ny": _log_int(rng, 20, hi), "method": "lm",
             "outer": outer, "inner": inner}
        if kind == "mesh":
            c["tiled"] = rng.random() < 0.5
        return c
    if kind == "volume":
        return {"kind": kind, "W": _log_int(rng, 10, 110), "H": _log_int(rng, 10, 110), "D": _log_int(rng, 10, 110),
                "method": "lm", "outer": outer, "inner": inner}
    if kind == "batch":
        return {"kind": kind, "n": _log_int(rng, 12, 96), "sizes_seed": rng.randrange(1 << 20), "lo": 32,
                "hi": _log_int(rng, 96, 512), "method": method, "outer": outer, "inner": rng.randint(6, 12),
                "form": rng.randint(0, 1)}
    return {"kind": "server", "n_warps": rng.randint(2, 10), "sizes_seed": rng.randrange(1 << 20), "lo": 64,
            "hi": _log_int(rng, 256, 1024), "n_meshes": rng.randint(1, 6), "level_lo": 4,
            "level_hi": rng.randint(4, 6), "outer": rng.randint(2, 4), "inner": 10}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _warp_input(W, H, seed, masked=False):
    """A W x H warp: handles as the batched workload counts them, pulled by up
    to 8 pixels (a 16th of the shorter side where that is less)."""
    rng = np.random.default_rng(seed)
    ys, xs = np.mgrid[0:H, 0:W]
    mask = None
    if masked:   # smooth regions cut out, about a fifth of the image
        mask = (synth.smooth_noise(W, H, 1, seed + 3, cell=48)[0] > 0.66).astype(np.uint8)
    n = synth.warp_handle_count(W, H)
    idx = np.unique(rng.integers(0, W * H, n))
    if masked:
        idx = idx[mask.reshape(-1)[idx] == 0]
    amp = min(8.0, min(W, H) / 16.0)
    tgt = rng.uniform(-amp, amp, size=(idx.size, 2)).astype(np.float32)
    return synth.WarpProblem(W, H, np.stack([xs, ys]).astype(np.float32), np.zeros((3, H, W), np.float32),
                             idx.astype(np.int32), tgt, mask, 1.0, 100.0, seed)


@functools.lru_cache(maxsize=4)
def _sphere(level):
    verts, faces = synth.icosphere(level)
    v0, v1 = synth.directed_edges(faces, verts.shape[0])
    return verts.T.astype(np.float32), v0, v1


@functools.lru_cache(maxsize=4)
def _sheet(nx, ny):
    """Triangulated nx x ny sheet, unit spacing, a shallow relief."""
    ys, xs = np.mgrid[0:ny, 0:nx]
    z = 0.7 * np.sin(0.21 * xs) * np.cos(0.17 * ys)
    U = (np.stack([xs, ys, z]).reshape(3, -1) / 8.0).astype(np.float32)
    k = ys * nx + xs
    pairs = [(k[:, :-1], k[:, 1:]), (k[:-1], k[1:]), (k[:-1, :-1], k[1:, 1:])]
    a = np.concatenate([p[0].reshape(-1) for p in pairs])
    b = np.concatenate([p[1].reshape(-1) for p in pairs])
    v0, v1 = np.concatenate([a, b]), np.concatenate([b, a])
    order = np.lexsort((v1, v0))
    return U, v0[order].astype(np.int32), v1[order].astype(np.int32)


def _mesh_input(case, seed, level=None):
    if (level if level is not None else case["level"]) >= 0:
        U, v0, v1 = _sphere(level if level is not None else case["level"])
    else:
        U, v0, v1 = _sheet(case["nx"], case["ny"])
    V = U.shape[1]
    rng = np.random.default_rng(seed)
    idx = np.sort(rng.choice(V, size=max(1, round(0.01 * V)), replace=False)).astype(np.int32)
    tgt = rng.uniform(-0.05, 0.05, size=(idx.size, 3)).astype(np.float32)
    if case["kind"] == "embedded":
        x0 = np.zeros((12, V), np.float32)
        x0[3] = x0[7] = x0[11] = 1.0
        return synth.EmbeddedProblem(V, U, v0, v1, x0, idx, tgt, 1.0, 100.0, 1.0, -1, seed)
    return synth.MeshProblem(V, U, v0, v1, np.zeros((6, V), np.float32), idx, tgt, 1.0, 100.0, -1, seed)


def _problem_inputs(case, seed):
    """The problem instances of a case (one, or the members of a batch / stream)."""
    kind = case["kind"]
    if kind in ("warp", "warp64"):
        return [_warp_input(case["W"], case["H"], seed, case["masked"])]
    if kind == "warp_graph":
        return [synth.warp_graph_from_grid(_warp_input(case["W"], case["H"], seed, case["masked"]))]
    if kind in ("poisson", "poisson64"):
        return [synth.poisson_problem(case["W"], case["H"], seed=seed)]
    if kind in ("mesh", "mesh64", "embedded"):
        return [_mesh_input(case, seed)]
    if kind == "volume":
        n = max(8, case["W"] * case["H"] * case["D"] // 128)
        return [synth.volume_problem(case["W"], case["H"], case["D"], n, seed=seed, max_off=0.5)]
    if kind == "batch":
        sides = synth.batch_sides(case["n"], case["lo"], case["hi"], seed=case["sizes_seed"])
        return [_warp_input(int(s), int(s), seed + 1 + i) for i, s in enumerate(sides)]
    # server: warps and meshes in turn, as they arrive
    sides = synth.batch_sides(case["n_warps"], case["lo"], case["hi"], seed=case["sizes_seed"])
    warps = [_warp_input(int(s), int(s), seed + 1 + i) for i, s in enumerate(sides)]
    span = case["level_hi"] - case["level_lo"] + 1
    meshes = [_mesh_input(case, seed + 101 + i, level=case["level_lo"] + i % span) for i in range(case["n_meshes"])]
    out = []
    for i in range(max(len(warps), len(meshes))):
        out += warps[i:i + 1] + meshes[i:i + 1]
    return out


def prepare(case, seed):
    seed = 1 + int(seed) % (1 << 30)
    probs = _problem_inputs(case, seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "server":
        st["templates"] = [api.make_descriptor(p, "cuda") + (p.kind,) for p in probs]
        st["server"] = api.Server(SERVER_BUDGET, outer=case["outer"], inner=case["inner"], rel_tol=SERVER_TOL,
                                  max_rounds=16)
        return st
    if kind == "batch":
        st["problems"] = [api.Problem(p) for p in probs]
        st["batch"] = api.Batch(st["problems"])
        st["x0"] = [g.x.clone() for g in st["problems"]]
        return st
    g = api.ProblemF64(probs[0]) if kind.endswith("64") else api.Problem(probs[0])
    if case.get("tiled"):
        g.set_apply_form(1)
    st["problem"] = g
    st["x0"] = g.x.clone()
    return st


def _answer(x, reports, outer, f64=False):
    as_type = np.float64 if f64 else np.float32
    # a request that converged early keeps its last energy
    return {"x": x,
            "energies": np.array([r["E_history"] + r["E_history"][-1:] * (outer - r["outer_done"]) for r in reports],
                                 as_type),
            "lambda": np.array([r["lambda_final"] for r in reports], as_type),
            "outer": np.array([r["outer_done"] for r in reports], np.int64),
            "accepted": np.array([r["accepted"] for r in reports], np.int64),
            "pcg": np.array([r["pcg_done"] for r in reports], np.int64)}


def run(state):
    case = state["case"]
    if case["kind"] == "server":
        srv = state["server"]
        tickets = [srv.submit_template(t) for t in state["templates"]]
        busy = True
        while busy:
            active, queued = srv.step()
            busy = active + queued > 0
        done = [srv.poll(t) for t in tickets]
        return _answer(torch.cat([x.reshape(-1) for _, x in done]), [r for r, _ in done],
                       case["outer"])
    kw = {"pcg_form": case["form"]} if "form" in case else {}
    if case["kind"] == "batch":
        for g, x0 in zip(state["problems"], state["x0"]):
            g.x.copy_(x0)
        b = state["batch"]
        reports, _ = (b.solve_gn if case["method"] == "gn" else b.solve_lm)(case["outer"], case["inner"], **kw)
        return _answer(torch.cat([g.x.reshape(-1) for g in state["problems"]]), reports, case["outer"])
    g = state["problem"]
    g.x.copy_(state["x0"])
    report = (g.solve_gn if case["method"] == "gn" else g.solve_lm)(case["outer"], case["inner"], **kw)
    return _answer(g.x, [report], case["outer"], f64=case["kind"].endswith("64"))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# Per unit (pixel, vertex, voxel) in float32 values: unknowns, constants (rest
# positions and, on edge lists, the neighbour indices of both edge directions),
# preconditioner entries, and the multiply-adds of one product J^T J p.
_UNIT = {"warp": (3, 2, 2, 60), "poisson": (4, 0.25, 0, 34), "mesh": (6, 3 + 14, 4, 300), "volume": (6, 3, 4, 300),
         "embedded": (12, 3 + 14, 10, 420), "warp_graph": (3, 2 + 10, 2, 60)}


def work(case):
    """A PCG iteration ends in sums over all unknowns that the next one needs,
    so each iteration reads and writes delta, r and p once, and reads M^-1, the
    constants and (except Poisson, which is linear) cos / sin of the angles or
    the matrices; an outer iteration also reads and writes the unknowns."""
    kind = case["kind"]
    base = {"warp64": "warp", "poisson64": "poisson", "mesh64": "mesh", "batch": "warp"}.get(kind, kind)
    size = 8 if kind.endswith("64") else 4

    def solve(base, units, outer, inner):
        nx, nc, nm, flops = _UNIT[base]
        state = {"warp": 2, "warp_graph": 2, "mesh": 6, "volume": 6, "embedded": 9}.get(base, 0)
        per_iter = (6 * nx + nc + nm + state) * size
        per_outer = (5 * nx + nc + nm) * size
        return units * (outer * (inner * per_iter + per_outer) + 2 * nx * size), \
            units * outer * (inner * (2 * flops + 10 * nx) + 4 * flops)

    outer, inner = case["outer"], case["inner"]
    if kind in ("warp", "warp64", "warp_graph", "batch", "poisson", "poisson64", "volume"):
        if kind == "batch":
            units = float((synth.batch_sides(case["n"], case["lo"], case["hi"], seed=case["sizes_seed"]) ** 2).sum())
        else:
            units = case["W"] * case["H"] * case.get("D", 1) * (0.3 if base == "poisson" else 1.0)
        b, f = solve(base, units, outer, inner)
    elif kind == "server":
        sides = synth.batch_sides(case["n_warps"], case["lo"], case["hi"], seed=case["sizes_seed"])
        b, f = solve("warp", float((sides ** 2).sum()), outer, inner)
        span = case["level_hi"] - case["level_lo"] + 1
        for i in range(case["n_meshes"]):
            mb, mf = solve("mesh", 10 * 4 ** (case["level_lo"] + i % span) + 2, outer, inner)
            b, f = b + mb, f + mf
    else:
        units = 10 * 4 ** case["level"] + 2 if case["level"] >= 0 else case["nx"] * case["ny"]
        b, f = solve(base, units, outer, inner)
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# the same solves in float64 torch
# ---------------------------------------------------------------------------
def _dot(a, b, seg, n):
    """Sums over the unknowns of each member (seg: member of each unit)."""
    t = (a * b).sum(0)
    return t.sum().reshape(1) if n == 1 else torch.zeros(n, dtype=t.dtype, device=t.device).index_add_(0, seg, t)


class _Residuals:
    """Edge residuals over explicit lists a -> b (ARAP in 2-D / 3-D, embedded
    deformation, Poisson differences), fit residuals, and for the embedded
    deformation the column constraints.  x: (nx, units) float64."""

    def __init__(self, kind, x, a, b, U, hidx, htgt, wreg, wfit, free=None):
        self.kind, self.x0, self.a, self.b, self.U = kind, x, a, b, U
        self.h, self.t, self.wreg, self.wfit, self.free = hidx, htgt, wreg, wfit, free
        self.v = None if U is None else U[:, a] - U[:, b]
        self.D = {"warp": 2, "poisson": x.shape[0]}.get(kind, 3)

    def _rot(self, x):
        """R v per edge and its derivative by each angle (or matrix row pattern)."""
        v, a = self.v, self.a
        if self.kind == "warp":
            c, s = torch.cos(x[2])[a], torch.sin(x[2])[a]
            return torch.stack([c * v[0] - s * v[1], s * v[0] + c * v[1]]), \
                [torch.stack([-s * v[0] - c * v[1], c * v[0] - s * v[1]])]
        c, s = torch.cos(x[3:6])[:, a], torch.sin(x[3:6])[:, a]

        def rx(w, c, s):
            return torch.stack([w[0], c * w[1] - s * w[2], s * w[1] + c * w[2]])

        def ry(w, c, s):
            return torch.stack([c * w[0] + s * w[2], w[1], c * w[2] - s * w[0]])

        def rz(w, c, s):
            return torch.stack([c * w[0] - s * w[1], s * w[0] + c * w[1], w[2]])

        z = torch.zeros_like(v[0])
        w = rx(v, c[0], s[0])
        y = ry(w, c[1], s[1])
        gx = torch.stack([z, -s[0] * v[1] - c[0] * v[2], c[0] * v[1] - s[0] * v[2]])
        gy = torch.stack([-s[1] * w[0] + c[1] * w[2], z, -c[1] * w[0] - s[1] * w[2]])
        gz = torch.stack([-s[2] * y[0] - c[2] * y[1], c[2] * y[0] - s[2] * y[1], z])
        return rz(y, c[2], s[2]), [rz(ry(gx, c[1], s[1]), c[2], s[2]), rz(gy, c[2], s[2]), gz]

    def linearize(self, x):
        """F at x, kept with what J needs."""
        D, a, b = self.D, self.a, self.b
        sw = math.sqrt(self.wreg)
        self.at = x
        d = x[:D, a] - x[:D, b]
        if self.kind == "poisson":
            self.g = []
            fe = d - (self.U[:, a] - self.U[:, b])
        elif self.kind == "embedded":
            R = x[3:].reshape(3, 3, -1)
            fe = sw * (d + self.v - torch.einsum("ijv,jv->iv", R[:, :, a], self.v))
        else:
            rv, g = self._rot(x)
            self.g = [-sw * t for t in g]
            fe = sw * (d + self.v - rv)
        fh = None if self.h is None else math.sqrt(self.wfit) * (x[:D, self.h] - self.t)
        fc = None
        if self.kind == "embedded":
            c = [R[:, k] for k in range(3)]
            fc = torch.stack([(c[0] * c[1]).sum(0), (c[0] * c[2]).sum(0), (c[1] * c[2]).sum(0),
                              (c[0] * c[0]).sum(0) - 1, (c[1] * c[1]).sum(0) - 1, (c[2] * c[2]).sum(0) - 1])
        return fe, fh, fc

    def j(self, p):
        D, a, b = self.D, self.a, self.b
        sw = 1.0 if self.kind == "poisson" else math.sqrt(self.wreg)
        fe = sw * (p[:D, a] - p[:D, b])
        fc = None
        if self.kind == "embedded":
            P, R = p[3:].reshape(3, 3, -1), self.at[3:].reshape(3, 3, -1)
            fe = fe - sw * torch.einsum("ijv,jv->iv", P[:, :, a], self.v)
            fc = torch.stack([(R[:, i] * P[:, k] + P[:, i] * R[:, k]).sum(0)
                              for i, k in ((0, 1), (0, 2), (1, 2), (0, 0), (1, 1), (2, 2))])
        else:
            for m, g in enumerate(self.g):
                fe = fe + g * p[D + m, a]
        fh = None if self.h is None else math.sqrt(self.wfit) * p[:D, self.h]
        return fe, fh, fc

    def jt(self, f):
        fe, fh, fc = f
        D, a, b = self.D, self.a, self.b
        sw = 1.0 if self.kind == "poisson" else math.sqrt(self.wreg)
        out = torch.zeros_like(self.x0)
        out[:D].index_add_(1, a, sw * fe)
        out[:D].index_add_(1, b, -sw * fe)
        if self.kind == "embedded":
            rows = out[3:].reshape(3, 3, -1)
            for i in range(3):
                rows[i].index_add_(1, a, -sw * fe[i] * self.v)
            R = self.at[3:].reshape(3, 3, -1)
            for t, (i, k) in enumerate(((0, 1), (0, 2), (1, 2), (0, 0), (1, 1), (2, 2))):
                rows[:, i] += fc[t] * R[:, k]
                rows[:, k] += fc[t] * R[:, i]
        else:
            for m, g in enumerate(self.g):
                out[D + m].index_add_(0, a, (g * fe).sum(0))
        if fh is not None:
            out[:D].index_add_(1, self.h, math.sqrt(self.wfit) * fh)
        return out if self.free is None else out * self.free

    def diag(self):
        D, a, b = self.D, self.a, self.b
        w = 1.0 if self.kind == "poisson" else self.wreg
        out = torch.zeros_like(self.x0)
        one = torch.full(a.shape, w, dtype=out.dtype, device=out.device)
        deg = torch.zeros_like(out[0]).index_add_(0, a, one).index_add_(0, b, one)
        if self.h is not None:
            deg.index_add_(0, self.h, torch.full(self.h.shape, self.wfit, dtype=out.dtype, device=out.device))
        out[:D] = deg
        if self.kind == "embedded":
            rows = out[3:].reshape(3, 3, -1)
            for i in range(3):
                rows[i].index_add_(1, a, w * self.v * self.v)
            R = self.at[3:].reshape(3, 3, -1)
            for i, k in ((0, 1), (0, 2), (1, 2)):
                rows[:, i] += R[:, k] ** 2
                rows[:, k] += R[:, i] ** 2
            for k in range(3):
                rows[:, k] += (2.0 * R[:, k]) ** 2
        else:
            for m, g in enumerate(self.g):
                out[D + m].index_add_(0, a, (g * g).sum(0))
        return out if self.free is None else out * self.free

    def energy(self, f, seg, n):
        """Sum of squares per member."""
        fe, fh, fc = f
        if n == 1:
            return sum((t * t).sum() for t in f if t is not None).reshape(1)
        e = torch.zeros(n, dtype=fe.dtype, device=fe.device).index_add_(0, seg[self.a], (fe * fe).sum(0))
        return e if fh is None else e.index_add_(0, seg[self.h], (fh * fh).sum(0))


def _exact_solve(S, x, seg, n, lm, outer, inner, tol=0.0):
    """GN / LM with Jacobi PCG over n members side by side; per member the
    energies (one that converged keeps its last) and the damping."""
    def wide(s):
        return s if n == 1 else s[seg]

    dev = x.device
    lam = torch.full((n,), 1e-3 if lm else 0.0, dtype=torch.float64, device=dev)
    nu = torch.full_like(lam, 2.0)
    done = torch.zeros(n, dtype=torch.bool, device=dev)
    hist = []
    for _ in range(outer):
        f = S.linearize(x)
        E = S.energy(f, seg, n)
        hist.append(E)
        dg = S.diag()
        damp = wide(lam) * dg.clamp(1e-6, 1e32) if lm else 0.0
        m = dg + damp
        minv = torch.where(m != 0, 1.0 / torch.where(m != 0, m, torch.ones_like(m)), torch.ones_like(m))
        r = -S.jt(f)
        d = torch.zeros_like(x)
        z = minv * r
        p = z
        rz = _dot(r, z, seg, n)
        for _ in range(inner):
            q = S.jt(S.j(p)) + damp * p
            alpha = rz / _dot(p, q, seg, n)
            d = d + wide(alpha) * p
            r = r - wide(alpha) * q
            z = minv * r
            new = _dot(r, z, seg, n)
            p = z + wide(new / rz) * p
            rz = new
        if not lm:
            x = x + d
            continue
        model = S.energy(tuple(None if u is None else u + w for u, w in zip(f, S.j(d))), seg, n)
        trial = S.energy(S.linearize(x + d), seg, n)
        rho = (E - trial) / (E - model)
        ok = (rho > 1e-3) & ~done
        grown = ~ok & ~done
        x = torch.where(wide(ok), x + d, x)
        fac = torch.clamp(1 - (2 * rho - 1) ** 3, min=1.0 / 3.0)
        lam = torch.where(ok, lam * fac, torch.where(grown, lam * nu, lam))
        nu = torch.where(ok, torch.full_like(nu, 2.0), torch.where(grown, nu * 2, nu))
        if tol > 0:
            done = done | (ok & ((E - trial).abs() / E < tol))
    hist.append(S.energy(S.linearize(x), seg, n))
    return x, torch.stack(hist, 1), lam


def _grid_edges(W, H, dev):
    k = torch.arange(W * H, device=dev).reshape(H, W)
    a = [k[:, :-1], k[:, 1:], k[:-1], k[1:]]
    b = [k[:, 1:], k[:, :-1], k[1:], k[:-1]]
    return torch.cat([t.reshape(-1) for t in a]), torch.cat([t.reshape(-1) for t in b])


def _exact_residuals(p, dev):
    def f64(t):
        return torch.as_tensor(np.asarray(t, np.float64), device=dev)

    def idx(t):
        return torch.as_tensor(np.asarray(t, np.int64), device=dev)

    x = f64(p.x0).reshape(p.x0.shape[0], -1)
    if p.kind in ("warp", "poisson"):
        a, b = _grid_edges(p.W, p.H, dev)
        gone = None if p.mask is None else idx(p.mask).reshape(-1) != 0
        if p.kind == "poisson":
            keep = ~gone[a]
            return _Residuals("poisson", x, a[keep], b[keep], f64(p.guide).reshape(4, -1), None, None, 1.0, 0.0,
                              (~gone).double()), x
        if gone is not None:
            keep = ~(gone[a] | gone[b])
            a, b = a[keep], b[keep]
        return _Residuals("warp", x, a, b, f64(p.urshape).reshape(2, -1), idx(p.handle_idx), f64(p.handle_target).T,
                          p.w_reg, p.w_fit), x
    if p.kind == "volume":
        k = torch.arange(p.V, device=dev).reshape(p.D, p.H, p.W)
        pairs = [(k[:, :, :-1], k[:, :, 1:]), (k[:, :-1], k[:, 1:]), (k[:-1], k[1:])]
        a = torch.cat([s.reshape(-1) for u, w in pairs for s in (u, w)])
        b = torch.cat([s.reshape(-1) for u, w in pairs for s in (w, u)])
    else:
        a, b = idx(p.v0), idx(p.v1)
    kind = {"warp_graph": "warp", "embedded": "embedded"}.get(p.kind, "mesh")
    return _Residuals(kind, x, a, b, f64(p.urshape), idx(p.handle_idx), f64(p.handle_target).T, p.w_reg, p.w_fit), x


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    seed = 1 + int(seed) % (1 << 30)
    probs = _problem_inputs(case, seed)
    outer, inner = case["outer"], case["inner"]
    kind = case["kind"]
    if kind in ("batch", "server"):
        lm, tol = (case["method"] == "lm", 0.0) if kind == "batch" else (True, SERVER_TOL)
        order, xs, hs, ls = [], [None] * len(probs), [None] * len(probs), [None] * len(probs)
        for group in ("warp", "mesh"):   # the members of one kind side by side
            ids = [i for i, p in enumerate(probs) if p.kind == group]
            if not ids:
                continue
            parts = [_exact_residuals(probs[i], dev)[0] for i in ids]
            sizes = [s.x0.shape[1] for s in parts]
            base = np.concatenate([[0], np.cumsum(sizes)])
            S = _Residuals(group, torch.cat([s.x0 for s in parts], 1),
                           torch.cat([s.a + int(o) for s, o in zip(parts, base)]),
                           torch.cat([s.b + int(o) for s, o in zip(parts, base)]),
                           torch.cat([s.U for s in parts], 1),
                           torch.cat([s.h + int(o) for s, o in zip(parts, base)]),
                           torch.cat([s.t for s in parts], 1), parts[0].wreg, parts[0].wfit)
            seg = torch.repeat_interleave(torch.arange(len(ids), device=dev), torch.tensor(sizes, device=dev))
            x, h, lam = _exact_solve(S, S.x0, seg, len(ids), lm, outer, inner, tol)
            for j, i in enumerate(ids):
                xs[i] = x[:, int(base[j]):int(base[j + 1])].reshape(-1)
                hs[i] = h[j]
                ls[i] = lam[j]
        return {"x": torch.cat(xs), "energies": torch.stack(hs), "lambda": torch.stack(ls), "outer": None,
                "accepted": None, "pcg": None}
    S, x = _exact_residuals(probs[0], dev)
    lm = case["method"] == "lm"
    x, hist, lam = _exact_solve(S, x, None, 1, lm, outer, inner)
    p = probs[0]
    return {"x": x.reshape(-1, p.H, p.W) if p.kind in ("warp", "poisson") else x, "energies": hist,
            "lambda": lam, "outer": None, "accepted": None, "pcg": None}
