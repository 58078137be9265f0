"""What the performance of this framework is measured on: the calls a user makes.

In situ, a simulation hands one velocity field per cycle to `Context.advect`
(one block) or `Context.advect_batch` (many blocks) and ends each interval
with `Context.end_interval`; with an interval's fields resident, one
`Context.interval_graph` call takes the place of the per-cycle calls.
`adjoint.flow_map` and `adjoint.ftle` are the differentiable forms. Post hoc,
the seed lattice's missing basis flows are filled (`bto_fill_delaunay`,
`bto_fill_lattice`) and pathlines stitched (`bto_stitch_pathlines_ex`).

Sizes follow the paper's workloads and this repository's benchmark and
tests: blocks of 32^3 to 128^3 cells and 128 x 256 x 128, reductions 1:1 to
1:64 (seed strides 1 to 4), intervals of 5 to 200 cycles, steps of a quarter
cell at the largest speed.

`listed()` names the cases, `draw(rng)` makes another one of the same ranges,
`prepare` makes its inputs on the GPU, `run` is one pass, `work` the bytes
and operations a pass cannot do without, and `exact` the same outputs in
64-bit torch arithmetic.
"""
import math

import numpy as np
import torch

from paper_2004_02003_gb300 import adjoint, bto

DEV = "cuda"
NODE_ALIGN = 64          # nodes: a block's field starts on a 256-byte boundary, as an allocation of its own does


def listed():
    return [
        # the smallest block of one rank, one launch per cycle: launches and latency decide
        {"name": "block32", "kind": "interval", "nx": 32, "ny": 32, "nz": 32, "blocks": 1, "stride": 2,
         "cycles": 50, "layout": "f3", "exits": False},
        # an uneven block of one rank in weak scaling (1:8, interval 25), termination locations kept
        {"name": "block_uneven_exits", "kind": "interval", "nx": 67, "ny": 61, "nz": 72, "blocks": 1, "stride": 2,
         "cycles": 25, "layout": "f3", "exits": True},
        # the jet's grid on one rank, 16-byte nodes, 1:8, interval 10
        {"name": "jet_f4", "kind": "interval", "nx": 128, "ny": 256, "nz": 128, "blocks": 1, "stride": 2,
         "cycles": 10, "layout": "f4", "exits": False},
        # a 128^3 block seeded at every node (1:1), interval 20
        {"name": "block128_1to1", "kind": "interval", "nx": 128, "ny": 128, "nz": 128, "blocks": 1, "stride": 1,
         "cycles": 20, "layout": "f3", "exits": False},
        # 256^3 cells as 8 blocks, 1:8: the benchmark's workload on a shorter interval
        {"name": "turb256", "kind": "interval", "nx": 128, "ny": 128, "nz": 128, "blocks": 8, "stride": 2,
         "cycles": 25, "layout": "f3", "exits": False},
        # the same blocks seeded at every node: 16.8M particles
        {"name": "turb256_1to1", "kind": "interval", "nx": 128, "ny": 128, "nz": 128, "blocks": 8, "stride": 1,
         "cycles": 10, "layout": "f3", "exits": False},
        # many uneven blocks of 16 to 96 cells per axis, strides 1, 2 and 4, the whole interval in one call
        {"name": "graph_uneven", "kind": "graph", "blocks": 96, "lo": 16, "hi": 96, "cycles": 32, "layout": "f3"},
        # one small block at 1:27 over a long interval in one call
        {"name": "graph_block64", "kind": "graph", "blocks": 1, "lo": 64, "hi": 64, "stride": 3, "cycles": 100,
         "layout": "f3"},
        # gradients of a loss on the end positions with respect to seeds and every cycle's field
        {"name": "gradients", "kind": "gradients", "nx": 64, "ny": 64, "nz": 64, "particles": 32768, "cycles": 200,
         "every": 16},
        # flow-map Jacobian and FTLE of a denser set of seeds
        {"name": "ftle", "kind": "ftle", "nx": 64, "ny": 64, "nz": 64, "particles": 100003, "cycles": 50, "every": 16},
        # the paper's reconstruction of the basis flows lost at block faces
        {"name": "delaunay128", "kind": "delaunay", "sx": 128, "sy": 128, "sz": 128, "reach": 6.0},
        # lattice fill of three intervals' basis flows, then pathlines through them
        {"name": "pathlines", "kind": "pathlines", "sx": 192, "sy": 200, "sz": 177, "reach": 5.0, "intervals": 3,
         "queries": 200000, "scheme": "trilinear"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["interval", "interval", "interval", "batch", "graph", "graph", "gradients", "ftle", "delaunay",
                       "pathlines"])
    if kind == "interval":
        return {"kind": "interval", "nx": _log_int(rng, 24, 160), "ny": _log_int(rng, 24, 160),
                "nz": _log_int(rng, 24, 160), "blocks": 1, "stride": rng.choice([1, 2, 2, 3, 4]),
                "cycles": _log_int(rng, 5, 50), "layout": rng.choice(["f3", "f3", "f4"]),
                "exits": rng.random() < 0.3}
    if kind == "batch":
        return {"kind": "interval", "nx": _log_int(rng, 24, 128), "ny": _log_int(rng, 24, 128),
                "nz": _log_int(rng, 24, 128), "blocks": rng.choice([2, 4, 8]), "stride": rng.choice([1, 2, 2, 3]),
                "cycles": _log_int(rng, 5, 25), "layout": rng.choice(["f3", "f3", "f4"]),
                "exits": rng.random() < 0.3}
    if kind == "graph":
        hi = _log_int(rng, 24, 96)
        return {"kind": "graph", "blocks": _log_int(rng, 1, 64), "lo": rng.randint(16, hi), "hi": hi,
                "cycles": _log_int(rng, 5, 64), "layout": rng.choice(["f3", "f3", "f4"])}
    if kind in ("gradients", "ftle"):
        return {"kind": kind, "nx": _log_int(rng, 24, 80), "ny": _log_int(rng, 24, 80), "nz": _log_int(rng, 24, 80),
                "particles": _log_int(rng, 2000, 200000), "cycles": _log_int(rng, 10, 100),
                "every": rng.choice([4, 8, 16, 16, 32])}
    if kind == "delaunay":
        return {"kind": "delaunay", "sx": rng.randint(24, 112), "sy": rng.randint(24, 112), "sz": rng.randint(24, 112),
                "reach": round(rng.uniform(1.5, 6.0), 2)}
    return {"kind": "pathlines", "sx": rng.randint(32, 224), "sy": rng.randint(32, 224), "sz": rng.randint(32, 224),
            "reach": round(rng.uniform(1.5, 6.0), 2), "intervals": rng.randint(1, 5),
            "queries": _log_int(rng, 1000, 1000000), "scheme": rng.choice(["trilinear", "barycentric"])}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
class _Modes:
    """Divergence-free random Fourier modes, |k| in [1, 16] over the unit
    domain, amplitude |k|^(-5/6), phases drifting per cycle."""

    def __init__(self, rs, m=48):
        d = rs.standard_normal((m, 3))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        kmag = rs.uniform(1.0, 16.0, size=m)
        e = np.cross(d, rs.standard_normal((m, 3)))
        e /= np.linalg.norm(e, axis=1, keepdims=True)
        self.k, self.e, self.amp = d * kmag[:, None], e, kmag ** (-5.0 / 6.0)
        self.phase, self.drift = rs.uniform(0, 2 * np.pi, m), rs.uniform(0, 0.05, m)
        self.scale = 1.0

    def basis(self, axes):
        """Per-axis phases of the nodes at `axes` (3 float64 arrays): the part that does not change with the cycle."""
        X, Y, Z = (torch.polar(torch.ones(len(a), len(self.amp), dtype=torch.float32, device=DEV),
                               (torch.tensor(a, device=DEV)[:, None] *
                                torch.tensor(2 * np.pi * self.k[:, i], device=DEV)[None]).float())
                   for i, a in enumerate(axes))
        T = (Z[:, None, :] * Y[None, :, :]).reshape(-1, len(self.amp))
        return torch.cat([T.real, -T.imag], dim=1).contiguous(), X

    def coefficients(self, X, cycle, comps):
        W = torch.tensor(self.scale * self.amp * np.exp(1j * (self.phase + cycle * self.drift)), device=DEV)
        e = torch.tensor(np.concatenate([self.e, np.zeros((len(self.amp), comps - 3))], axis=1), device=DEV)
        G = (X.T[:, :, None] * (W[:, None] * e).to(torch.complex64)[:, None, :]).reshape(len(self.amp), -1)
        return torch.cat([G.real, G.imag], dim=0).contiguous()

    def normalise(self):
        g = np.linspace(0.0, 1.0, 33)
        A, X = self.basis((g, g, g))
        u = (A @ self.coefficients(X, 0, 3)).view(-1, 3)
        self.scale = float(1.0 / u.norm(dim=1).max())


def _layout(case):
    """Blocks of a case: extents, first cell in the domain, strides, cell side and the domain's cells. The sizes are
    the case's, whatever the seed of its inputs."""
    if case["kind"] == "graph":
        nb = case["blocks"]
        rs = np.random.RandomState(nb + 1000 * case["lo"] + 100000 * case["hi"] + case["cycles"])
        ext = []
        for _ in range(nb):
            e = rs.randint(case["lo"], case["hi"] + 1, size=3)
            ext.append([int(max(v, -(-int(e.max()) // 3))) for v in e])          # aspect ratios up to 3
        strides = [int(case["stride"]) if "stride" in case else int(rs.choice([1, 2, 4])) for _ in range(nb)]
        side = 256
        first = [[int(rs.randint(0, max(1, side - v))) for v in e] for e in ext]
    else:
        n, nb = (case["nx"], case["ny"], case["nz"]), case["blocks"]
        grid = (min(nb, 2), 2 if nb >= 4 else 1, 2 if nb >= 8 else 1)
        ext, strides = [list(n)] * nb, [case["stride"]] * nb
        first = [[(b % grid[0]) * n[0], (b // grid[0]) % grid[1] * n[1], b // (grid[0] * grid[1]) * n[2]]
                 for b in range(nb)]
        side = max(g * v for g, v in zip(grid, n))
    return ext, first, strides, float(np.float32(1.0 / side)), side


def _fields(modes, ext, first, side, cycles, comps):
    """[cycles, nodes of all blocks, comps] float32 and each block's first node."""
    start, total = [], 0
    for e in ext:
        start.append(total)
        total += -(-((e[0] + 1) * (e[1] + 1) * (e[2] + 1)) // NODE_ALIGN) * NODE_ALIGN
    buf = torch.zeros((cycles, total, comps), dtype=torch.float32, device=DEV)
    for e, f, s in zip(ext, first, start):
        A, X = modes.basis([(f[i] + np.arange(e[i] + 1)) / side for i in range(3)])
        for c in range(cycles):
            out = buf[c, s:s + A.shape[0] * X.shape[0]].view(A.shape[0], X.shape[0] * comps)
            torch.matmul(A, modes.coefficients(X, c, comps), out=out)
    return buf, start


def _interval_inputs(case, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    modes = _Modes(rs)
    modes.normalise()
    ext, first, strides, h, side = _layout(case)
    buf, start = _fields(modes, ext, first, side, case["cycles"], 4 if case["layout"] == "f4" else 3)
    origins = [[f[i] * h for i in range(3)] for f in first]
    return {"ext": ext, "origins": origins, "h": h, "strides": strides, "buf": buf, "start": start, "dt": 0.25 * h}


def _adjoint_inputs(case, seed):
    """The time-dependent ABC flow on its natural period, random seeds away from the faces."""
    rs = np.random.RandomState(seed % (1 << 31))
    n = (case["nx"], case["ny"], case["nz"])
    h = float(np.float32(2 * np.pi / 64))
    a, b, c = math.sqrt(3.0), math.sqrt(2.0), 1.0
    shift = rs.uniform(0, 2 * np.pi, 3)
    x, y, z = (torch.arange(n[i] + 1, dtype=torch.float64, device=DEV) * h + shift[i] for i in range(3))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    fields = torch.empty((case["cycles"], n[2] + 1, n[1] + 1, n[0] + 1, 3), dtype=torch.float32, device=DEV)
    for k in range(case["cycles"]):
        s = 0.1 * math.sin(2 * np.pi * 0.01 * k)
        fields[k, ..., 0] = a * torch.sin(z + s) + c * torch.cos(y + s)
        fields[k, ..., 1] = b * torch.sin(x + s) + a * torch.cos(z + s)
        fields[k, ..., 2] = c * torch.sin(y + s) + b * torch.cos(x + s)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    u = torch.rand((case["particles"], 3), generator=gen, device=DEV)
    seeds = (u * 0.9 + 0.05) * torch.tensor([v * h for v in n], dtype=torch.float32, device=DEV)
    return {"n": n, "h": h, "fields": fields, "seeds": seeds, "dt": 0.01}


def _basis_flows(case, seed, intervals):
    """Basis flows of a global seed lattice cut into 2 x 2 x 2 blocks: smooth displacements of up to `reach` lattice
    units, missing where the end lies outside the seed's block, plus a few stray holes."""
    S = (case["sx"], case["sy"], case["sz"])
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rs = np.random.RandomState(seed % (1 << 31))
    ax = [torch.arange(S[i], dtype=torch.float32, device=DEV) for i in range(3)]
    j = torch.stack(torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")[::-1], dim=-1)
    half = torch.tensor([-(-v // 2) for v in S], dtype=torch.float32, device=DEV)
    last = torch.tensor([v - 1 for v in S], dtype=torch.float32, device=DEV)
    upper = j >= half
    lo = torch.where(upper, half, torch.zeros_like(half))
    hi = torch.where(upper, last, half)
    side = float(max(S))
    flows = []
    for _ in range(intervals):
        modes = _Modes(rs, 24)
        modes.normalise()
        A, X = modes.basis([np.arange(S[i]) / side for i in range(3)])
        d = (A @ modes.coefficients(X, 0, 3)).view(S[2], S[1], S[0], 3) * case["reach"]
        e = j + d
        valid = ((e >= lo) & (e <= hi)).all(dim=-1) & (torch.rand(e.shape[:-1], generator=gen, device=DEV) > 5e-4)
        flows.append((torch.minimum(torch.maximum(e, lo), hi).contiguous().view(-1, 3),
                      valid.to(torch.uint8).contiguous().view(-1)))
    return S, flows


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("interval", "graph"):
        s = _interval_inputs(case, seed)
        nb, L, h = len(s["ext"]), case["cycles"], s["h"]
        if nb == 1:
            ctx = bto.Context(s["ext"][0], s["origins"][0], (h, h, h), s["strides"][0], L)
        else:
            ctx = bto.Context.batch(s["ext"], s["origins"], [(h, h, h)] * nb, s["strides"], L)
        if case["layout"] == "f4":
            ctx.set_layout(bto.BTO_FIELD_F4_AOS)
        node = s["buf"].stride(1) * 4
        ptrs = [[s["buf"][c].data_ptr() + node * b for b in s["start"]] for c in range(L)]
        table = torch.tensor(ptrs, dtype=torch.int64, device=DEV)
        if kind == "graph":
            return {"kind": kind, "ctx": ctx, "table": table, "dt": s["dt"], "keep": s["buf"]}
        return {"kind": kind, "ctx": ctx, "dt": s["dt"], "keep": s["buf"], "exits": case["exits"], "batch": nb > 1,
                "fields": list(table) if nb > 1 else list(s["buf"])}
    if kind in ("gradients", "ftle"):
        s = _adjoint_inputs(case, seed)
        h = s["h"]
        tape = adjoint.Tape(s["n"], (0.0, 0.0, 0.0), (h, h, h), case["particles"], case["cycles"], case["every"])
        grad = kind == "gradients"
        return {"kind": kind, "tape": tape, "dt": s["dt"], "seeds": s["seeds"].requires_grad_(grad),
                "fields": s["fields"].requires_grad_(grad)}
    if kind == "delaunay":
        S, flows = _basis_flows(case, seed, 1)
        return {"kind": kind, "S": S, "ends": flows[0][0], "valid": flows[0][1]}
    S, flows = _basis_flows(case, seed, case["intervals"])
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    start = torch.rand((case["queries"], 3), generator=gen, device=DEV) * torch.tensor(
        [v - 1 for v in S], dtype=torch.float32, device=DEV)
    return {"kind": kind, "S": S, "flows": flows, "start": start,
            "scheme": bto.BTO_STITCH_BARYCENTRIC if case["scheme"] == "barycentric" else bto.BTO_STITCH_TRILINEAR}


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "interval":
        ctx, dt = s["ctx"], s["dt"]
        if s["batch"]:
            for f in s["fields"]:
                ctx.advect_batch(f, dt)
        else:
            for f in s["fields"]:
                ctx.advect(f, dt)
        return ctx.end_interval(exits=s["exits"])
    if kind == "graph":
        s["ctx"].interval_graph(s["table"], s["dt"])
        return s["ctx"].end_interval()
    if kind == "gradients":
        seeds, fields = s["seeds"], s["fields"]
        ends, valid, exit_cycle = adjoint.flow_map(seeds, fields, s["tape"], s["dt"])
        loss = (((ends - seeds) ** 2).sum(dim=1) * valid).sum()
        g_seeds, g_fields = torch.autograd.grad(loss, (seeds, fields))
        return {"ends": ends, "valid": valid, "exit_cycle": exit_cycle, "g_seeds": g_seeds, "g_fields": g_fields}
    if kind == "ftle":
        ends, valid, jac, ftle = adjoint.ftle(s["tape"], s["seeds"], s["fields"], s["dt"])
        return {"ends": ends, "valid": valid, "jac": jac, "ftle": ftle}
    if kind == "delaunay":
        out, status = torch.empty_like(s["ends"]), torch.empty_like(s["valid"])
        bto.bto_fill_delaunay(s["S"], s["ends"], s["valid"], out, status)
        return {"filled": out, "status": status}
    filled, statuses = [], []
    for ends, valid in s["flows"]:
        out, status = torch.empty_like(ends), torch.empty_like(valid)
        bto.bto_fill_lattice(s["S"], ends, valid, out, status)
        filled.append(out)
        statuses.append(status)
    K, nq = len(filled), s["start"].shape[0]
    table = torch.tensor([f.data_ptr() for f in filled], dtype=torch.int64, device=DEV)
    path = torch.empty((K + 1, nq, 3), dtype=torch.float32, device=DEV)
    bto.bto_stitch_pathlines_ex(s["S"], (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), K, table, nq, s["start"], path, s["scheme"])
    return {"filled": filled, "status": statuses, "path": path}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
STEP_FLOPS = 4 * 7 * 3 * 3 + 60          # four trilinear samples of three components, and the RK4 combination


def work(case):
    kind = case["kind"]
    if kind in ("interval", "graph"):
        ext, _, strides, _, _ = _layout(case)
        seeds = [math.prod(-(-v // st) for v in e) for e, st in zip(ext, strides)]
        nodes = sum(min(math.prod(v + 1 for v in e), 8 * p) for e, p in zip(ext, seeds))   # 8 nodes a seed at most
        P, L = sum(seeds), case["cycles"]
        per_cycle = (16 if case["layout"] == "f4" else 12) * nodes
        if kind == "interval":           # positions are kept between the calls
            per_cycle += 24 * P
        return {"bytes": L * per_cycle + P * (29 + (16 if case.get("exits") else 0)), "flops": L * P * STEP_FLOPS}
    if kind in ("gradients", "ftle"):
        P, L = case["particles"], case["cycles"]
        nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        fields = 12 * L * min(nodes, 8 * P)
        if kind == "gradients":          # fields in, their gradients out; forward, and twice as much back
            return {"bytes": fields + 12 * L * nodes + P * (12 + 17 + 12), "flops": 3 * L * P * STEP_FLOPS}
        return {"bytes": fields + P * (12 + 13 + 36 + 4), "flops": 7 * L * P * STEP_FLOPS}
    P = case["sx"] * case["sy"] * case["sz"]
    if kind == "delaunay":
        return {"bytes": 26 * P, "flops": 0}
    K, nq = case["intervals"], case["queries"]
    corners = 4 if case["scheme"] == "barycentric" else 8
    return {"bytes": 26 * P * K + nq * (12 + K * (12 * corners + 12)), "flops": nq * K * 3 * 2 * corners}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _cell64(x, n):
    """Cell and fractions of points in cell units, clamped into the block."""
    x = torch.minimum(torch.clamp(x, min=0.0), n)
    i = torch.minimum(torch.floor(x), n - 1)
    return i.long(), x - i


def _sample64(field, x, n, nn, base):
    """Trilinear sample of `field` [nodes, >= 3] at x [P, 3]; n, nn: cells and nodes per axis, base: first node."""
    i, f = _cell64(x, n)
    v = 0.0
    for c in (0, 1):
        for b in (0, 1):
            for a in (0, 1):
                node = base + (i[:, 0] + a) + nn[:, 0] * ((i[:, 1] + b) + nn[:, 1] * (i[:, 2] + c))
                w = ((f[:, 0] if a else 1 - f[:, 0]) * (f[:, 1] if b else 1 - f[:, 1]) *
                     (f[:, 2] if c else 1 - f[:, 2]))
                v = v + w[:, None] * torch.index_select(field, 0, node)[:, :3]
    return v


def _inside64(x, n):
    return ((x >= 0) & (x <= n)).all(dim=1)


def _advect64(fields, x, n, base, s, alive):
    """One RK4 step per field with the closed-box tests. Returns positions, exit cycle (-1 while alive), the first
    outside point and its stage."""
    nn = n.long() + 1
    exit_cycle = torch.where(alive, -1, 0)
    q, stage = torch.zeros_like(x), torch.zeros_like(exit_cycle)
    for c, f in enumerate(fields):
        f = f.double()
        ok = alive

        def test(p, k):
            nonlocal ok, q, stage
            out = ok & ~_inside64(p, n)
            q, stage = torch.where(out[:, None], p.detach(), q), torch.where(out, k, stage)
            ok = ok & ~out

        k1 = _sample64(f, x, n, nn, base)
        p = x + 0.5 * s * k1
        test(p, 1)
        k2 = _sample64(f, p, n, nn, base)
        p = x + 0.5 * s * k2
        test(p, 2)
        k3 = _sample64(f, p, n, nn, base)
        p = x + s * k3
        test(p, 3)
        k4 = _sample64(f, p, n, nn, base)
        p = x + s / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        test(p, 4)
        x = torch.where(ok[:, None], p, x)
        exit_cycle = torch.where(alive & ~ok, c, exit_cycle)
        alive = ok
    return x, exit_cycle, q, stage


def _exact_interval(case, seed):
    s = _interval_inputs(case, seed)
    h, out = s["h"], []
    o32 = [[float(np.float32(v)) for v in o] for o in s["origins"]]
    parts = []
    for b, (e, st) in enumerate(zip(s["ext"], s["strides"])):
        ax = [torch.arange(0, e[i], st, dtype=torch.float64, device=DEV) for i in range(3)]
        j = torch.stack(torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")[::-1], dim=-1).reshape(-1, 3)
        one = torch.ones((j.shape[0], 1), dtype=torch.float64, device=DEV)
        parts.append((j, one * torch.tensor(e, dtype=torch.float64, device=DEV),
                      one * torch.tensor(o32[b], dtype=torch.float64, device=DEV),
                      torch.full((j.shape[0],), s["start"][b], dtype=torch.int64, device=DEV)))
    x0, n, origin, base = (torch.cat([p[k] for p in parts]) for k in range(4))
    step = float(np.float32(s["dt"])) / h
    exits = bool(case.get("exits"))
    for at in range(0, x0.shape[0], 1 << 21):
        cut = slice(at, at + (1 << 21))
        x, e, q, stage = _advect64(list(s["buf"]), x0[cut], n[cut], base[cut], step,
                                   torch.ones(x0[cut].shape[0], dtype=torch.bool, device=DEV))
        got = [x * h + origin[cut]]
        if exits:
            d = q - x
            t = torch.where(q > n[cut], (n[cut] - x) / d, torch.where(q < 0, -x / d, torch.ones_like(d)))
            t = t.amin(dim=1).clamp(0.0, 1.0)
            nan = torch.full_like(t, float("nan"))
            pos = torch.minimum((x + t[:, None] * d).clamp(min=0.0), n[cut]) * h + origin[cut]
            left = e >= 0
            got += [torch.where(left[:, None], pos, nan[:, None]),
                    torch.where(left, e + t * torch.where(stage <= 2, 0.5, 1.0), nan)]
        out.append(got)
    r = {"seeds": x0 * h + origin, "ends": torch.cat([g[0] for g in out]), "valid": None, "exit_cycle": None}
    if exits:
        r["exit_pos"], r["exit_time"] = (torch.cat([g[k] for g in out]) for k in (1, 2))
    return r


def _exact_adjoint(case, seed):
    s = _adjoint_inputs(case, seed)
    P, h, grad = case["particles"], s["h"], case["kind"] == "gradients"
    seeds = s["seeds"].double().requires_grad_(True)
    fields = [f.double().view(-1, 3).requires_grad_(grad) for f in s["fields"]]
    n = torch.tensor(s["n"], dtype=torch.float64, device=DEV).expand(P, 3)
    base = torch.zeros(P, dtype=torch.int64, device=DEV)
    step = float(np.float32(s["dt"])) / h
    x0 = seeds / h
    x, e, _, _ = _advect64(fields, x0, n, base, step, _inside64(x0, n))
    ends = x * h
    valid = e < 0
    if grad:
        loss = (((ends - seeds) ** 2).sum(dim=1) * valid).sum()
        got = torch.autograd.grad(loss, [seeds] + fields)
        return {"ends": ends.detach(), "valid": None, "exit_cycle": None, "g_seeds": got[0],
                "g_fields": torch.stack([g.view(s["fields"].shape[1:]) for g in got[1:]])}
    jac = torch.stack([torch.autograd.grad(ends[:, a].sum(), seeds, retain_graph=True)[0] for a in range(3)], dim=1)
    J = jac.cpu().numpy()
    lam = np.linalg.eigvalsh(np.einsum("pka,pkb->pab", J, J))[:, -1]
    T = abs(float(np.float32(s["dt"])) * case["cycles"])
    ftle = np.where(valid.cpu().numpy(), 0.5 * np.log(np.maximum(lam, 1e-300)) / T, np.nan)
    return {"ends": ends.detach(), "valid": None, "jac": jac, "ftle": ftle}


def _fill_lattice64(S, ends, valid):
    """Missing entries from the closest valid neighbours along the axis where the two are closest together."""
    e, v = ends.double().view(S[2], S[1], S[0], 3), valid.view(S[2], S[1], S[0]) != 0
    big = 1 << 30
    best = torch.full(v.shape, big, dtype=torch.int64, device=DEV)
    out = torch.where(v[..., None], e, torch.full_like(e, float("nan")))
    for axis in (0, 1, 2):
        dim = 2 - axis
        at = torch.arange(S[axis], device=DEV).view([-1 if d == dim else 1 for d in range(3)]).expand(v.shape)
        left = torch.where(v, at, -1).cummax(dim=dim).values
        right = torch.where(v, at, big).flip(dim).cummin(dim=dim).values.flip(dim)
        has = ~v & (left >= 0) & (right < big)
        gap = torch.where(has, right - left, big)
        take = has & (gap < best)
        best = torch.where(take, gap, best)
        li, ri = left.clamp(min=0), right.clamp(max=S[axis] - 1)
        el = torch.gather(e, dim, li[..., None].expand(e.shape))
        er = torch.gather(e, dim, ri[..., None].expand(e.shape))
        wl = (ri - at).double() / gap.double()
        out = torch.where(take[..., None], wl[..., None] * el + (1 - wl)[..., None] * er, out)
    return out.view(-1, 3)


def _stitch64(S, flows, start, barycentric):
    x, path = start.double(), [start.double()]
    n = torch.tensor([v - 1 for v in S], dtype=torch.float64, device=DEV)
    for E in flows:
        i, f = _cell64(torch.nan_to_num(x), n.expand(x.shape))
        ok = _inside64(x, n)
        if barycentric:
            t, ax = torch.sort(f, dim=1, descending=True, stable=True)
            w = torch.stack([1 - t[:, 0], t[:, 0] - t[:, 1], t[:, 1] - t[:, 2], t[:, 2]], dim=1)
            j, y = i.clone(), 0.0
            for m in range(4):
                if m:
                    j = j + torch.nn.functional.one_hot(ax[:, m - 1], 3)
                y = y + w[:, m:m + 1] * E[j[:, 0] + S[0] * (j[:, 1] + S[1] * j[:, 2])]
        else:
            nn = (n.long() + 1).expand(x.shape)
            y = _sample64(E, torch.nan_to_num(x), n.expand(x.shape), nn, torch.zeros_like(i[:, 0]))
        x = torch.where(ok[:, None], y, torch.full_like(y, float("nan")))
        path.append(x)
    return torch.stack(path)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("interval", "graph"):
        return _exact_interval(case, seed)
    if kind in ("gradients", "ftle"):
        return _exact_adjoint(case, seed)
    if kind == "delaunay":               # a triangulation of millions of points takes minutes without this framework
        return None
    s = prepare(case, seed)
    filled = [_fill_lattice64(s["S"], e, v) for e, v in s["flows"]]
    return {"filled": filled, "status": [None] * len(filled),
            "path": _stitch64(s["S"], filled, s["start"], case["scheme"] == "barycentric")}
