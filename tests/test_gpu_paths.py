"""GPU: the routes a call takes by its sizes, types and alignment give what the
general route or the oracle gives, at the sizes where a route begins, ends or
leaves a remainder.
"""
import numpy as np
import pytest

import oracle
from paper_2004_02003_gb300 import adjoint, bto, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    from paper_2004_02003_gb300 import build
    build.build()
    bto.load()


def _fields(n, L, seed, comps=3):
    """Per-cycle node fields of a block of n cells on the unit box, on the device."""
    import torch
    modes = inputs.fourier_modes(seed, m=10, kmax=4.0)
    h = (1.0 / max(n),) * 3
    out = []
    for c in range(L):
        f = inputs.fourier_field(modes, n, (0.0, 0.0, 0.0), h, c)
        if comps == 4:
            f = np.concatenate([f, np.zeros(f.shape[:-1] + (1,), f.dtype)], axis=-1)
        out.append(torch.from_numpy(np.ascontiguousarray(f, dtype=np.float32)).cuda())
    return out, h


def _numpy(out):
    return {k: v.cpu().numpy() for k, v in out.items()}


# Seeds: a single one, around one unit of 32, around a region of 128, a wide
# row with a remainder, and the last count taken by four lanes per particle
# (112 slots per SM: 17,024 on 152 SMs) with the first beyond it.
@pytest.mark.parametrize("n,stride", [((1, 1, 1), 1), ((31, 1, 1), 1), ((32, 2, 1), 1), ((43, 3, 1), 1), ((67, 9, 5), 2),
                                      ((38, 28, 16), 1), ((38, 28, 17), 1), ((50, 41, 30), 1)])
@pytest.mark.parametrize("comps,ppt", [(3, 0), (3, 1), (3, 2), (3, 4), (4, 2)])
def test_interval_in_one_launch_equals_per_cycle_calls(n, stride, comps, ppt):
    import torch
    L, dt = 9, 0.03
    fields, h = _fields(n, L, 31 + n[0], comps)
    table = torch.tensor([f.data_ptr() for f in fields], dtype=torch.int64, device="cuda")
    got = []
    for graph in (False, True):
        ctx = bto.Context(n, (0, 0, 0), h, stride, L)
        if comps == 4:
            ctx.set_layout(bto.BTO_FIELD_F4_AOS)
        if ppt:
            ctx.set_launch(128, ppt)
        for _ in range(2):                       # the second interval starts from the seeds again
            if graph:
                ctx.interval_graph(table, dt)
            else:
                for f in fields:
                    ctx.advect(f, dt)
            act = torch.zeros((ctx.P, 4), device="cuda")
            live = ctx.copy_active(act)          # the list itself: survivors in order
            out = _numpy(ctx.end_interval(exits=True))
            got.append((live, act.cpu().numpy(), out))
        ctx.check()
        ctx.close()
    for live, act, out in got[1:]:
        assert live == got[0][0]
        assert np.array_equal(act.view(np.int32), got[0][1].view(np.int32))
        for k, v in out.items():
            assert np.array_equal(v, got[0][2][k], equal_nan=True), k


# The interval's end writes outputs and the next seeds in one pass; the
# allocation-free interval writes them by its own kernels. Widths: whole runs
# of 32 seeds, and runs that end inside a unit.
@pytest.mark.parametrize("n,stride", [((32, 5, 3), 1), ((64, 4, 4), 2), ((33, 7, 5), 1), ((95, 3, 2), 3)])
def test_interval_end_equals_allocation_free_interval(n, stride):
    import torch
    L, dt = 8, 0.04
    fields, h = _fields(n, L, 77 + n[0])
    table = torch.tensor([f.data_ptr() for f in fields], dtype=torch.int64, device="cuda")
    ctx = bto.Context(n, (0, 0, 0), h, stride, L)
    for _ in range(2):
        for f in fields:
            ctx.advect(f, dt)
        out = _numpy(ctx.end_interval(exits=True))
        P = ctx.P
        ref = {"seeds": torch.empty((P, 3), device="cuda"), "ends": torch.empty((P, 3), device="cuda"),
               "valid": torch.empty(P, dtype=torch.uint8, device="cuda"),
               "exit_cycle": torch.empty(P, dtype=torch.int32, device="cuda")}
        bto.bto_interval_noalloc(n, (0, 0, 0), h, stride, L, table, dt, ref["seeds"], ref["ends"], ref["valid"],
                                 ref["exit_cycle"])
        for k, v in _numpy(ref).items():
            assert np.array_equal(out[k], v), k
        left = out["valid"] == 0
        assert left.any() and np.isfinite(out["exit_pos"][left]).all() and np.isnan(out["exit_pos"][~left]).all()
        assert np.isfinite(out["exit_time"][left]).all() and np.isnan(out["exit_time"][~left]).all()
    ctx.close()


# Particles are independent: their ends and seed gradients do not depend on
# the others, so not on whether the list is sorted by cell (2048 on) or takes
# four lanes per particle (up to 132 per SM).
@pytest.mark.parametrize("P", [1, 33, 2047, 2048, 20064, 20065, 45001])
def test_tape_results_do_not_depend_on_the_number_of_particles(P):
    import torch
    n, L, dt = (24, 20, 17), 21, 0.02
    fields, h = _fields(n, L, 5)
    F = torch.stack(fields)
    rng = np.random.default_rng(3)
    box = np.asarray(n) * np.asarray(h)
    x = rng.uniform(-0.02, 1.02, size=(45001, 3)) * box      # some start outside
    g = rng.standard_normal((45001, 3))
    runs = []
    for count in (45001, P):
        tape = adjoint.Tape(n, (0, 0, 0), h, count, L, 5)
        s = torch.from_numpy(x[:count].astype(np.float32)).cuda().requires_grad_(True)
        ends, valid, exit_cycle = adjoint.flow_map(s, F, tape, dt)
        gs, = torch.autograd.grad((ends * torch.from_numpy(g[:count].astype(np.float32)).cuda()).sum(), s)
        _, _, jac, ftle = adjoint.ftle(tape, s.detach(), F, dt)
        runs.append([v.detach().cpu().numpy()[:P] for v in (ends, valid, exit_cycle, gs, jac, ftle)])
        tape.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b, equal_nan=True)


# Segments of 26, 62 and 194 cycles: two, three and nine chunks of 24, restarted
# every 24 cycles and, the longest, every 48.
@pytest.mark.parametrize("L", [450, 2600, 26000])
def test_tape_segments_longer_than_the_scatter_keeps_positions_for(L):
    # An affine field has one Jacobian everywhere, so the FP32 path cannot sit
    # in another cell with another derivative. Each of the L steps adds about
    # 10 roundings of 6e-8: 2.7e-4 relative at 450.
    import torch
    tol = 6e-7 * L
    n, h, dt = ((8, 8, 8) if L < 1000 else (4, 4, 4)), (1.0,) * 3, 4.5 / L
    A = np.array([[0.05, 0.25, 0.0], [-0.25, 0.025, 0.125], [0.0, -0.125, -0.05]])
    c = np.asarray(n) / 2.0
    field = inputs.affine_field(n, (0, 0, 0), h, A, -A @ c)
    rng = np.random.default_rng(9)
    x0 = c + rng.uniform(-0.2, 0.2, size=(40, 3)) * n       # these stay in the block
    up = rng.standard_normal((40, 3))
    g = oracle.Grid.make(n, (0, 0, 0), h)
    st, lam, gF = oracle.vjp(g, lambda k: field, dt, x0.astype(np.float32).astype(np.float64), L, up,
                             want_field_grads=True)
    assert st.valid.all()
    tape = adjoint.Tape(n, (0, 0, 0), h, 40, L, 16)
    s = torch.from_numpy(x0.astype(np.float32)).cuda().requires_grad_(True)
    F = torch.from_numpy(np.repeat(np.asarray(field, dtype=np.float32)[None], L, axis=0)).cuda().requires_grad_(True)
    ends, valid, exit_cycle = adjoint.flow_map(s, F, tape, dt)
    gs, gf = torch.autograd.grad((ends * torch.from_numpy(up.astype(np.float32)).cuda()).sum(), (s, F))
    tape.close()
    assert np.array_equal(exit_cycle.cpu().numpy(), st.exit_cycle)
    assert np.max(np.abs(gs.cpu().numpy() - lam)) <= tol * np.max(np.abs(lam))
    gF = np.stack(gF)
    got = gf.cpu().numpy().reshape(gF.shape)
    assert np.max(np.abs(got - gF)) <= tol * np.max(np.abs(gF))


# Lattice fill: tiles of 512 entries and their remainder, searches that end
# within and beyond the first 16 points, on either side, axes one or two
# points long, and pointers that are not 16-byte aligned.
@pytest.mark.parametrize("S", [(1, 1, 1), (511, 1, 1), (8, 8, 8), (513, 1, 1), (2, 40, 21), (37, 34, 2), (64, 48, 5)])
@pytest.mark.parametrize("shift", [0, 1])
def test_lattice_fill_routes_match_oracle(S, shift):
    import torch
    rng = np.random.default_rng(int(np.prod(S)) + shift)
    P = int(np.prod(S))
    ends = rng.standard_normal((P, 3)).astype(np.float32)
    valid = (rng.random(P) > 0.1).astype(np.uint8) * rng.integers(1, 256, P).astype(np.uint8)
    v3 = valid.reshape(S[2], S[1], S[0])
    v3[:, :, S[0] // 4:S[0] // 4 + 17] = 0           # 17 and 34 points: beyond the first look
    v3[:, S[1] // 8:S[1] // 8 + 34, :] *= (rng.random((S[2], min(34, S[1] - S[1] // 8), S[0])) > 0.97)
    out_o, st_o = oracle.fill_lattice(S, ends.astype(np.float64), (valid != 0).astype(np.uint8))

    def dev(a):
        t = torch.empty(a.size + 4, dtype=torch.from_numpy(a).dtype, device="cuda")
        v = t[shift:shift + a.size].view(a.shape)
        v.copy_(torch.from_numpy(a))
        return v
    out = dev(np.zeros((P, 3), np.float32))
    st = dev(np.full(P, 9, np.uint8))
    bto.bto_fill_lattice(S, dev(ends), dev(valid), out, st)
    st_g, out_g = st.cpu().numpy(), out.cpu().numpy()
    assert np.array_equal(st_g, st_o)
    ok = st_o > 0
    if ok.any():
        # one product and one fused product and add of values below 5
        assert np.max(np.abs(out_g[ok] - out_o[ok])) < 5 * 3 * 2.0 ** -24
    assert np.all(np.isnan(out_g[~ok]))


# Delaunay fill: interiors of one point, tiles with a remainder, lattices two
# points thick (boundary only), and faces wider than a window of 25.
@pytest.mark.parametrize("S,frac", [((3, 3, 3), 0.1), ((9, 5, 3), 0.15), ((8, 4, 4), 0.2), ((17, 6, 5), 0.25),
                                    ((30, 28, 2), 0.3), ((33, 7, 4), 0.35)])
def test_delaunay_fill_tile_edges_match_oracle(S, frac):
    import torch
    rng = np.random.default_rng(int(np.prod(S)))
    P = int(np.prod(S))
    v = rng.random(P) >= frac
    X = oracle.lattice_coords(S, np.arange(P)).astype(np.float64)
    ends = np.where(v[:, None], X + 0.2 * np.sin(X[:, [1, 2, 0]]), np.nan).astype(np.float32)
    ref, st_o = oracle.fill_delaunay(S, ends.astype(np.float64), v)
    e = torch.from_numpy(ends).cuda()
    d = torch.from_numpy(v.astype(np.uint8)).cuda()
    out, st = torch.empty_like(e), torch.empty_like(d)
    bto.bto_fill_delaunay(S, e, d, out, st)
    assert np.array_equal(st.cpu().numpy(), st_o)
    filled = st_o == 2
    got = out.cpu().numpy()
    if filled.any():
        assert np.max(np.abs(got[filled] - ref[filled])) <= 2e-6 * np.abs(ref[filled]).max()
    assert np.array_equal(got[st_o == 1], ends[st_o == 1]) and np.all(np.isnan(got[st_o == 0]))
