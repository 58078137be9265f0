"""GPU: the Delaunay fill's routes by lattice size, shape and alignment give the
same bytes. Above four tiles of 8 x 2 x 2 entries for each CTA in flight the
tiles with missing entries are listed in the output's plane z = 0; a call whose
output overlaps its input takes every tile instead, as small lattices do.
"""
import numpy as np
import pytest

from paper_2004_02003_gb300 import bto

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    from paper_2004_02003_gb300 import build
    build.build()
    bto.load()


def _lattice(S, holes, seed):
    """Basis flows of lattice S (z, y, x order) and valid flags by a pattern of holes."""
    rng = np.random.default_rng(seed)
    v = np.ones(S[::-1], dtype=np.uint8)
    if holes == "sparse":
        v[rng.random(v.shape) < 0.002] = 0
    elif holes == "slabs":
        v[S[2] // 2 - 1:S[2] // 2 + 2] = 0
        v[:, S[1] // 3] = 0
        v[:, :, :2] = 0
        v[rng.random(v.shape) < 0.001] = 0
    elif holes == "all":
        v[:] = 0
    ends = rng.standard_normal((int(np.prod(S)), 3)).astype(np.float32)
    ends[v.reshape(-1) == 0] = np.nan
    return ends, v.reshape(-1)


# Lattices listed (more than 2,432 tiles on 152 SMs): sizes that divide into
# groups of four tiles and that leave ragged ones, thin ones, and deep ones
# whose groups take several tiles along z; and one just below.
@pytest.mark.parametrize("S", [(64, 64, 48), (67, 45, 53), (200, 131, 3), (5, 40, 1200), (9, 3, 9001), (96, 101, 16)])
@pytest.mark.parametrize("holes", ["none", "sparse", "slabs", "all"])
def test_listed_tiles_equal_every_tile(S, holes):
    import torch
    ends, valid = _lattice(S, holes, S[0])
    P = int(np.prod(S))
    v = torch.from_numpy(valid).cuda()
    want = torch.from_numpy(ends).cuda()                  # in place: every tile has a CTA
    st_want = torch.full((P,), 9, dtype=torch.uint8, device="cuda")
    bto.bto_fill_delaunay(S, want, v, want, st_want)
    want, st_want = want.cpu().numpy(), st_want.cpu().numpy()
    ok = valid != 0
    assert np.array_equal(want[ok], ends[ok]) and np.all(st_want[ok] == 1) and np.all(st_want[~ok] != 1)
    assert np.all(np.isnan(want[st_want == 0])) and not np.isnan(want[st_want == 2]).any()
    if holes == "sparse":
        assert (st_want == 2).sum() > 0.9 * (~ok).sum()
    for shift, status in ((0, True), (0, False), (1, True), (3, True)):
        src = torch.full((3 * P + 8,), 5.0, device="cuda")[shift:shift + 3 * P]
        src.copy_(torch.from_numpy(ends).cuda().view(-1))
        flags = torch.full((P + 8,), 1, dtype=torch.uint8, device="cuda")[shift:shift + P]
        flags.copy_(v)
        store = torch.full((3 * P + 64,), 5.0, device="cuda")
        out = store[shift:shift + 3 * P]
        st_store = torch.full((P + 64,), 9, dtype=torch.uint8, device="cuda")
        st = st_store[shift:shift + P]
        bto.bto_fill_delaunay(S, src, flags, out, st if status else None)
        assert np.array_equal(out.cpu().numpy().reshape(-1, 3).view(np.int32), want.view(np.int32)), (shift, status)
        assert bool((store[:shift] == 5.0).all()) and bool((store[shift + 3 * P:] == 5.0).all())
        if status:
            assert np.array_equal(st.cpu().numpy(), st_want)
        assert bool((st_store[:shift] == 9).all()) and bool((st_store[shift + P:] == 9).all())


# A lattice one point thick has no tetrahedra: the copy finishes it. Whole
# tiles of 512 entries and a remainder, aligned and not.
@pytest.mark.parametrize("S", [(512, 3, 1), (1, 77, 45), (41, 1, 25), (1, 1, 1)])
@pytest.mark.parametrize("shift", [0, 1])
def test_flat_lattice(S, shift):
    import torch
    ends, valid = _lattice(S, "sparse", 3)
    P = int(np.prod(S))
    valid[::5] = 0
    src = torch.empty(3 * P + 8, device="cuda")[shift:shift + 3 * P]
    src.copy_(torch.from_numpy(ends).view(-1))
    v = torch.from_numpy(valid).cuda()
    out, st = torch.full((P, 3), 5.0, device="cuda"), torch.full((P,), 9, dtype=torch.uint8, device="cuda")
    bto.bto_fill_delaunay(S, src, v, out, st)
    out, st = out.cpu().numpy(), st.cpu().numpy()
    ok = valid != 0
    assert np.array_equal(out[ok], ends[ok]) and np.isnan(out[~ok]).all()
    assert np.array_equal(st, valid)


# Captured into a CUDA graph, the fill's launches and the list's clearing replay
# on whatever the buffers then hold.
@pytest.mark.parametrize("S", [(67, 45, 53), (33, 31, 29), (40, 1, 25)])
def test_fill_replays_from_a_captured_graph(S):
    import torch
    P = int(np.prod(S))
    ends, valid = torch.zeros((P, 3), device="cuda"), torch.ones(P, dtype=torch.uint8, device="cuda")
    out, st = torch.empty_like(ends), torch.empty_like(valid)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bto.bto_fill_delaunay(S, ends, valid, out, st)
    for holes in ("slabs", "none", "sparse"):
        e, v = _lattice(S, holes, 5)
        ends.copy_(torch.from_numpy(e))
        valid.copy_(torch.from_numpy(v))
        graph.replay()
        want, st_want = torch.empty_like(ends), torch.empty_like(valid)
        torch.cuda.synchronize()
        bto.bto_fill_delaunay(S, ends, valid, want, st_want)
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int32), want.view(torch.int32)) and torch.equal(st, st_want)
