"""GPU: an interval's results depend on the fields it is given and on nothing
that an earlier call left in the context.
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


def _uniform(n, v):
    """Node field of a block of n cells: velocity v along x, on the device."""
    import torch
    f = torch.zeros((n[2] + 1, n[1] + 1, n[0] + 1, 3), dtype=torch.float32, device="cuda")
    f[..., 0] = v
    return f


# Autotune's trials run on fields that empty the block, as a caller may tune on
# others than the run's; then an interval in which nobody leaves, one in which
# the particles near a face leave (some of the groups lose a part, others
# nothing), and one at rest again. Row widths: whole runs of 32 seeds, and runs
# that end inside a group.
@pytest.mark.parametrize("n", [(64, 5, 4), (43, 7, 3)])
def test_intervals_after_autotune_on_other_fields(n):
    import torch
    L, dt, h = 4, 0.25, (1.0, 1.0, 1.0)
    out_all = _uniform(n, 8.0 * n[0])
    speeds = [0.0, 3.0, 0.0]
    tune = torch.tensor([out_all.data_ptr()] * L, dtype=torch.int64, device="cuda")
    got = []
    for tuned in (False, True):
        ctx = bto.Context(n, (0, 0, 0), h, 1, L)
        if tuned:
            ctx.autotune(tune, L, dt)
        res = []
        for v in speeds:
            f = _uniform(n, v)
            for _ in range(L):
                ctx.advect(f, dt)
            res.append({k: a.cpu().numpy() for k, a in ctx.end_interval(exits=True).items()})
        ctx.check()
        ctx.close()
        got.append(res)
    for v, want, have in zip(speeds, *got):
        assert (want["valid"] == 0).any() == (v > 0) and (want["valid"] == 1).any()
        for k in want:
            assert np.array_equal(want[k], have[k], equal_nan=True), (v, k)


# With ingest each launch holds one block: the launch shape follows the largest
# block while it is on, unless the caller has set one, and the results do not
# depend on it. The blocks hold seeds on either side of the lines (65,536 and
# 750,000), and the context enough for another shape without ingest.
@pytest.mark.parametrize("nb,n,shape", [(40, 26, (128, 1)), (12, 41, (128, 2)), (1, 91, (256, 4))])
def test_ingest_takes_the_launch_shape_of_its_blocks(nb, n, shape):
    import torch
    L, dt, h = 3, 0.4, (1.0, 1.0, 1.0)
    f = _uniform((n, n, n), 1.5)
    f[..., 1] = torch.linspace(-2, 2, n + 1, device="cuda")[:, None, None]
    table = torch.full((nb,), f.data_ptr(), dtype=torch.int64, device="cuda")
    ctx = bto.Context.batch([(n, n, n)] * nb, [(0.0, 0.0, 0.0)] * nb, [h] * nb, [1] * nb, L)
    plain = ctx.launch()
    got = []
    for mode in ("plain", "ingest", "plain", "set"):
        if mode == "set":
            ctx.set_launch(128, 4)
            bto.bto_set_ingest(ctx.handle, 1)
            assert ctx.launch()["particles_per_thread"] == 4
        else:
            bto.bto_set_ingest(ctx.handle, int(mode == "ingest"))
            now = ctx.launch()
            assert now == plain if mode == "plain" else (now["threads_per_cta"], now["particles_per_thread"]) == shape
        for _ in range(L):
            ctx.advect_batch(table, dt)
        got.append({k: v.cpu().numpy() for k, v in ctx.end_interval().items()})
    ctx.check()
    ctx.close()
    assert (got[0]["valid"] == 0).any() and (got[0]["valid"] == 1).any()
    for other in got[1:]:
        for k in other:
            assert np.array_equal(got[0][k], other[k]), k
