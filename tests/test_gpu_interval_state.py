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
