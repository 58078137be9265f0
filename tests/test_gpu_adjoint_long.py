"""GPU: field gradients of long intervals, whose segments the scatter takes in
chunks restarted from positions kept on the way, to a bound that does not grow
with the interval.

Every cycle's field is uniform and every position a multiple of 1/4, so that
positions are exact in FP32 and in the reference alike, the flow's Jacobian is
the identity, and a cycle's gradient has the closed form: each stage's trilinear
weights times its share of the step. A chunk restarted from a wrong position
lands in other cells.
"""
import numpy as np
import pytest

from paper_2004_02003_gb300 import adjoint, bto

pytestmark = pytest.mark.gpu

N = (9, 8, 7)        # cells


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    from paper_2004_02003_gb300 import build
    build.build()
    bto.load()


def walk(L, seed):
    """Steps of L cycles (cells) that keep every particle at [1/2, n - 1/2], and the displacement before each."""
    rng = np.random.default_rng(seed)
    step, at = np.empty((L, 3)), np.zeros((L + 1, 3))
    for a in range(3):
        room = N[a] / 2 - 1.0
        for c in range(L):
            v = rng.choice((-0.5, -0.25, 0.25, 0.5))
            step[c, a] = v if abs(at[c, a] + v) <= room else -v
            at[c + 1, a] = at[c, a] + step[c, a]
    return step, at[:-1]


def expected(x0, g, step, at):
    """Field gradients of sum(g . end) and the sums of their terms' magnitudes: [L, nodes, 3] each."""
    nn = np.asarray(N) + 1
    out = np.zeros((step.shape[0], int(nn.prod()), 3))
    mag = np.zeros_like(out)
    cycles = np.arange(step.shape[0])
    for p in range(x0.shape[0]):
        for at_step, share in ((0.0, 1 / 6), (0.5, 1 / 3), (0.5, 1 / 3), (1.0, 1 / 6)):
            x = x0[p] + at + at_step * step
            i = np.minimum(x.astype(np.int64), np.asarray(N) - 1)
            f = x - i
            for k in range(8):
                d = np.array([k & 1, k >> 1 & 1, k >> 2 & 1])
                w = np.where(d, f, 1.0 - f).prod(axis=1)
                node = (i + d) @ np.array([1, nn[0], nn[0] * nn[1]])
                t = share * w[:, None] * g[p]
                out[cycles, node] += t
                mag[cycles, node] += np.abs(t)
    return out, mag


# One chunk of 24 a segment; two; a segment of 62 restarted at every chunk
# (positions 24 apart); of 194, 48 apart, so that every second chunk starts
# between two kept positions.
@pytest.mark.parametrize("L", [30, 450, 2600, 26000])
def test_field_gradients_of_long_segments(L):
    import torch
    P, h, dt = 5, (1.0, 1.0, 1.0), 1.0
    step, at = walk(L, L)
    rng = np.random.default_rng(1)
    x0 = np.asarray(N) / 2 + rng.integers(-1, 2, size=(P, 3)) * 0.25
    g = rng.integers(-8, 9, size=(P, 3)) / 4.0
    fields = torch.empty((L, N[2] + 1, N[1] + 1, N[0] + 1, 3), device="cuda")
    fields[:] = torch.from_numpy(step.astype(np.float32)).cuda()[:, None, None, None, :]
    grad = torch.zeros_like(fields)

    def table(t):
        return torch.from_numpy(t.data_ptr() + np.arange(L) * t.stride(0) * 4).cuda()

    tape = adjoint.Tape(N, (0.0, 0.0, 0.0), h, P, L)
    seeds = torch.from_numpy(x0.astype(np.float32)).cuda()
    ends, valid = torch.empty((P, 3), device="cuda"), torch.empty(P, dtype=torch.uint8, device="cuda")
    g_ends, g_seeds = torch.from_numpy(g.astype(np.float32)).cuda(), torch.empty((P, 3), device="cuda")
    ft, gt = table(fields), table(grad)
    bto.bto_tape_forward(tape.handle, seeds, ft, dt, ends, valid, None)
    bto.bto_tape_backward(tape.handle, g_ends, g_seeds, gt)
    torch.cuda.synchronize()
    tape.close()
    assert bool(valid.all())
    assert np.array_equal(ends.cpu().numpy(), (x0 + at[-1] + step[-1]).astype(np.float32))
    assert np.array_equal(g_seeds.cpu().numpy(), g.astype(np.float32))
    # a term's weight and share are rounded at most six times and up to 20
    # terms of each particle are added: 32 roundings of 2^-24
    got = grad.cpu().numpy().reshape(L, -1, 3)
    for c0 in range(0, L, 10000):
        c = slice(c0, c0 + 10000)
        want, mag = expected(x0, g, step[c], at[c])
        assert np.all(np.abs(got[c] - want) <= 32 * 2.0 ** -24 * mag)
