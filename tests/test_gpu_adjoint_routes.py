"""GPU: a tape's results by the routes that its forward takes by the numbers of
cycles and particles.
"""
import numpy as np
import pytest

from paper_2004_02003_gb300 import adjoint, bto, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    from paper_2004_02003_gb300 import build
    build.build()
    bto.load()


def _tape(n, h, fields, seeds, dt):
    """Ends, valid, exit cycles, seed gradients and field gradients of a loss that weighs the first 300 particles."""
    import torch
    s, F = seeds.clone().requires_grad_(True), fields.clone().requires_grad_(True)
    tape = adjoint.Tape(n, (0.0, 0.0, 0.0), h, seeds.shape[0], fields.shape[0])
    ends, valid, exit_cycle = adjoint.flow_map(s, F, tape, dt)
    w = torch.zeros_like(ends)
    w[:300] = torch.linspace(-1.0, 2.0, 900, device="cuda").view(300, 3)
    gs, gF = torch.autograd.grad((ends * w).sum(), (s, F))
    torch.cuda.synchronize()
    tape.close()
    return [v[:300].detach().cpu().numpy() for v in (ends, valid, exit_cycle, gs)] + [gF.cpu().numpy()]


# Around the counts from which on a forward sorts its particles by cell: none
# in one or two cycles, 400,000 particle-cycles below ten, 2,048 particles from
# ten on. A particle's results do not depend on the others, so 300 particles
# alone, in the caller's order, give the same bits. Field gradients are sums
# over atomics in any order: of at most 300 x 4 terms a node and component,
# each of both sides within 1,200 2^-24 of the sum of their magnitudes, which
# the node sums of |w| dt bound.
@pytest.mark.parametrize("L,P", [(1, 3000), (2, 3000), (3, 133333), (3, 133334), (9, 44444), (9, 44445), (10, 2047),
                                 (10, 2048)])
def test_results_do_not_depend_on_the_sort(L, P):
    import torch
    n, dt = (24, 20, 17), 0.03
    h = (1.0 / max(n),) * 3
    modes = inputs.fourier_modes(5, m=10, kmax=4.0)
    fields = torch.stack([torch.from_numpy(np.ascontiguousarray(inputs.fourier_field(modes, n, (0.0, 0.0, 0.0), h, c),
                                                                dtype=np.float32)).cuda() for c in range(L)])
    rng = np.random.default_rng(11)
    x = rng.uniform(-0.02, 1.02, size=(P, 3)) * np.asarray(n) * np.asarray(h)     # some start outside
    seeds = torch.from_numpy(x.astype(np.float32)).cuda()
    want, got = _tape(n, h, fields, seeds[:300], dt), _tape(n, h, fields, seeds, dt)
    for a, b in zip(want[:4], got[:4]):
        assert np.array_equal(a, b)
    tol = 2 * 1200 * 2.0 ** -24 * np.abs(want[4]).max() * 4
    assert np.abs(want[4]).max() > 0 and np.abs(want[4] - got[4]).max() <= tol
