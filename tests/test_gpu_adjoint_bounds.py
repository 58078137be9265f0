"""GPU: a backward call stays inside the block's nodes whatever the fields hold
when it runs.
"""
import numpy as np
import pytest

from paper_2004_02003_gb300 import adjoint, bto

pytestmark = pytest.mark.gpu

GUARD = 1 << 20      # floats on either side of the gradient fields


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    from paper_2004_02003_gb300 import build
    build.build()
    bto.load()


# The fields are written between forward and backward, as a simulation with a
# ring of field buffers may do: points that the forward never sampled, beyond
# each face, far out, and not a number. The gradient of a node outside the
# block would land in the guards around the gradient fields. Segments of one
# chunk and of more; the particle counts of the caller's order and the sorted.
@pytest.mark.parametrize("P,L", [(300, 30), (3000, 30), (300, 450)])
@pytest.mark.parametrize("velocity", [(-0.3, 0.0, 0.0), (0.0, -40.0, 0.0), (0.0, 3.0, 50.0), (-1e30, 1e30, 0.0),
                                      (float("inf"), float("-inf"), 0.0), (float("nan"), 1.0, -1.0)])
def test_backward_on_fields_written_since_the_forward(P, L, velocity):
    import torch
    n, h, dt = (16, 12, 10), (1.0, 1.0, 1.0), 0.5
    shape = (L, n[2] + 1, n[1] + 1, n[0] + 1, 3)
    fields = torch.zeros(shape, device="cuda")
    table = torch.tensor([f.data_ptr() for f in fields], dtype=torch.int64, device="cuda")
    rng = np.random.default_rng(P + L)
    seeds = torch.from_numpy((rng.uniform(0, 1, (P, 3)) * n).astype(np.float32)).cuda()
    ends, valid = torch.empty((P, 3), device="cuda"), torch.empty(P, dtype=torch.uint8, device="cuda")
    store = torch.full((2 * GUARD + fields.numel(),), 7.0, device="cuda")
    grad = store[GUARD:GUARD + fields.numel()].view(shape)
    gtable = torch.tensor([g.data_ptr() for g in grad], dtype=torch.int64, device="cuda")
    g_ends, g_seeds = torch.ones((P, 3), device="cuda"), torch.empty((P, 3), device="cuda")
    jac = torch.empty((P, 9), device="cuda")
    tape = adjoint.Tape(n, (0.0, 0.0, 0.0), h, P, L)

    def sweep():
        grad.zero_()
        bto.bto_tape_jacobian(tape.handle, jac)
        bto.bto_tape_backward(tape.handle, g_ends, g_seeds, gtable)
        torch.cuda.synchronize()
        return g_seeds.clone(), jac.clone(), grad.clone()

    bto.bto_tape_forward(tape.handle, seeds, table, dt, ends, valid, None)
    assert bool(valid.all())
    first = sweep()
    for k in range(3):
        fields[..., k] = velocity[k]
    sweep()
    assert bool((store[:GUARD] == 7.0).all()) and bool((store[GUARD + fields.numel():] == 7.0).all())
    # and the tape is as good as new: the first forward's gradients again
    fields.zero_()
    bto.bto_tape_forward(tape.handle, seeds, table, dt, ends, valid, None)
    for a, b in zip(first[:2], sweep()[:2]):
        assert torch.equal(a, b)
    # at rest every particle's weights add up to dt in each cycle and component
    assert torch.allclose(grad.double().sum(dim=(1, 2, 3)), torch.full((L, 3), dt * P, dtype=torch.float64,
                                                                       device="cuda"), rtol=1e-5)
    tape.close()
