"""Bounds-checked build of libbto (BTO_CHECK_BOUNDS) on the calls that take all
cycles in one launch, the tape and the listed Delaunay fill: no failed check,
clear error words, and the product build's outputs. The checked calls run in a
child process.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def scenarios():
    """Whole-interval calls with one lane and with four per particle, F3 and F4, tapes of one chunk a segment and of
    more with the field gradients, a Delaunay fill whose tiles are listed and a flat one."""
    import torch
    from paper_2004_02003_gb300 import adjoint, bto, inputs
    torch.cuda.set_device(0)
    out = {}

    def fields(n, h, L, comps=3):
        modes = inputs.fourier_modes(7, m=12, kmax=5.0)
        f = [inputs.fourier_field(modes, n, (0, 0, 0), h, c) for c in range(L)]
        if comps == 4:
            f = [np.concatenate([a, np.zeros(a.shape[:-1] + (1,), a.dtype)], -1) for a in f]
        return torch.from_numpy(np.ascontiguousarray(np.stack(f), dtype=np.float32)).cuda()

    def table(f):
        return torch.tensor([v.data_ptr() for v in f], dtype=torch.int64, device="cuda")

    for n, comps, tag in (((38, 28, 16), 3, "quad3_"), ((23, 9, 31), 4, "quad4_"), ((50, 41, 30), 3, "lane3_"),
                          ((50, 41, 30), 4, "lane4_")):
        h, L = (1.0 / max(n),) * 3, 9
        f = fields(n, h, L, comps)
        ctx = bto.Context(n, (0, 0, 0), h, 1, L)
        if comps == 4:
            ctx.set_layout(bto.BTO_FIELD_F4_AOS)
        ctx.interval_graph(table(f), 0.03)
        o = ctx.end_interval(exits=True)
        ctx.check()
        out.update({tag + k: v.cpu().numpy() for k, v in o.items()})
        ctx.close()
    for P, L, tag in ((700, 30, "tape_quad_"), (30000, 30, "tape_lane_"), (500, 450, "tape_long_")):
        n = (24, 20, 17)
        h = (1.0 / max(n),) * 3
        f = fields(n, h, L)
        rng = np.random.default_rng(L)
        seeds = torch.from_numpy((rng.uniform(-0.02, 1.02, (P, 3)) * np.asarray(n) * h).astype(np.float32)).cuda()
        tape = adjoint.Tape(n, (0, 0, 0), h, P, L)
        ends, valid, jac, _ = adjoint.ftle(tape, seeds, f, 0.01)
        s, F = seeds.requires_grad_(True), f.requires_grad_(True)
        e2, v2, x2 = adjoint.flow_map(s, F, tape, 0.01)
        gs, gF = torch.autograd.grad((e2 ** 2).sum(), (s, F))
        for k, v in (("ends", ends), ("valid", valid), ("jac", jac), ("exit", x2), ("gs", gs), ("gF_", gF)):
            out[tag + k] = v.detach().cpu().numpy()
        tape.close()
    for S, tag in (((64, 64, 48), "listed_"), ((41, 29, 1), "flat_")):
        rng = np.random.default_rng(S[0])
        P = int(np.prod(S))
        valid = (rng.random(S[::-1]) > 0.01).astype(np.uint8)
        valid[:, S[1] // 2 - 1:S[1] // 2 + 2] = 0
        ends = torch.from_numpy(rng.standard_normal((P, 3)).astype(np.float32)).cuda()
        v = torch.from_numpy(valid.reshape(-1)).cuda()
        filled, status = torch.empty_like(ends), torch.empty_like(v)
        bto.bto_fill_delaunay(S, ends, v, filled, status)
        out[tag + "filled"], out[tag + "status"] = filled.cpu().numpy(), status.cpu().numpy()
    torch.cuda.synchronize()
    return out


@pytest.mark.gpu
def test_bounds_checked_routes_count_nothing_and_match_product(cuda_device, tmp_path):
    from paper_2004_02003_gb300 import bto, build
    build.build()
    check_lib = build.build(check_bounds=True)
    dst = str(tmp_path / "checked.npz")
    r = subprocess.run([sys.executable, os.path.abspath(__file__), dst], env=dict(os.environ, BTO_LIBRARY=check_lib),
                       cwd=ROOT, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=600)
    assert r.returncode == 0, r.stdout.decode(errors="replace")[-3000:]
    bto.load()
    assert not bto.bto_check_bounds_build()
    want, got = scenarios(), np.load(dst)
    assert set(got.files) == set(want)
    for k in want:
        if k.endswith("gF_"):
            # sums by atomics in any order: a few hundred terms a node at most
            assert np.abs(got[k] - want[k]).max() <= 500 * 2.0 ** -24 * np.abs(want[k]).max() * 8, k
        else:
            assert np.array_equal(got[k], want[k], equal_nan=True), k


# The checks of the tape's kernels have a counter of their own, which the
# build's count includes.
def test_the_count_includes_every_translation_unit():
    csrc = os.path.join(ROOT, "paper_2004_02003_gb300", "csrc")
    api = open(os.path.join(csrc, "bto_api.cu")).read()
    for name in sorted(os.listdir(csrc)):
        text = open(os.path.join(csrc, name)).read()
        if name.endswith(".cu") and ("BTO_IN_BOUNDS(" in text or "bto_device.cuh" in text) and "noalloc" not in name:
            unit = "bounds_failures_" + name[len("bto_"):-len(".cu")]
            assert f"BTO_BOUNDS_ACCESSOR({unit})" in text, name
            assert f"bto::{unit}(" in api, name


if __name__ == "__main__":
    from paper_2004_02003_gb300 import bto
    bto.load()
    assert bto.bto_check_bounds_build(), "BTO_LIBRARY is not the bounds-checked build"
    bto.bto_bounds_failures(reset=True)
    res = scenarios()
    fails = bto.bto_bounds_failures()
    assert fails == 0, f"{fails} bounds checks failed"
    np.savez(sys.argv[1], **res)
