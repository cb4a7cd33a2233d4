"""Chained passes (programmatic dependent launches) of small plans give the bits of unchained ones
(needs a GPU).  Launch events turn chaining off, so the same plan runs both ways; the repeated
forward / inverse pairs on one set of buffers would show a pass that starts before its input is
complete or overwrites what the previous pass still reads."""
import numpy as np
import pytest
import torch

from gpu_util import bits

pytestmark = pytest.mark.gpu

CASES = [((32, 32, 32), (2, 2), "c2c"), ((60, 72, 100), (2, 2), "c2c"),       # largest carve-out
         ((64, 64, 128), (2, 2), "c2c"), ((65, 64, 128), (2, 3), "c2c"),      # 4 MiB, just above
         ((42, 127, 64), (3, 4), "c2c"),                                      # Bluestein between two lengths
         ((24, 512, 30), (2, 2), "c2c"), ((16, 17, 18, 19), (2, 3, 2), "c2c"),  # unchained passes in the chain
         ((128, 128, 256), (2, 4), "c2c"), ((96, 100, 128), (2, 4), "r2c"), ((64, 128, 240), (8,), "r2c")]


@pytest.mark.parametrize("shape,grid,kind", CASES)
@pytest.mark.parametrize("graphs", [True, False])
def test_chained_equals_unchained(cuda_device, shape, grid, kind, graphs):
    from paper_1804_09536_gb300.plan import Plan
    real = kind == "r2c"
    p = Plan(shape, grid, kind=kind, device=cuda_device, graphs=graphs)
    gen = torch.Generator(device="cpu").manual_seed(3)
    x = torch.randn(p.stage_elems(0, real), 1 if real else 2, generator=gen).to(cuda_device)
    x = x.reshape(-1) if real else torch.view_as_complex(x)

    def rounds(n, events):
        a, y = x.clone(), p.empty_stage(p.g)
        seen = []
        evs = {s: [torch.cuda.Event(enable_timing=True) for _ in range(p.num_launches(s) + 1)] for s in (-1, 1)}
        for _ in range(n):
            for sign, src, dst in ((-1, a, y), (1, y, a)):
                if events:
                    p.set_launch_events(evs[sign])
                (p.forward if sign < 0 else p.inverse)(src, out=dst, keep_input=not real)
                if not (real and sign > 0):  # a c2r backward leaves its input undefined
                    seen.append(dst.clone())
        p.set_launch_events([])
        torch.cuda.synchronize()
        return seen + [a]

    want, got = rounds(6, True), rounds(6, False)
    assert p.device_status() == 0
    for k, (w, g) in enumerate(zip(want, got)):
        assert np.array_equal(bits(w), bits(g)), k


@pytest.mark.parametrize("shape,grid", [((64, 64, 64), (2, 2)), ((96, 96, 96), (2, 2)), ((128, 128, 128), (2, 4)),
                                        ((256, 32, 256), (2, 2))])
def test_tma_tiles_of_small_plans(cuda_device, shape, grid):
    """The TMA-staged tiles that small plans run only when timed: the bits of a plan without TMA."""
    from paper_1804_09536_gb300.plan import Plan
    pt, pp = Plan(shape, grid, device=cuda_device), Plan(shape, grid, device=cuda_device, tma=False)
    gen = torch.Generator(device="cpu").manual_seed(4)
    x = torch.view_as_complex(torch.randn(pt.stage_elems(0), 2, generator=gen)).to(cuda_device)
    for sign in (-1, 1):
        assert any("_tma_" in n for n, _ in pt.launch_info(sign))
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(pt.num_launches(sign) + 1)]
        pt.set_launch_events(evs)
        got = (pt.forward if sign < 0 else pt.inverse)(x)
        pt.set_launch_events([])
        want = (pp.forward if sign < 0 else pp.inverse)(x.clone())
        torch.cuda.synchronize()
        assert np.array_equal(bits(got), bits(want))
    assert pt.device_status() == 0
