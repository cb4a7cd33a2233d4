"""GPU parity of the gathering passes over the number of parts (needs a GPU): one round of placing
lanes, two, the most a CTA holds, and more (the row-table pass), with empty and uneven parts."""
import numpy as np
import pytest

from oracle import redistribute as R
from paper_1804_09536_gb300 import inputs
from gpu_util import RTOL_FP32, bits, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,grid", [((70, 256, 24), (32,)), ((70, 256, 17), (40,)), ((70, 256, 24), (64,)),
                                        ((90, 256, 24), (80,)), ((20, 400, 33), (24,)),   # empty parts of axis 0
                                        ((40, 128, 130), (5, 7)), ((12, 11, 128, 60), (2, 3, 4))])
def test_parts(cuda_device, shape, grid):
    from paper_1804_09536_gb300.plan import Plan
    g = len(grid)
    x = inputs.uniform_complex(shape, seed=len(shape)).numpy()
    b0 = R.scatter(x, grid, 0)
    p = Plan(shape, grid, device=cuda_device, tma=False)
    y = p.forward(to_dev(b0, cuda_device))
    yu = p.forward(to_dev(b0, cuda_device), mode="unfused")
    back = p.inverse(y.clone())
    want = R.scatter(np.fft.fftn(x.astype(np.complex128)) / x.size, grid, g)
    assert rel_l2(y.cpu().numpy(), want) <= RTOL_FP32
    assert rel_l2(back.cpu().numpy(), b0) <= RTOL_FP32
    assert np.array_equal(bits(y), bits(yu))


@pytest.mark.parametrize("shape,grid", [((512, 512, 32), (1, 2)), ((512, 512, 32), (1, 3)),   # three stages
                                        ((400, 400, 40), (3, 2)), ((384, 384, 48), (1, 3))])
def test_column_blocks(cuda_device, shape, grid):
    """Whole and partial column blocks of plans too large to chain their passes."""
    from paper_1804_09536_gb300.plan import Plan
    x = inputs.uniform_complex(shape, seed=len(shape)).numpy()
    b0 = R.scatter(x, grid, 0)
    p = Plan(shape, grid, device=cuda_device, tma=False)
    y = p.forward(to_dev(b0, cuda_device))
    assert rel_l2(y.cpu().numpy(), R.scatter(np.fft.fftn(x.astype(np.complex128)) / x.size, grid, len(grid))) <= RTOL_FP32
    assert np.array_equal(bits(y), bits(p.forward(to_dev(b0, cuda_device), mode="unfused")))
    assert rel_l2(p.inverse(y).cpu().numpy(), b0) <= RTOL_FP32


@pytest.mark.parametrize("L", [120, 224, 324, 441, 490, 784, 800, 864, 875, 900, 980, 1008])
def test_row_tables_and_gathering_agree(cuda_device, L):
    """Rows that gather only in chained calls: a call with launch events is not chained and runs row tables."""
    import torch
    from paper_1804_09536_gb300.plan import Plan
    for shape, grid in (((5, L, 64), (3, 2)), ((4, L, 35), (1, 3))):
        x = inputs.uniform_complex(shape, seed=L).numpy()
        p = Plan(shape, grid, device=cuda_device, tma=False)
        for sign in (-1, 1):
            b = to_dev(R.scatter(x, grid, 0 if sign < 0 else 2), cuda_device)
            want = (p.forward if sign < 0 else p.inverse)(b.clone())
            events = [torch.cuda.Event(enable_timing=True) for _ in range(p.num_launches(sign) + 1)]
            p.set_launch_events(events)
            got = (p.forward if sign < 0 else p.inverse)(b)
            p.set_launch_events([])
            f = np.fft.fftn(x.astype(np.complex128)) / x.size if sign < 0 else np.fft.ifftn(x.astype(np.complex128)) * x.size
            assert rel_l2(got.cpu().numpy(), R.scatter(f, grid, 2 if sign < 0 else 0)) <= RTOL_FP32, (shape, sign)
            assert np.array_equal(bits(got), bits(want)), (shape, sign)
