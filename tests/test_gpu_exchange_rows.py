"""Exchange rows of every kind through the copy kernel, bit for bit (needs a GPU)."""
import numpy as np
import pytest

from oracle import redistribute as R
from paper_1804_09536_gb300 import inputs
from gpu_util import bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,grid", [((6, 9, 1), (2, 3)), ((4, 6, 3), (1, 3)), ((8, 16, 66), (2, 2)),   # rows of 1, 1 and 33
                                        ((3, 5, 4100), (3, 1)), ((2, 130, 257), (2, 4)), ((5, 3, 8192), (2, 1))])
def test_exchange_row_lengths(cuda_device, shape, grid):
    """Rows of one element, odd, longer than a task and split."""
    from paper_1804_09536_gb300.plan import Plan
    x = inputs.uniform_complex(shape, seed=5).numpy()
    p = Plan(shape, grid, device=cuda_device)
    stages = [R.scatter(x, grid, s) for s in range(3)]
    for v, w in ((2, 1), (1, 0), (0, 1), (1, 2)):
        got = p.redistribute(v, w, to_dev(stages[2 - v], cuda_device))
        assert np.array_equal(bits(got), stages[2 - w].view(np.uint8)), (v, w)


@pytest.mark.parametrize("shape,grid", [((5, 7, 33), (1, 3)), ((25, 5, 37), (2, 3)), ((9, 15, 27), (3, 3))])
@pytest.mark.parametrize("mode", ["unfused", "packed"])
def test_exchange_odd_stage(cuda_device, shape, grid, mode):
    """An odd number of elements: the second workspace buffer of the unfused and packed paths is
    only 8-byte aligned, whatever the parity of a copy task's own offsets."""
    from paper_1804_09536_gb300.plan import Plan
    p = Plan(shape, grid, device=cuda_device)
    x = to_dev(R.scatter(inputs.uniform_complex(shape, seed=6).numpy(), grid, 0), cuda_device)
    y = p.forward(x)
    assert np.array_equal(bits(p.forward(x, mode=mode)), bits(y))
    assert np.array_equal(bits(p.inverse(y.clone(), mode=mode)), bits(p.inverse(y.clone())))
