"""Partial transforms of plans whose whole transform is unsupported (needs a GPU)."""
import numpy as np
import pytest

from oracle import dft, redistribute as R
from paper_1804_09536_gb300 import inputs
from gpu_util import RTOL_FP32, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,grid,kind", [((20, 200), (2,), "r2c"), ((8, 60, 200), (2,), "r2c"),
                                             ((20, 4099), (3,), "c2c"), ((64, 128, 4160), (2, 2), "c2c")])
def test_partial_beside_a_length_without_a_plan(cuda_device, shape, grid, kind):
    from paper_1804_09536_gb300 import TfftError
    from paper_1804_09536_gb300.plan import Plan
    p = Plan(shape, grid, kind=kind, device=cuda_device)
    cshape = shape[:-1] + (shape[-1] // 2 + 1,) if kind == "r2c" else shape
    x = inputs.uniform_complex(cshape, seed=9).numpy()
    d, g = len(shape), len(grid)
    for s in range(g + 1):
        b = R.scatter(x, grid, s)
        cut = [i if i < g - s else i + 1 for i in range(g)]
        for axis in set(range(d - 1)) - set(cut):
            for sign in (-1, 1):
                t = to_dev(b, cuda_device)
                p.partial(s, axis, sign, t)
                want = dft._transform_ranks(b.astype(np.complex128), cshape, grid, s, axis, sign)
                assert rel_l2(t.cpu().numpy(), want) <= RTOL_FP32, (s, axis, sign)
        if kind == "c2c" and d - 1 not in cut:
            with pytest.raises(TfftError):
                p.partial(s, d - 1, -1, to_dev(b, cuda_device))
