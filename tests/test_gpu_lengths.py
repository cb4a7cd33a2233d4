"""GPU parity of every compiled line length (needs a GPU): the length as a contiguous and as a
strided axis, on uneven blocks, with partial tiles at the edges of columns and of line groups."""
import numpy as np
import pytest

from oracle import redistribute as R
from paper_1804_09536_gb300 import inputs
from gpu_util import RTOL_FP32, bits, rel_l2, to_dev
from test_radices_host import _rows

pytestmark = pytest.mark.gpu

LENGTHS = sorted({r[0] for r in _rows("TFFT_CONTIG_LINES")} | {r[0] for r in _rows("TFFT_STRIDED_LINES")})


@pytest.mark.parametrize("shape,grid", [((5, 37), (2, 3)), ((3, 33), (3, 1))])
@pytest.mark.parametrize("part", range(4))
def test_every_length(cuda_device, shape, grid, part):
    from paper_1804_09536_gb300.plan import Plan
    for L in LENGTHS[part::4]:
        for full in ((L,) + shape, (shape[0], L, shape[1]), shape + (L,)):
            x = inputs.uniform_complex(full, seed=L).numpy()
            b0 = R.scatter(x, grid, 0)
            p = Plan(full, grid, device=cuda_device)
            y = p.forward(to_dev(b0, cuda_device))
            yu = p.forward(to_dev(b0, cuda_device), mode="unfused")
            back = p.inverse(y.clone())
            want = R.scatter(np.fft.fftn(x.astype(np.complex128)) / x.size, grid, 2)
            assert rel_l2(y.cpu().numpy(), want) <= RTOL_FP32, full
            assert rel_l2(back.cpu().numpy(), b0) <= RTOL_FP32, full
            assert np.array_equal(bits(y), bits(yu)), full
            assert p.device_status() == 0
