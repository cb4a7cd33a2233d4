"""GPU parity of the Bluestein and Rader passes (needs a GPU): the largest and the smallest line
length of every compiled convolution length, and every prime with a Rader pass, contiguous and strided, on uneven
blocks with partial tiles."""
import os
import re

import numpy as np
import pytest

from oracle import redistribute as R
from paper_1804_09536_gb300 import inputs
from gpu_util import RTOL_FP32, bits, rel_l2, to_dev
from test_radices_host import CSRC

pytestmark = pytest.mark.gpu


def _lengths():
    """(N, M) just inside both ends of every convolution length's range, N prime-like (not 7-smooth)."""
    text = open(os.path.join(CSRC, "tfft_blue.cuh")).read()
    body = text[text.index("#define TFFT_BLUE_STRIDED"):].split("\n\n")[0]
    ms = sorted(int(m) for m in re.findall(r"X\((\d+),", body))

    def smooth(n):
        for f in (2, 3, 5, 7):
            while n % f == 0:
                n //= f
        return n == 1

    out = []
    for lo, m in zip([16] + ms, ms):
        ns = [n for n in range(lo // 2 + 1, (m + 1) // 2 + 1) if not smooth(n)]
        out += sorted({ns[0], ns[-1]}) if ns else []
    return out


def _rader():
    text = open(os.path.join(CSRC, "tfft_blue.cuh")).read()
    body = text[text.index("#define TFFT_RADER_STRIDED"):].split("\n\n")[0]
    return [int(m) + 1 for m in re.findall(r"X\((\d+),", body)]


LENGTHS = sorted(set(_lengths() + _rader()))


@pytest.mark.parametrize("N", LENGTHS)
def test_bluestein_lengths(cuda_device, N):
    from paper_1804_09536_gb300.plan import Plan
    for full, grid in (((N, 5, 19), (2, 3)), ((3, N, 19), (3, 1)), ((5, 7, N), (2, 3))):
        x = inputs.uniform_complex(full, seed=N).numpy()
        b0 = R.scatter(x, grid, 0)
        p = Plan(full, grid, device=cuda_device)
        assert any(n.endswith((f"bluestein_L{N}", f"rader_L{N}")) for n, _ in p.launch_info(-1))
        y = p.forward(to_dev(b0, cuda_device))
        yu = p.forward(to_dev(b0, cuda_device), mode="unfused")
        back = p.inverse(y.clone())
        want = R.scatter(np.fft.fftn(x.astype(np.complex128)) / x.size, grid, 2)
        assert rel_l2(y.cpu().numpy(), want) <= RTOL_FP32, full
        assert rel_l2(back.cpu().numpy(), b0) <= RTOL_FP32, full
        assert np.array_equal(bits(y), bits(yu)), full
