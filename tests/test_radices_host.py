"""The butterflies of tfft_common.cuh against the exact DFT, and the lengths whose plans changed
route when the composed radices came in (CPU only)."""
import ctypes
import math
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1804_09536_gb300", "csrc")
RADICES = [2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16, 18, 20, 21, 24, 25, 27, 28, 30, 32]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists("/usr/local/cuda/include/vector_types.h"):
        pytest.skip("no host C++ compiler or CUDA headers")
    out = str(tmp_path_factory.mktemp("dft") / "libdft.so")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", "/usr/local/cuda/include",
                    os.path.join(HERE, "native", "dft_radices.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("radix", RADICES)
def test_radix_matches_dft(lib, radix):
    rng = np.random.default_rng(radix)
    x = (rng.standard_normal(radix) + 1j * rng.standard_normal(radix)).astype(np.complex64)
    got = x.copy()
    assert lib.dft_radix(radix, got.ctypes.data_as(ctypes.c_void_p)) == 0
    k = np.arange(radix)
    want = np.exp(-2j * np.pi * (np.outer(k, k) % radix) / radix) @ x.astype(np.complex128)
    # a few roundings of 2^-24 per level of the butterfly
    assert np.linalg.norm(got - want) <= 2.0 ** -24 * (2 + 2 * math.log2(radix)) * np.linalg.norm(want)


def _rows(name):
    text = open(os.path.join(CSRC, "tfft_spec_table.h")).read()
    body = text[text.index("#define " + name):].split("\n\n")[0]
    return [tuple(int(v) for v in m.split(",")) for m in re.findall(r"X\(([\d, ]+)\)", body)]


@pytest.mark.parametrize("name", ["TFFT_CONTIG_LINES", "TFFT_STRIDED_LINES"])
def test_table_rows(name):
    """Radices multiply to the length; threads, registers and shared memory within a CTA's limits."""
    rows = _rows(name)
    assert len({r[0] for r in rows}) == len(rows) >= 120
    for L, T, W, ctas, *rad in rows:
        assert math.prod(rad) == L and set(rad) <= set(RADICES)
        assert 32 < T * W <= 1024 and ctas >= 1
        held = max(-(-(L // r) // T) * r for r in rad)
        assert held <= 32
        smem = (W * (L + L // 2) * 8) if name == "TFFT_CONTIG_LINES" else L * W * 8 + 16 * L + 256
        assert smem <= 227 * 1024


def test_routes_that_stay():
    """Lengths refused before are refused; a prime whose N - 1 factors takes Rader's strided pass."""
    from paper_1804_09536_gb300 import TfftError
    from paper_1804_09536_gb300.plan import Plan
    for shape, kind in [((2058, 8), "c2c"), ((4097, 8), "c2c"), ((16, 200), "r2c"), ((16, 180), "r2c"), ((16, 84), "r2c")]:
        p = Plan(shape, (2,), kind=kind, bind=False)
        with pytest.raises(TfftError):
            p.num_launches(-1)
    names = [n for n, _ in Plan((42, 127, 256), (3, 4), bind=False).launch_info(-1)]
    assert names == ["fft_contig_L256", "fft_strided_rader_L127", "fft_strided_L42"]
