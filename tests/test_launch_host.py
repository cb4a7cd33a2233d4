"""What the library launches, on a CUDA runtime of host memory (CPU only).

tests/native/fake_cuda.cpp, linked with the library's own objects in place of cudart, runs plans and
calls as they are and records each launch, so that the tables a kernel would read can be checked
against the state buffer they have to lie in.
"""
import ctypes
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1804_09536_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1804_09536_gb300 import _lib, build
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists("/usr/local/cuda/include/cuda_runtime.h"):
        pytest.skip("no host C++ compiler or CUDA headers")
    build.build()
    d = tmp_path_factory.mktemp("fake")
    out, script = str(d / "libtfft_fake.so"), d / "exports.map"
    script.write_text("{ global: tfft_*; fake_*; local: *; };")  # the fake runtime serves these objects alone
    objs = [os.path.join(build.BUILD, u[1]) for u in build._units()]
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", "/usr/local/cuda/include",
                    os.path.join(HERE, "native", "fake_cuda.cpp"), *objs, f"-Wl,--version-script={script}", "-Wl,-z,defs",
                    "-o", out], check=True)
    so = ctypes.CDLL(out)
    for name, args in _lib.SIGNATURES.items():
        fn = getattr(so, name)
        fn.argtypes, fn.restype = args, _lib._RESTYPE.get(name, ctypes.c_int)
    yield so
    os.remove(out)


def _aligned(nbytes):
    raw = np.zeros(nbytes + 256, np.uint8)
    off = -raw.ctypes.data % 256
    return raw[off:off + nbytes]


class Fake:
    """A plan bound to host memory of exactly the state's size."""

    def __init__(self, lib, shape, grid, kind="c2c", precision=0, flags=0):
        self.lib, self.shape, self.grid, self.h = lib, shape, grid, ctypes.c_void_p()
        assert lib.tfft_plan_create(ctypes.byref(self.h), len(shape), (ctypes.c_int64 * len(shape))(*shape), len(grid),
                                    (ctypes.c_int * len(grid))(*grid), int(kind == "r2c"), precision, flags) == 0
        nb = ctypes.c_size_t()
        assert lib.tfft_plan_state_bytes(self.h, ctypes.byref(nb)) == 0
        self.state = _aligned(nb.value)
        assert lib.tfft_plan_bind(self.h, self.state.ctypes.data, nb.value, None) == 0
        (twiddles,) = self.launches()  # one launch makes every twiddle table, one per grid row
        assert "k_twiddles" in twiddles[0]
        self.tables = twiddles[2]

    def __del__(self):
        self.lib.tfft_plan_destroy(self.h)

    def launches(self):
        """(kernel, grid x, grid y, threads, table address, number of column blocks, merged blocks) since the last call."""
        buf = ctypes.create_string_buffer(1 << 16)
        assert self.lib.fake_launches(buf, len(buf)) < len(buf)
        rows = [r.split("|", 6) for r in buf.value.decode().splitlines()]
        return [(r[6], *map(int, r[:6])) for r in rows]

    def execute(self, sign=-1, events=False):
        """The launches of one call on distinct buffers (no kernel runs)."""
        n, nb = ctypes.c_int(), ctypes.c_size_t()
        assert self.lib.tfft_plan_num_launches(self.h, sign, 0, ctypes.byref(n)) == 0
        ev = (ctypes.c_void_p * (n.value + 1))(*[256] * (n.value + 1))
        assert self.lib.tfft_plan_set_launch_events(self.h, ev, n.value + 1 if events else 0) == 0
        assert self.lib.tfft_plan_workspace_bytes(self.h, 0, 1, ctypes.byref(nb)) == 0
        at = 1 << 40  # addresses only
        assert self.lib.tfft_execute(self.h, sign, 0, at, 2 * at, 3 * at, nb.value, None) == 0
        return self.launches()

    def names(self, sign=-1):
        n, b = ctypes.c_int(), ctypes.c_int64()
        assert self.lib.tfft_plan_num_launches(self.h, sign, 0, ctypes.byref(n)) == 0
        out = []
        for k in range(n.value):
            buf = ctypes.create_string_buffer(64)
            assert self.lib.tfft_plan_launch_info(self.h, sign, 0, k, buf, 64, ctypes.byref(b)) == 0
            out.append(buf.value.decode())
        return out

    def column_blocks(self, launch):
        """The column blocks a strided launch reads, which have to lie in the state; None where it reads none."""
        kernel, _, _, _, addr, n, _ = launch
        if "strided" not in kernel or "k_strided_merged" in kernel or "RankGroupTiles" in kernel:
            return None
        lo = self.state.ctypes.data
        assert lo <= addr and addr + 8 * n <= lo + self.state.size, f"{kernel}: column blocks outside the state"
        return self.state[addr - lo:addr - lo + 8 * n].view(np.int32).reshape(-1, 2)


@pytest.mark.parametrize("shape,grid,kind", [((60, 200), (2,), "r2c"), ((20, 200), (2,), "r2c"), ((8, 60, 200), (2,), "r2c"),
                                             ((22, 18, 200), (2, 2), "r2c"), ((20, 4099), (2,), "c2c"),
                                             ((20, 4099, 18), (3, 2), "c2c"), ((64, 128, 4160), (2, 2), "c2c"),
                                             ((96, 64, 4160), (2,), "c2c"), ((18, 4099, 20, 22), (2, 2, 2), "c2c")])
def test_partial_of_a_plan_that_does_not_transform(lib, shape, grid, kind):
    """A length without a plan stops the whole transform, not the partial ones along the other axes."""
    p = Fake(lib, shape, grid, kind)
    n = ctypes.c_int()
    assert lib.tfft_plan_num_launches(p.h, -1, 0, ctypes.byref(n)) == 2
    _partials(lib, p, shape, grid, kind)


@pytest.mark.parametrize("shape,grid,kind,precision", [((64, 96, 64), (2, 2), "c2c", 0), ((20, 127, 33), (3, 2), "c2c", 0),
                                                       ((512, 256, 64), (2,), "c2c", 1), ((256, 512, 128), (2, 2), "c2c", 1),
                                                       ((60, 64, 128), (2, 2), "r2c", 0), ((20, 96, 18, 22), (2, 2), "c2c", 0),
                                                       ((384, 30, 17), (), "c2c", 0), ((18, 200), (3,), "c2c", 0)])
def test_partial_of_a_plan(lib, shape, grid, kind, precision):
    _partials(lib, Fake(lib, shape, grid, kind, precision), shape, grid, kind)


def _partials(lib, p, shape, grid, kind):
    """Every partial transform along a strided axis reads column blocks of the state: whole columns,
    each once."""
    d, g = len(shape), len(grid)
    columns = shape[-1] // 2 + 1 if kind == "r2c" else shape[-1]
    x = _aligned(256)  # no kernel runs
    ran = 0
    for stage in range(g + 1):
        cut = [i if i < g - stage else i + 1 for i in range(g)]
        for axis in range(d - 1):
            for sign in (-1, 1):
                rc = lib.tfft_partial(p.h, stage, axis, sign, x.ctypes.data, None)
                launched = p.launches()
                if axis in cut or shape[axis] == 4099:
                    assert rc != 0 and not launched
                    continue
                assert rc == 0 and len(launched) == 1
                ran += 1
                blocks = p.column_blocks(launched[0])
                if blocks is not None:
                    at = 0
                    for c, w in blocks:
                        assert c == at and w > 0
                        at += w
                    assert at == columns
    assert ran > 0


def test_smoke_reaches_a_tma_staged_pass(lib):
    """The second case of smoke() launches the TMA kernel, not only a plan that names it."""
    import __graft_entry__ as entry
    p = Fake(lib, entry.TMA_SHAPE, entry.TMA_GRID)
    assert "fft_strided_tma_L512" in p.names()
    assert [k for k, *_ in p.execute() if "k_strided_tma<512" in k]


@pytest.mark.parametrize("shape,grid", [((64, 64, 64), (2, 2)), ((96, 96, 96), (2, 2)), ((128, 128, 128), (2, 4)),
                                        ((32, 64, 128), (2, 2)), ((32, 512, 64), (2, 2)), ((256, 128, 256), (2, 4)),
                                        ((60, 64, 100), (2, 3))])
def test_timed_launches_are_the_named_ones(lib, shape, grid):
    """A call with launch events runs the kernels launch_info() names, TMA-staged ones where it says so."""
    p = Fake(lib, shape, grid)
    for sign in (-1, 1):
        for name, (kernel, *_) in zip(p.names(sign), p.execute(sign, events=True)):
            assert ("_tma_" in name) == ("k_strided_tma<" in kernel), (name, kernel)
            assert ("_groups" in name) == ("RankGroupTiles" in kernel), (name, kernel)
            assert ("contig" in name) == ("contig" in kernel), (name, kernel)


@pytest.mark.parametrize("ask,threads", [("512:16", 16), ("512:16:32", 16), ("512:16:16", 32), ("256:16", 16),
                                         ("512:16:24", 16)])  # 24 is not compiled: the default
def test_tuning_variable(lib, monkeypatch, ask, threads):
    """TFFT_TMA_W="length:width:elements per thread" picks the TMA-staged variant of a length."""
    monkeypatch.setenv("TFFT_TMA_W", ask)
    p = Fake(lib, (32, 512, 64), (2, 2))
    kernels = [k for k, *_ in p.execute() if "k_strided_tma<512" in k]
    assert kernels and f"k_strided_tma<512, {threads}, 16," in kernels[0], kernels


@pytest.mark.parametrize("L,tables", [(240, 2), (256, 2), (512, 1), (1024, 1), (2048, 2), (20, 1)])
def test_stage_tables_made_are_read(lib, L, tables):
    """A contiguous pass has a stage table in the state when its kernel reads one, and only then;
    512 and 1024 read the roots, 20 has no compiled row."""
    p = Fake(lib, (L,), ())
    assert p.tables == tables
    (launch,) = p.execute()
    assert ("k_contig_spec" in launch[0]) == (L != 20)
    at = launch[4] - p.state.ctypes.data
    assert 0 <= at and at + 8 * L <= p.state.size if tables == 2 else launch[4] == 0


@pytest.mark.parametrize("L,whole,partial", [(64, True, True), (160, True, True), (240, True, True), (400, True, True),
                                             (245, True, False), (560, True, False), (1024, True, False),
                                             (60, False, False), (120, False, False), (224, False, False),
                                             (324, False, False), (490, False, False), (784, False, False),
                                             (864, False, False), (1008, False, False)])
def test_gathering_rows(lib, L, whole, partial):
    """Outside chained calls a cut pass runs gathering tiles where its row gains from them."""
    for K, want in ((128, whole), (127, partial)):
        p = Fake(lib, ((1 << 23) // (L * K) + 1, L, K), (2, 2), flags=8)  # too large to chain, no TMA
        kernels = [k for k, *_ in p.execute() if f"strided_spec<{L}," in k or f"strided_gather<{L}," in k]
        assert len(kernels) == 1 and ("gather" in kernels[0]) == want, (K, kernels)


def test_capture_ends_when_a_launch_throws(lib):
    """The second identical call captures its launches; one that runs out of host memory there leaves
    no capture open, and the next call captures and replays as usual."""
    p = Fake(lib, (32, 32, 32), (2, 2))
    lib.fake_graphs(1)
    try:
        assert len(p.execute()) == 3
        lib.fake_fail_launch(2)
        nb = ctypes.c_size_t()
        assert lib.tfft_plan_workspace_bytes(p.h, 0, 1, ctypes.byref(nb)) == 0
        at = 1 << 40
        assert lib.tfft_execute(p.h, -1, 0, at, 2 * at, 3 * at, nb.value, None) != 0
        assert not lib.fake_capturing()
        p.launches()
        assert [k for k, *_ in p.execute()][-1] == "graph"
        assert [k for k, *_ in p.execute()] == ["graph"]
    finally:
        lib.fake_fail_launch(0)
        lib.fake_graphs(0)
