"""The grid's integer arithmetic, compiled for the host, against Python integers: records of the
fixed format (valid and not) and the cell size at the ends of its range."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2106_03636_gb300 import _build

SOURCE = """
#include "o2tpc_internal.cuh"
using namespace o2tpc;
extern "C" int t_decode_fixed(const uint32_t* w, const int* npads, int* o) {
  return decode_fixed(w[0], w[1], w[2], npads, o[0], o[1], o[2], o[3]) ? 1 : 0;
}
extern "C" int t_drift_bins(float range, int count, int nz) { return drift_bins(range, count, nz); }
extern "C" int t_cell_height(int zmin, int zmax, int nz) { return cell_height(zmin, zmax, nz); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid")
    (d / "grid.cu").write_text(SOURCE)
    cmd = [_build._nvcc()] + _build.ARCH + ["-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", _build.CSRC, "-I",
                                            _build.INCLUDE, str(d / "grid.cu"), "-o", str(d / "grid.so")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(d / "grid.so"))


def test_fixed_records(lib):
    """Valid records give their values, others row 0 with a time that a valid record can have."""
    rng = np.random.default_rng(1)
    w = rng.integers(0, 1 << 32, (4000, 3), dtype=np.uint64).astype(np.uint32)
    w[:2000, 0] &= 0x3FFFFFFF
    w[:1000, 2] = rng.integers(0, 36, 1000) << 8 | rng.integers(0, 152, 1000)
    w[0], w[1], w[2], w[3] = (0x3FFFFFFF, 0xFFFF, 151 | 35 << 8), (0x40000000, 0, 0), (0, 0, 152), (0, 0, 36 << 8)
    w[4], w[5] = (0xFFFFFFFF,) * 3, (0x80000000, 0, 0)
    npads = np.arange(152, dtype=np.int32) + 60
    out = (ctypes.c_int * 4)()
    nok = 0
    for a, b, c in w.tolist():
        ok = lib.t_decode_fixed((ctypes.c_uint32 * 3)(a, b, c), npads.ctypes.data_as(ctypes.c_void_p), out)
        s, r, y, z = out
        want = (c >> 8 & 255) < 36 and (c & 255) < 152 and a < 1 << 30
        assert ok == want
        assert (s, r) == ((c >> 8 & 255, c & 255) if want else (0, 0))
        assert y == (b & 0xFFFF) - 32 * int(npads[r])
        assert 0 <= z < 1 << 30 and (z == a or not want)
        nok += ok
    assert nok > 900


@pytest.mark.parametrize("zmin,zmax", [(0, 0), (0, 1), (-5, 1000000), (0, (1 << 30) - 1), (-(1 << 30), 1 << 30),
                                       (-(1 << 31), (1 << 31) - 1), (-(1 << 31) + 7, (1 << 31) - 9)])
def test_cell_height(lib, zmin, zmax):
    """ceil(range / nz), also where range + nz - 1 does not fit 32 bits."""
    for nz in (1, 2, 3, 7, 1000, 8214, (1 << 20) - 1, 1 << 20):
        want = (zmax - zmin + nz) // nz
        assert lib.t_cell_height(zmin, zmax, nz) & 0xFFFFFFFF == want & 0xFFFFFFFF


@pytest.mark.parametrize("nz", [1, 2, 1000, 536870, 536871, 1 << 20])
def test_drift_bins(lib, nz):
    """The least of 62 units a bin, a bin a hit and 4000 a cell row, also past 2^31 of these."""
    lib.t_drift_bins.argtypes = [ctypes.c_float, ctypes.c_int, ctypes.c_int]
    for count in (1, 100, 40000000):
        for rng in (1.0, 61.0, 6200.0, 2.0 ** 31):
            got = lib.t_drift_bins(rng, count, nz)
            want = max(1, min(int(np.float32(rng) * np.float32(1 / 62)), count, nz * 4000))
            assert abs(got - want) <= (rng > 2 ** 24)
