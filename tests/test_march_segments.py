"""The rule that cuts the marching axis of a 2D / 3D step into segments
(csrc/sv_march.h), compiled on the host: every grid gets a count the launch
accepts, no segment longer than the configuration's cap, and enough blocks to
reach every SM where the grid has the planes for it."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1805_03442_gb300", "csrc")
SMS = 152


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("march")
    src, so = d / "m.cpp", d / "m.so"
    src.write_text("""#include "sv_march.h"
extern "C" int segs(int cx, int cy, int step, int occ, int dim, int64_t nx, int64_t ny, int64_t nz,
                    int64_t cap, int sms) {
  const sv::MarchShape g = {cx, cy, step, 2.0, occ, {1.0, 1.3, 2.0}, 0};
  const int64_t n[3] = {nx, ny, nz};
  return sv::march_segments(g, dim, n, cap, sms);
}""")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    f = ctypes.CDLL(str(so)).segs
    f.argtypes = [ctypes.c_int] * 5 + [ctypes.c_int64] * 4 + [ctypes.c_int]
    return f


@pytest.mark.parametrize("shape", [(126, 0, 2, 3), (126, 0, 1, 2), (32, 13, 1, 1), (14, 14, 1, 1)])
@pytest.mark.parametrize("cap", [64, 128, 256, 512])
def test_every_grid_gets_a_valid_count(rule, shape, cap):
    dim = 2 if shape[1] == 0 else 3
    for nx in (1, 5, 126, 127, 500, 8192):
        for m in (1, 2, 3, 5, 63, 64, 65, 500, 513, 8192):
            ny, nz = (m, 1) if dim == 2 else (13, m)
            s = rule(*shape, dim, nx, ny, nz, cap, SMS)
            assert 1 <= s <= m
            assert -(-m // s) <= cap
            # segment k holds planes [k m / s, (k + 1) m / s): none is empty
            assert all((k + 1) * m // s > k * m // s for k in range(s))


@pytest.mark.parametrize("shape,n", [((126, 0, 1, 2), (500, 500, 1)), ((126, 0, 2, 3), (1000, 700, 1)),
                                     ((32, 13, 1, 1), (64, 48, 200))])
def test_small_grids_reach_most_sms(rule, shape, n):
    dim = 2 if shape[1] == 0 else 3
    tiles = -(-n[0] // shape[0]) * (1 if dim == 2 else -(-n[1] // shape[1]))
    s = rule(*shape, dim, *n, 256, SMS)
    assert tiles * s >= 0.9 * SMS
