"""Which colour classes the tensor-core sweeps take: exactly those whose four products fit
the shared memory that their launches ask for, whatever the number of columns.  The plan
(host code) is compiled alone and compared with the sizes written out here."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2310_15458_gb300", "csrc")
LIMIT = 222 * 1024
SRC = r"""
#include "tw_plan.h"
extern "C" int fits(int n, int r, int c, int real) { return tw_shape_fits(n, r, c, real); }
extern "C" int group(int op, int n, int r, int c, int real) { return tw_group(op, n, r, c, real); }
extern "C" int plan(int op, int n, int r, int c, int gw, int real, int* out) {
  const TwPlan p = tw_plan_op(op, n, r, c, gw, real);
  out[0] = p.rows8; out[1] = p.nst; out[2] = p.nstr; out[3] = p.smem;
  return TW_MAXN;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(SRC)
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "p.so"), str(d / "p.cpp")], check=True)
    return ctypes.CDLL(str(d / "p.so"))


def bytes_of(rows, k, gw, stretch, nst):
    """nst stages of 8 slices of 2-byte digits, 32 entries a slice; 4-byte places and exponents."""
    rows8 = min(128, -(-rows // 8) * 8)
    stage = 8 * 32 * 2 * (rows8 + 2 * gw)
    stretches = -(-k // stretch) + 1
    return nst * stage + 4 * (k + stretches * (128 + 2 * gw)) + (128 - rows8) * 64


@pytest.mark.parametrize("real", [True, False])
def test_plan_and_rule(lib, real):
    out = (ctypes.c_int * 4)()
    maxn = lib.plan(0, 1, 1, 1, 32, real, out)
    seen = set()
    for n in sorted({1, 2, 4, 8, 9, 33, 64, 100, 121, 127, 128, 129, 144, 256, 257, 400, 1000, 1024, 1025, 2000, maxn, maxn + 1}):
        for r in sorted({1, n // 2 + 1, n}):
            for c in (0, 1, 100, 383, 385, 900, 1200, 1400, 1500, 1600, 1709, 1750, 2000, 3000, 4999, 5200, 5600, 5700, 6000, 6001, 9000):
                stretch = 48 if not real else 64 if n > 128 else 384
                shapes = [(r, n), (max(1, c), r), (r, c), (n, r)]
                fits = n <= maxn and c <= 6000 and all(bytes_of(m, k, 16, stretch, 2) <= LIMIT for m, k in shapes)
                assert bool(lib.fits(n, r, c, real)) == fits, (n, r, c)
                seen.add(fits)
                if not fits:
                    continue
                for op, (m, k) in enumerate(shapes):
                    most = lib.group(op, n, r, c, real)
                    assert most == (32 if bytes_of(m, k, 32, stretch, 2) <= LIMIT else 16)
                    for gw in (16, 32)[:most // 16]:
                        lib.plan(op, n, r, c, gw, real, out)
                        assert 2 <= out[1] <= 4 and out[3] == bytes_of(m, k, gw, stretch, out[1]) <= LIMIT, (op, n, r, c, gw)
    assert seen == {True, False}
