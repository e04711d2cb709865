"""The eight group sums of a digit product joined into one integer (the Schur update).

Over K entries a group sum reaches 10 2^12 K, so beyond K = 102 it may pass 2^22, up to
which an FP32 integer can be read off by adding 1.5 2^23.  The join must be exact on both
sides of that, for sums at their bounds and for random ones: W = sum_u G_u 2^(39 - 7u),
the last pair (G_6 2^7 + G_7) rounded to a multiple of 2^10.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2310_15458_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "common.cuh"
__global__ void k_join(const float* g, long long* w, int n, int K) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) w[i] = oz_join_k(K, [&](int u) { return g[8 * i + u]; });
}
extern "C" int join(const float* g, long long* w, int n, int K) {
  k_join<<<(n + 127) / 128, 128>>>(g, w, n, K);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("join")
    (d / "join.cu").write_text(SRC)
    so = str(d / "join.so")
    subprocess.run([B._nvcc(), *B.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC,
                    "-I", os.path.join(B.HERE, "..", "include"), "-shared", "-Xcompiler", "-fPIC", "-o", so,
                    str(d / "join.cu")], check=True)
    lib = ctypes.CDLL(so)
    lib.join.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    return lib


@pytest.mark.parametrize("K", [16, 64, 96, 112, 128, 256, 368, 384])
def test_group_sums_join_exactly(lib, K):
    bound = np.array([4 if u == 0 else 3 + u for u in range(8)], dtype=np.int64) * 4096 * K
    rng = np.random.default_rng(K)
    g = [bound, -bound, bound * (-1) ** np.arange(8), bound - 1, 0 * bound]
    g += [bound * np.where(np.arange(8) == u, s, 0) for u in range(8) for s in (1, -1)]
    g += [rng.integers(-bound, bound + 1) for _ in range(1000)]
    g = np.array(g)
    want = [sum(int(r[u]) << (39 - 7 * u) for u in range(6)) + ((int(r[6]) * 128 + int(r[7]) + 512) >> 10) for r in g]
    gd = torch.from_numpy(g.astype(np.float32)).cuda()
    w = torch.empty(len(g), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.join(gd.data_ptr(), w.data_ptr(), len(g), K) == 0
    assert w.cpu().tolist() == want
