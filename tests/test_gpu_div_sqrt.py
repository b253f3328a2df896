"""The circle fits' division and square root on the integer pipe give the IEEE
results: compiled into a small kernel of their own and compared bit for bit
with the compiler's on random significands (dense, sparse, next to a power of
two, squares and their neighbours), over exponents inside and outside the range
the fast path takes, zeros, infinities and NaN included."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import build as B  # noqa: E402

SRC = """
#include "ebit_device.cuh"
__global__ void k(const double* a, const double* b, double* o, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  o[t] = ebit::d_div(a[t], b[t]);
  o[n + t] = a[t] / b[t];
  o[2 * n + t] = ebit::d_sqrt(a[t]);
  o[3 * n + t] = sqrt(a[t]);
  o[4 * n + t] = ebit::d_scale<2>(a[t]);
  o[5 * n + t] = 4.0 * a[t];
  o[6 * n + t] = ebit::d_scale<-1>(a[t]);
  o[7 * n + t] = 0.5 * a[t];
}
extern "C" int run(const double* a, const double* b, double* o, long long n) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(a, b, o, n);
  return (int)cudaDeviceSynchronize();
}
"""


def _values(rng, n, span):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 6, n)
    cut = rng.integers(0, 52, n).astype(np.uint64)
    low = (np.uint64(1) << cut) - np.uint64(1)
    m = np.where(kind == 0, m & ~low, np.where(kind == 1, (m | low) & np.uint64((1 << 52) - 1), m))
    m = np.where(kind == 2, m % np.uint64(4), np.where(kind == 3, np.uint64((1 << 52) - 1) - m % np.uint64(4), m))
    e = (1023 + rng.integers(-span, span + 1, n)).astype(np.uint64)
    x = (m | (e << np.uint64(52)) | (rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63))).view(np.float64)
    with np.errstate(over="ignore"):
        square = x * x
    sq = square.view(np.uint64) + rng.integers(0, 3, n).astype(np.uint64) - np.uint64(1)
    return np.where((kind == 4) & (span < 500), sq.view(np.float64), x)


def test_division_and_square_root_are_ieee(tmp_path):
    src, lib = tmp_path / "t.cu", tmp_path / "t.so"
    src.write_text(SRC)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", "-I", B.CSRC, str(src), "-o", str(lib)], check=True)
    run = ctypes.CDLL(os.fspath(lib)).run
    run.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_longlong]
    rng = np.random.default_rng(11)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.3e-308, 1.7e308])
    for span in (40, 400, 1022):
        n = 4_000_000
        a, b = _values(rng, n, span), _values(rng, n, span)
        a[:64], b[:64] = np.repeat(special, 8), np.tile(special, 8)
        ta, tb = (torch.from_numpy(t).cuda() for t in (a, b))
        o = torch.empty(8 * n, dtype=torch.float64, device="cuda")
        assert run(ta.data_ptr(), tb.data_ptr(), o.data_ptr(), n) == 0
        got = o.view(4, 2, n)
        for q, name in enumerate(("division", "square root", "times 4", "half")):
            x, y = got[q, 0], got[q, 1]
            same = (x.view(torch.int64) == y.view(torch.int64)) | (x.isnan() & y.isnan())
            assert bool(same.all()), name
