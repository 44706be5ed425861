"""Reciprocal and reciprocal square root in integers (fp64_int.cuh) against the
correctly rounded quotient and against extended precision: both ends of the
mantissa, powers of two, every exponent they accept, both signs."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "fp64_int.cuh"
__global__ void k(int n, const double *x, double *near, double *exact, double *rs, int *range) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  range[i] = cagb::int_range(x[i]);
  exact[i] = cagb::recip_exact_or_zero(x[i]);
  near[i] = range[i] ? cagb::recip_near(x[i]) : 0.0;
  rs[i] = range[i] ? cagb::rsqrt_near(fabs(x[i])) : 0.0;
}
extern "C" int run(int n, const double *x, double *near, double *exact, double *rs, int *range) {
  k<<<(n + 255) / 256, 256>>>(n, x, near, exact, rs, range);
  return (int)cudaDeviceSynchronize();
}
"""


def values():
    g = np.random.default_rng(5)
    ends = np.arange(4096, dtype=np.uint64)
    mant = np.concatenate([ends, (1 << 52) - 1 - ends, (1 << 51) - 2048 + ends, ends << np.uint64(40),
                           g.integers(0, 1 << 52, 400000, dtype=np.uint64)])
    expo = g.integers(64, 0x7ff - 64, mant.size, dtype=np.uint64)
    expo[:8] = [64, 0x7ff - 65, 1023, 1024, 1022, 65, 66, 0x7ff - 66]
    sign = g.integers(0, 2, mant.size, dtype=np.uint64)
    x = ((sign << np.uint64(63)) | (expo << np.uint64(52)) | mant).view(np.float64)
    out = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1.7e308, 2.0 ** (63 - 1023), 2.0 ** 1023])
    return np.concatenate([x, out]), x.size


def test_integer_reciprocals(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, so = tmp_path / "k.cu", tmp_path / "libk.so"
    src.write_text(SRC)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-cudart", "shared", "-I", os.path.join(ROOT, "paper_1303_5837_gb300", "csrc"), "-o", str(so),
                    str(src)], check=True)
    x, inside = values()
    X = torch.from_numpy(x).cuda()
    near, exact, rs = (torch.empty_like(X) for _ in range(3))
    rng = torch.empty(x.size, dtype=torch.int32, device="cuda")
    run = ctypes.CDLL(str(so)).run
    assert run(x.size, *(ctypes.c_void_p(t.data_ptr()) for t in (X, near, exact, rs, rng))) == 0
    near, exact, rs, rng = (t.cpu().numpy() for t in (near, exact, rs, rng))
    assert rng[:inside].all() and not rng[inside:].any()
    assert not exact[inside:].any()                       # outside the range: left to the library
    got = exact[:inside]
    sure = got != 0
    assert np.array_equal(got[sure], (1.0 / x[:inside])[sure])      # IEEE division rounds correctly
    assert sure.mean() > 0.93                             # 1 in 20 is too near a tie to tell
    v = x[:inside].astype(np.longdouble)
    assert np.abs(near[:inside] * v - 1).max() <= 1.02 * 2.0 ** -53
    a = np.abs(v)
    assert np.abs(rs[:inside].astype(np.longdouble) ** 2 * a - 1).max() <= 2.1001 * 2.0 ** -53
