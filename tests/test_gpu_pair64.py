"""The scalar building blocks of csrc/pair64.cuh against CUDA's own correctly
rounded operations, over all exponents: a small program that includes the header
is compiled for the test."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "paper_1007_3458_gb300/csrc/pair64.cuh"
using namespace qym;
__global__ void k(long n, const double *x, const double *y, double *o, float *f) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double a = x[i], b = y[i];
    double ir;
    o[i] = p64::rcp(a);             o[n + i] = 1.0 / a;
    o[2 * n + i] = p64::sqrt_rcp(a, ir); o[3 * n + i] = sqrt(a);
    o[4 * n + i] = ir;              o[5 * n + i] = 1.0 / sqrt(a);
    o[6 * n + i] = p64::div(b, a, p64::rcp(a)); o[7 * n + i] = b / a;
    o[8 * n + i] = p64::rsqrt64(a); o[9 * n + i] = rsqrt(a);
    const float2 s = p64::split2(a);
    f[i] = p64::to_float(a);        f[n + i] = (float)a;
    f[2 * n + i] = s.x;             f[3 * n + i] = s.y;
    f[4 * n + i] = (float)(a - (double)(float)a);
    f[5 * n + i] = p64::norm_up(a, b, 0.0);
}
extern "C" int run(long n, const double *x, const double *y, double *o, float *f) {
    k<<<(unsigned)((n + 255) / 256), 256>>>(n, x, y, o, f);
    return (int)cudaDeviceSynchronize();
}
"""


def _values(rng, n):
    """Positive doubles: random mantissas over all exponents and around 1, powers of
    two and their neighbours, the ends of the range, zeros, infinities, NaN."""
    u = rng.integers(0, 1 << 63, n, dtype=np.uint64)
    near = rng.uniform(0.5, 4.0, n)
    p = 2.0 ** rng.integers(-1022, 1023, 4000).astype(float)
    edge = np.concatenate([p, np.nextafter(p, 0), np.nextafter(p, np.inf), [0.0, np.inf, np.nan, 5e-324, 2.3e-308,
                          1.797e308, 2.0 ** -149, 2.0 ** -126, 2.0 ** 127, 3.4e38, 3.5e38]])
    return np.concatenate([u.view(np.float64), near, edge])


def test_scalar_operations(tmp_path):
    """Reciprocal, square root, the root's reciprocal and quotients carry the bits of
    CUDA's IEEE forms, the reciprocal square root lies within an ulp of the library's
    (2 ulp, so 3 in all), the float conversions and the two-float split are the
    nearest floats, and norm_up bounds the norm from above within 1e-6."""
    torch = pytest.importorskip("torch")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, lib = tmp_path / "p.cu", tmp_path / "p.so"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", ROOT, "-shared",
                    "-Xcompiler", "-fPIC", str(src), "-o", str(lib)], check=True)
    rng = np.random.default_rng(1)
    x = _values(rng, 1 << 20)
    y = rng.permutation(x) * rng.choice([-1.0, 1.0], len(x))
    n = len(x)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    o = torch.empty((10, n), dtype=torch.float64, device="cuda")
    f = torch.empty((6, n), dtype=torch.float32, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert ctypes.CDLL(str(lib)).run(ctypes.c_long(n), p(xd), p(yd), p(o), p(f)) == 0
    o, f = o.cpu().numpy(), f.cpu().numpy()
    same = lambda a, b: (a == b) | (np.isnan(a) & np.isnan(b))
    for k, name in ((0, "reciprocal"), (2, "square root"), (4, "reciprocal of the root"), (6, "quotient")):
        bad = ~same(o[k], o[k + 1])
        assert not bad.any(), (name, int(bad.sum()), x[bad][:4].tolist(), y[bad][:4].tolist())
    fin = np.isfinite(o[9]) & (o[9] > 0)
    assert np.all(same(o[8], o[9])[~fin])
    assert np.all(np.abs(o[8] - o[9])[fin] <= 3 * np.spacing(o[9][fin]))
    assert np.all(same(f[0], f[1])) and np.all(same(f[2], f[1]))
    normal = np.isfinite(f[1]) & (x >= 2.0 ** -88)
    assert np.array_equal(f[3][normal], f[4][normal])
    with np.errstate(over="ignore", invalid="ignore"):
        r = np.hypot(x, np.abs(y))
    inside = np.isfinite(r) & (r > 2.0 ** -120) & (r < 2.0 ** 126)
    up = f[5].astype(np.float64)
    assert np.all(up[inside] >= r[inside]) and np.all(up[inside] <= r[inside] * (1 + 1e-6))
    low = np.isfinite(r) & (r <= 2.0 ** -120)
    assert np.all(up[low] >= r[low])
