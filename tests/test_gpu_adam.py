"""The Adam update of eight parameters at a time (adam_many: quotients and root from hardware approximations
and a residual step each) against the update of one in IEEE operations (adam_one), on the device, over
magnitudes from zero and subnormals to the largest, infinities and NaN."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "sur_adam.cuh"
using namespace es;
__global__ void both(int n, const float* p, const float* g, const float* m, const float* v, float* many, float* one, AdamStep w)
{
    const int i = 8 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n) return;
    float P[8], G[8], M[8], V[8];
    for (int k = 0; k < 8; ++k) { P[k] = p[i + k]; G[k] = g[i + k]; M[k] = m[i + k]; V[k] = v[i + k]; }
    adam_many<8>(P, G, M, V, w);
    for (int k = 0; k < 8; ++k) { many[i + k] = P[k]; many[n + i + k] = M[k]; many[2 * n + i + k] = V[k]; }
    for (int k = 0; k < 8; ++k) {
        float a = p[i + k], b = m[i + k], c = v[i + k];
        adam_one(a, g[i + k], b, c, w.lr, w.b1, w.b2, w.eps, w.c1, w.c2);
        one[i + k] = a; one[n + i + k] = b; one[2 * n + i + k] = c;
    }
}
extern "C" int run(int n, const float* p, const float* g, const float* m, const float* v, float* many, float* one, float lr, int t)
{
    both<<<(n / 8 + 127) / 128, 128>>>(n, p, g, m, v, many, one, adam_step(lr, 0.9f, 0.999f, 1e-8f, t));
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_04874_gb300 import build as b
    d = tmp_path_factory.mktemp("adam")
    src, so = d / "adam.cu", d / "libadam.so"
    src.write_text(SOURCE)
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", str(so), str(src)], check=True)
    vp = ctypes.c_void_p
    lib = ctypes.CDLL(os.fspath(so))
    lib.run.argtypes = [ctypes.c_int] + [vp] * 6 + [ctypes.c_float, ctypes.c_int]
    return lib


@pytest.mark.parametrize("t", [1, 2, 37, 1000, 200000])
@pytest.mark.parametrize("lr", [2e-6, 1e-2])
@pytest.mark.parametrize("span", [2, 30])
def test_many_equals_one(lib, t, lr, span):
    """Both moments to one rounding of their two terms; the parameter to its own rounding plus four last bits of
    the step (three quotients and a root), and 2^-99 where quotients underflow.  What is not finite is not
    finite in the same way."""
    import torch
    n = 1 << 20
    rng = np.random.default_rng(t + span)
    draw = lambda: rng.standard_normal(n) * 10.0 ** rng.uniform(-span, span / 2, n)
    p, g, m = (draw().astype(np.float32) for _ in range(3))
    v = np.abs(draw()).astype(np.float32)
    special = np.array([0.0, -0.0, 1e-45, -1e-40, 1.17e-38, 1e19, 3e38, -3e38, np.inf, -np.inf, np.nan], np.float32)
    for a in (p, g, m, v):  # about one group of eight in sixteen holds one or more
        at = rng.integers(0, n, n // 512)
        a[at] = rng.choice(special, len(at))
    v = np.abs(v)
    dev = [torch.from_numpy(a).cuda() for a in (p, g, m, v)]
    many, one = torch.empty(3 * n, device="cuda"), torch.empty(3 * n, device="cuda")
    assert lib.run(n, *(ctypes.c_void_p(a.data_ptr()) for a in dev), many.data_ptr(), one.data_ptr(), lr, t) == 0
    a, b = (x.cpu().numpy().reshape(3, n) for x in (many, one))
    finite = np.isfinite(b)
    assert np.array_equal(np.isfinite(a), finite)
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[~finite & ~np.isnan(b)], b[~finite & ~np.isnan(b)])
    a, b = a.astype(np.float64), b.astype(np.float64)
    p, g, m, v = (x.astype(np.float64) for x in (p, g, m, v))
    with np.errstate(all="ignore"):
        for i, size in ((1, np.abs(0.9 * m) + np.abs(0.1 * g)), (2, 0.999 * v + 0.001 * g * g)):
            ok = finite[i]
            assert np.all((np.abs(a[i] - b[i]) <= 2.0 ** -23 * size + 2.0 ** -148)[ok])
        ok = finite[0]
        step = np.abs(b[0] - p) + 2.0 ** -24 * np.abs(p)
        assert np.all((np.abs(a[0] - b[0]) <= 2.0 ** -23 * np.abs(b[0]) + 2.0 ** -21 * step + 2.0 ** -99)[ok])
