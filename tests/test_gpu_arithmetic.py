"""The short arithmetic sequences of the device code (les_fp64.cuh, les_fused.cuh, les_pair.cuh) over the exponents
they may meet and at special values, each against higher precision at the bound that its comment states, and the FP64
ones no further off than CUDA's own functions where they replace them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2212_12365_gb300", "csrc")
SRC = r"""
#include "les_fp64.cuh"
#include "les_bc.cuh"
#include "les_fused.cuh"
#include "les_pair.cuh"
using namespace les;
__global__ void k64(const double *x, int n, double *o)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v[8] = {rcp64(x[i]), rcp64_1(x[i]), rsqrt64(x[i]), sqrt64(x[i]), twice_sqrt64(x[i]), half_sqrt64(x[i]),
                         sqrt(x[i]), rsqrt(x[i])};
    for (int f = 0; f < 8; ++f) o[f * n + i] = v[f];
}
__global__ void k32(const float *x, int n, float *o)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 p = f2(x[i], x[n - 1 - i]); // the other lane holds something else
    const float v[5] = {rcp2(p).x, rsqa(x[i]), rcbrt2(p).x, sqrtp2(p).x, sqrt2(p).x};
    for (int f = 0; f < 5; ++f) o[f * n + i] = v[f];
}
__global__ void kpair(const float *a, const float *b, int n, float *o) // a, b: [2][n] pairs
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    typedef Num<float> A;
    const FloatPair p{a[i], a[n + i]}, q{b[i], b[n + i]};
    const FloatPair v[4] = {A::add(p, q), A::sub(p, q), A::mulp(p, q), A::mul(a[i], q)};
    for (int f = 0; f < 4; ++f) {
        o[2 * f * n + i] = v[f].h;
        o[(2 * f + 1) * n + i] = v[f].l;
    }
}
// energy_pair of a state at rest but for rho u: 1/rho, and the internal energy
__global__ void kenergy(const float *q, int n, float *o)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float Q[5] = {q[i], q[n + i], q[2 * n + i], q[3 * n + i], q[4 * n + i]};
    FloatPair rr, ei;
    energy_pair(Q, rr, ei);
    o[i] = rr.h;
    o[n + i] = rr.l;
    o[2 * n + i] = ei.h;
    o[3 * n + i] = ei.l;
}
extern "C" int run(int which, const void *a, const void *b, int n, void *o)
{
    const int g = (n + 255) / 256;
    if (which == 0) k64<<<g, 256>>>((const double *)a, n, (double *)o);
    else if (which == 1) k32<<<g, 256>>>((const float *)a, n, (float *)o);
    else if (which == 3) kenergy<<<g, 256>>>((const float *)a, n, (float *)o);
    else kpair<<<g, 256>>>((const float *)a, (const float *)b, n, (float *)o);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_2212_12365_gb300 import build
    d = tmp_path_factory.mktemp("arith")
    (d / "a.cu").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-I",
                    inc, str(d / "a.cu"), "-o", str(d / "a.so")], check=True)
    f = ctypes.CDLL(str(d / "a.so")).run
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def call(which, a, b, rows):
        n = a.shape[-1]
        ta, tb = torch.from_numpy(a).cuda(), None if b is None else torch.from_numpy(b).cuda()
        o = torch.empty((rows, n), dtype=ta.dtype, device="cuda")
        torch.cuda.synchronize()
        assert f(which, ta.data_ptr(), 0 if b is None else tb.data_ptr(), n, o.data_ptr()) == 0
        return o.cpu().numpy()
    return call


def _ulps(got, exact, kind):
    """Error in units in the last place of the exact value."""
    return np.abs((got.astype(np.longdouble) - exact) / np.spacing(np.abs(exact.astype(kind)))).astype(float)


def test_fp64_sequences(run):
    g = np.random.default_rng(0)
    e = np.concatenate([np.repeat(np.arange(-1021, 1022), 200), g.integers(-12, 12, 600000)])
    x = np.ldexp(1.0 + g.random(e.size), e - 1)
    x = np.concatenate([x, np.ldexp(1.0, np.arange(-1021, 1021)), np.nextafter(np.ldexp(1.0, np.arange(-1020, 1021)), 0)])
    v = run(0, x, None, 8)
    X = x.astype(np.longdouble)
    root, one = np.sqrt(X), np.longdouble(1)
    assert _ulps(v[0], one / X, np.float64).max() <= 0.53  # the cubic step leaves 2^-60
    assert np.abs((v[1] * X - 1).astype(float)).max() <= 2.0 ** -39
    assert _ulps(v[2], one / root, np.float64).max() <= 1.03
    for f, scale in ((3, 1), (4, 2), (5, 0.5)):
        # no further from the root than the correctly rounded one but for 2^-58; near the smallest numbers the
        # residual x - t^2 is rounded to a subnormal
        u = _ulps(v[f], root * scale, np.float64)
        assert u[x >= 2.0 ** -1000].max() <= 0.53 and u.max() <= 1.03, f
    assert _ulps(v[6], root, np.float64).max() <= 0.5 + 1e-6


def test_fp64_roots_at_special_values(run):
    x = np.array([0.0, -0.0, np.inf, np.nan, -1.0, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0), 5e-324, np.finfo(float).max])
    v = run(0, x, None, 8)
    with np.errstate(invalid="ignore"):
        exact = np.sqrt(x)
    for f, scale in ((3, 1.0), (4, 2.0), (5, 0.5)):
        want = exact * scale
        want[6:8] = 0.0  # below the normal range
        np.testing.assert_array_equal(v[f], want)
    np.testing.assert_array_equal(v[6], exact)


def test_fp32_sequences(run):
    g = np.random.default_rng(1)
    e = np.concatenate([np.repeat(np.arange(-124, 125), 2000), g.integers(-8, 8, 600000)])
    x = np.ldexp(1.0 + g.random(e.size), e - 1).astype(np.float32)
    v = run(1, x, None, 5)
    X = x.astype(np.float64)
    ok = X < 2.0 ** 125
    assert _ulps(v[0][ok], (1 / X)[ok].astype(np.longdouble), np.float32).max() <= 1.5
    assert _ulps(v[1], (1 / np.sqrt(X)).astype(np.longdouble), np.float32).max() <= 2.5
    assert _ulps(v[2], np.cbrt(1 / X.astype(np.longdouble)), np.float32).max() <= 2.0
    for f in (3, 4):
        assert _ulps(v[f], np.sqrt(X).astype(np.longdouble), np.float32).max() <= 3.0
    zero = run(1, np.zeros(4, np.float32), None, 5)
    assert (zero[4] == 0).all()  # no strain; a spectral radius on the axis of a polar mesh


def test_pairs_of_floats(run):
    g = np.random.default_rng(2)
    n = 400000

    def pair():
        d = g.normal(size=n) * 2.0 ** g.integers(-12, 13, n)
        h = d.astype(np.float32)
        return np.stack([h, (d - h).astype(np.float32)])
    a, b = pair(), pair()
    b[:, ::5] = -a[:, ::5] * np.float32(1 + 2 ** -12)  # near cancellation
    v = run(2, a, b, 8).astype(np.longdouble)
    A, B = (t[0].astype(np.longdouble) + t[1] for t in (a, b))
    a0 = a[0].astype(np.longdouble)
    for f, (exact, scale) in enumerate(((A + B, abs(A) + abs(B)), (A - B, abs(A) + abs(B)), (A * B, abs(A * B)), (a0 * B, abs(a0 * B)))):
        rel = np.abs((v[2 * f] + v[2 * f + 1] - exact) / scale).astype(float).max()
        assert rel <= 2.0 ** -45, (f, np.log2(rel))  # 48 bits less the roundings of the low parts


def test_energy_in_pairs_of_floats(run):
    """1/rho and e - rho u^2 / 2 of the FP32 boundary pass, whose differences to the ambient values matter."""
    g = np.random.default_rng(3)
    n = 400000
    q = np.stack([g.uniform(0.3, 4.0, n), *(g.normal(size=(3, n)) * 10.0 ** g.uniform(-7, 0, n)), g.uniform(3.0, 8.0, n)]).astype(np.float32)
    v = run(3, q, None, 4).astype(np.longdouble)
    Q = q.astype(np.longdouble)
    assert np.abs(((v[0] + v[1]) * Q[0] - 1).astype(float)).max() <= 2.0 ** -46  # the last bit of the low part
    e = Q[4] - (Q[1] ** 2 + Q[2] ** 2 + Q[3] ** 2) / (2 * Q[0])
    scale = Q[4] + (Q[1] ** 2 + Q[2] ** 2 + Q[3] ** 2) / (2 * Q[0])
    assert np.abs(((v[2] + v[3] - e) / scale).astype(float)).max() <= 2.0 ** -44  # five pair operations
