"""The arithmetic that the kernels build on, one function at a time: reciprocals and
reciprocal roots from a seed, conversions by integers, and the digits and digit sums
of the column kernels.  A harness is compiled from the kernels' own headers.

Bounds: rcp_nr2 and rsqrt_nr end in one rounded fma on a correction below 2^-22, whose
own errors are 2^-22 of that rounding (rsqrt_nr's residual carries the rounding of q y,
half of it in the result): 2^-53 and 1.5 2^-53 relative, 1e-3 of it to spare; rcp_rn is
the rounded reciprocal; ff_top half a unit of single precision, ff_split2 2^-47; digits
and their sums are exact, seven digits of a three-float entry within 2^-55."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIB = os.path.join(ROOT, "paper_2108_04209_gb300", "_lib")

HARNESS = r"""
#include "fmm_impl.cuh"
__global__ void k_all(int n, const double *x, const int *k, double *o)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    o[i] = rcp_nr2(x[i]);
    o[n + i] = rcp_any(x[i]);
    o[2 * n + i] = rsqrt_nr(fabs(x[i]));
    o[3 * n + i] = rsqrt_any(fabs(x[i]));
    o[4 * n + i] = ff_top(x[i], k[i]);
    const ff_f2 s = ff_split2(x[i], k[i]);
    o[5 * n + i] = (double)s.x + (double)s.y;
    o[6 * n + i] = ff_up(ff_top(x[i], k[i]), -k[i]);
    o[7 * n + i] = rcp_rn(x[i]);
}
__global__ void k_dig(int n, const double *y, double *d, const float *t, double *c)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned short g[CM_D];
    cm_digits(y[i], g);
    for (int s = 0; s < CM_D; s++) d[i * CM_D + s] = (double)__uint_as_float((unsigned)g[s] << 16);
    float f[CM_D];
    cm_cut({t[3 * i], t[3 * i + 1], t[3 * i + 2]}, f);
    for (int s = 0; s < CM_D; s++) c[i * CM_D + s] = (double)f[s];
}
__global__ void k_sum(int n, const float *a, long long *hi, long long *lo, double *v)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float b[CM_D][4] = {};
    for (int s = 0; s < CM_D; s++) b[s][1] = a[i * CM_D + s];
    CmSum m = {0, 0};
    cm_add(m, b, 1);
    hi[i] = m.hi;
    lo[i] = m.lo;
    v[i] = cm_value(m);
}
extern "C" {
void h_all(int n, const double *x, const int *k, double *o) { k_all<<<(n + 127) / 128, 128>>>(n, x, k, o); }
void h_dig(int n, const double *y, double *d, const float *t, double *c) { k_dig<<<(n + 127) / 128, 128>>>(n, y, d, t, c); }
void h_sum(int n, const float *a, long long *hi, long long *lo, double *v) { k_sum<<<(n + 127) / 128, 128>>>(n, a, hi, lo, v); }
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    import paper_2108_04209_gb300._lib as L
    L.lib()                                        # built, and its symbols' file known
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("arith")
    (d / "h.cu").write_text(HARNESS)
    cmd = [nvcc, "-shared", str(d / "h.cu"), "-o", str(d / "h.so"), "-gencode", "arch=compute_103a,code=sm_103a", "-O1",
           "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(ROOT, "paper_2108_04209_gb300", "csrc"), "-L", LIB, "-l:libsuperdc.so",
           "-Xlinker", "-rpath," + LIB]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return ctypes.CDLL(str(d / "h.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _values(rng):
    e = np.concatenate([rng.uniform(-1000, 1000, 4000), rng.uniform(-2, 2, 4000)])
    x = rng.choice([-1.0, 1.0], e.size) * rng.uniform(1, 2, e.size) * 2.0 ** np.floor(e)
    near = np.concatenate([2.0 ** np.arange(-40, 40.0), np.nextafter(2.0 ** np.arange(-40, 40.0), 0), [1.5, -3.0, 1 / 3]])
    return np.concatenate([x, near])


def test_reciprocals_and_conversions(harness):
    L = np.longdouble
    if np.finfo(L).nmant < 100:
        pytest.skip("long double is not quadruple precision here")
    x = _values(np.random.default_rng(1))
    n = len(x)
    k = -np.floor(np.log2(np.abs(x))).astype(np.int32) + np.random.default_rng(2).integers(-20, 20, n).astype(np.int32)
    xg, kg = torch.from_numpy(x).cuda(), torch.from_numpy(k).cuda()
    o = torch.empty(8, n, dtype=torch.float64, device="cuda")
    harness.h_all(n, _p(xg), _p(kg), _p(o))
    torch.cuda.synchronize()
    rcp, rany, rsq, rsany, top, split, up, rn = (v.astype(L) for v in o.cpu().numpy())
    xl = x.astype(L)
    u = L(2.0) ** -53 * (1 + L(1e-3))
    assert np.all(np.abs(rcp * xl - 1) <= u)
    assert np.all(np.abs(rany * xl - 1) <= u)
    assert np.array_equal(rn.astype(np.float64), 1.0 / x)
    for r in (rsq, rsany):
        assert np.all(np.abs(r * np.sqrt(np.abs(xl)) - 1) <= 1.5 * u)
    v = xl * L(2.0) ** k
    assert np.all(np.abs(top - v) <= L(2.0) ** -24 * np.abs(v))
    assert np.all(np.abs(split - v) <= L(2.0) ** -47 * np.abs(v))
    assert np.array_equal(up, top * L(2.0) ** -k)


def test_digits_are_exact(harness):
    rng = np.random.default_rng(3)
    y = np.concatenate([rng.uniform(-1, 1, 4000), rng.standard_normal(2000) * 1e-3, [1.0, -1.0, 0.0, 0.5, -0.5, 127.5 / 128,
                        2.0 ** -55, 2.0 ** -56, 1 - 2.0 ** -53, -1 + 2.0 ** -53], 2.0 ** -np.arange(1, 56.0)])
    n = len(y)
    t = np.zeros((n, 3), np.float32)
    t[:, 0] = y
    r = y - t[:, 0]
    t[:, 1] = r
    t[:, 2] = (r - t[:, 1]) + rng.uniform(-1, 1, n) * 2.0 ** -52 * np.abs(y)      # a third part below the second's unit
    yg, tg = torch.from_numpy(y).cuda(), torch.from_numpy(t).cuda()
    d, c = (torch.empty(n, 7, dtype=torch.float64, device="cuda") for _ in range(2))
    harness.h_dig(n, _p(yg), _p(d), _p(tg), _p(c))
    torch.cuda.synchronize()
    grid = 2.0 ** -(8 * np.arange(1, 8) - 1.0)
    for got, want in ((d.cpu().numpy(), y), (c.cpu().numpy(), None)):
        q = got / grid
        assert np.array_equal(q, np.round(q)) and np.all(np.abs(q) <= 256)
        q = q.astype(np.int64)                     # the sum in units of the last digit, exact
        tot = sum(int(2 ** (8 * (6 - s))) * q[:, s] for s in range(7))
        if want is not None:
            assert np.array_equal(tot, np.rint(want * 2.0 ** 55).astype(np.int64))
            assert np.all(np.abs(q) <= 128)
        else:
            err = [abs(int(tot[i]) - sum(Fraction(float(p)) for p in t[i]) * 2 ** 55) for i in range(n)]
            assert max(err) <= 1


def test_digit_sums_are_exact(harness):
    """Accumulators as the products leave them: multiples of the order's unit below 2^24 units."""
    rng = np.random.default_rng(4)
    n = 3000
    units = np.array([2.0 ** -(14 + 8 * s) for s in range(7)])
    q = rng.integers(-(2 ** 24) + 1, 2 ** 24, (n, 7))
    q[:7] = np.eye(7, dtype=np.int64) * (2 ** 24 - 1)
    a = torch.from_numpy((q * units).astype(np.float32)).cuda()
    hi, lo = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    v = torch.empty(n, dtype=torch.float64, device="cuda")
    harness.h_sum(n, _p(a), _p(hi), _p(lo), _p(v))
    torch.cuda.synchronize()
    exact = [sum(int(q[i, s]) << (8 * (6 - s)) for s in range(7)) for i in range(n)]       # in units of 2^-62
    got = [(int(h) << 32) + int(w) for h, w in zip(hi.cpu(), lo.cpu())]
    assert got == exact
    e = np.array([float(x) for x in exact]) * 2.0 ** -62
    assert np.all(np.abs(v.cpu().numpy() - e) <= 2.0 ** -52 * np.abs(e) + 2.0 ** -85)
