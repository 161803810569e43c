"""The FP64 reciprocal, quotient and roots of the flux arithmetic themselves
(csrc/physics.cuh), against exact values over the exponent range, and the
logarithmic mean where the sum of two densities is near the end of that range.

Bounds, relative, in units of 2^-53 (half the spacing of doubles at 1).  The seed
of a step has 20 significant bits, so its relative error d is below 2^-19.
  reciprocal  the step's first term left out is e^3, e = d: 2^-57; e and e + e^2
              are rounded relative to themselves; the final fma rounds once:
              1 + 2^-4
  quotient    that and one product: 2 + 2^-4
  root^-1     e = 1 - x y^2 is formed from the rounded product x y (one rounding
              relative to 1, halved by e/2), the first term left out is 5 e^3/16
              with e = 2 d: 2^-54 5/16, and the final fma: 1/2 + 0.16 + 1
  root        that and one product: 2.66
  corrected   root and quotient by their residuals, which are exact to 2^-53 of
              themselves: the square of the error corrected (2^-104) and one
              rounding, 1 + 2^-20, where the residual is a normal number
"""
import ctypes as C
import subprocess

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2206_09733_gb300 as hs  # noqa: E402
from paper_2206_09733_gb300 import build as hsbuild  # noqa: E402

SOURCE = r'''
#include "physics.cuh"
using namespace hs3d;
__global__ void k_steps(const double *a, const double *x, long long n, double *out)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    const double r[10] = {rcp_fast(v), rsqrt_fast(v), sqrt_fast(v), div_(a[i], v),
                          1.0 / v, 1.0 / sqrt(v), sqrt(v), a[i] * (1.0 / v), root(v), quotient(a[i], v)};
    for (int k = 0; k < 10; ++k) out[k * n + i] = r[k];
}
extern "C" int run_steps(const double *a, const double *x, long long n, double *out)
{
    k_steps<<<(unsigned)((n + 255) / 256), 256>>>(a, x, n, out);
    cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
'''


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("steps")
    src, lib = d / "steps.cu", d / "libsteps.so"
    src.write_text(SOURCE)
    subprocess.check_call([hsbuild.nvcc()] + hsbuild._flags(False) + ["-I", hsbuild.CSRC, "-shared", str(src), "-o", str(lib)])
    f = C.CDLL(str(lib)).run_steps
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_longlong, C.c_void_p]

    def run(a, x):
        ad, xd = torch.from_numpy(a).cuda(), torch.from_numpy(x).cuda()
        out = torch.empty((10, x.size), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert f(ad.data_ptr(), xd.data_ptr(), x.size, out.data_ptr()) == 0
        return out.cpu().numpy()
    return run


def plain(x):
    """Arguments that take the step: biased exponents 2 .. 0x7fb."""
    e = (x.view(np.uint64) >> np.uint64(52)) & np.uint64(0x7ff)
    return (e >= 2) & (e <= 0x7fb)


def test_steps_against_exact_values(steps):
    rng = np.random.default_rng(17)
    n = 1 << 20
    ex = rng.integers(2, 0x7fc, size=n).astype(np.uint64)
    ex[: n // 2] = rng.integers(0x3ff - 40, 0x3ff + 40, size=n // 2)   # the range of flow states, more densely
    x = ((ex << np.uint64(52)) | rng.integers(0, 1 << 52, size=n, dtype=np.uint64)).view(np.float64)
    x[:4] = [2.0 ** -1021, np.nextafter(2.0 ** 1021, 0), 1.0, np.nextafter(1.0, 2.0)]
    assert plain(x).all()
    a = rng.uniform(0.5, 2.0, size=n)
    got = steps(a, x)
    xl, al = x.astype(np.longdouble), a.astype(np.longdouble)
    exact = [1 / xl, 1 / np.sqrt(xl), np.sqrt(xl), al / xl]
    for k, (name, bound) in enumerate((("reciprocal", 1.0625), ("inverse root", 1.66), ("root", 2.66),
                                       ("quotient", 2.0625))):
        err = np.abs((got[k] - exact[k]) / exact[k]).max() * 2.0 ** 53
        ieee = np.abs((got[4 + k] - exact[k]) / exact[k]).max() * 2.0 ** 53
        print(f"{name}: {float(err):.3f} (CUDA's operations: {float(ieee):.3f}) x 2^-53")
        assert err <= bound, (name, float(err))


def test_corrected_root_and_quotient(steps):
    rng = np.random.default_rng(19)
    n = 1 << 20
    x = np.ldexp(rng.uniform(1.0, 2.0, size=n), rng.integers(-400, 400, size=n))
    a = np.ldexp(rng.uniform(1.0, 2.0, size=n), rng.integers(-400, 400, size=n))
    got = steps(a, x)
    xl, al = x.astype(np.longdouble), a.astype(np.longdouble)
    for v, exact in ((got[8], np.sqrt(xl)), (got[9], al / xl)):
        assert np.abs((v - exact) / exact).max() * 2.0 ** 53 <= 1 + 2.0 ** -20


def test_arguments_outside_the_steps_take_the_ieee_operations(steps):
    rng = np.random.default_rng(18)
    x = np.concatenate([[0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1021, 0),
                         2.0 ** 1021, -1.0, -2.0 ** 1021, np.finfo(float).max],
                        rng.integers(1, 1 << 53, size=500).astype(np.uint64).view(np.float64)])
    a = np.ones_like(x)
    got = steps(a, x)
    same = lambda p, q: (p.view(np.uint64) == q.view(np.uint64)) | (np.isnan(p) & np.isnan(q))  # noqa: E731
    # (a reciprocal may be taken of negative arguments, a root not)
    step = plain(np.abs(x))
    assert same(got[0], got[4])[~step].all() and same(got[3], got[7])[~step].all()
    step = plain(x) & (x > 0)
    assert same(got[1], got[5])[~step].all() and same(got[2], got[6])[~step].all()
    assert same(got[8], got[6])[~step].all()
    # a quotient by an infinite value is zero, by zero or one that overflows infinite
    assert (got[9][np.isinf(x)] == 0).all() and np.isinf(got[9][x == 0]).all()
    big, small = np.full(1, 1e300), np.full(1, 1e-300)
    assert np.isposinf(steps(big, small)[9]).all()


def test_logarithmic_mean_of_densities_whose_sum_is_near_the_largest_double():
    """rho_L + rho_R above 2^1022, where 1/(rho_L + rho_R) is subnormal; slow flow and
    a small pressure keep every flux in range.  Each variable's residual by itself:
    the mass row is the logarithmic mean's."""
    om = O.Mesh(2, 3, 2, 3, lo=(0.0,) * 3, hi=(10.0,) * 3, amp=0.05)
    gm = hs.Mesh(2, 3, 2, 3, lo=(0.0,) * 3, hi=(10.0,) * 3, amp=0.05)
    rng = np.random.default_rng(5)
    dims = (om.shape[0],) + tuple(om.shape[2:])
    rho = np.ldexp(np.where(rng.random(dims) < 0.5, 1.1, 1.1 * 1.015), 1021)
    p = np.ldexp(rng.uniform(1.0, 1.3, size=dims), 1000)
    v = rng.uniform(0.5e-9, 1e-9, size=(3,) + dims)
    u0 = np.empty(om.shape)
    u0[:, 0] = rho
    for c in range(3):
        u0[:, 1 + c] = rho * v[c]
    u0[:, 4] = p / 0.4 + 0.5 * rho * (v ** 2).sum(0)
    ref = om.residual(O.Cfg("euler", "ec", "ec"), u0)
    u = torch.from_numpy(u0).cuda()
    r = torch.empty_like(u)
    gm.residual(hs.solver_cfg("euler", "ec", "ec", "fp64"), u, r)
    out = r.cpu().numpy()
    for k in range(5):
        a, b = np.ldexp(out[:, k], -1000), np.ldexp(ref[:, k], -1000)
        assert np.isfinite(b).all() and np.linalg.norm(a - b) / np.linalg.norm(b) < 1e-12, k
