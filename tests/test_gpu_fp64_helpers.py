"""The scalar helpers of the FP64 integrator against CUDA's and numpy's results: the
reciprocal, quotient and inverse square root that stand for CUDA's, FP32 <-> FP64 by
integer operations, and the step controller's factor; and a trace whose absolute
tolerance is subnormal."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2309_08655_gb300 import build as B  # noqa: E402
from paper_2309_08655_gb300 import inputs as I  # noqa: E402
from paper_2309_08655_gb300 import rt  # noqa: E402

from . import gpu_util as G  # noqa: E402

SRC = r"""
#include "rt_integrator.cuh"
using namespace rtk;
__global__ void apply(int op, long n, const double* a, const double* b, double* out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const double x = a[i], y = b[i];
    if (op == 0) out[i] = recip(x);
    if (op == 1) out[i] = quotient(x, y);
    if (op == 2) out[i] = widen(narrow(x));
    if (op == 3) out[i] = step_factor_sq(x, y != 0.0, false);
    if (op == 4) out[i] = max_abs(x, y);
    if (op == 5) out[i] = 1.0 / x;
    if (op == 6) out[i] = inv_sqrt(x);
    if (op == 7) out[i] = rsqrt(x);
  }
}
extern "C" int run(int op, long n, const double* a, const double* b, double* out) {
  apply<<<64, 128>>>(op, n, a, b, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    B.build()
    assert torch.cuda.is_available()
    d = tmp_path_factory.mktemp("helpers")
    src, so = os.path.join(d, "helpers.cu"), os.path.join(d, "helpers.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-I", B.INCLUDE, "-I", B.CSRC, "-I", B.BUILD, src, "-o",
                    so], check=True, capture_output=True)
    L = ctypes.CDLL(so)

    def call(op, a, b=None):
        a = torch.as_tensor(np.asarray(a, dtype=np.float64)).to(G.dev())
        b = torch.ones_like(a) if b is None else torch.as_tensor(
            np.asarray(b, dtype=np.float64)).to(G.dev())
        out = torch.empty_like(a)
        code = L.run(op, ctypes.c_long(a.numel()), *(ctypes.c_void_p(t.data_ptr())
                                                     for t in (a, b, out)))
        assert code == 0
        return out.cpu().numpy()
    return call


def _positive(n, lo, hi, seed):
    rng = np.random.default_rng(seed)
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


SPECIAL = np.array([0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1030, 2.0 ** -1022, 1e-308, 2.0 ** -101,
                    2.0 ** -100, 2.0 ** 100, np.nextafter(2.0 ** 100, 0), 2.0 ** 1022, 1.7e308,
                    np.inf, -np.inf, np.nan, -1.0, -3.5, 1.0, 1 + 2.0 ** -52, 2 - 2.0 ** -52])


def test_reciprocal_and_quotient(run):
    x = np.concatenate([_positive(200000, -1000, 1000, 1), _positive(200000, -100, 100, 2)])
    # the corrected reciprocal is off by the last multiply-add's rounding: at most one
    # unit in the last place of the correctly rounded 1/x, as CUDA gives it
    ref = run(5, x)
    assert (np.abs(run(0, x) - ref) <= np.spacing(ref)).all()
    one = run(0, SPECIAL)
    with np.errstate(all="ignore"):
        want = 1.0 / SPECIAL
        inside = (SPECIAL >= 2.0 ** -100) & (SPECIAL < 2.0 ** 100)
        np.testing.assert_array_equal(one[~inside], want[~inside])
        assert (np.abs(one[inside] / want[inside] - 1) <= 2.0 ** -52).all()
        e = np.concatenate([_positive(400000, -60, 60, 3), np.resize([0.0, 1e-300, -2.0], 21)])
        b = np.concatenate([x, SPECIAL])
        q, want = run(1, e, b), e / b
    fin = np.isfinite(want) & (np.abs(want) > 1e-290)
    # two roundings more: the product's, and half of the reciprocal's unit
    assert (np.abs(q[fin] / want[fin] - 1) <= 2.0 ** -51).all()
    far = (b < 2.0 ** -100) | (b >= 2.0 ** 100) | np.isnan(b)
    np.testing.assert_array_equal(q[far], want[far])


def test_inverse_square_root(run):
    x = np.concatenate([_positive(200000, -1000, 1000, 6), _positive(200000, -100, 100, 7)])
    want = 1 / np.sqrt(x.astype(np.longdouble))
    # 2^-53 of the last multiply-add, half of that of y^2 (it enters e, and y (1 + e/2) half
    # of e) and 2^-58 of the series
    assert (np.abs(run(6, x) / want - 1) <= 2.0 ** -52).all()
    x = np.concatenate([x, SPECIAL])
    outside = ~((x >= 2.0 ** -100) & (x < 2.0 ** 100))
    np.testing.assert_array_equal(run(6, x)[outside], run(7, x)[outside])


def test_narrow_and_widen(run):
    x = np.concatenate([_positive(100000, -126, 127, 4) * np.resize([1.0, -1.0], 100000)])
    got = run(2, x)
    # toward zero: the leading 24 bits
    want = (x.view(np.int64) & ~np.int64((1 << 29) - 1)).view(np.float64)
    np.testing.assert_array_equal(got, want)
    assert not run(2, np.ldexp([1.0, 1.99, -1.5], -127)).any()
    np.testing.assert_array_equal(run(2, [0.0, 5e-324, 2.0 ** 128, -1e300, np.inf, -np.inf, np.nan]),
                                  [0.0, 0.0, np.inf, -np.inf, np.inf, -np.inf, np.nan])
    a, b = np.array([1.0, -3.0, 0.0, np.inf, 2.0]), np.array([-2.0, 1.0, -0.0, 1.0, np.nan])
    np.testing.assert_array_equal(run(4, a, b), [2.0, 3.0, 0.0, np.inf, np.nan])


def test_step_factor(run):
    q = np.concatenate([_positive(200000, -60, 60, 5), [1e-300, 1e-12, 1e12, 1e300, 0.0],
                        np.array([5.0, 0.2]) ** -10 * 0.9 ** 10, [1.0]])
    with np.errstate(divide="ignore"):
        want = np.clip(0.9 * q.astype(np.longdouble) ** np.longdouble(-0.1), 0.2, 5.0)
    # the series' remainder is below 1e-17, the tenth power's rounding below 3 units of
    # 2^-53, divided by ten; the estimate's own products add two
    got = run(3, q, np.ones_like(q))
    assert (np.abs(got / want - 1) <= 1e-15).all()
    assert (got >= 0.2).all() and (got <= 5.0).all()
    np.testing.assert_array_equal(run(3, q, np.zeros_like(q)), np.minimum(got, 1.0))


@pytest.mark.parametrize("tail,rotation", [(1, 0), (31, 0), (0, 1)])
def test_subnormal_absolute_tolerance(tail, rotation):
    """Rays in the plane of the axis keep y = k_y = 0 exactly: their error scale is atol
    alone, and 0 / atol is 0 however small atol is."""
    kw = dict(I.star_config0(), phase_mode=0, psi=0.0, theta_m=0.0, rotation=rotation)
    u = I.sample_uniforms(4, 64)
    star, st0, w, s0, _ = G.gpu_sample(kw, u)
    st0[1] = 0.0
    st0[4] = 0.0
    out = []
    for atol in (1e-290, 1e-310, 5e-324):
        st, s = st0.clone(), s0.clone()
        rt.rt_trace_forward(star, 64, st, s, opts=rt.make_opts(rtol=1e-6, atol=atol, tail=tail,
                                                               max_steps=2000))
        out.append((st, s))
    assert (out[0][1] == rt.RAY_ESCAPED).any()
    for st, s in out[1:]:
        assert torch.equal(s, out[0][1]) and torch.equal(st, out[0][0])
