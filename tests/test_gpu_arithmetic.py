"""Pieces of the kernels' device arithmetic on arrays, against NumPy."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2008_11607_gb300 import build as B
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def device(tmp_path_factory):
    torch = torch_cuda()
    so = str(tmp_path_factory.mktemp("arithmetic") / "device_arithmetic.so")
    subprocess.run([B.nvcc(), "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(B.ROOT, "include"),
                    "-I", B.CSRC, os.path.join(HERE, "device_arithmetic.cu"), "-o", so] + B.ARCH, check=True)
    lib = ctypes.CDLL(so)

    def call(name, n, *arrays, out):
        dev = [torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda() for a in arrays]
        res = torch.zeros(out, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert getattr(lib, name)(n, *[ctypes.c_void_p(d.data_ptr()) for d in dev], ctypes.c_void_p(res.data_ptr())) == 0
        return res.cpu().numpy()

    return call


def _monomials(f):
    """Monomial coefficients of the polynomial of degree 15 through f at Chebyshev nodes."""
    x = np.cos(math.pi * (2 * np.arange(16) + 1) / 32)
    return np.polynomial.chebyshev.cheb2poly(np.polynomial.chebyshev.chebfit(x, f(x), 15))


POLYNOMIALS = {
    # one pole at the nearest distance that a cell has, 5.13 half-widths
    "pole": (_monomials(lambda t: 1.0 / (5.13 ** 2 + t * t)), _monomials(lambda t: t / (5.13 ** 2 + t * t))),
    # e^{ix} on the half-widths 1/2 (h = 0.5), 1 and 2 (h = 2)
    "wave_half": (_monomials(lambda t: np.cos(0.5 * t)), _monomials(lambda t: np.sin(0.5 * t))),
    "wave_one": (_monomials(np.cos), _monomials(np.sin)),
    "wave_two": (_monomials(lambda t: np.cos(2.0 * t)), _monomials(lambda t: np.sin(2.0 * t))),
}


@pytest.mark.parametrize("name", sorted(POLYNOMIALS))
def test_cell_polynomial_in_pairs(device, name):
    """Horner's rule of degree n = 15 in double-float (u = 2^-47): within gamma_2n sum |c_i t^i|
    (Higham, Accuracy and Stability of Numerical Algorithms, Section 5.1), and n + 1 more
    roundings for the factors t and the coefficient."""
    re, im = POLYNOMIALS[name]
    t = np.linspace(-1.0, 1.0, 4001)
    got = device("device_horner", len(t), re, im, t, out=(len(t), 2))
    for c, v in ((re, got[:, 0]), (im, got[:, 1])):
        ref = np.polynomial.polynomial.polyval(t.astype(np.longdouble), c.astype(np.longdouble))
        bound = 46 * 2.0 ** -47 * np.polynomial.polynomial.polyval(np.abs(t), np.abs(c))
        assert np.all(np.abs(v - ref) <= bound + 2.0 ** -126)  # and the least that FP32 holds


def test_reciprocal_and_roots_over_their_exponents(device):
    """rcp64 and sqrt_rsqrt64 against NumPy's correctly rounded 1 / x and sqrt(x) in extended
    precision: one unit in the last place, 2^-52 relative (half of it the final rounding, the
    rest the residual's rounding and the seed's third-order remainder, 2^-57)."""
    rng = np.random.default_rng(5)
    ends = [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, math.sqrt(2.0)]
    m = np.concatenate([rng.uniform(1.0, 2.0, 100000), np.repeat(ends, 400)])
    e = np.concatenate([rng.integers(-929, 930, 100000), np.tile(np.linspace(-929, 929, 400).astype(int), len(ends))])
    x = np.concatenate([np.ldexp(m, e), rng.uniform(0.1, 1e7, 100000)])  # the last: what the sums meet
    assert x.min() > 1e-280 and x.max() < 1e280
    got = device("device_reciprocals", len(x), x, out=(len(x), 3))
    X = x.astype(np.longdouble)
    for v, ref in zip(got.T, (1.0 / X, np.sqrt(X), 1.0 / np.sqrt(X))):
        assert np.max(np.abs(v - ref) / ref) <= 2.0 ** -52
