"""The FP64 arithmetic the kernels carry themselves, against exact values: the
reciprocal and inverse root from the hardware's estimate, the half-range moments
on both sides of |z| = 1, and the integer conversions between FP32 and FP64
against the conversion instructions, pattern by pattern."""
import ctypes as C
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
U = 2.0 ** -53


@pytest.fixture(scope="module")
def arith(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_09965_gb300 import build
    so = str(tmp_path_factory.mktemp("arith") / "arith.so")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC,
                    "-I", os.path.join(ROOT, "include"), "-o", so, os.path.join(HERE, "arith.cu")], check=True)
    return C.CDLL(so)


def ptr(t):
    return C.c_void_p(t.data_ptr())


def sample(rng, n, lo, hi):
    """Positive doubles, exponents lo to hi, with mantissas about the ends."""
    m = np.concatenate([rng.random(n), 1.0 - 2.0 ** -rng.uniform(20, 52, n // 4), 2.0 ** -rng.uniform(20, 52, n // 4),
                        np.zeros(n // 4)])
    return (1.0 + m) * 2.0 ** rng.integers(lo, hi + 1, m.size).astype(float)


def test_reciprocal_and_inverse_root(arith):
    """The estimate has 20 mantissa bits of an argument cut to 20, so e is at
    most 2^-19 (2^-18 for the root, whose residual has r squared).  The rest of
    the third-order step is then e^3 = 2^-57 and 5/16 e^3 = 2^-55.7; the last
    rounding adds 2^-53 and, for the root, the product x r another 2^-54."""
    import torch
    rng = np.random.default_rng(3)
    x = sample(rng, 400000, -1020, 1020)
    x[:2000] = np.arange(1, 2001)
    for sign in (1.0, -1.0):
        d = torch.from_numpy(sign * x).cuda()
        r, q = torch.empty_like(d), torch.empty_like(d)
        assert arith.arith_recip(x.size, ptr(d), ptr(r), ptr(q)) == 0
        r, q, X = r.cpu().numpy(), q.cpu().numpy(), x.astype(np.longdouble)
        assert np.abs(r * (sign * X) - 1).max() < 1.1 * U
        if sign > 0:
            assert np.abs(q * np.sqrt(X) - 1).max() < 2 * U
        else:
            assert np.isnan(q).all()


def exact_half(z):
    """erfc(-z) / 2 and exp(-z^2) of a double to 50 digits."""
    getcontext().prec = 80
    z = Decimal(float(z))
    t = z * z
    term, total, k = z, z, 0
    while abs(term) > Decimal(10) ** -75:
        k += 1
        term = -term * t / k
        total += term / (2 * k + 1)
    pi = Decimal("3.14159265358979323846264338327950288419716939937510582097494459230781640628620899862803")
    return (1 + 2 * total / pi.sqrt()) / 2, (-t).exp()


def test_half_range_moments(arith):
    """m0 = (1 +- erf z) / 2 and m1 = U m0 +- exp(-z^2) / (2 sqrt(pi lambda))
    over u > 0 and u < 0.  Below |z| = 1 m0 is 0.5 plus a product: absolute
    errors (four units, 2^-53 each, of the sum's, the product's and the
    polynomial's roundings).  Beyond, the library's erfc (5 ulp at most by its
    documentation) is as accurate relative to itself; its argument z is the same
    double here.  exp(-t) of a rounded t moves by t units."""
    import torch
    rng = np.random.default_rng(5)
    th = 10.0 ** rng.uniform(-3, 3, 600)
    z = np.concatenate([rng.uniform(-1, 1, 250), rng.uniform(-5, 5, 200), 1.0 + rng.uniform(-1e-3, 1e-3, 50),
                        -1.0 + rng.uniform(-1e-3, 1e-3, 50), 10.0 ** rng.uniform(-18, -1, 47), [0.0, -0.0, 1.0]])
    u = z * np.sqrt(2.0 * th)
    u[-1] = np.nextafter(np.sqrt(2.0 * th[-1]), 10)
    du, dt, out = torch.from_numpy(u).cuda(), torch.from_numpy(th).cuda(), torch.empty((600, 6), dtype=torch.float64,
                                                                                      device="cuda")
    assert arith.arith_half(600, ptr(du), ptr(dt), ptr(out)) == 0
    for k, (sl, isp, p0, p1, n0, n1) in enumerate(out.cpu().numpy()):
        assert abs(sl * np.sqrt(2 * np.longdouble(th[k])) - 1) < 3 * U
        zz = sl * u[k]                              # the kernel's product
        plus, ex = exact_half(zz)
        t, near = zz * zz, zz * zz < 1.0
        for m0, m1, sgn in ((p0, p1, 1), (n0, n1, -1)):
            e0 = plus if sgn > 0 else 1 - plus
            bar0 = 4 * U if near else 12 * U * float(e0)
            assert abs(Decimal(float(m0)) - e0) <= Decimal(bar0), (zz, sgn)
            e1 = Decimal(float(u[k])) * e0 + sgn * ex * Decimal(float(isp)) / 2
            bar1 = abs(u[k]) * bar0 + 0.5 * isp * float(ex) * (6 + 2 * t) * U + 2 * U * abs(float(e1))
            assert abs(Decimal(float(m1)) - e1) <= Decimal(float(bar1)), (zz, sgn)
    ends = torch.tensor([np.inf, -np.inf, np.nan, 60.0, -60.0], dtype=torch.float64, device="cuda")
    out = torch.empty((5, 6), dtype=torch.float64, device="cuda")
    assert arith.arith_half(5, ptr(ends), ptr(torch.full_like(ends, 0.5)), ptr(out)) == 0
    o = out.cpu().numpy()
    assert o[0, 2] == 1 and o[0, 4] == 0 and o[1, 2] == 0 and o[1, 4] == 1 and np.isnan(o[2, 2:]).all()
    assert o[3, 2] == 1 and o[3, 4] == 0 and o[3, 3] == 60 and o[4, 4] == 1 and o[4, 5] == -60


def test_conversions_are_the_instructions(arith):
    """widen and narrow give the conversion instructions' bits: every FP32
    pattern (signed zeros, subnormals, infinities, NaN payloads), alone and in
    runs; every upper word of an FP64 one with lower words at and about the ties."""
    import torch
    bad = torch.zeros(2, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert arith.arith_conversions(ptr(bad)) == 0
    assert bad.tolist() == [0, 0]
