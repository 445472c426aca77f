"""Rounding error of the FP64 band-passed wavelet (csrc/wavelet.cu): against the
same definition in extended precision (numpy's long double) with the library's
own FP64 coefficients, the scan is no further off than the plain FP64 recursion
in transposed direct form with a zero at 1 and one at -1 in every section, one
sample after another: the production bands, finer time steps, other orders and
bands over several octaves; and it stays within 1e-13 of the peak (a host model
of it has at most 2.4e-14). The coefficients come from the library's source,
compiled here with a small wrapper."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import wavelet as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2605_30541_gb300 as p
    p.abi.load()
    return p


@pytest.fixture(scope="module")
def design(pkg, tmp_path_factory):
    from paper_2605_30541_gb300 import build as b
    d = tmp_path_factory.mktemp("design")
    src, lib = str(d / "design.cu"), str(d / "design.so")
    with open(src, "w") as f:
        f.write('#include "wavelet.cu"\n'
                'void gsim::set_thread_error(const char *) {}\n'
                'extern "C" void design(int n, double lo, double hi, double fs, double *out) {\n'
                '    const auto s = gsim::butter_bandpass(n, lo, hi, fs);\n'
                '    *out++ = s[0].b0;\n'
                '    for (const auto &q : s) *out++ = q.a1, *out++ = q.a2;\n}\n')
    subprocess.run([b._nvcc()] + b.ARCH + b.FLAGS + ["-I", b.CSRC, "-shared", src, "-o", lib], check=True)
    fn = ctypes.CDLL(lib).design
    fn.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_double, ctypes.c_void_p]

    def coefficients(order, lo, hi, fs):
        out = np.zeros(1 + 2 * order)
        fn(order, lo, hi, fs, out.ctypes.data)
        return out[0], out[1::2], out[2::2]
    return coefficients


def wavelet(T, order, lo, hi, f0, dt, nt, coef):
    """The definition with all arithmetic in type T."""
    g, a1, a2 = (np.asarray(c).astype(T) for c in coef)
    pi = T(3.14159265358979323846) if T is np.float64 else 4 * np.arctan(T(1))
    pad = 3 * (2 * order + 1)
    a = (pi * T(f0) * (np.arange(nt).astype(T) * T(dt) - 1 / T(f0))) ** 2
    x = (1 - 2 * a) * np.exp(-a)
    x = np.concatenate([2 * x[0] - x[pad:0:-1], x, 2 * x[-1] - x[-2:-pad - 2:-1]])
    for _ in range(2):
        z1, z2, out = [T(0)] * order, [T(0)] * order, np.empty_like(x)
        z1[0] = z2[0] = -g * x[0]
        for i in range(len(x)):
            v = g * x[i]
            for k in range(order):
                y = v + z1[k]
                z1[k], z2[k], v = z2[k] - a1[k] * y, -v - a2[k] * y, y
            out[i] = v
        x = out[::-1]
    x = x[pad:pad + nt]
    return x * (np.sqrt((T(hi) - T(lo)) / 24) / np.sqrt(np.sum(x * x)))


@pytest.mark.parametrize("order,lo,hi,f0,dt,nt", [(4, *b, 1e-3, 8001) for b in W.BANDS] +
                         [(4, 3.0, 6.0, 4.5, 2.5e-4, 16001), (4, 3.0, 6.0, 4.5, 1e-4, 40001), (4, 5.0, 200.0, 80.0, 1e-3, 3001),
                          (2, 3.0, 12.0, 7.5, 1e-3, 8001), (8, 3.0, 12.0, 7.5, 1e-3, 8001), (12, 3.0, 25.0, 14.0, 1e-3, 8001),
                          (16, 3.0, 25.0, 14.0, 1e-3, 8001), (4, 2.0, 1500.0, 10.0, 2.5e-4, 4777),
                          (8, 2.0, 1500.0, 10.0, 2.5e-4, 4777), (16, 5.0, 400.0, 20.0, 1e-3, 4000), (3, 3.0, 15.0, 8.0, 2.5e-4, 3001),
                          (5, 100.0, 180.0, 140.0, 1e-3, 2000), (1, 3.0, 12.0, 7.5, 1e-3, 1001)])
def test_no_further_off_than_the_plain_recursion(pkg, design, order, lo, hi, f0, dt, nt):
    coef = design(order, lo, hi, 1.0 / dt)
    ref = wavelet(np.longdouble, order, lo, hi, f0, dt, nt, coef)
    plain = wavelet(np.float64, order, lo, hi, f0, dt, nt, coef)
    g = pkg.bandpass_ricker(nt, dt, f0, lo, hi, order=order, dtype="float64").cpu().numpy()
    peak = np.abs(ref).max()
    e, e0 = float(np.abs(g - ref).max() / peak), float(np.abs(plain - ref).max() / peak)
    print("order %d %g-%g Hz dt %g nt %d: plain %.1e scan %.1e" % (order, lo, hi, dt, nt, e0, e))
    assert e <= min(e0, 1e-13)
