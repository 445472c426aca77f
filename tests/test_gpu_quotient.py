"""The sponge's quotient (quot1, quot2 in csrc/stencil.cuh) against the division,
bit for bit, over normal, subnormal, huge and non-finite numerators, subnormal
quotients, quotients within two units of a tie, and divisors from just above 1
to 2^20 (and just below 1, where an absorbing layer with R > 1 lies). The
header is compiled here into a small kernel."""
import ctypes
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "stencil.cuh"
using namespace gsim;
__device__ unsigned mix(unsigned long long x) {
    x ^= x >> 33; x *= 0xff51afd7ed558ccdULL; x ^= x >> 33; x *= 0xc4ceb9fe1a85ec53ULL; x ^= x >> 33;
    return (unsigned)x;
}
__device__ float unit(unsigned r) { return (r >> 8) * 0x1p-24f; }  // [0, 1)
__device__ float divisor(int kind, unsigned r) {
    switch (kind) {
        case 0: return 1.f + 5.f * unit(r);
        case 1: return 1.f + (r & 63) * 0x1p-23f;
        case 2: return ldexpf(1.f + unit(r), r % 20);
        default: return 1.f - 0.5f * unit(r);
    }
}
__device__ float numerator(int kind, unsigned r, unsigned s, float d) {
    switch (kind) {
        case 0: return __uint_as_float(r);                                       // any bits
        case 1: return __uint_as_float((r & 0x80000000u) | (r & 0x03ffffffu));   // below 2^-118
        case 2: {                                                                // near a tie of the quotient
            const float q = __uint_as_float((0x3f800000u + ((s % 40u) << 23)) | (r & 0x7fffffu));
            const double m = ((double)q + 0.5 * ldexp(1.0, ilogbf(q) - 23)) * d;
            return __uint_as_float(__float_as_uint((float)m) + (s >> 8) % 5u - 2u);
        }
        case 3: {                                                                // near a tie of a subnormal quotient
            const double m = ((r >> 8) % 0x1000000u + 0.5) * 0x1p-149 * d;
            return __uint_as_float(__float_as_uint((float)m) + (s >> 8) % 5u - 2u);
        }
        case 4: return __uint_as_float(r & 31u);                                 // the smallest
        default: return __uint_as_float((r & 0x80000000u) | 0x6b800000u | (r & 0x17ffffffu));  // 2^88 and more
    }
}
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (a != a && b != b); }
__global__ void check(int tk, int dk, unsigned long long seed, unsigned long long n, unsigned long long *bad) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned a = mix(seed + 4 * i), b = mix(seed + 4 * i + 1), c = mix(seed + 4 * i + 2), e = mix(seed + 4 * i + 3);
        const float d0 = divisor(dk, a), d1 = divisor(dk, b), t0 = numerator(tk, c, e, d0), t1 = numerator(tk, e, c, d1);
        const float r0 = t0 / d0, r1 = t1 / d1;
        const float2 q = quot2(make_float2(t0, t1), make_float2(d0, d1), make_float2(1.f / d0, 1.f / d1));
        if (!same(quot1(t0, d0), r0) || !same(quot1(t1, d1), r1) || !same(q.x, r0) || !same(q.y, r1)) atomicAdd(bad, 1ULL);
    }
}
extern "C" int run(int tk, int dk, unsigned long long seed, unsigned long long n, void *bad) {
    check<<<1216, 256>>>(tk, dk, seed, n, static_cast<unsigned long long *>(bad));
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2605_30541_gb300 import build as b
    d = tmp_path_factory.mktemp("quotient")
    src, lib = str(d / "quotient.cu"), str(d / "quotient.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([b._nvcc()] + b.ARCH + b.FLAGS + ["-I", b.CSRC, "-shared", src, "-o", lib], check=True)
    fn = ctypes.CDLL(lib).run
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_ulonglong, ctypes.c_ulonglong, ctypes.c_void_p]

    def mismatches(tk, dk, n):
        bad = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        assert fn(tk, dk, 1000003 * (8 * tk + dk), n, bad.data_ptr()) == 0
        return int(bad.item())
    return mismatches


@pytest.mark.parametrize("numerators", ["any", "small", "tie", "subnormal tie", "smallest", "huge"])
@pytest.mark.parametrize("divisors", ["[1, 6)", "just above 1", "[1, 2^20)", "(0.5, 1]"])
def test_is_the_division(run, numerators, divisors):
    tk = ["any", "small", "tie", "subnormal tie", "smallest", "huge"].index(numerators)
    dk = ["[1, 6)", "just above 1", "[1, 2^20)", "(0.5, 1]"].index(divisors)
    assert run(tk, dk, 1 << 26) == 0
