"""The exact mode's straight-line division, square root and branch-free series
against CUDA's IEEE operations and the series in their plain form, bit for bit:
over every significand, every uniform, and every float where that is the domain."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2012_14332_gb300 import build as _build  # noqa: E402

_SRC = r"""
#include "abc_model.cuh"
using namespace abcgb;
using namespace abcgb::exact;
namespace plain {
__device__ float log2x(float x)
{
    const uint32_t b = __float_as_uint(x);
    int e = (int)(b >> 23) - 127;
    float m = __uint_as_float((b & 0x007FFFFFu) | 0x3F800000u);
    if (m > 0x1.6a09e6p+0f) { m = m * 0.5f; e += 1; }
    const float s = __fdiv_rn(__fsub_rn(m, 1.0f), __fadd_rn(m, 1.0f)), s2 = __fmul_rn(s, s);
    const float q = madd(madd(madd(madd(kL9, s2, kL7), s2, kL5), s2, kL3), s2, kL1);
    return __fadd_rn((float)e, __fmul_rn(s, q));
}
__device__ float exp2x(float y)
{
    if (!(y < 127.5f)) return __int_as_float(0x7F800000);
    if (y < -125.5f) return 0.0f;
    const float kf = rintf(y), t = __fmul_rn(__fsub_rn(y, kf), kLn2);
    const float q = madd(madd(madd(madd(madd(madd(madd(kE7, t, kE6), t, kE5), t, kE4), t, kE3), t, kE2), t, 1.f), t, 1.f);
    return __fmul_rn(q, __uint_as_float((uint32_t)((int)kf + 127) << 23));
}
__device__ void sincospix(float v, float& s_out, float& c_out)
{
    const float qf = rintf(__fmul_rn(v, 2.0f)), w = __fsub_rn(v, __fmul_rn(qf, 0.5f));
    const float t = __fmul_rn(w, kPi), t2 = __fmul_rn(t, t);
    const float sn = __fadd_rn(__fmul_rn(t, __fmul_rn(madd(madd(madd(kS9, t2, kS7), t2, kS5), t2, kS3), t2)), t);
    const float cs = __fadd_rn(__fmul_rn(madd(madd(madd(madd(kC10, t2, kC8), t2, kC6), t2, kC4), t2, kC2), t2), 1.0f);
    switch ((int)qf & 3) {
    case 0: s_out = sn; c_out = cs; break;
    case 1: s_out = cs; c_out = -sn; break;
    case 2: s_out = -sn; c_out = -cs; break;
    default: s_out = -cs; c_out = sn; break;
    }
}
}
__device__ bool differ(float a, float b) { return __float_as_uint(a) != __float_as_uint(b) && !(a != a && b != b); }
__device__ uint32_t mix(uint32_t h) { h ^= h >> 16; h *= 0x7FEB352Du; h ^= h >> 15; h *= 0x846CA68Bu; return h ^ h >> 16; }
__global__ void check(unsigned long long* bad)
{
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x, first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long n[8] = {};
    for (uint64_t i = first; i < (1ull << 24); i += step) {
        const uint32_t m = (uint32_t)i & 0x7FFFFFu;
        const float b = __uint_as_float(0x3F800000u + (uint32_t)i);                     // [1, 4)
        n[0] += differ(exact::rcp_rn(b), __frcp_rn(b));
        for (int e = -60; e <= 58; e += 59) n[1] += differ(exact::sqrt_rn(ldexpf(b, e & ~1)), __fsqrt_rn(ldexpf(b, e & ~1)));
        if (i < (1u << 23)) {
            const float f = __uint_as_float(m + 0x3F3504F4u);                           // log2x's (sqrt 1/2, sqrt 2]
            n[2] += differ(exact::div_rn(f - 1.0f, f + 1.0f), __fdiv_rn(f - 1.0f, f + 1.0f));
            const float u = uniform01(m);
            const float r2 = __fmul_rn(kNeg2Ln2, plain::log2x(u));
            n[3] += differ(exact::sqrt_rn(__fmul_rn(kNeg2Ln2, exact::log2x(u))), __fsqrt_rn(r2));
            float s, c, s1, c1;
            exact::sincospix(2.0f * u, s, c);
            plain::sincospix(2.0f * u, s1, c1);
            n[4] += differ(s, s1) + differ(c, c1);
        }
    }
    for (uint64_t i = first; i < (1ull << 32); i += step) {
        const float x = __uint_as_float((uint32_t)i);
        n[5] += differ(exact::exp2x(x), plain::exp2x(x));
        if (x >= 0x1p-126f && x < __int_as_float(0x7F800000)) n[6] += differ(exact::log2x(x), plain::log2x(x));
        // a pair of the quotient's range: random significands, exponents and sign
        const uint32_t p = mix((uint32_t)i), q = mix((uint32_t)i ^ 0x9E3779B9u);
        const float a = __uint_as_float((p & 0x807FFFFFu) | ((67u + (p >> 23) % 120u) << 23));
        const float d = __uint_as_float((q & 0x007FFFFFu) | ((126u + (q >> 23) % 61u) << 23));
        n[7] += differ(exact::div_rn(a, d), __fdiv_rn(a, d));
    }
    for (int k = 0; k < 8; ++k)
        if (n[k]) atomicAdd(bad + k, n[k]);
}
extern "C" int exact_math_check(void* bad) { check<<<1216, 256>>>((unsigned long long*)bad); return (int)cudaDeviceSynchronize(); }
"""


def test_straight_line_forms_equal_the_ieee_ones():
    build_dir = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_build")
    os.makedirs(build_dir, exist_ok=True)
    src, so = os.path.join(build_dir, "exact_math.cu"), os.path.join(build_dir, "libexact_math.so")
    with open(src, "w") as f:
        f.write(_SRC)
    subprocess.check_call([_build.nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-fmad=false", "-std=c++17",
                           "-I", _build.CSRC, "-shared", "-Xcompiler", "-fPIC", "-o", so, src])
    bad = torch.zeros(8, dtype=torch.int64, device="cuda")
    assert ctypes.CDLL(so).exact_math_check(ctypes.c_void_p(bad.data_ptr())) == 0
    names = ("reciprocal", "square root", "log2 quotient", "Box-Muller radius", "sin and cos", "exp2", "log2", "quotient")
    assert dict(zip(names, bad.tolist())) == dict.fromkeys(names, 0)
