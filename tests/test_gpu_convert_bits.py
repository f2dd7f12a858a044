"""narrow() and widen(), the conversions between double and float in integer arithmetic,
against the casts bit for bit (NaN: against being NaN): rounding ties, carries into the
exponent, both ends of float's normal range, zeros of both signs, subnormals, infinities
and NaN, alone and beside ordinary numbers.  A CUDA program around the library's header,
16 M groups of four numbers of pseudo-random bits bent into those classes."""
import shutil
import subprocess

import pytest

from paper_1011_0911_gb300 import build_lib

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "lqcd_internal.cuh"
typedef unsigned long long u64;
constexpr int NCLASS = 10;
__device__ u64 bits(u64 &z)   // SplitMix64
{
    u64 y = (z += 0x9E3779B97F4A7C15ull);
    y = (y ^ (y >> 30)) * 0xBF58476D1CE4E5B9ull;
    y = (y ^ (y >> 27)) * 0x94D049BB133111EBull;
    return y ^ (y >> 31);
}
__device__ double number(int cls, u64 y)
{
    const u64 sm = 0x800fffffffffffffull;   // sign and mantissa
    const u64 e = y >> 52;
    switch (cls) {
        case 0: y = (y & sm) | (0x3e0 + e % 64) << 52; break;                              // ordinary
        case 1: y = (y & sm) | (0x380 + e % 3) << 52; break;                               // 2^-127 .. 2^-124
        case 2: y = (y & sm) | (0x47d + e % 3) << 52; break;                               // 2^126 .. 2^129
        case 3: y = (y & (sm & ~0x1fffffffull)) | 0x10000000ull | (0x3e0 + e % 64) << 52; break;   // ties
        case 4: y = (y & 0x8000000000000000ull) | 0x000fffffe0000000ull | (y & 0x1fffffffull) |    // carries,
                    (0x381 + e % 254) << 52; break;                                        // the last to infinity
        case 5: y = (y & sm) | (0x360 + e % 32) << 52; break;                              // subnormal floats and less
        case 6: y &= sm; break;                                                            // subnormal doubles
        case 7: y &= 0x8000000000000000ull; break;                                         // zeros
        case 8: y = (y & 0x8000000000000000ull) | 0x7ff0000000000000ull; break;            // infinities
        default: y = (y & sm) | 0x7ff0000000000001ull; break;                              // NaN
    }
    return __longlong_as_double((long long)y);
}
__global__ void check(u64 *bad)
{
    u64 z = (blockIdx.x * (u64)blockDim.x + threadIdx.x) << 20;
    for (int it = 0; it < 64; it++) {
        double x[4];
        float f[4], g[4];
        const u64 r = bits(z);
        // three of four groups hold one class beside ordinary numbers, the fourth any
        for (int i = 0; i < 4; i++) {
            const int any = (int)((r >> (8 * i)) % NCLASS);
            x[i] = number((r >> 62) == 3 || (int)(r >> 60 & 3) == i ? any : 0, bits(z));
            // floats: the casts of the same numbers, and any bits
            g[i] = (it & 1) ? (float)x[i] : __uint_as_float((unsigned)bits(z));
        }
        narrow(x, f);
        for (int i = 0; i < 4; i++) {
            const float want = (float)x[i];
            if (want == want ? __float_as_uint(f[i]) != __float_as_uint(want) : f[i] == f[i]) atomicAdd(bad, 1ull);
        }
        double w[4];
        widen(g, w);
        for (int i = 0; i < 4; i++) {
            const double want = (double)g[i];
            if (want == want ? __double_as_longlong(w[i]) != __double_as_longlong(want) : w[i] == w[i])
                atomicAdd(bad + 1, 1ull);
        }
    }
}
int main()
{
    u64 *d, h[2];
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
    check<<<1024, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_same_bits_as_the_casts(tmp_path):
    src, exe = tmp_path / "convert.cu", tmp_path / "convert"
    src.write_text(PROGRAM)
    subprocess.run(["nvcc"] + build_lib.ARCH + build_lib.FLAGS + [str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "0"]
