// FP64 values as integers relative to a power of two: the conversions shared by the emulated
// products (oz_gemm.cu) and the fixed-point factorisation (ldl_fix.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace thc {

constexpr int kNanExp = 1 << 20;             // exponent of a NaN or an infinity
constexpr int kZeroExp = -5000;              // exponent of a zero

// Exponent E of a double, |x| in [2^(E-1), 2^E); kZeroExp for zero, kNanExp for inf and NaN.
__device__ __forceinline__ int dbl_exp(double x) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF);
    if (ex == 0x7FF) return kNanExp;
    if (ex == 0) {
        const long long m = b & 0xFFFFFFFFFFFFFLL;
        return m ? 64 - __clzll(m) - 1074 : kZeroExp;
    }
    return ex - 1022;
}

// round(x 2^(62 - e)) for |x| < 2^e, formed exactly from the bits of x (|.| <= 2^62); a value that
// is too large, a NaN or an infinity gives some value.
__device__ __forceinline__ long long fixed62(double x, int e) {
    const long long b = __double_as_longlong(x);
    int ex = (int)((b >> 52) & 0x7FF);
    long long m = b & 0xFFFFFFFFFFFFFLL;
    if (ex)
        m |= 1LL << 52;
    else
        ex = 1;
    const int sh = (ex - 1022) - e + 9;  // <= 9 for a normal x (a subnormal m has fewer bits)
    long long X = 0;
    if (sh >= 0)
        X = (long long)((unsigned long long)m << min(sh, 62));
    else if (sh > -54)
        X = (m + (1LL << (-sh - 1))) >> (-sh);
    return b < 0 ? -X : X;
}

// The eight signed base-256 digits of four fixed-point values (|X| <= 2^62), as BF16, written to
// out[a * stride .. + 3]. Adding 128 to every byte carries the signed digits out: digit a is then
// byte 7 - a minus 128, and an integer byte becomes a float without a conversion instruction as
// (2^23 + byte) - (2^23 + 128).
__device__ __forceinline__ void store_fixed4(const long long (&X)[4], uint16_t* __restrict__ out, size_t stride) {
    unsigned long long w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = (unsigned long long)X[i] + 0x8080808080808080ULL;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int byte = 7 - a;
        float f[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t half = byte < 4 ? (uint32_t)w[i] : (uint32_t)(w[i] >> 32);
            f[i] = __uint_as_float(__byte_perm(half, 0x4B000000u, 0x7440 + (byte & 3))) - 8388736.0f;
        }
        uint2 p;
        p.x = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);
        p.y = __byte_perm(__float_as_uint(f[2]), __float_as_uint(f[3]), 0x7632);
        *reinterpret_cast<uint2*>(out + (size_t)a * stride) = p;
    }
}

}  // namespace thc
