// Error-free digit splitting for the FP64-accurate tensor-core kernels
// (jk_split.cu, df_split.cu): fixed-point digits of base 512 as FP16, and the
// issue of MMAs whose descriptors live in uniform registers.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "umma.cuh"

namespace esmf {
namespace split {

// Polls after which a wait of these kernels gives up (every wait is far shorter).
constexpr uint32_t POLLS = 1u << 22;
__device__ __forceinline__ bool wait_for(uint64_t *bar, uint32_t parity, const volatile int *abort) {
    return umma::mbar_wait(bar, parity, abort, POLLS);
}

// ---- densities that digits serve: the largest element in [2^DMIN, 2^DMAX), where
// the exponents of all products and the squares behind norms stay in FP64's
// range; top is a density's largest exponent field, 0 for a zero one
constexpr int DMIN = -500, DMAX = 500;
__device__ __forceinline__ bool beyond_digits(int top) {
    return top != 0 && (top > 1022 + DMAX || top <= 1022 + DMIN);
}
// exponent field of x, 1 for subnormal numbers, 0 for zero: |x| < 2^(field - 1022)
__device__ __forceinline__ int field_of(double x) {
    const int f = (__double2hiint(x) >> 20) & 0x7ff;
    return x != 0.0 ? max(f, 1) : 0;
}

// ---- digits.  x 2^(BITS - e) rounded to an integer of magnitude at most
// 2^BITS, for |x| < 2^e, e = emax - 1022 with emax the largest exponent field
// of the tile (at least some minimum, so that sh below stays meaningful).  The shift runs on twice the result,
// so that the last bit shifted out rounds; zeros (exponent field 0) shift out.
template <int BITS>
__device__ __forceinline__ long long fixed_point(uint32_t lo, uint32_t hi, int emax) {
    const int sh = min(emax - (int)((hi >> 20) & 0x7ffu), 63);
    const unsigned long long mant = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const unsigned long long r = (((mant << (BITS - 52)) >> sh) + 1) >> 1;
    const long long sg = (int)hi >> 31;
    return ((long long)r ^ sg) - sg;
}
// the same for one FP32 part of a double-FP32 value; emax counts in FP64 bias
template <int BITS>
__device__ __forceinline__ long long fixed_point_f(float x, int emax) {
    const uint32_t b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xffu);
    const int sh = min(emax - 896 - max(e, 1), 63);      // subnormal parts have the exponent of field 1
    const unsigned long long mant = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
    const unsigned long long r = (((mant << (BITS - 23)) >> sh) + 1) >> 1;
    const long long sg = (int)b >> 31;
    return ((long long)r ^ sg) - sg;
}

// Balanced digits of X, |X| <= 2^(9 N - 1): X + sum_k 256 512^k has the digits
// u_i of base 512 (u_0 up to 512), x_i = u_i - 256.  Words of three digits,
// w[0] = u_0 u_1 u_2 and so on.
template <int N>
__device__ __forceinline__ void digit_words(long long X, uint32_t *w) {
    unsigned long long B = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) B += 256ull << (9 * k);
    const unsigned long long Y = (unsigned long long)X + B;
    w[0] = (uint32_t)(Y >> (9 * N - 27));
    w[1] = (uint32_t)(Y >> (9 * N - 54)) & 0x7ffffffu;
    if (N > 6) w[2] = (uint32_t)Y & 0x1ffu;
}
// digit i of two values as packed FP16: FP16 holds 1024 + u exactly with the
// bits 0x6400 | u, and subtracting 1280 leaves u - 256
template <int I>
__device__ __forceinline__ uint32_t digit_pair(const uint32_t *wa, const uint32_t *wb) {
    constexpr int s = I == 6 ? 0 : 18 - 9 * (I % 3);
    constexpr uint32_t mask = I == 0 ? 0x3ffu : 0x1ffu;
    const uint32_t a = wa[I / 3], b = wb[I / 3];
    const uint32_t u = ((a >> s) & mask) | ((s > 16 ? b >> (s - 16) : b << (16 - s)) & (mask << 16)) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&u), __floats2half2_rn(1280.f, 1280.f));
    return *reinterpret_cast<const uint32_t *>(&h);
}

// a warp-uniform value in a uniform register (the reduction's result is one)
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_or_sync(0xffffffffu, x); }

// MMA issued by the lane whose `lead` is set; descriptors as low and high words
__device__ __forceinline__ void mma_pred(uint32_t lead, uint32_t dtmem, uint32_t alo, uint32_t ahi, uint32_t blo,
                                         uint32_t bhi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p, q;\n.reg .b64 a, b;\nsetp.ne.b32 p, %6, 0;\nsetp.ne.b32 q, %7, 0;\n"
        "mov.b64 a, {%1, %2};\nmov.b64 b, {%3, %4};\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}" ::"r"(dtmem),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate), "r"(lead));
}

}  // namespace split
}  // namespace esmf
