// Helpers of the inverse paths of gbs_dequantize (gbs_tc_uvinv.cu, gbs_rowinv.cu): packed codes -> packed halves without a
// conversion instruction, exact half-precision butterfly steps, and the stores of scaled values.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace {

__device__ __forceinline__ unsigned hadd2(unsigned a, unsigned b)
{
    unsigned d;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ unsigned hsub2(unsigned a, unsigned b)
{
    unsigned d;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ unsigned hmul2(unsigned a, unsigned b)
{
    unsigned d;
    asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ unsigned hfma2(unsigned a, unsigned b, unsigned c)
{
    unsigned d;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// -a, which an addition or FMA takes as a modifier of its operand
__device__ __forceinline__ unsigned hneg2(unsigned a)
{
    unsigned d;
    asm("neg.f16x2 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
// (lo, hi) -> (lo + hi, lo - hi)
__device__ __forceinline__ unsigned hpair(unsigned v)
{
    const __half2 h = *reinterpret_cast<const __half2*>(&v);
    const __half2 r = __hfma2(__high2half2(h), __halves2half2(__ushort_as_half(0x3c00), __ushort_as_half(0xbc00)), __low2half2(h));
    return *reinterpret_cast<const unsigned*>(&r);
}

// Codes 8 o .. 8 o + 7 of a row segment of NW packed words -> four halves' pairs (code 8 o + i, code 8 o + 4 + i), i < 4, after the
// butterflies over i (H_4).  Each half is the integer q + 2^(b-1) (UNSIGNED_FIELDS: the code itself) times 2^-24: a field in the
// low bits of a subnormal; LIFT: times 2^-10 instead, which the first stage brings in.
// Fields are masked where they stand, and where one stands higher than bit 0 the multiplication of an FMA in the first stages
// takes the power of two out again (exact): one shift per eight codes instead of three, and no separate pass to lift the halves.
// 8192 x 3584, 3 bits, groups of 128 -> bf16: 27.5 -> 27.0 us; groups of 32: 28.1 -> 27.5; 262 144 x 128, 4 bits: 19.16 -> 19.10.
template <int BITS, bool UNSIGNED_FIELDS, int NW, bool LIFT>
__device__ __forceinline__ void rotate_octet(const unsigned* w, int o, unsigned h[4])
{
    constexpr unsigned NEG = 0x80008000u;
    if (BITS == 4) {
        constexpr unsigned F = LIFT ? 0x64006400u : 0x2c002c00u;             // 2^14 or 1, over the 2^4 that b and d stand high
        const unsigned x = w[o] ^ (UNSIGNED_FIELDS ? 0u : 0x88888888u), y = x >> 8;
        unsigned a = x & 0x000f000fu, c = y & 0x000f000fu;
        const unsigned b = x & 0x00f000f0u, d = y & 0x00f000f0u;
        if (LIFT) { a = hmul2(a, 0x74007400u); c = hmul2(c, 0x74007400u); }
        const unsigned s0 = hfma2(b, F, a), s1 = hfma2(b, F ^ NEG, a), s2 = hfma2(d, F, c), s3 = hfma2(d, F ^ NEG, c);
        h[0] = hadd2(s0, s2); h[1] = hadd2(s1, s3); h[2] = hsub2(s0, s2); h[3] = hsub2(s1, s3);
    } else {
        constexpr unsigned F = LIFT ? 0x68006800u : 0x30003000u;             // 2^14 or 1, over 2^3
        constexpr unsigned G = LIFT ? 0x5c005c00u : 0x24002400u;             // the same over 2^6
        const int at = 24 * (o & 3), k = 3 * (o >> 2) + (at >> 5);
        const unsigned g = (at & 31) == 0 ? w[k] : ((o & 3) == 3 ? w[k] >> 8 : __funnelshift_r(w[k], w[k + 1 < NW ? k + 1 : k], at & 31));
        const unsigned x = ((g & 0xfffu) | ((g << 4) & 0x0fff0000u)) ^ (UNSIGNED_FIELDS ? 0u : 0x09240924u);
        unsigned a = x & 0x00070007u;
        const unsigned b = x & 0x00380038u, c = x & 0x01c001c0u, d = (x >> 3) & 0x01c001c0u;
        if (LIFT) a = hmul2(a, 0x74007400u);
        const unsigned s0 = hfma2(b, F, a), s1 = hfma2(b, F ^ NEG, a), s2 = hadd2(c, d), s3 = hsub2(c, d);
        h[0] = hfma2(s2, G, s0); h[1] = hfma2(s3, G, s1); h[2] = hfma2(s2, G ^ NEG, s0); h[3] = hfma2(s3, G ^ NEG, s1);
    }
}

// sixteen values as the output type's words
__device__ __forceinline__ void pack_values(const float f[16], unsigned w[16], float)
{
#pragma unroll
    for (int e = 0; e < 16; ++e) w[e] = __float_as_uint(f[e]);
}
__device__ __forceinline__ void pack_values(const float f[16], unsigned w[16], __nv_bfloat16)
{
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
        w[e] = *reinterpret_cast<const unsigned*>(&b2);
    }
}

// 32 bytes: one store where the address allows (a full DRAM sector per thread), else two
__device__ __forceinline__ void store32(void* p, const unsigned w[8], bool wide)
{
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                     "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
    } else {
        reinterpret_cast<uint4*>(p)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(p)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

// dst[i] = f[i], N a multiple of 16
template <int N>
__device__ __forceinline__ void store_values(float* dst, const float f[N], bool wide)
{
#pragma unroll
    for (int c = 0; c < N / 8; ++c) {
        unsigned w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(f[8 * c + e]);
        store32(dst + 8 * c, w, wide);
    }
}
template <int N>
__device__ __forceinline__ void store_values(__nv_bfloat16* dst, const float f[N], bool wide)
{
#pragma unroll
    for (int c = 0; c < N / 16; ++c) {
        unsigned w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(f[16 * c + 2 * e], f[16 * c + 2 * e + 1]);
            w[e] = *reinterpret_cast<const unsigned*>(&b2);
        }
        store32(dst + 16 * c, w, wide);
    }
}

}  // namespace
