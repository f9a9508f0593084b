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
// (lo, hi) -> (lo + hi, lo - hi)
__device__ __forceinline__ unsigned hpair(unsigned v)
{
    const __half2 h = *reinterpret_cast<const __half2*>(&v);
    const __half2 r = __hfma2(__high2half2(h), __halves2half2(__ushort_as_half(0x3c00), __ushort_as_half(0xbc00)), __low2half2(h));
    return *reinterpret_cast<const unsigned*>(&r);
}

// Codes 8 o .. 8 o + 7 of a row segment of NW packed words -> h[i] = (code 8 o + i, code 8 o + 4 + i), i < 4, each half
// the integer q + 2^(b-1) (UNSIGNED_FIELDS: the code itself) times 2^-24: the field in the low bits of a subnormal.
template <int BITS, bool UNSIGNED_FIELDS, int NW>
__device__ __forceinline__ void unpack_octet(const unsigned* w, int o, unsigned h[4])
{
    if (BITS == 4) {
        const unsigned x = w[o] ^ (UNSIGNED_FIELDS ? 0u : 0x88888888u);
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = (x >> (4 * i)) & 0x000f000fu;
    } else {
        const int b = 24 * (o & 3), k = 3 * (o >> 2) + (b >> 5);
        const unsigned g = (b & 31) == 0 ? w[k] : ((o & 3) == 3 ? w[k] >> 8 : __funnelshift_r(w[k], w[k + 1 < NW ? k + 1 : k], b & 31));
        const unsigned x = ((g & 0xfffu) | ((g << 4) & 0x0fff0000u)) ^ (UNSIGNED_FIELDS ? 0u : 0x09240924u);
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = (x >> (3 * i)) & 0x00070007u;
    }
}

__device__ __forceinline__ void st_shared_v4(unsigned addr, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
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
