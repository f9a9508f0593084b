// Shared by the two tile kernels of the quantized matmul (gbs_tc_qgemm.cu, gbs_tc_qgemm2.cu): parameters, unpacking of a row's 128 codes,
// the epilogue of 32 tokens.
#pragma once

#include "gbs_internal.h"
#include "gbs_qfields.cuh"
#include "gbs_tc_common.cuh"

struct QgemmParams {
    long long n_tok, n_out;
    int n;                              // tokens per tile (MMA N)
    int xbox;                           // token rows a load brings: n, or all tokens if they are fewer
    int m_tiles, tiles;                 // channel tiles, all tiles
    int kblocks;                        // d' / 128
    const float* sx;
    const float* sw;
    void* out;
    long long out_stride;               // elements
    int* status;
};

constexpr int GBS_QGEMM2_MAX_TOKENS = 256;      // tokens per tile of the pairs' kernel
// How many pairs of the device's SMs can run the pairs' kernel (gbs_tc_qgemm2.cu) at once; 0 where a cluster of two cannot be launched.
int gbs_tc_qgemm2_pairs(const gbs_plan* px);
// That kernel, on `pairs` of them at most.  P: tokens per tile (a multiple of 32, 64 at least), tiles of 256 channels; xmap's boxes hold P.xbox <= P.n / 2 rows.
int gbs_tc_qgemm2(const gbs_plan* px, const gbs_plan* pw, const CUtensorMap& wmap, const CUtensorMap& xmap, const QgemmParams& P, int pairs,
                  int out_dtype, cudaStream_t stream);

namespace {

constexpr int KB = 128;                 // codes per step and row: one 128-byte line of int8

// Instruction descriptor, kind::i8: int32 accumulate, signed 8-bit A and B, both K-major, M x N.
__host__ __device__ constexpr unsigned instr_desc_i8(int M, int N)
{
    return (2u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ uint4 ld_shared_v4(unsigned addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
// 8 registers -> 8 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_st8(unsigned taddr, const unsigned r[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                 ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr) : "memory");
}
// 16 columns of this thread's TMEM lane -> 16 registers
__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}

// The packed 128 codes of row r of a stage.  Four-bit rows are 64 bytes with the 64-byte swizzle (eight rows side by side hit
// all banks), three-bit rows 48 bytes plain (48-byte steps do so by themselves).
template <int BITS>
__device__ __forceinline__ void load_row128(unsigned rows, int r, uint4 w[BITS])
{
#pragma unroll
    for (int c = 0; c < BITS; ++c)
        w[c] = ld_shared_v4(rows + (unsigned)r * (16u * BITS) + (unsigned)((BITS == 4 ? c ^ ((r >> 1) & 3) : c) << 4));
}
// Codes 32 c .. 32 c + 31 of it -> eight words of int8.
template <int BITS, bool GATHER>
__device__ __forceinline__ void unpack32(const uint4 w[BITS], int c, unsigned v[8])
{
    const unsigned f[16] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w,
                            w[2].x, w[2].y, w[2].z, w[2].w, w[BITS - 1].x, w[BITS - 1].y, w[BITS - 1].z, w[BITS - 1].w};
    unsigned p[BITS];
    if (GATHER) {
        gather_octets<BITS>(f + BITS * c, p);
    } else {
#pragma unroll
        for (int i = 0; i < BITS; ++i) p[i] = f[BITS * c + i];
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) field_pair<BITS>(p, o, v[2 * o], v[2 * o + 1]);
}

// 32 accumulator columns (tokens t .. t + 31) of this thread's channel o, scaled and stored.
template <int BITS_BOTH, typename OutT>
__device__ __forceinline__ void store_tokens(unsigned taddr, long long t, long long o, float dw, int lane, const QgemmParams& P)
{
    // the int8 operands were q * 2^(8 - bits): take the two powers of two out again (exact)
    const float dx_l = t + lane < P.n_tok ? __ldg(P.sx + t + lane) * (1.f / (float)(1 << (16 - BITS_BOTH))) : 0.f;
    OutT* dst = reinterpret_cast<OutT*>(P.out) + t * P.out_stride + o;
    const int cols = (int)((P.n_tok - t) < 32 ? (P.n_tok - t) : 32);
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
        unsigned v[16];
        tmem_ld16(taddr + (unsigned)(16 * hf), v);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const float dx = __shfl_sync(0xffffffffu, dx_l, 16 * hf + e);
            const float f = (float)(int)v[e] * (dx * dw);
            if (16 * hf + e < cols && o < P.n_out) {
                if (sizeof(OutT) == 4) *reinterpret_cast<float*>(dst) = f;
                else *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(f);
            }
            dst += P.out_stride;
        }
    }
}

}  // namespace
