// gbs_quantized_matmul for a few tokens (a decoding step): out[t][o] = Delta_x[t] Delta_w[o] sum_j q_x[t][j] q_w[o][j] with
// n_tokens <= 64 (Section 4.2, Eq. (2)); the tile kernel of gbs_tc_qgemm.cu serves larger batches, and wide outputs (the rule is there).
//
// With this few tokens the call reads the packed weights once and does little with them, so what bounds it is how much of
// the chip reads at once and how many latencies follow one another, not the tensor pipe.  A 128 x 256 output tile per CTA
// put a 4096-channel layer on 16 SMs with 32 dependent steps each (31.6 us for 16 tokens).  Here a CTA takes 16 or 32 output
// channels and its eight warps split the contraction, so the same layer is 128 - 256 CTAs and every warp has its share of the
// weights in flight at once.
//   * Operands go from global memory to registers to mma.sync (m16n8k32, int8 x int8 -> int32), with no shared memory between:
//     a dot product does not see the order of its terms, so the codes of a thread's packed word simply ARE its fragment --
//     even fields one register, odd fields the other -- as long as both operands use the same order.  tcgen05 would want the
//     unpacked operands in shared memory and 128 rows; this is not its shape.
//   * A field moved to the top of its byte is the int8 q * 2^(8-b); the scale takes the powers of two out exactly.
//   * The eight partial sums meet in shared memory as integers (exact, any order).
#include <cuda_bf16.h>
#include <string.h>

#include "gbs_internal.h"
#include "gbs_qfields.cuh"

namespace {

constexpr int WARPS = 8;
constexpr int KB = 128;                 // codes per step and row: four threads x 32 codes

struct QgemvParams {
    long long n_out;
    int n_tok;
    int kblocks;                        // d' / 128
    int rbx, rbw;                       // bytes per row of packed codes
    const unsigned char* cx;
    const unsigned char* cw;
    const float* sx;
    const float* sw;
    void* out;
    long long out_stride;               // elements
};

// 32 codes of one row: packed words, then eight registers of four int8
template <int BITS> struct Packed {
    unsigned w[BITS];
    __device__ __forceinline__ void load(const unsigned char* p)
    {
        if (BITS == 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
            w[0] = v.x; w[1] = v.y; w[2] = v.z; w[BITS - 1] = v.w;
        } else {
#pragma unroll
            for (int i = 0; i < BITS; ++i) w[i] = __ldg(reinterpret_cast<const unsigned*>(p) + i);
        }
    }
};

template <int BITS>
__device__ __forceinline__ void gather_in_place(unsigned w[BITS])
{
    unsigned p[BITS];
    gather_octets<BITS>(w, p);
#pragma unroll
    for (int i = 0; i < BITS; ++i) w[i] = p[i];
}

__device__ __forceinline__ void mma_s8(int c[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// MT tiles of 16 output channels x NT tiles of 8 tokens per CTA; PF steps of every operand row in flight per thread
template <int XBITS, int WBITS, typename OutT, int MT, int NT, int PF>
__global__ void __launch_bounds__(32 * WARPS) k_qgemv(const __grid_constant__ QgemvParams P)
{
    // More than 16 tokens: the scales are fetched before the contraction, not behind it, where their latency would be one more in the chain.  (Up
    // to 16 the end is short and blocks come in several waves: 8 tokens -> 14336 9.25 us as it is, 9.75 with the scales first.)
    constexpr bool SCALES_FIRST = MT > 1;
    __shared__ int sums[16 * MT][8 * NT + 1];
    __shared__ float scale_w[SCALES_FIRST ? 16 * MT : 1], scale_x[SCALES_FIRST ? 8 * NT : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tig = lane & 3;
    const long long o0 = (long long)blockIdx.x * (16 * MT);
    for (int i = threadIdx.x; i < 16 * MT * (8 * NT + 1); i += 32 * WARPS) (&sums[0][0])[i] = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the int8 operands are q * 2^(8 - bits): the token's scale takes the two powers of two out again (exact)
    constexpr float OUT = 1.f / (float)(1 << (16 - XBITS - WBITS));
    if constexpr (SCALES_FIRST)
        for (int i = threadIdx.x; i < 16 * MT + 8 * NT; i += 32 * WARPS) {
            const int t = i - 16 * MT;
            if (t < 0) scale_w[i] = o0 + i < P.n_out ? __ldg(P.sw + o0 + i) : 0.f;
            else scale_x[t] = t < P.n_tok ? __ldg(P.sx + t) * OUT : 0.f;
        }

    // rows beyond the last are read as the last one; their sums are not stored
    const unsigned char* wp[2 * MT];
    const unsigned char* xp[NT];
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) {
        const long long o = o0 + 8 * i + g;
        wp[i] = P.cw + (o < P.n_out ? o : P.n_out - 1) * P.rbw + tig * (32 * WBITS / 8);
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        const int t = 8 * i + g;
        xp[i] = P.cx + (long long)(t < P.n_tok ? t : P.n_tok - 1) * P.rbx + tig * (32 * XBITS / 8);
    }
    int acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[m][n][e] = 0;

    const int kb1 = (warp + 1) * P.kblocks / WARPS;
    for (int kb0 = warp * P.kblocks / WARPS; kb0 < kb1; kb0 += PF) {
        Packed<WBITS> w[PF][2 * MT];
        Packed<XBITS> x[PF][NT];
#pragma unroll
        for (int p = 0; p < PF; ++p) {
            const int kb = kb0 + p < kb1 ? kb0 + p : kb1 - 1;             // a step beyond the share repeats the last loads
#pragma unroll
            for (int i = 0; i < 2 * MT; ++i) w[p][i].load(wp[i] + kb * (KB * WBITS / 8));
#pragma unroll
            for (int i = 0; i < NT; ++i) x[p][i].load(xp[i] + kb * (KB * XBITS / 8));
        }
#pragma unroll
        for (int p = 0; p < PF; ++p) {
            if (kb0 + p < kb1) {
                if (XBITS == 3 || WBITS == 3) {
#pragma unroll
                    for (int i = 0; i < 2 * MT; ++i) gather_in_place<WBITS>(w[p][i].w);
#pragma unroll
                    for (int n = 0; n < NT; ++n) gather_in_place<XBITS>(x[p][n].w);
                }
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    unsigned a[2 * MT][2];
#pragma unroll
                    for (int i = 0; i < 2 * MT; ++i) field_pair<WBITS>(w[p][i].w, o, a[i][0], a[i][1]);
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        unsigned b0, b1;
                        field_pair<XBITS>(x[p][n].w, o, b0, b1);
#pragma unroll
                        for (int m = 0; m < MT; ++m)
                            mma_s8(acc[m][n], a[2 * m][0], a[2 * m + 1][0], a[2 * m][1], a[2 * m + 1][1], b0, b1);
                    }
                }
            }
        }
    }
    __syncthreads();                                                      // the sums are zeroed
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) atomicAdd(&sums[16 * m + g + 8 * (e >> 1)][8 * n + 2 * tig + (e & 1)], acc[m][n][e]);
    __syncthreads();
    for (int i = threadIdx.x; i < 16 * MT * P.n_tok; i += 32 * WARPS) {
        const int oi = i % (16 * MT), t = i / (16 * MT);
        const long long o = o0 + oi;
        if (o >= P.n_out) continue;
        float v;                                                          // (both forms in one expression: 8 tokens -> 512 2.41 us instead of 2.24)
        if constexpr (SCALES_FIRST) {
            v = (float)sums[oi][t] * (scale_x[t] * scale_w[oi]);
        } else {
            const float dx = __ldg(P.sx + t) * OUT;
            v = (float)sums[oi][t] * (dx * __ldg(P.sw + o));
        }
        OutT* dst = reinterpret_cast<OutT*>(P.out) + (long long)t * P.out_stride + o;
        if (sizeof(OutT) == 4) *reinterpret_cast<float*>(dst) = v;
        else *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(v);
    }
}

template <int XB, int WB, typename OutT>
cudaError_t launch(const QgemvParams& P, bool pdl, cudaStream_t stream)
{
    // 16 channels per CTA while the tokens are few: more CTAs than SMs already at 4096 channels.  Beyond 16 tokens the
    // token codes, read by every CTA, are the larger traffic: 32 channels halve it.
    void (*kernel)(const QgemvParams);
    int ch = 16;
    if (P.n_tok <= 8) kernel = k_qgemv<XB, WB, OutT, 1, 1, 4>;
    else if (P.n_tok <= 16) kernel = k_qgemv<XB, WB, OutT, 1, 2, 4>;
    else if (P.n_tok <= 32) { kernel = k_qgemv<XB, WB, OutT, 2, 4, 2>; ch = 32; }
    else {
        // Two steps of four-bit rows in flight where a warp has more than two (64 tokens -> 4096 channels, 5120 wide: 9.60 us with one and 8.90 with two;
        // 4096: 8.12, 7.90; 2560: 6.96, 6.59; 2048: 5.31, 5.42; 1024: 3.71, 4.38).  Three bits: one (4096 wide, with the layer's other launch: 11.8, 12.7).
        kernel = k_qgemv<XB, WB, OutT, 2, 8, 1>;
        if constexpr (XB == 4 && WB == 4)
            if (P.kblocks > 2 * WARPS) kernel = k_qgemv<XB, WB, OutT, 2, 8, 2>;
        ch = 32;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((P.n_out + ch - 1) / ch));
    cfg.blockDim = dim3(32 * WARPS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P);
}

}  // namespace

int gbs_qgemv(const gbs_plan* px, const void* codes_x, const float* scales_x, int n_tokens, const gbs_plan* pw, const void* codes_w,
              const float* scales_w, int64_t n_out, void* out, int out_dtype, int64_t out_row_stride, cudaStream_t stream)
{
    QgemvParams P;
    memset(&P, 0, sizeof(P));
    P.n_out = n_out;
    P.n_tok = n_tokens;
    P.kblocks = px->d_pad / KB;
    P.rbx = px->d_pad * px->bits / 8;
    P.rbw = pw->d_pad * pw->bits / 8;
    P.cx = (const unsigned char*)codes_x;
    P.cw = (const unsigned char*)codes_w;
    P.sx = scales_x;
    P.sw = scales_w;
    P.out = out;
    P.out_stride = out_row_stride;
    const bool f32 = out_dtype == GBS_DTYPE_F32, pdl = px->pdl != 0;
    cudaError_t e;
    if (px->bits == 4) {
        if (pw->bits == 4) e = f32 ? launch<4, 4, float>(P, pdl, stream) : launch<4, 4, __nv_bfloat16>(P, pdl, stream);
        else e = f32 ? launch<4, 3, float>(P, pdl, stream) : launch<4, 3, __nv_bfloat16>(P, pdl, stream);
    } else {
        if (pw->bits == 4) e = f32 ? launch<3, 4, float>(P, pdl, stream) : launch<3, 4, __nv_bfloat16>(P, pdl, stream);
        else e = f32 ? launch<3, 3, float>(P, pdl, stream) : launch<3, 3, __nv_bfloat16>(P, pdl, stream);
    }
    return (int)e;
}
