// Inverse path of gbs_dequantize for d' = 128 rows (KV entries) with one scale per row (group 0 or 128), symmetric or
// asymmetric quantizer:
//     xhat = (H_128^T yhat / sqrt(128))[0:d],   yhat = q * Delta   or   code * Delta + lo
// (Section 2.1 / 5.1; inverse by the transpose, Section 2.3; H_128 of Eq. (1) is symmetric).
//
// One thread owns one row.  A packed field k, masked into the low bits of a 16-bit half, IS the subnormal half-precision
// number k * 2^-24, and sums of 128 fields of at most 15 stay below 2048 * 2^-24: every one of the seven butterfly stages
// is exact in packed half arithmetic, two coordinates per instruction, with no conversion before and one to fp32 after.
// Symmetric codes are stored as q + 2^(b-1); the offset adds 128 * 2^(b-1) to coordinate 0 and nothing elsewhere, where
// one exact subtraction removes it.  The only rounding is the product with Delta / sqrt(128) (and the output type's).
//
// The rows leave through shared memory: a thread's stores to its own row touch 32 rows per instruction and took 73 % of the L1 data
// pipe, so the warp puts 128-byte pieces of its rows there with the 128-byte swizzle (eight lanes side by side hit all banks) and one TMA
// store carries each piece of all 32 rows.
// What bounds it: HBM (48 or 64 bytes read and 256 or 512 written per row).  About 7 issue slots per value without any
// barrier or tensor-core round trip; the tensor-core form this replaces waited on that round trip with 16
// warps per SM.  262 144 rows, 4 bits, asymmetric -> bf16: 33.2 us in that form, 18.6 with stores by each thread, 16.0 now (5.4 TB/s).
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_tc_common.cuh"
#include "gbs_tc_inv.cuh"

namespace {

constexpr int DP = 128;
constexpr int RI_THREADS = 32;        // single warps: a finished one makes room for the next at once (blocks of 128: 19.6 us, 19.15 so)
constexpr int RI_BLOCKS = 20;         // per SM: 102 registers per thread, of which 64 hold the row
constexpr int BOX_BYTES = 32 * 128;   // one store: 128 bytes of 32 rows

struct RowInvParams {
    long long n_rows;
    int d;                            // output width, a multiple of 32
    float norm;                       // 1 / sqrt(128)
    const unsigned char* codes;
    const float* scales;              // Delta per row, or (Delta, lo) per row
};

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(smem_u32(src)), "r"(c0), "r"(c1) : "memory");
}

template <int BITS, bool ASYM, typename OutT>
__global__ void __launch_bounds__(RI_THREADS, RI_BLOCKS) k_row_inv(const __grid_constant__ CUtensorMap omap, const __grid_constant__ RowInvParams P)
{
    __shared__ __align__(1024) unsigned char stage[2 * BOX_BYTES];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long row = (long long)blockIdx.x * RI_THREADS + threadIdx.x;
    const bool live = row < P.n_rows;                        // the last block's other rows are left out of its stores
    constexpr int NW = DP * BITS / 32;                       // packed words of a row
    unsigned w[NW];
    const uint4* src = reinterpret_cast<const uint4*>(P.codes + row * (NW * 4));
#pragma unroll
    for (int i = 0; i < NW / 4; ++i) {
        const uint4 v = live ? __ldg(src + i) : make_uint4(0u, 0u, 0u, 0u);
        w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
    }
    float delta = 0.f, lo = 0.f;
    if (ASYM) {
        const float2 sl = live ? __ldg(reinterpret_cast<const float2*>(P.scales) + row) : make_float2(0.f, 0.f);
        delta = sl.x; lo = sl.y;
    } else if (live) {
        delta = __ldg(P.scales + row);
    }
    // h[4 o + i] = (coordinate 8 o + i, coordinate 8 o + 4 + i)
    unsigned h[64];
#pragma unroll
    for (int o = 0; o < 16; ++o) rotate_octet<BITS, ASYM, NW, false>(w, o, h + 4 * o);
#pragma unroll
    for (int i = 0; i < 64; ++i) h[i] = hpair(h[i]);
#pragma unroll
    for (int s = 4; s < 64; s <<= 1)
#pragma unroll
        for (int i = 0; i < 64; ++i)
            if ((i & s) == 0) {
                const unsigned a = h[i], b = h[i + s];
                h[i] = hadd2(a, b);
                h[i + s] = hsub2(a, b);
            }
    float sc = delta * P.norm * 16777216.f;                  // the halves are integers times 2^-24
    const float add0 = ASYM ? 128.f * lo * P.norm : 0.f;
    constexpr float OFF0 = (ASYM ? 0.f : 128.f * (float)(1 << (BITS - 1))) / 16777216.f;
    float off0 = OFF0;
    if (!(fabsf(sc) <= 3.4028234e38f)) {
        // a scale beyond 2^107: the halves as the integers they stand for (below 2048), exactly
#pragma unroll
        for (int i = 0; i < 64; ++i) h[i] = hmul2(hmul2(h[i], 0x6c006c00u), 0x6c006c00u);                      // 2^12 twice
        sc = delta * P.norm;
        off0 = OFF0 * 16777216.f;
    }
    // Through shared memory, 128-byte pieces of the block's 32 rows with the 128-byte swizzle (a store instruction's lanes then hit
    // different banks), and out by TMA: 16 KB for fp32 go in two halves.
    constexpr int PER_BOX = 128 / (int)sizeof(OutT);         // coordinates: 64 or 32
    const unsigned line = smem_u32(stage) + threadIdx.x * 128u, swz = threadIdx.x & 7u;
#pragma unroll
    for (int c = 0; c < 8; ++c) {                            // sixteen coordinates each
        if (c * 16 >= P.d) break;
        float f[16];
#pragma unroll
        for (int o = 0; o < 2; ++o)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&h[8 * c + 4 * o + i]));
                f[8 * o + i] = v.x;
                f[8 * o + 4 + i] = v.y;
            }
        if (c == 0) f[0] -= off0;
#pragma unroll
        for (int e = 0; e < 16; ++e) f[e] = (c == 0 && e == 0) ? fmaf(f[0], sc, add0) : f[e] * sc;
        unsigned w32[16];
        pack_values(f, w32, OutT());
        const int box = c * 16 / PER_BOX;
        const unsigned chunk0 = (unsigned)(c * 16 % PER_BOX * (int)sizeof(OutT)) / 16u;
#pragma unroll
        for (unsigned k = 0; k < sizeof(OutT); ++k)
            st_shared_v4(line + (box & 1) * BOX_BYTES + (((chunk0 + k) ^ swz) << 4), make_uint4(w32[4 * k], w32[4 * k + 1], w32[4 * k + 2], w32[4 * k + 3]));
        const bool last = (c + 1) * 16 >= P.d;
        if (c == 7 || last || (sizeof(OutT) == 4 && c == 3)) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (threadIdx.x == 0) {
                const int first = box & ~1;
                tma_store_2d(&omap, stage, first * PER_BOX, (int)(blockIdx.x * RI_THREADS));
                if (box & 1) tma_store_2d(&omap, stage + BOX_BYTES, box * PER_BOX, (int)(blockIdx.x * RI_THREADS));
                asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group.read 0;" ::: "memory");
            }
            __syncwarp();                                    // the bytes have left, also before the block ends
        }
    }
}

typedef void (*RowInvKernel)(const CUtensorMap, const RowInvParams);

}  // namespace

// What this path serves: d' = 128 (the ROW family) with one scale (pair) per row and whole 32-value output chunks, as many rows as the
// stores' 32-bit coordinates count.
bool gbs_rowinv_serves(const gbs_plan* p, const float* scales, int64_t n_rows)
{
    if (p->variant != GBS_VARIANT_TC_ROW || !(p->group == 0 || p->group == DP) || p->d % 32 != 0 || n_rows > 0x7fffffff || !get_encode())
        return false;
    return !(p->asym && (reinterpret_cast<uintptr_t>(scales) & 7u));        // (Delta, lo) pairs are read as one 8-byte word
}

int gbs_rowinv_dequantize(const gbs_plan* p, const void* codes, const float* scales, int64_t n_rows, void* out,
                          int out_dtype, cudaStream_t stream)
{
    static const RowInvKernel table[2][2][2] = {
        {{k_row_inv<3, false, float>, k_row_inv<3, false, __nv_bfloat16>}, {k_row_inv<3, true, float>, k_row_inv<3, true, __nv_bfloat16>}},
        {{k_row_inv<4, false, float>, k_row_inv<4, false, __nv_bfloat16>}, {k_row_inv<4, true, float>, k_row_inv<4, true, __nv_bfloat16>}}};
    const long long blocks = (n_rows + RI_THREADS - 1) / RI_THREADS;
    RowInvParams P;
    memset(&P, 0, sizeof(P));
    P.n_rows = n_rows;
    P.d = p->d;
    P.norm = p->norm;
    P.codes = (const unsigned char*)codes;
    P.scales = scales;
    const bool f32 = out_dtype == GBS_DTYPE_F32;
    CUtensorMap omap;
    const cuuint64_t gdim[2] = {(cuuint64_t)p->d, (cuuint64_t)n_rows};
    const cuuint64_t gstr[1] = {(cuuint64_t)p->d * (f32 ? 4 : 2)};
    const cuuint32_t box[2] = {f32 ? 32u : 64u, RI_THREADS}, estr[2] = {1, 1};
    if (get_encode()(&omap, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, out, gdim, gstr, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return (int)cudaErrorInvalidValue;
    {
        // room for all blocks' stages, once per device (not a stream operation)
        static std::mutex mu;
        static bool done[64] = {false};
        std::lock_guard<std::mutex> lock(mu);
        if (!(p->device >= 0 && p->device < 64 && done[p->device])) {
            for (int i = 0; i < 8; ++i) {
                const cudaError_t e = cudaFuncSetAttribute(table[i >> 2][i >> 1 & 1][i & 1], cudaFuncAttributePreferredSharedMemoryCarveout,
                                                           cudaSharedmemCarveoutMaxShared);
                if (e != cudaSuccess) return (int)e;
            }
            if (p->device >= 0 && p->device < 64) done[p->device] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(RI_THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p->pdl ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, table[p->bits - 3][p->asym ? 1 : 0][f32 ? 0 : 1], omap, P);
}
