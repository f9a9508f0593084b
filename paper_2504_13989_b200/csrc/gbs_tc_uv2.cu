// Tensor-core rotate-quantize of bf16 rows with d' = 64 U, U = m * 2^j <= 128 (4096 < d' <= 8192, e.g. 8192 and 5120).
//
// The row is a U x 64 matrix X and Y = A X H_64, A = H_m (x) H_{2^j}, as in gbs_tc_uv.cu with twice the columns.  A lane of the
// contraction's result holds 64 values; two warps share it, one taking the sums and one the differences of its two halves (the
// first stage of H_64) and both finishing with H_32 in registers, so that a thread again owns 32 consecutive output coordinates
// and every value leaves TMEM once per warp, nothing goes back.  (The three-sweep wide kernel that ran these widths moves
// every value through TMEM five times.)
//   * TMA brings two tokens per tile (zero-filled beyond d: Section 4.2), N-major with the 128-byte swizzle; U / 16 MMAs of
//     N = 128, four stages in shared memory and in TMEM.
//   * Sixteen warps: (lane quadrant q, token t, half).  Where U leaves a quadrant without rows (U <= 96, e.g. 80 for 5120) the
//     rows move on by one quadrant from tile to tile, so that every warp, and every scheduler with it, rests equally often: the
//     image of A stands twice in shared memory, one below the other, and a tile's MMAs start 32 rows higher than the last.
//   * Maxima: one scale per token over the warps of the token (named barrier), or one per group of 64 * 2^g coordinates over
//     2^g lanes and the two halves (shuffles and a barrier of the pair).  Delta, rounding, clipping, packing as everywhere
//     (Sections 2.1, 3.1).
// What bounds it: instruction issue, as for the narrower widths.  8192 rows, 4 bits, one scale per token, called back to back for
// seconds: 8192 wide 46.8 us on the three-sweep kernel, 42.5 here; 5120 wide 41.1 -> 34.8; 5120 wide, 3 bits, groups of 128: 44.1 -> 30.4.
// In bursts, on a cool GPU: 35.0, 32.1 and 27.6.
// Every wait is bounded; an expired wait records a code in the plan's status word.  A warp whose wait ran out brings a pattern no
// maximum can have to the barrier it shares, and all who meet it there leave their loop with it.  With one scale per token they go on
// bringing it to the barriers of the tiles that are left: a warp that rested in this tile knows nothing of it yet and will wait for
// them.  (The two warps of a group always have rows in the same tiles.)
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_tc_common.cuh"

namespace {

constexpr int V = 64, TOK = 2, UMAX = 128;
constexpr int NCOLS = TOK * V;
constexpr int STAGES = 4;                          // in shared memory and in TMEM; as many as quadrants: see `slab` below
constexpr int TMEM_COLS = STAGES * NCOLS;
constexpr int A_BLOCK = UMAX * 128;                // 64 columns of the image of A
constexpr int STAGE_BYTES_MAX = TOK * UMAX * V * 2;
constexpr int EPI_WARPS = 16;
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr unsigned POISON = 0xffffffffu;           // no maximum of absolute values has the sign bit set

struct __align__(1024) Smem {
    unsigned char a[2][2][A_BLOCK];                // [64-column block][copy]
    unsigned char b[STAGES][STAGE_BYTES_MAX];
    // Maxima exchanged between warps, a place and a barrier of their own for each of four tiles: warps rest in different tiles,
    // but of the three tiles between two uses of a place any two warps share one, whose barrier orders them.
    union {
        unsigned tok[STAGES][TOK][8];              // [token][slab and half]
        unsigned grp[STAGES][8][2][16];            // [quadrant and token][half][group]
    } red;
    unsigned long long full[STAGES], empty[STAGES], tfull[STAGES], tempty[STAGES];
    unsigned long long abar;
    unsigned tmem_base;
    volatile int abort_flag;
};

struct Uv2Params {
    long long n_rows;
    int n_tiles;                  // ceil(n_rows / TOK)
    int U, Upad, ksteps;
    int slabs;                    // lane quadrants with rows: ceil(U / 32)
    int d_pad;
    int code_row_bytes;
    int spr;                      // scales per row
    int glog;                     // log2 of the u-rows per group
    float c_scale, c_half, norm;
    const unsigned char* a_img;
    unsigned char* codes;
    float* scales;
    float* y_opt;
    int* status;
};

template <int BITS, bool GROUPED, bool WANT_Y>
__global__ void __launch_bounds__(THREADS, 1) k_tc_uv2(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ Uv2Params P)
{
    extern __shared__ unsigned char smem_raw[];
    Smem* S = reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const unsigned stage_bytes = (unsigned)(TOK * P.Upad * V * 2);
    const bool rotate = P.slabs < 4;
    const int n_mine = (P.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // tiles of this CTA

    int it_p = 0;                                  // producer iterations already issued
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&S->full[s], 1);
        mbar_init(&S->abar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_arrive_expect_tx(&S->abar, 4 * A_BLOCK);
        for (int kb = 0; kb < 2; ++kb)             // plan-owned, immutable: needs no ordering
            for (int c = 0; c < 2; ++c) bulk_load(S->a[kb][c], P.a_img + kb * A_BLOCK, A_BLOCK, &S->abar);
        // programmatic dependent launch: until the wait below returns an earlier kernel may still be writing the rows; only L2
        // is filled before it
        tma_prefetch_3d(&tmap, 0, 0, blockIdx.x * TOK);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (; it_p < STAGES && it_p < n_mine; ++it_p) {
            mbar_arrive_expect_tx(&S->full[it_p], stage_bytes);
            tma_load_3d(S->b[it_p], &tmap, &S->full[it_p], 0, 0, ((int)blockIdx.x + it_p * (int)gridDim.x) * TOK);
        }
    }
    if (threadIdx.x == 64) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S->empty[s], 1);
            mbar_init(&S->tfull[s], 1);
            mbar_init(&S->tempty[s], (unsigned)(2 * TOK * P.slabs));
        }
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&S->tmem_base, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned tmem_base = S->tmem_base;

    if (warp == 0) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) {
            int it = it_p;
            for (; it < n_mine; ++it) {
                const int s = it % STAGES;
                if (!mbar_wait(&S->abort_flag, &S->empty[s], ((it / STAGES) & 1) ^ 1, P.status, 1)) break;
                mbar_arrive_expect_tx(&S->full[s], stage_bytes);
                tma_load_3d(S->b[s], &tmap, &S->full[s], 0, 0, ((int)blockIdx.x + it * (int)gridDim.x) * TOK);
            }
            if (S->abort_flag) drain_copies(S->full, STAGES, it);
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        constexpr unsigned IDESC = instr_desc(UMAX, NCOLS);
        const unsigned long long ad0 = smem_desc(smem_u32(S->a[0][0]), 16, 1024, 2);
        const unsigned long long bd0 = smem_desc(smem_u32(S->b[0]), (unsigned)(P.Upad * V * 2), 8 * V * 2, 2);
        bool ok = mbar_wait_warp(&S->abort_flag, &S->abar, 0, P.status, 6);
        for (int it = 0; ok && it < n_mine; ++it) {
            const int s = it % STAGES;
            const unsigned ph = (it / STAGES) & 1;
            if (!mbar_wait_warp(&S->abort_flag, &S->full[s], ph, P.status, 2)) break;
            if (!mbar_wait_warp(&S->abort_flag, &S->tempty[s], ph ^ 1, P.status, 3)) break;
            tc_fence_after();
            // lane quadrant q receives slab (q - it) mod 4 of A's rows
            unsigned long long ad = ad0 + (rotate ? (unsigned long long)(((4 - (it & 3)) & 3) * 32 * 128 / 16) : 0ull);
            unsigned long long bd = bd0 + (unsigned long long)(s * STAGE_BYTES_MAX / 16);
            const unsigned d_tmem = tmem_base + s * NCOLS;
            for (int ks = 0; ks < P.ksteps; ++ks) {
                umma_f16(d_tmem, ad, bd, IDESC, ks != 0 ? 1u : 0u);
                ad += ks == 3 ? (2 * A_BLOCK - 96) / 16 : 2;
                bd += 16 * V * 2 / 16;
            }
            umma_commit(&S->empty[s]);
            umma_commit(&S->tfull[s]);
        }
    } else {
        // ------------------------------ epilogue ------------------------------
        const int q = warp & 3;                    // TMEM lane quadrant this warp may access
        const int w = (warp - 2) >> 2;
        const int t = w >> 1, half = w & 1;        // token slot of its tiles, half of a lane's 64 outputs
        const unsigned taddr0 = tmem_base + ((unsigned)(q * 32) << 16) + t * V;
        const float sign = half ? -1.f : 1.f;
        const int gl = 1 << P.glog;                // lanes per group
        const long long row_step = (long long)gridDim.x * TOK;
        long long row = (long long)blockIdx.x * TOK + t;
        int it = 0;
        for (; it < n_mine; ++it, row += row_step) {
            const int s = it % STAGES;
            // A warp without rows in this tile has none in any tile of this stage (there are as many stages as quadrants), so it
            // takes part in every phase of the barriers it waits for.
            const int slab = rotate ? (q - it) & 3 : q;
            if (slab >= P.slabs) continue;
            const int up = slab * 32 + lane;       // u'
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&S->abort_flag, &S->tfull[s], (it / STAGES) & 1, P.status, 4, false));
            unsigned r[32];
            unsigned mb = POISON;
            if (ok) {
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    unsigned hi[16];
                    tmem_ld16_issue(taddr0 + s * NCOLS + 16 * h, r + 16 * h);
                    tmem_ld16_issue(taddr0 + s * NCOLS + 32 + 16 * h, hi);
                    tmem_ld_wait16x2(r + 16 * h, hi);
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        r[16 * h + e] = __float_as_uint(fmaf(__uint_as_float(hi[e]), sign, __uint_as_float(r[16 * h + e])));
                }
                // the accumulators are in registers: hand the TMEM stage back to the MMA issuer
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->tempty[s]);
                mb = __float_as_uint(fwht32_absmax(r));
            }
            if (GROUPED) {
                // a group is 2^glog adjacent lanes of both warps
                if (ok) {
                    switch (P.glog) {
                        case 5: mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 16));   // fall through
                        case 4: mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 8));    // fall through
                        case 3: mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 4));    // fall through
                        case 2: mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 2));    // fall through
                        default: mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 1));
                    }
                }
                unsigned (*slot)[16] = S->red.grp[s][q * 2 + t];
                if ((lane & (gl - 1)) == 0) slot[half][lane >> P.glog] = mb;
                asm volatile("bar.sync %0, 64;" ::"r"(1 + q * 2 + t) : "memory");
                mb = max(mb, slot[half ^ 1][lane >> P.glog]);
                if (__any_sync(0xffffffffu, mb == POISON)) break;
            } else {
                if (ok) mb = __reduce_max_sync(0xffffffffu, mb);
                unsigned* slot = S->red.tok[s][t];
                if (lane == 0) slot[slab * 2 + half] = mb;
                asm volatile("bar.sync %0, %1;" ::"r"(1 + t * STAGES + s), "r"(64 * P.slabs) : "memory");
                const uint4 m0 = *reinterpret_cast<const uint4*>(slot), m1 = *reinterpret_cast<const uint4*>(slot + 4);
                mb = max(max(m0.x, m0.y), max(m0.z, m0.w));
                if (P.slabs > 2) mb = max(mb, max(m1.x, m1.y));
                if (P.slabs > 3) mb = max(mb, max(m1.z, m1.w));
                if (mb == POISON) break;
            }
            const float M = __uint_as_float(mb);
            // an all-zero token or group has every value at zero: any finite factor gives code 0.  (No lower limit above that: a group
            // of tiny values is quantized like any other.)
            const float a1 = M > 0.f ? __fdividef(P.c_half, M) : 0.f;
            unsigned out[BITS];
            quantize_pack32<BITS>(r, a1, out);
            if (up < P.U && row < P.n_rows) {
                const int out0 = up * V + half * 32;
                unsigned* dst = reinterpret_cast<unsigned*>(P.codes + row * P.code_row_bytes + out0 / 8 * BITS);
                if (BITS == 4) {
                    *reinterpret_cast<uint4*>(dst) = make_uint4(out[0], out[1], out[2], out[BITS - 1]);
                } else {
                    dst[0] = out[0]; dst[1] = out[1]; dst[2] = out[2];
                }
                if (GROUPED ? (half == 0 && (lane & (gl - 1)) == 0) : out0 == 0)
                    P.scales[row * P.spr + (GROUPED ? up >> P.glog : 0)] = P.c_scale * M;
                if (WANT_Y) {
                    float4* yo = reinterpret_cast<float4*>(P.y_opt + row * (long long)P.d_pad + out0);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        yo[i] = make_float4(__uint_as_float(r[4 * i]) * P.norm, __uint_as_float(r[4 * i + 1]) * P.norm,
                                            __uint_as_float(r[4 * i + 2]) * P.norm, __uint_as_float(r[4 * i + 3]) * P.norm);
                }
            }
        }
        if (!GROUPED) {
            // after an expired wait: the barriers of the tiles that are left
            for (++it; it < n_mine; ++it) {
                const int s = it % STAGES, slab = rotate ? (q - it) & 3 : q;
                if (slab >= P.slabs) continue;
                if (lane == 0) S->red.tok[s][t][slab * 2 + half] = POISON;
                asm volatile("bar.sync %0, %1;" ::"r"(1 + t * STAGES + s), "r"(64 * P.slabs) : "memory");
            }
        }
    }

    // ---- teardown: every role leaves its loop (normally or through the abort flag), then TMEM is freed
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

typedef void (*Uv2Kernel)(const CUtensorMap, const Uv2Params);
Uv2Kernel kernel_of(int bits, bool grouped, bool want_y)
{
    static const Uv2Kernel table[2][2][2] = {
        {{k_tc_uv2<3, false, false>, k_tc_uv2<3, false, true>}, {k_tc_uv2<3, true, false>, k_tc_uv2<3, true, true>}},
        {{k_tc_uv2<4, false, false>, k_tc_uv2<4, false, true>}, {k_tc_uv2<4, true, false>, k_tc_uv2<4, true, true>}}};
    return table[bits - 3][grouped ? 1 : 0][want_y ? 1 : 0];
}

}  // namespace

// The wide plans this kernel serves: those whose image of A has U = d' / 64 rows (bf16 rows; a group is at least two lanes and
// at most a warp's).
bool gbs_tc_uv2_supported(const gbs_plan* p)
{
    return p->variant == GBS_VARIANT_TC_UVM && p->uvm_glog == 1 && !p->asym &&
           (p->group == 0 || (p->group >= 2 * V && p->group <= 32 * V)) && p->smem_optin >= (int)sizeof(Smem) + 1024;
}

int gbs_tc_uv2_rotate_quantize(const gbs_plan* p, const void* x, int64_t n_rows, int64_t stride, void* codes, float* scales,
                               float* y_opt, cudaStream_t stream)
{
    EncodeTiledFn encode = get_encode();
    if (!encode) return (int)cudaErrorNotSupported;
    if (n_rows > (int64_t)0x7fffffff - TOK) return (int)cudaErrorInvalidValue;      // TMA coordinates are 32-bit
    Uv2Params P;
    memset(&P, 0, sizeof(P));
    P.U = p->d_pad / V;
    P.Upad = (P.U + 15) & ~15;
    CUtensorMap tmap;
    const cuuint64_t gdim[3] = {(cuuint64_t)V, (cuuint64_t)(p->d / V), (cuuint64_t)n_rows};
    const cuuint64_t gstr[2] = {(cuuint64_t)(V * 2), (cuuint64_t)(stride * 2)};
    const cuuint32_t box[3] = {V, (cuuint32_t)P.Upad, TOK}, estr[3] = {1, 1, 1};
    if (encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return (int)cudaErrorInvalidValue;
    P.n_rows = n_rows;
    P.n_tiles = (int)((n_rows + TOK - 1) / TOK);
    P.ksteps = P.Upad / 16;
    P.slabs = (P.U + 31) / 32;
    P.d_pad = p->d_pad;
    P.code_row_bytes = p->d_pad * p->bits / 8;
    P.spr = p->group ? p->d_pad / p->group : 1;
    while (p->group && (V << P.glog) < p->group) ++P.glog;
    P.c_scale = p->c_scale;
    P.c_half = (float)(1.0 / (2.0 * (double)p->alpha));
    P.norm = p->norm;
    P.a_img = p->d_aimg;
    P.codes = (unsigned char*)codes;
    P.scales = scales;
    P.y_opt = y_opt;
    P.status = p->d_status;
    const int smem = (int)sizeof(Smem) + 1024;
    {
        // opt in to the large dynamic shared memory once per device (not a stream operation)
        static std::mutex mu;
        static bool done[64] = {false};
        std::lock_guard<std::mutex> lock(mu);
        if (!(p->device >= 0 && p->device < 64 && done[p->device])) {
            for (int i = 0; i < 8; ++i) {
                const cudaError_t e = cudaFuncSetAttribute(kernel_of(3 + (i & 1), (i & 2) != 0, (i & 4) != 0), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
                if (e != cudaSuccess) return (int)e;
            }
            if (p->device >= 0 && p->device < 64) done[p->device] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(P.n_tiles < p->sm_count ? P.n_tiles : p->sm_count));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p->pdl ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, kernel_of(p->bits, p->group != 0, y_opt != nullptr), tmap, P);
}
