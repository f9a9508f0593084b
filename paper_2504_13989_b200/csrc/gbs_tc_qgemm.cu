// gbs_quantized_matmul: the consumer on the other side of the path (Section 4.2, Eq. (2); Section 2.3.1).
//
// The online path leaves, per token, b-bit codes q_x and one scale Delta_x of the rotated, zero-padded activation
// H x_pad / sqrt(d'); the weights W (one row per output channel) go through the same rotation and quantizer once,
// offline (gbs_weight_rotate_quantize), leaving codes q_w and one scale Delta_w per output channel.  Because the
// rotation is orthogonal and the padding adds zeros, (H x_pad)^T (H w_pad) / d' = x^T w (Eq. (2)), so the layer's
// output is, up to quantization error,
//
//        out[t][o] = Delta_x[t] * Delta_w[o] * sum_j q_x[t][j] * q_w[o][j],
//
// an INTEGER contraction over the d' codes followed by one multiplication per output.  The rotated activation never
// exists in memory as floats: this kernel reads the packed codes of both operands.  (Up to 64 tokens: gbs_qgemv.cu.)
//
//   * Output channels are the rows of the MMA (TMEM lane = channel), tokens its columns: a tile is 128 channels x up to 256
//     tokens on one SM.
//   * Packed codes arrive by TMA (128 codes of every row per step, several steps ahead).  Twenty-four warps unpack, one thread
//     per row: a field moved to the top bits of its byte IS the int8 q * 2^(8-b) (the epilogue removes the power of two).
//     Weights go to TENSOR MEMORY (a thread's 128 int8 are 32 columns of its lane), tokens to 128-byte-swizzled K-major rows in
//     shared memory; both use the same order of the codes, which a dot product does not see.
//   * One thread issues tcgen05.mma kind::i8 (int32 accumulators, exact).  Consecutive tiles use accumulators that overlap by
//     half (or not at all, up to 128 tokens); four epilogue warps drain the shared half first, so that the next tile starts
//     early.  Lanes of a warp hold consecutive channels, so every store instruction writes 64 or 128 contiguous bytes.
// What bounds it: narrow tiles, the latencies a warp set goes through per step (about 1200 cycles: packed codes, a free stage,
// its stores becoming visible to the tensor cores; two or three sets take turns).  256-token tiles, the shared-memory port:
// 24 KB of packed codes in and out and 32 KB of int8 in and out are about 900 of a step's 1016 cycles, the tensor pipe 512.
// 4096 x 4096 x 4096, 4 bits: 139 us (one 128 x 256 tile per CTA, both operands in shared memory, packed codes by global
// loads), 63 us now; 56 on pairs of SMs (gbs_tc_qgemm2.cu), which outputs of that size take.
// Every wait is bounded; an expired wait records a code in the activation plan's status word.
#include <math.h>
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_qgemm.cuh"

namespace {

constexpr int TM = 128;                 // output channels per tile
constexpr int UNPACK_WARPS = 24;
constexpr int EPI_WARPS = 4;
constexpr int THREADS = 32 * (2 + UNPACK_WARPS + EPI_WARPS);
constexpr int TMEM_COLS = 512;
constexpr int MAX_STAGES = 6;

// TW warps of a set unpack tokens (32 rows each), four unpack weights.  Sets take alternate steps; a stage belongs to one set,
// which therefore takes part in every phase of the barriers it waits for.
template <int TW> struct Shape {
    static constexpr int SETS = UNPACK_WARPS / (4 + TW);            // TW = 4: three, TW = 8: two
    static constexpr int STAGES = TW == 8 ? 4 : 6;
    static constexpr int TN = 32 * TW;                              // tokens per tile at most
    static constexpr int P_STAGE = (TM + TN) * 64;                  // packed bytes of a stage (64 or 48 per row)
    static constexpr int B_STAGE = TN * KB;                         // int8 tokens of a stage
    static constexpr int ACC_STEP = 128;                            // second accumulator's first column
    static constexpr int A_COL0 = TW == 8 ? 384 : 256;              // weights: 32 columns per stage
    static constexpr int SMEM = 1024 + STAGES * (P_STAGE + B_STAGE) + 512;
    static_assert(STAGES % SETS == 0 && A_COL0 + 32 * STAGES <= TMEM_COLS, "stages");
};

struct Ctl {
    unsigned long long pfull[MAX_STAGES], pempty[MAX_STAGES], ofull[MAX_STAGES], oempty[MAX_STAGES], tfull[2], tempty[2], tshared;
    unsigned tmem_base;
    volatile int abort_flag;
};

// A from tensor memory, B from shared memory
__device__ __forceinline__ void umma_i8_ts(unsigned d_tmem, unsigned a_tmem, unsigned long long b_desc, unsigned idesc, unsigned accumulate)
{
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

template <int XBITS, int WBITS, typename OutT, int TW>
__global__ void __launch_bounds__(THREADS, 1) k_tc_qgemm(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap,
                                                         const __grid_constant__ QgemmParams P)
{
    typedef Shape<TW> SH;
    constexpr int STAGES = SH::STAGES, SETS = SH::SETS, SET_WARPS = 4 + TW;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* sm_b = base;
    unsigned char* sm_p = base + STAGES * SH::B_STAGE;                            // a stage: weight rows, then token rows
    Ctl* S = reinterpret_cast<Ctl*>(sm_p + STAGES * SH::P_STAGE);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    constexpr int WB = WBITS * 16, XB = XBITS * 16;                               // packed bytes per row and step

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S->pfull[s], 1);
            mbar_init(&S->pempty[s], SET_WARPS);
            mbar_init(&S->ofull[s], SET_WARPS);
            mbar_init(&S->oempty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&S->tfull[a], 1);
            mbar_init(&S->tempty[a], EPI_WARPS);
        }
        mbar_init(&S->tshared, EPI_WARPS);
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&S->tmem_base, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = S->tmem_base;
    // programmatic dependent launch: the codes may still be being written until this returns
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int first = (int)blockIdx.x, step = (int)gridDim.x;
    const int n_mine = first < P.tiles ? (P.tiles - first + step - 1) / step : 0;

    if (warp == 0) {
        // ------------------------------ TMA producer (packed codes) ------------------------------
        if (lane == 0) {
            int c = 0;
            bool ok = true;
            for (int i = 0; ok && i < n_mine; ++i) {
                const int tile = first + i * step, mt = tile % P.m_tiles, nt = tile / P.m_tiles;
                for (int kb = 0; kb < P.kblocks; ++kb, ++c) {
                    const int s = c % STAGES;
                    if (!mbar_wait(&S->abort_flag, &S->pempty[s], ((c / STAGES) & 1) ^ 1, P.status, 1)) { ok = false; break; }
                    mbar_arrive_expect_tx(&S->pfull[s], (unsigned)(TM * WB + P.xbox * XB));
                    tma_load_2d(sm_p + s * SH::P_STAGE, &wmap, &S->pfull[s], kb * WB, mt * TM);
                    tma_load_2d(sm_p + s * SH::P_STAGE + TM * 64, &xmap, &S->pfull[s], kb * XB, nt * P.n);
                }
            }
            if (!ok) drain_copies(S->pfull, STAGES, c);
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        {
            const unsigned idesc = instr_desc_i8(TM, P.n);
            int c = 0;
            bool ok = true;
            for (int i = 0; ok && i < n_mine; ++i) {
                const int a = i & 1;
                if (!mbar_wait_warp(&S->abort_flag, &S->tempty[a], ((i >> 1) & 1) ^ 1, P.status, 3)) break;
                // the columns shared with the tile before are drained first
                if (TW == 8 && !mbar_wait_warp(&S->abort_flag, &S->tshared, (i & 1) ^ 1, P.status, 3)) break;
                for (int kb = 0; kb < P.kblocks; ++kb, ++c) {
                    const int s = c % STAGES;
                    if (!mbar_wait_warp(&S->abort_flag, &S->ofull[s], (c / STAGES) & 1, P.status, 2)) { ok = false; break; }
                    tc_fence_after();
                    // an instruction takes 32 codes: eight columns of the weights' lanes, 32 bytes of the tokens' lines
                    const unsigned long long bd = smem_desc(smem_u32(sm_b + s * SH::B_STAGE), 16, 1024, 2);
#pragma unroll
                    for (int ks = 0; ks < KB / 32; ++ks)
                        umma_i8_ts(tmem_base + a * SH::ACC_STEP, tmem_base + SH::A_COL0 + s * 32 + ks * 8, bd + (unsigned long long)(2 * ks),
                                   idesc, (kb | ks) != 0 ? 1u : 0u);
                    umma_commit(&S->oempty[s]);
                }
                if (ok) umma_commit(&S->tfull[a]);
            }
        }
    } else if (warp < 2 + UNPACK_WARPS) {
        // ------------------------------ unpack ------------------------------
        // Sets take alternate steps, so that one set's waits are covered by the others' work.
        const int set = (warp - 2) / SET_WARPS, member = (warp - 2) % SET_WARPS;
        const bool weights = member < 4;
        const int r = weights ? (warp & 3) * 32 + lane : (member - 4) * 32 + lane;     // weights: the warp's own lane quadrant
        const unsigned lane_base = tmem_base + ((unsigned)((warp & 3) * 32) << 16) + SH::A_COL0;
        const int total = n_mine * P.kblocks;
        const bool have = weights || r < P.n;
        for (int c = set; c < total; c += SETS) {
            const int s = c % STAGES;
            const unsigned ph = (unsigned)(c / STAGES) & 1u;
            bool ok = mbar_wait(&S->abort_flag, &S->pfull[s], ph, P.status, 4);
            if (!__all_sync(0xffffffffu, ok)) break;                             // a warp leaves as one
            const unsigned rows = smem_u32(sm_p + s * SH::P_STAGE);
            if (weights) {
                uint4 w[WBITS];
                load_row128<WBITS>(rows, r, w);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->pempty[s]);
                ok = mbar_wait(&S->abort_flag, &S->oempty[s], ph ^ 1u, P.status, 5);
                if (!__all_sync(0xffffffffu, ok)) break;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    unsigned v[8];
                    unpack32<WBITS, XBITS == 3 || WBITS == 3>(w, k, v);
                    tmem_st8(lane_base + s * 32 + k * 8, v);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
            } else {
                uint4 w[XBITS];
                if (have) load_row128<XBITS>(rows + TM * 64, r, w);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->pempty[s]);
                ok = mbar_wait(&S->abort_flag, &S->oempty[s], ph ^ 1u, P.status, 5);
                if (!__all_sync(0xffffffffu, ok)) break;
                if (have) {
                    const unsigned line = smem_u32(sm_b + s * SH::B_STAGE) + (unsigned)r * 128u;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        unsigned v[8];
                        unpack32<XBITS, XBITS == 3 || WBITS == 3>(w, k, v);
                        st_shared_v4(line + (unsigned)(((2 * k) ^ (r & 7)) << 4), make_uint4(v[0], v[1], v[2], v[3]));
                        st_shared_v4(line + (unsigned)(((2 * k + 1) ^ (r & 7)) << 4), make_uint4(v[4], v[5], v[6], v[7]));
                    }
                }
                // make the generic-proxy writes visible to the tensor cores' (async proxy) reads, then signal
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&S->ofull[s]);
        }
    } else {
        // ------------------------------ epilogue: lane = output channel, column = token ------------------------------
        const int q = warp & 3;
        for (int i = 0; i < n_mine; ++i) {
            const int tile = first + i * step, mt = tile % P.m_tiles, nt = tile / P.m_tiles, a = i & 1;
            const long long o = (long long)mt * TM + q * 32 + lane;
            const long long t0 = (long long)nt * P.n;
            const float dw = o < P.n_out ? __ldg(P.sw + o) : 0.f;
            const bool ok = mbar_wait(&S->abort_flag, &S->tfull[a], (i >> 1) & 1, P.status, 6);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            // TMEM columns [128, 256) belong to both accumulators of a wide tile: the upper half of the even ones, the lower
            // half of the odd ones, drained first
            const int shift = (TW == 8 && a == 0) ? 128 : 0;
            for (int j = 0; j < SH::TN; j += 32) {
                const int c0 = TW == 8 ? (j + shift) & 255 : j;
                if (TW == 8 && j == 128) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&S->tshared);
                }
                if (c0 >= P.n) continue;
                store_tokens<XBITS + WBITS, OutT>(tmem_base + ((unsigned)(q * 32) << 16) + (unsigned)(a * SH::ACC_STEP + c0), t0 + c0, o, dw, lane, P);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S->tempty[a]);
        }
    }

    // ---- teardown: every role has left its loop (normally or after a wait expired); TMEM is freed
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

typedef void (*QgemmKernel)(const CUtensorMap, const CUtensorMap, const QgemmParams);
template <int TW>
QgemmKernel pick(int xbits, int wbits, int out_dtype)
{
    static const QgemmKernel table[2][2][2] = {
        {{k_tc_qgemm<3, 3, float, TW>, k_tc_qgemm<3, 3, __nv_bfloat16, TW>}, {k_tc_qgemm<3, 4, float, TW>, k_tc_qgemm<3, 4, __nv_bfloat16, TW>}},
        {{k_tc_qgemm<4, 3, float, TW>, k_tc_qgemm<4, 3, __nv_bfloat16, TW>}, {k_tc_qgemm<4, 4, float, TW>, k_tc_qgemm<4, 4, __nv_bfloat16, TW>}}};
    return table[xbits - 3][wbits - 3][out_dtype == GBS_DTYPE_F32 ? 0 : 1];
}

// Tokens per tile, and whether tiles are 256 channels on a pair of SMs (gbs_tc_qgemm2.cu) or 128 on one.  A step of 128 codes was measured at
// 600 cycles up to 96 tokens and 2.6 more per token beyond (1016 at 256) on one SM, at 500 and 0.9 per token on a pair, whose start and end take
// 3500 cycles longer (2000 where a side has three bits: their step on one SM is the slower one); tiles go in waves over the SMs.  (4096
// wide, 4 bits: 400 tokens -> 4096 15.3 us on one and 15.5 on pairs, 520: 17.4 and 16.3, 2048: 34.9 and 31.5; 130 -> 9472: 13.6 and 15.1,
// 260: 17.1 and 16.1; 3 bits: 2048 -> 1024 16.5 and 16.1, 100 -> 14336 18.1 and 16.6.)  The width with the least total is taken: 256 where the output fills the chip, narrow
// tiles on more SMs where it does not.  `pairs`: how many there are; where clusters of two cannot be launched, none.
int pick_tokens(long long n_tok, long long n_out, int kblocks, bool three, int sm_count, int pairs, bool& on_pairs)
{
    double best = 0.0;
    int n_best = 0;
    on_pairs = false;
    for (int n = 32; n <= 256; n += 32) {
        const long long tiles = ((n_out + TM - 1) / TM) * ((n_tok + n - 1) / n);
        const long long waves = (tiles + sm_count - 1) / sm_count;
        const double unit = n <= 96 ? 600.0 : 600.0 + 2.6 * (n - 96);
        const double cost = (double)waves * kblocks * unit + 8.0 * n;
        if (n_best == 0 || cost < best) { best = cost; n_best = n; }
    }
    for (int n = 64; pairs > 0 && n <= GBS_QGEMM2_MAX_TOKENS; n += 32) {
        const long long tiles = ((n_out + 2 * TM - 1) / (2 * TM)) * ((n_tok + n - 1) / n);
        const long long waves = (tiles + pairs - 1) / pairs;
        const double cost = (double)waves * kblocks * (500.0 + 0.9 * n) + 8.0 * n + (three ? 2000.0 : 3500.0);
        if (cost < best) { best = cost; n_best = n; on_pairs = true; }
    }
    return n_best;
}

// Whether the few-token kernel (gbs_qgemv.cu) is the faster one, by cycles per step of 128 codes.  Tiles of 128 channels come in waves over
// the SMs, 600 cycles each whatever they hold, with much the same start.  The few-token kernel's 17 - 64 tokens come in waves of 32 channels
// per SM (4736 on 148): 300 cycles each up to 32 tokens, 600 up to 64.  So 32 tokens go to the tiles beyond two such waves and 64 beyond one.
// Up to 16 tokens, and up to 32 with three bits on a side, the time was measured to grow with the channels of an SM.  Four bits: up to 8
// tokens never go to the tiles, up to 16 beyond 18 200 channels until the tiles' second wave begins (18 944), and so on in every wave.
// Three bits: up to 8 tokens likewise beyond 17 100, 16 beyond 8800, 32 beyond 7800.  4096 wide, weights not in L2, few-token kernel and tiles, four
// bits: 20 tokens -> 9472: 10.6 and 11.7 us, 10 240: 14.1 and 11.8; 32 -> 8704: 10.3 and 11.6, 9472: 10.6 and 11.7, 10 240: 14.0 and 11.8; 64 -> 4736:
// 8.1 and 11.6, 5760: 14.1 and 11.6; three bits: 20 -> 7168: 11.2 and 12.5, 10 240: 16.0 and 12.7; 32 -> 7168: 12.3 and 12.5, 9472: 12.0 and 12.6,
// 10 240: 17.3 and 12.7; 64 -> 4736: 10.1 and 12.4, 5760: 18.8 and 12.5.
bool few_tokens(long long n_tok, long long n_out, bool three, int sm_count)
{
    if (n_tok > GBS_QGEMV_MAX_TOKENS) return false;
    const long long tiles = (n_out + TM - 1) / TM, tile_waves = (tiles + sm_count - 1) / sm_count;
    if (n_tok > 32 || (n_tok > 16 && !three)) {
        const long long waves = (n_out + 32ll * sm_count - 1) / (32ll * sm_count);
        return waves * (n_tok > 32 ? 600 : 300) <= 600 * tile_waves;
    }
    // per channel of the whole chip, on 148 SMs
    static const double per_channel[2][3] = {{0.021, 0.033, 0.0}, {0.035, 0.068, 0.077}};
    const double cycles = per_channel[three ? 1 : 0][n_tok <= 8 ? 0 : n_tok <= 16 ? 1 : 2] * 148.0 / sm_count;
    return (double)n_out * cycles <= 600.0 * (double)tile_waves;
}

bool encode_codes(EncodeTiledFn encode, CUtensorMap* map, const void* codes, int64_t rows, int row_bytes, int bits, int box_rows)
{
    const cuuint64_t gdim[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
    const cuuint64_t gstr[1] = {(cuuint64_t)row_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)(bits * 16), (cuuint32_t)box_rows}, estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(codes), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  bits == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

extern "C" int gbs_matmul_rule(int64_t n_tokens, int64_t n_out, int kblocks, int three, int sm_count, int pairs, int* tile_tokens)
{
    *tile_tokens = (int)n_tokens;
    if (few_tokens(n_tokens, n_out, three != 0, sm_count)) return GBS_MATMUL_FEW_TOKENS;
    bool on_pairs;
    *tile_tokens = pick_tokens(n_tokens, n_out, kblocks, three != 0, sm_count, pairs, on_pairs);
    return on_pairs ? GBS_MATMUL_PAIRS : GBS_MATMUL_TILES;
}

extern "C" int gbs_quantized_matmul(const gbs_plan_t* px, const void* codes_x, const float* scales_x, int64_t n_tokens,
                                    const gbs_plan_t* pw, const void* codes_w, const float* scales_w, int64_t n_out,
                                    void* out, int out_dtype, int64_t out_row_stride, void* cuda_stream)
{
    if (!px || !pw) return GBS_ERR_INVALID_ARG;
    if (out_dtype != GBS_DTYPE_F32 && out_dtype != GBS_DTYPE_BF16) return GBS_ERR_INVALID_ARG;
    if (n_tokens < 0 || n_out < 0 || out_row_stride < n_out) return GBS_ERR_INVALID_ARG;
    if (px->d_pad != pw->d_pad || px->d != pw->d || px->m != pw->m) return GBS_ERR_INVALID_ARG;   // one rotation for both sides
    if (px->device != pw->device) return GBS_ERR_INVALID_ARG;
    // one symmetric scale per token and per output channel, so that the scales leave the contraction
    if (px->group != 0 || pw->group != 0 || px->asym || pw->asym) return GBS_ERR_UNSUPPORTED;
    if (px->d_pad % KB != 0) return GBS_ERR_UNSUPPORTED;
    if (px->smem_optin < (int)(Shape<8>::SMEM)) return GBS_ERR_UNSUPPORTED;
    if (n_tokens == 0 || n_out == 0) return GBS_OK;
    if (n_tokens > (int64_t)0x7fffffff - 256 || n_out > (int64_t)0x7fffffff - 256) return GBS_ERR_INVALID_ARG;   // TMA coordinates are 32-bit
    if (!codes_x || !scales_x || !codes_w || !scales_w || !out) return GBS_ERR_INVALID_ARG;
    const int esz = out_dtype == GBS_DTYPE_F32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(codes_x) & 15u) || (reinterpret_cast<uintptr_t>(codes_w) & 15u) ||
        (reinterpret_cast<uintptr_t>(out) & (uintptr_t)(esz - 1)) ||
        (reinterpret_cast<uintptr_t>(scales_x) & 3u) || (reinterpret_cast<uintptr_t>(scales_w) & 3u))
        return GBS_ERR_ALIGNMENT;
    gbs_device_guard guard;
    if (guard.enter(px->device) != cudaSuccess) { cudaGetLastError(); return GBS_ERR_CUDA; }

    // a few tokens are bound by latencies: no 128-channel tile, the whole chip on the weight rows
    if (few_tokens(n_tokens, n_out, px->bits == 3 || pw->bits == 3, px->sm_count)) {
        const int e = gbs_qgemv(px, codes_x, scales_x, (int)n_tokens, pw, codes_w, scales_w, n_out, out, out_dtype, out_row_stride,
                                static_cast<cudaStream_t>(cuda_stream));
        if (e != 0) cudaGetLastError();
        return e == 0 ? GBS_OK : GBS_ERR_CUDA;
    }
    EncodeTiledFn encode = get_encode();
    if (!encode) return GBS_ERR_CUDA;
    QgemmParams P;
    memset(&P, 0, sizeof(P));
    P.n_tok = n_tokens;
    P.n_out = n_out;
    P.kblocks = px->d_pad / KB;
    P.sx = scales_x;
    P.sw = scales_w;
    P.out = out;
    P.out_stride = out_row_stride;
    P.status = px->d_status;
    const int pairs = gbs_tc_qgemm2_pairs(px);
    bool on_pairs;
    P.n = pick_tokens(n_tokens, n_out, P.kblocks, px->bits == 3 || pw->bits == 3, px->sm_count, pairs, on_pairs);
    const int box_rows = on_pairs ? P.n / 2 : P.n;                   // an SM of a pair brings half the tokens
    // Rows of a box beyond the tensor's end are slow to fill where no swizzle is set (16 of 32 rows of three-bit codes: 15.8 us instead
    // of 12.2 at 14336 channels).  What shared memory holds beyond the box goes into sums that are not stored.  (A map of its own for
    // the last of several token tiles costs other calls as much as it gains.)
    P.xbox = n_tokens < box_rows ? (int)n_tokens : box_rows;
    const int channels = on_pairs ? 2 * TM : TM;
    P.m_tiles = (int)((n_out + channels - 1) / channels);
    const long long tiles = (long long)P.m_tiles * ((n_tokens + P.n - 1) / P.n);
    if (tiles > 0x7fffffff / 2) return GBS_ERR_INVALID_ARG;
    P.tiles = (int)tiles;
    CUtensorMap wmap, xmap;
    if (!encode_codes(encode, &wmap, codes_w, n_out, pw->d_pad * pw->bits / 8, pw->bits, TM) ||
        !encode_codes(encode, &xmap, codes_x, n_tokens, px->d_pad * px->bits / 8, px->bits, P.xbox))
        return GBS_ERR_CUDA;
    if (on_pairs) {
        const int e = gbs_tc_qgemm2(px, pw, wmap, xmap, P, pairs, out_dtype, static_cast<cudaStream_t>(cuda_stream));
        if (e != 0) cudaGetLastError();
        return e == 0 ? GBS_OK : GBS_ERR_CUDA;
    }
    const bool wide = P.n > 128;
    const int smem = wide ? Shape<8>::SMEM : Shape<4>::SMEM;
    QgemmKernel kernel = wide ? pick<8>(px->bits, pw->bits, out_dtype) : pick<4>(px->bits, pw->bits, out_dtype);
    {
        // opt in to the large dynamic shared memory once per device and instantiation (not a stream operation)
        static std::mutex mu;
        static bool done[64][16] = {{false}};
        const int ki = (wide ? 8 : 0) + (px->bits - 3) * 4 + (pw->bits - 3) * 2 + (out_dtype == GBS_DTYPE_F32 ? 0 : 1);
        std::lock_guard<std::mutex> lock(mu);
        if (!(px->device >= 0 && px->device < 64 && done[px->device][ki])) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
                cudaGetLastError();
                return GBS_ERR_CUDA;
            }
            if (px->device >= 0 && px->device < 64) done[px->device][ki] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(P.tiles < px->sm_count ? P.tiles : px->sm_count));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = static_cast<cudaStream_t>(cuda_stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = px->pdl ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, kernel, wmap, xmap, P) != cudaSuccess) { cudaGetLastError(); return GBS_ERR_CUDA; }
    return GBS_OK;
}

// Weight side of Eq. (2): every row of W (one output channel, width d) is zero-padded, rotated and quantized like a
// token row -- round to nearest, one scale per output channel when the plan has group 0.
extern "C" int gbs_weight_rotate_quantize(const gbs_plan_t* plan, const void* w, int w_dtype, int64_t n_out,
                                          int64_t w_row_stride, void* codes, float* scales, void* cuda_stream)
{
    if (!plan) return GBS_ERR_INVALID_ARG;
    if (plan->asym) return GBS_ERR_UNSUPPORTED;
    return gbs_rotate_quantize(plan, w, w_dtype, n_out, w_row_stride, codes, scales, nullptr, cuda_stream);
}
