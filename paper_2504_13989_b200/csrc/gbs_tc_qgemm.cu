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
//   * Output channels are the rows of the MMA (TMEM lane = channel), tokens its columns.  A tile is 128 channels x N tokens
//     on one SM, or 256 x N on a pair of SMs (cta_group::2): each SM unpacks 128 rows of weights and half of the tokens, so
//     a code of either operand is unpacked once per 256 outputs of the other.
//   * Packed codes arrive by TMA (128 codes of every row per step, four steps ahead).  Sixteen warps unpack, one thread per row:
//     a field moved to the top bits of its byte IS the int8 q * 2^(8-b) (the epilogue removes the power of two).  Weights go to
//     TENSOR MEMORY (a thread's 128 int8 are 32 columns of its lane), tokens to 128-byte-swizzled K-major rows in shared memory;
//     both use the same order of the codes inside a word (even fields, then odd), which a dot product does not see.
//   * One thread issues tcgen05.mma kind::i8 (int32 accumulators, exact); two accumulators in TMEM, so that four epilogue
//     warps convert and store a tile while the next one is contracted.  Lanes of a warp hold consecutive channels, so every
//     store instruction writes 64 or 128 contiguous bytes of one token's row.
// What bounds it: the shared-memory port (per step and SM: packed codes in and out, token operand in and out) about level
// with the tensor pipe for pairs.  The single-SM kernel before it fetched packed codes with global loads, kept both operands in
// shared memory and held the L1 74 % busy: 139 us for 4096 x 4096 x 4096 at 4 bits.
// Every wait is bounded; an expired wait records a code in the activation plan's status word.
#include <math.h>
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_qfields.cuh"
#include "gbs_tc_common.cuh"

namespace {

constexpr int KB = 128;                 // codes per step and row: one 128-byte line of int8
constexpr int ROWS = 128;               // rows of each operand one SM unpacks at most
constexpr int STAGES = 4;               // of packed codes, and of unpacked operands; even: see `set` below
constexpr int P_OPERAND = ROWS * 64;    // packed bytes of one operand's rows in a stage (64 or 48 per row)
constexpr int B_STAGE = ROWS * KB;      // 16 KB of int8
constexpr int SETS = 2;                 // warp sets that take alternate steps
constexpr int UNPACK_WARPS = 8 * SETS;  // per set: four for the weights (one per TMEM lane quadrant), four for the tokens
constexpr int EPI_WARPS = 4;
constexpr int THREADS = 32 * (2 + UNPACK_WARPS + EPI_WARPS);
constexpr int TMEM_COLS = 512;
constexpr int ACC_COLS = 192;           // columns of an accumulator: two of them, and STAGES x 32 columns of weights
constexpr int A_COL0 = 2 * ACC_COLS;

struct __align__(1024) Smem {
    unsigned char p[STAGES][2][P_OPERAND];
    unsigned char b[STAGES][B_STAGE];
    unsigned long long pfull[STAGES], pempty[STAGES], ofull[STAGES], oempty[STAGES], tfull[2], tempty[2];
    unsigned tmem_base;
    volatile int abort_flag;
};

struct QgemmParams {
    long long n_tok, n_out;
    int n;                              // tokens per tile (MMA N)
    int m_tiles, tiles;                 // channel tiles, all tiles
    int kblocks;                        // d' / 128
    const float* sx;
    const float* sw;
    void* out;
    long long out_stride;               // elements
    int* status;
};

// Instruction descriptor, kind::i8: int32 accumulate, signed 8-bit A and B, both K-major, M x N.
__host__ __device__ constexpr unsigned instr_desc_i8(int M, int N)
{
    return (2u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

// A from tensor memory, B from shared memory
template <int CG>
__device__ __forceinline__ void umma_i8_ts(unsigned d_tmem, unsigned a_tmem, unsigned long long b_desc, unsigned idesc, unsigned accumulate)
{
    if (CG == 2)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
                     ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
                     ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// completion of the MMAs so far, on this barrier of every SM of the pair
template <int CG>
__device__ __forceinline__ void commit_all(void* bar)
{
    if (CG == 2)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                     ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
    else
        umma_commit(bar);
}
template <int CG>
__device__ __forceinline__ void tmem_alloc_cg(unsigned* slot)
{
    if (CG == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        tmem_alloc(slot, TMEM_COLS);
    }
}
template <int CG>
__device__ __forceinline__ void tmem_dealloc_cg(unsigned addr)
{
    if (CG == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(TMEM_COLS) : "memory");
    else tmem_dealloc(addr, TMEM_COLS);
}
// arrive on a barrier of the pair's first SM (the one that issues the MMAs)
template <int CG>
__device__ __forceinline__ void arrive_leader(void* bar)
{
    if (CG == 2) {
        unsigned a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(bar)), "r"(0));
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(a) : "memory");
    } else {
        mbar_arrive(bar);
    }
}
__device__ __forceinline__ bool try_wait_cluster(void* bar, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(WAIT_HINT_NS) : "memory");
    return ok != 0;
}
// bounded wait for arrivals of either SM of the pair
template <int CG>
__device__ __forceinline__ bool wait_pair(volatile int* abort_flag, void* bar, unsigned parity, int* status, int code)
{
    if (CG == 1) return mbar_wait(abort_flag, bar, parity, status, code);
    if (try_wait_cluster(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned i = 1;; ++i) {
        if (try_wait_cluster(bar, parity)) return true;
        if ((i & 15u) == 0) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > WAIT_LIMIT_NS) break;
        }
    }
    *abort_flag = 1;
    atomicCAS(status, 0, code);
    return false;
}
template <int CG>
__device__ __forceinline__ void pair_sync()
{
    if (CG == 2) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void st_shared_v4(unsigned addr, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(unsigned addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
// 32 registers -> 32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_st32(unsigned taddr, const unsigned r[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
        ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]), "r"(taddr) : "memory");
}

// The 128 codes of row r in a packed stage -> 32 words of int8: per octet of codes the even fields, then the odd ones.
// Four-bit rows are 64 bytes with the 64-byte swizzle (eight rows side by side hit all banks), three-bit rows 48 bytes plain
// (48-byte steps do so by themselves).
template <int BITS>
__device__ __forceinline__ void unpack_row128(unsigned rows, int r, unsigned v[32])
{
    if (BITS == 4) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint4 w = ld_shared_v4(rows + (unsigned)r * 64u + (unsigned)((c ^ ((r >> 1) & 3)) << 4));
            fields_to_int8<4>(w.x, v[8 * c], v[8 * c + 1]);
            fields_to_int8<4>(w.y, v[8 * c + 2], v[8 * c + 3]);
            fields_to_int8<4>(w.z, v[8 * c + 4], v[8 * c + 5]);
            fields_to_int8<4>(w.w, v[8 * c + 6], v[8 * c + 7]);
        }
    } else {
        unsigned w[12];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const uint4 x = ld_shared_v4(rows + (unsigned)r * 48u + 16u * c);
            w[4 * c] = x.x; w[4 * c + 1] = x.y; w[4 * c + 2] = x.z; w[4 * c + 3] = x.w;
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const unsigned w0 = w[3 * g], w1 = w[3 * g + 1], w2 = w[3 * g + 2];
            fields_to_int8<3>(w0, v[8 * g], v[8 * g + 1]);                       // bits above 24 are dropped by the masks
            fields_to_int8<3>(__funnelshift_r(w0, w1, 24), v[8 * g + 2], v[8 * g + 3]);
            fields_to_int8<3>(__funnelshift_r(w1, w2, 16), v[8 * g + 4], v[8 * g + 5]);
            fields_to_int8<3>(w2 >> 8, v[8 * g + 6], v[8 * g + 7]);
        }
    }
}

template <int XBITS, int WBITS, typename OutT, int CG>
__global__ void __launch_bounds__(THREADS, 1) k_tc_qgemm(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap,
                                                         const __grid_constant__ QgemmParams P)
{
    extern __shared__ unsigned char smem_raw[];
    Smem* S = reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = CG == 2 ? (int)(blockIdx.x & 1) : 0;
    const int first = (int)blockIdx.x / CG, step = (int)gridDim.x / CG;          // tiles first, first + step, ..
    const int nb = P.n / CG;                                                      // token rows this SM unpacks
    constexpr int WB = WBITS * 16, XB = XBITS * 16;                               // packed bytes per row and step

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S->pfull[s], 1);
            mbar_init(&S->pempty[s], 8);
            mbar_init(&S->ofull[s], 8 * CG);
            mbar_init(&S->oempty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&S->tfull[a], 1);
            mbar_init(&S->tempty[a], EPI_WARPS * CG);
        }
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc_cg<CG>(&S->tmem_base);
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    pair_sync<CG>();                                                             // the peer's barriers are ready
    tc_fence_after();
    const unsigned tmem_base = S->tmem_base;
    // programmatic dependent launch: the codes may still be being written until this returns
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int n_mine = first < P.tiles ? (P.tiles - first + step - 1) / step : 0;

    if (warp == 0) {
        // ------------------------------ TMA producer (packed codes) ------------------------------
        if (lane == 0) {
            int c = 0;
            bool ok = true;
            for (int i = 0; ok && i < n_mine; ++i) {
                const int tile = first + i * step, mt = tile % P.m_tiles, nt = tile / P.m_tiles;
                const int w0 = (mt * CG + rank) * ROWS, x0 = nt * P.n + rank * nb;
                for (int kb = 0; kb < P.kblocks; ++kb, ++c) {
                    const int s = c % STAGES;
                    if (!mbar_wait(&S->abort_flag, &S->pempty[s], ((c / STAGES) & 1) ^ 1, P.status, 1)) { ok = false; break; }
                    mbar_arrive_expect_tx(&S->pfull[s], (unsigned)(ROWS * WB + nb * XB));
                    tma_load_2d(S->p[s][0], &wmap, &S->pfull[s], kb * WB, w0);
                    tma_load_2d(S->p[s][1], &xmap, &S->pfull[s], kb * XB, x0);
                }
            }
            if (!ok) drain_copies(S->pfull, STAGES, c);
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer (the pair's first SM) ------------------------------
        if (lane == 0 && rank == 0) {
            const unsigned idesc = instr_desc_i8(ROWS * CG, P.n);
            int c = 0;
            bool ok = true;
            for (int i = 0; ok && i < n_mine; ++i) {
                const int a = i & 1;
                if (!wait_pair<CG>(&S->abort_flag, &S->tempty[a], ((i >> 1) & 1) ^ 1, P.status, 3)) break;
                for (int kb = 0; kb < P.kblocks; ++kb, ++c) {
                    const int s = c % STAGES;
                    if (!wait_pair<CG>(&S->abort_flag, &S->ofull[s], (c / STAGES) & 1, P.status, 2)) { ok = false; break; }
                    tc_fence_after();
                    // an instruction takes 32 codes: eight columns of the weights' lanes, 32 bytes of the tokens' lines
                    const unsigned long long bd = smem_desc(smem_u32(S->b[s]), 16, 1024, 2);
#pragma unroll
                    for (int ks = 0; ks < KB / 32; ++ks)
                        umma_i8_ts<CG>(tmem_base + a * ACC_COLS, tmem_base + A_COL0 + s * 32 + ks * 8, bd + (unsigned long long)(2 * ks),
                                       idesc, (kb | ks) != 0 ? 1u : 0u);
                    commit_all<CG>(&S->oempty[s]);
                }
                if (ok) commit_all<CG>(&S->tfull[a]);
            }
        }
    } else if (warp < 2 + UNPACK_WARPS) {
        // ------------------------------ unpack ------------------------------
        // Two sets of eight warps take alternate steps, so that one set's waits (packed codes, a free stage, its own stores
        // becoming visible) are covered by the other's work.  STAGES is even: a stage belongs to one set, which therefore takes
        // part in every phase of the barriers it waits for.
        const int set = (warp - 2) >> 3, role = ((warp - 2) >> 2) & 1, q = warp & 3, r = q * 32 + lane;
        const unsigned lane_base = tmem_base + ((unsigned)(q * 32) << 16) + A_COL0;
        const int total = n_mine * P.kblocks;
        const bool have = role == 0 || r < nb;
        for (int c = set; c < total; c += SETS) {
            const int s = c % STAGES;
            const unsigned ph = (unsigned)(c / STAGES) & 1u;
            bool ok = mbar_wait(&S->abort_flag, &S->pfull[s], ph, P.status, 4);
            if (!__all_sync(0xffffffffu, ok)) break;                             // a warp leaves as one
            unsigned v[32];
            if (role == 0) unpack_row128<WBITS>(smem_u32(S->p[s][0]), r, v);
            else if (have) unpack_row128<XBITS>(smem_u32(S->p[s][1]), r, v);
            __syncwarp();
            if (lane == 0) mbar_arrive(&S->pempty[s]);
            ok = mbar_wait(&S->abort_flag, &S->oempty[s], ph ^ 1u, P.status, 5);
            if (!__all_sync(0xffffffffu, ok)) break;
            if (role == 0) {
                tc_fence_after();
                tmem_st32(lane_base + s * 32, v);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
            } else {
                if (have) {
                    const unsigned line = smem_u32(S->b[s]) + (unsigned)r * 128u;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        st_shared_v4(line + (unsigned)((k ^ (r & 7)) << 4), make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]));
                }
                // make the generic-proxy writes visible to the tensor cores' (async proxy) reads, then signal
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) arrive_leader<CG>(&S->ofull[s]);
        }
    } else {
        // ------------------------------ epilogue: lane = output channel, column = token ------------------------------
        const int q = warp & 3;
        for (int i = 0; i < n_mine; ++i) {
            const int tile = first + i * step, mt = tile % P.m_tiles, nt = tile / P.m_tiles, a = i & 1;
            const long long o = (long long)(mt * CG + rank) * ROWS + q * 32 + lane;
            const long long t0 = (long long)nt * P.n;
            const float dw = o < P.n_out ? __ldg(P.sw + o) : 0.f;
            const bool ok = mbar_wait(&S->abort_flag, &S->tfull[a], (i >> 1) & 1, P.status, 6);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            for (int c0 = 0; c0 < P.n; c0 += 32) {
                unsigned v[32];
                tmem_ld32_issue(tmem_base + ((unsigned)(q * 32) << 16) + (unsigned)(a * ACC_COLS + c0), v);
                // the int8 operands were q * 2^(8 - bits): take the two powers of two out again (exact)
                const float dx_l = t0 + c0 + lane < P.n_tok ? __ldg(P.sx + t0 + c0 + lane) * (1.f / (float)(1 << (16 - XBITS - WBITS))) : 0.f;
                tmem_ld_wait(v);
                const int cols = (int)((P.n_tok - t0 - c0) < 32 ? (P.n_tok - t0 - c0) : 32);
                OutT* dst = reinterpret_cast<OutT*>(P.out) + (t0 + c0) * P.out_stride + o;
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float dx = __shfl_sync(0xffffffffu, dx_l, e);
                    const float f = (float)(int)v[e] * (dx * dw);
                    if (e < cols && o < P.n_out) {
                        if (sizeof(OutT) == 4) *reinterpret_cast<float*>(dst) = f;
                        else *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(f);
                    }
                    dst += P.out_stride;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_leader<CG>(&S->tempty[a]);
        }
    }

    // ---- teardown: every role has left its loop (normally or after a wait expired); no SM of a pair leaves before the other
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    pair_sync<CG>();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_cg<CG>(tmem_base);
    }
}

typedef void (*QgemmKernel)(const CUtensorMap, const CUtensorMap, const QgemmParams);
template <int CG>
QgemmKernel pick(int xbits, int wbits, int out_dtype)
{
    static const QgemmKernel table[2][2][2] = {
        {{k_tc_qgemm<3, 3, float, CG>, k_tc_qgemm<3, 3, __nv_bfloat16, CG>}, {k_tc_qgemm<3, 4, float, CG>, k_tc_qgemm<3, 4, __nv_bfloat16, CG>}},
        {{k_tc_qgemm<4, 3, float, CG>, k_tc_qgemm<4, 3, __nv_bfloat16, CG>}, {k_tc_qgemm<4, 4, float, CG>, k_tc_qgemm<4, 4, __nv_bfloat16, CG>}}};
    return table[xbits - 3][wbits - 3][out_dtype == GBS_DTYPE_F32 ? 0 : 1];
}

// Tile shape.  A step of 128 codes keeps the tensor pipe busy for 2 N cycles whatever the pairing, and the unpacking warps for
// about 300 + N; tiles go in waves over the SMs (or pairs).  The shape with the least total is taken: pairs with N = 192
// where the output fills the chip, single SMs with narrow tiles where it does not.
void pick_tile(long long n_tok, long long n_out, int kblocks, int sm_count, int* cg_out, int* n_out_cols)
{
    double best = 0.0;
    *cg_out = 0;
    for (int cg = 1; cg <= 2; ++cg)
        for (int n = 32; n <= (cg == 2 ? ACC_COLS : ROWS); n += 32) {
            const long long tiles = ((n_out + ROWS * cg - 1) / (ROWS * cg)) * ((n_tok + n - 1) / n);
            const long long waves = (tiles + sm_count / cg - 1) / (sm_count / cg);
            const double unit = 2.0 * n > 300.0 + n ? 2.0 * n : 300.0 + n;
            const double cost = (double)waves * kblocks * unit + 8.0 * n;
            if (*cg_out == 0 || cost < best) { best = cost; *cg_out = cg; *n_out_cols = n; }
        }
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
    if (px->smem_optin < (int)(sizeof(Smem) + 1024)) return GBS_ERR_UNSUPPORTED;
    if (n_tokens == 0 || n_out == 0) return GBS_OK;
    if (!codes_x || !scales_x || !codes_w || !scales_w || !out) return GBS_ERR_INVALID_ARG;
    const int esz = out_dtype == GBS_DTYPE_F32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(codes_x) & 15u) || (reinterpret_cast<uintptr_t>(codes_w) & 15u) ||
        (reinterpret_cast<uintptr_t>(out) & (uintptr_t)(esz - 1)) ||
        (reinterpret_cast<uintptr_t>(scales_x) & 3u) || (reinterpret_cast<uintptr_t>(scales_w) & 3u))
        return GBS_ERR_ALIGNMENT;
    gbs_device_guard guard;
    if (guard.enter(px->device) != cudaSuccess) { cudaGetLastError(); return GBS_ERR_CUDA; }

    // up to 64 tokens the call is bound by reading the weights: no 128-token tile, the whole chip on the weight rows (crossover
    // in gbs_qgemv.cu)
    if (n_tokens <= GBS_QGEMV_MAX_TOKENS) {
        const int e = gbs_qgemv(px, codes_x, scales_x, (int)n_tokens, pw, codes_w, scales_w, n_out, out, out_dtype, out_row_stride,
                                static_cast<cudaStream_t>(cuda_stream));
        if (e != 0) cudaGetLastError();
        return e == 0 ? GBS_OK : GBS_ERR_CUDA;
    }
    EncodeTiledFn encode = get_encode();
    if (!encode) return GBS_ERR_CUDA;
    if (n_tokens > (int64_t)0x7fffffff - 256 || n_out > (int64_t)0x7fffffff - 256) return GBS_ERR_INVALID_ARG;   // TMA coordinates are 32-bit
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
    int cg = 1;
    pick_tile(n_tokens, n_out, P.kblocks, px->sm_count, &cg, &P.n);
    P.m_tiles = (int)((n_out + ROWS * cg - 1) / (ROWS * cg));
    const long long tiles = (long long)P.m_tiles * ((n_tokens + P.n - 1) / P.n);
    if (tiles > 0x7fffffff / 2) return GBS_ERR_INVALID_ARG;
    P.tiles = (int)tiles;
    CUtensorMap wmap, xmap;
    if (!encode_codes(encode, &wmap, codes_w, n_out, pw->d_pad * pw->bits / 8, pw->bits, ROWS) ||
        !encode_codes(encode, &xmap, codes_x, n_tokens, px->d_pad * px->bits / 8, px->bits, P.n / cg))
        return GBS_ERR_CUDA;
    const int smem = (int)sizeof(Smem) + 1024;
    QgemmKernel kernel = cg == 2 ? pick<2>(px->bits, pw->bits, out_dtype) : pick<1>(px->bits, pw->bits, out_dtype);
    {
        // opt in to the large dynamic shared memory once per device and instantiation (not a stream operation)
        static std::mutex mu;
        static bool done[64][16] = {{false}};
        const int ki = (cg - 1) * 8 + (px->bits - 3) * 4 + (pw->bits - 3) * 2 + (out_dtype == GBS_DTYPE_F32 ? 0 : 1);
        std::lock_guard<std::mutex> lock(mu);
        if (!(px->device >= 0 && px->device < 64 && done[px->device][ki])) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
                cudaGetLastError();
                return GBS_ERR_CUDA;
            }
            if (px->device >= 0 && px->device < 64) done[px->device][ki] = true;
        }
    }
    const int slots = px->sm_count / cg;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cg * (P.tiles < slots ? P.tiles : slots)));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = static_cast<cudaStream_t>(cuda_stream);
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (cg == 2) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = 2;
        attr[na].val.clusterDim.y = attr[na].val.clusterDim.z = 1;
        ++na;
    }
    if (px->pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)na;
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
