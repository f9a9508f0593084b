// gbs_quantized_matmul on pairs of SMs: tiles of 256 channels x up to 256 tokens (the arithmetic is that of gbs_tc_qgemm.cu).
//
// One SM's tile of 128 x 256 is bound by its shared-memory port: 24 KB of packed codes in and out and 32 KB of unpacked tokens in and
// out per step of 128 codes, about 900 cycles against 512 of the tensor pipe.  A pair shares the tokens: each SM unpacks its own 128
// channels (to its tensor memory) and half of the tokens (to its shared memory), and tcgen05.mma with cta_group::2 reads each half once
// for both.  16 KB in, out, in and out again are 512 cycles.
//   * Roles per SM: a producer, twenty-four unpacking warps in three sets that take every third step (four warps for channels, four
//     for tokens), four epilogue warps; the pair's first SM issues all MMAs.  Accumulators overlap by half as there.
//   * Both SMs' unpacking warps arrive at the issuer's barriers (cluster scope, see pair_arrive); commits are multicast to both.
//   * A set serves every third step and a stage of operands every fourth, so barriers are indexed by the step modulo twelve: each
//     waiter then takes part in every phase of the barriers it waits for.
// What bounds it: with 256 tokens a step takes about 730 cycles at 1.9 GHz, 512 of them the tensor pipe's, at the 1 kW limit (with a quarter of
// the MMAs 4096^3 takes 52.6 instead of 56 us; more stages of either kind, running indices and unpacking before the wait for a free
// stage change nothing or cost time); 256 tiles are 3.5 waves over 74 pairs and count as four.
// 4096 x 4096 x 4096: 4 bits 63.5 -> 55.9 us (2.46 POP/s, 0.74 of twice the measured bf16 rate), 3 bits 71.9 -> 60.3.  300 tokens -> 14336:
// 29.3 -> 26.2 and 33.6 -> 28.1.  1000 -> 4096: 19.7 -> 18.3 and 22.0 -> 19.4.
// Every wait is bounded; an expired wait records a code in the activation plan's status word, and both SMs come to the last barrier.
#include <string.h>

#include <mutex>

#include "gbs_qgemm.cuh"

namespace {

constexpr int TM = 128;                 // output channels of an SM: half a tile
constexpr int TN = 128;                 // tokens of an SM at most: half a tile
constexpr int SETS = 3, SET_WARPS = 8;
constexpr int UNPACK_WARPS = SETS * SET_WARPS;
constexpr int EPI_WARPS = 4;
constexpr int THREADS = 32 * (2 + UNPACK_WARPS + EPI_WARPS);
constexpr int TMEM_COLS = 512;
constexpr int STAGES = 4;               // of operands: unpacked tokens in shared memory, channels in tensor memory
constexpr int P_STAGES = 6;             // of packed codes
constexpr int BARS = 12;                // a multiple of SETS, STAGES and P_STAGES
constexpr int P_STAGE = (TM + TN) * 64;
constexpr int B_STAGE = TN * KB;
constexpr int ACC_STEP = 128;           // second accumulator's first column
constexpr int A_COL0 = 384;             // channels: 32 columns per stage
constexpr int SMEM = 1024 + STAGES * B_STAGE + P_STAGES * P_STAGE + 1024;

struct Ctl {
    unsigned long long pfull[BARS], pempty[BARS], oempty[BARS], tfull[2];
    unsigned long long ofull[BARS], tempty[2], tshared;           // used in the issuer's SM, with arrivals from both
    unsigned tmem_base;
    volatile int abort_flag;
};
static_assert(sizeof(Ctl) <= 1024, "control block");

__device__ __forceinline__ void pair_mma(unsigned d_tmem, unsigned a_tmem, unsigned long long b_desc, unsigned idesc, unsigned accumulate)
{
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
                 "@q tcgen05.mma.cta_group::2.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives at this barrier of both SMs when the MMAs issued so far are complete
__device__ __forceinline__ void pair_commit(void* bar)
{
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
                 "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
                 ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}

// Arrivals at the issuer's barriers and waits on barriers that the other SM's threads or commits arrive at.  Between threads of two CTAs the
// scope has to be the cluster's; what is ordered is named by the fences around them, as PTX's patterns for tcgen05 have it:
//   * tensor memory (channels written by tcgen05.st, accumulators read by tcgen05.ld): tcgen05.wait, tcgen05.fence::before_thread_sync and a
//     relaxed arrival; a relaxed wait and tcgen05.fence::after_thread_sync.  The same wait and fence stand behind a commit.
//   * tokens written to shared memory: fence.proxy.async by each lane, then one release per warp; the issuer acquires before it lets the
//     tensor cores (async proxy) read both SMs' shared memory.  Before a stage is written again the warps acquire behind the commit's wait.
// The fences are the ones restricted to shared memory: with them 4096^3 takes 55.9 us at 4 bits and 60.3 at 3 (56.1 and 59.8 with
// arrivals and waits of CTA scope; 700 tokens -> 9088 at 3 bits: 28.8 and 28.1).  An arrival with .release.cluster orders the writer's global accesses as well: 98.9 us.
__device__ __forceinline__ void pair_arrive(unsigned bar_addr)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_addr) : "memory");
}
__device__ __forceinline__ void release_tokens()
{
    asm volatile("fence.proxy.async::generic.release.sync_restrict::shared::cta.cluster;" ::: "memory");
}
__device__ __forceinline__ void acquire_tokens()
{
    asm volatile("fence.proxy.async::generic.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory");
}
__device__ __forceinline__ void acquire_stage()
{
    asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory");
}
__device__ __forceinline__ bool pair_try_wait(void* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(WAIT_HINT_NS) : "memory");
    return ok != 0;
}
// bounded, like mbar_wait
__device__ __noinline__ bool pair_wait_slow(volatile int* abort_flag, void* bar, unsigned parity, int* status, int code)
{
    const unsigned long long t0 = global_ns();
    for (unsigned i = 1;; ++i) {
        if (pair_try_wait(bar, parity)) return true;
        if ((i & 15u) == 0) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > WAIT_LIMIT_NS) break;
        }
    }
    *abort_flag = 1;
    atomicCAS(status, 0, code);
    return false;
}
__device__ __forceinline__ bool pair_wait(volatile int* abort_flag, void* bar, unsigned parity, int* status, int code)
{
    if (pair_try_wait(bar, parity)) return true;
    return pair_wait_slow(abort_flag, bar, parity, status, code);
}

template <int XBITS, int WBITS, typename OutT>
__global__ void __launch_bounds__(THREADS, 1) k_tc_qgemm2(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap,
                                                          const __grid_constant__ QgemmParams P)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* sm_b = base;
    unsigned char* sm_p = base + STAGES * B_STAGE;                                // a stage: channel rows, then token rows
    Ctl* S = reinterpret_cast<Ctl*>(sm_p + P_STAGES * P_STAGE);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();
    constexpr int WB = WBITS * 16, XB = XBITS * 16;                               // packed bytes per row and step

    if (threadIdx.x == 0) {
        for (int b = 0; b < BARS; ++b) {
            mbar_init(&S->pfull[b], 1);
            mbar_init(&S->pempty[b], SET_WARPS);
            mbar_init(&S->ofull[b], 2 * SET_WARPS);
            mbar_init(&S->oempty[b], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&S->tfull[a], 1);
            mbar_init(&S->tempty[a], 2 * EPI_WARPS);
        }
        mbar_init(&S->tshared, 2 * EPI_WARPS);
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S->tmem_base)), "r"((unsigned)TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    cluster_sync();                                                               // the peer's barriers are ready too
    tc_fence_after();
    const unsigned tmem_base = S->tmem_base;
    // programmatic dependent launch: the codes may still be being written until this returns
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int first = (int)blockIdx.x / 2, step = (int)gridDim.x / 2;
    const int n_mine = first < P.tiles ? (P.tiles - first + step - 1) / step : 0;
    const int total = n_mine * P.kblocks;
    const int half = P.n / 2;                                                     // tokens of this SM

    if (warp == 0) {
        // ------------------------------ TMA producer (packed codes) ------------------------------
        if (lane == 0) {
            int c = 0;
            bool ok = true;
            for (int i = 0; ok && i < n_mine; ++i) {
                const int tile = first + i * step, mt = tile % P.m_tiles, nt = tile / P.m_tiles;
                for (int kb = 0; kb < P.kblocks; ++kb, ++c) {
                    const int s = c % P_STAGES, b = c % BARS, before = c - P_STAGES;
                    if (before >= 0 && !mbar_wait(&S->abort_flag, &S->pempty[before % BARS], (unsigned)(before / BARS) & 1u, P.status, 1)) { ok = false; break; }
                    mbar_arrive_expect_tx(&S->pfull[b], (unsigned)(TM * WB + P.xbox * XB));
                    tma_load_2d(sm_p + s * P_STAGE, &wmap, &S->pfull[b], kb * WB, (2 * mt + rank) * TM);
                    tma_load_2d(sm_p + s * P_STAGE + TM * 64, &xmap, &S->pfull[b], kb * XB, nt * P.n + rank * half);
                }
            }
            if (!ok) drain_copies(S->pfull, BARS, c);
            // The last stages are not used again, but the commits that free them arrive here too: not after this block has ended.  (Leaving
            // those commits out costs a branch per step: 4096^3, 4 bits: 59.1 us instead of 56.1.)
            for (int l = c < STAGES ? 0 : c - STAGES; ok && l < c; ++l)
                ok = pair_wait(&S->abort_flag, &S->oempty[l % BARS], (unsigned)(l / BARS) & 1u, P.status, 5);
        }
    } else if (warp == 1 && rank == 0) {
        // ------------------------------ MMA issuer ------------------------------
        const unsigned idesc = instr_desc_i8(2 * TM, P.n);
        int c = 0;
        bool ok = true;
        for (int i = 0; ok && i < n_mine; ++i) {
            const int a = i & 1;
            ok = pair_wait(&S->abort_flag, &S->tempty[a], (unsigned)((i >> 1) & 1) ^ 1u, P.status, 3);
            // the columns shared with the tile before are drained first
            ok = ok && pair_wait(&S->abort_flag, &S->tshared, (unsigned)(i & 1) ^ 1u, P.status, 3);
            if (!__all_sync(0xffffffffu, ok)) break;
            for (int kb = 0; kb < P.kblocks; ++kb, ++c) {
                const int s = c % STAGES, b = c % BARS;
                const unsigned ph = (unsigned)(c / BARS) & 1u;
                ok = pair_wait(&S->abort_flag, &S->ofull[b], ph, P.status, 2);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                acquire_tokens();
                tc_fence_after();
                // an instruction takes 32 codes: eight columns of the channels' lanes, 32 bytes of the tokens' lines
                const unsigned long long bd = smem_desc(smem_u32(sm_b + s * B_STAGE), 16, 1024, 2);
#pragma unroll
                for (int ks = 0; ks < KB / 32; ++ks)
                    pair_mma(tmem_base + a * ACC_STEP, tmem_base + A_COL0 + s * 32 + ks * 8, bd + (unsigned long long)(2 * ks), idesc,
                             (kb | ks) != 0 ? 1u : 0u);
                pair_commit(&S->oempty[b]);
            }
            if (ok) pair_commit(&S->tfull[a]);
        }
    } else if (warp >= 2 && warp < 2 + UNPACK_WARPS) {
        // ------------------------------ unpack ------------------------------
        const int set = (warp - 2) / SET_WARPS, member = (warp - 2) % SET_WARPS;
        const bool channels = member < 4;
        const int r = channels ? (warp & 3) * 32 + lane : (member - 4) * 32 + lane;      // channels: the warp's own lane quadrant
        const unsigned lane_base = tmem_base + ((unsigned)((warp & 3) * 32) << 16) + A_COL0;
        const bool have = channels || r < half;
        const unsigned ofull0 = peer_addr(smem_u32(&S->ofull[0]), 0u);       // the issuer's
        constexpr bool GATHER = XBITS == 3 || WBITS == 3;
        for (int c = set; c < total; c += SETS) {
            const int b = c % BARS, before = c - STAGES;
            bool ok = mbar_wait(&S->abort_flag, &S->pfull[b], (unsigned)(c / BARS) & 1u, P.status, 4);
            if (!__all_sync(0xffffffffu, ok)) break;                             // a warp leaves as one
            const unsigned rows = smem_u32(sm_p + (c % P_STAGES) * P_STAGE);
            if (channels) {
                uint4 w[WBITS];
                load_row128<WBITS>(rows, r, w);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->pempty[b]);
                ok = before < 0 || pair_wait(&S->abort_flag, &S->oempty[before % BARS], (unsigned)(before / BARS) & 1u, P.status, 5);
                if (!__all_sync(0xffffffffu, ok)) break;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    unsigned v[8];
                    unpack32<WBITS, GATHER>(w, k, v);
                    tmem_st8(lane_base + (c % STAGES) * 32 + k * 8, v);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
            } else {
                uint4 w[XBITS];
                if (have) load_row128<XBITS>(rows + TM * 64, r, w);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->pempty[b]);
                ok = before < 0 || pair_wait(&S->abort_flag, &S->oempty[before % BARS], (unsigned)(before / BARS) & 1u, P.status, 5);
                if (!__all_sync(0xffffffffu, ok)) break;
                acquire_stage();
                if (have) {
                    const unsigned line = smem_u32(sm_b + (c % STAGES) * B_STAGE) + (unsigned)r * 128u;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        unsigned v[8];
                        unpack32<XBITS, GATHER>(w, k, v);
                        st_shared_v4(line + (unsigned)(((2 * k) ^ (r & 7)) << 4), make_uint4(v[0], v[1], v[2], v[3]));
                        st_shared_v4(line + (unsigned)(((2 * k + 1) ^ (r & 7)) << 4), make_uint4(v[4], v[5], v[6], v[7]));
                    }
                }
                // make the generic-proxy writes visible to the tensor cores' (async proxy) reads, then signal
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) {
                if (!channels) release_tokens();
                pair_arrive(ofull0 + 8u * (unsigned)b);
            }
        }
    } else if (warp >= 2) {
        // ------------------------------ epilogue: lane = output channel, column = token ------------------------------
        const int q = warp & 3;
        const unsigned tempty0 = peer_addr(smem_u32(&S->tempty[0]), 0u), tshared0 = peer_addr(smem_u32(&S->tshared), 0u);
        for (int i = 0; i < n_mine; ++i) {
            const int tile = first + i * step, mt = tile % P.m_tiles, nt = tile / P.m_tiles, a = i & 1;
            const long long o = (long long)(2 * mt + rank) * TM + q * 32 + lane;
            const long long t0 = (long long)nt * P.n;
            const float dw = o < P.n_out ? __ldg(P.sw + o) : 0.f;
            const bool ok = pair_wait(&S->abort_flag, &S->tfull[a], (unsigned)(i >> 1) & 1u, P.status, 6);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            // columns [128, 256) belong to both accumulators: the upper half of the even tiles', the lower half of the odd ones',
            // drained first
            const int shift = a == 0 ? 128 : 0;
            for (int j = 0; j < 2 * TN; j += 32) {
                const int c0 = (j + shift) & 255;
                if (j == 128) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) pair_arrive(tshared0);
                }
                if (c0 >= P.n || t0 + c0 >= P.n_tok) continue;
                store_tokens<XBITS + WBITS, OutT>(tmem_base + ((unsigned)(q * 32) << 16) + (unsigned)(a * ACC_STEP + c0), t0 + c0, o, dw, lane, P);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) pair_arrive(tempty0 + 8u * (unsigned)a);
        }
    }

    // ---- teardown: every role has left its loop (normally or after a wait expired), in both SMs; TMEM is freed
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((unsigned)TMEM_COLS) : "memory");
    }
}

typedef void (*PairKernel)(const CUtensorMap, const CUtensorMap, const QgemmParams);

PairKernel pick(int xbits, int wbits, int out_dtype)
{
    static const PairKernel table[2][2][2] = {
        {{k_tc_qgemm2<3, 3, float>, k_tc_qgemm2<3, 3, __nv_bfloat16>}, {k_tc_qgemm2<3, 4, float>, k_tc_qgemm2<3, 4, __nv_bfloat16>}},
        {{k_tc_qgemm2<4, 3, float>, k_tc_qgemm2<4, 3, __nv_bfloat16>}, {k_tc_qgemm2<4, 4, float>, k_tc_qgemm2<4, 4, __nv_bfloat16>}}};
    return table[xbits - 3][wbits - 3][out_dtype == GBS_DTYPE_F32 ? 0 : 1];
}

// attr[0]: clusters of two
cudaLaunchConfig_t pair_config(cudaLaunchAttribute attr[2], int pairs)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

int gbs_tc_qgemm2_pairs(const gbs_plan* px)
{
    // once per device (not a stream operation): the large dynamic shared memory, and how many clusters there is room for
    static std::mutex mu;
    static int known[64] = {0};                     // pairs + 1
    std::lock_guard<std::mutex> lock(mu);
    const bool keep = px->device >= 0 && px->device < 64;
    if (keep && known[px->device] != 0) return known[px->device] - 1;
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 8 && e == cudaSuccess; ++i)
        e = cudaFuncSetAttribute(pick(3 + (i >> 2), 3 + (i >> 1 & 1), i & 1 ? GBS_DTYPE_BF16 : GBS_DTYPE_F32), cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    int pairs = 0;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = pair_config(attr, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&pairs, pick(4, 4, GBS_DTYPE_BF16), &cfg);
    if (e != cudaSuccess) { cudaGetLastError(); return 0; }
    if (pairs > px->sm_count / 2) pairs = px->sm_count / 2;
    if (keep) known[px->device] = pairs + 1;
    return pairs;
}

int gbs_tc_qgemm2(const gbs_plan* px, const gbs_plan* pw, const CUtensorMap& wmap, const CUtensorMap& xmap, const QgemmParams& P, int pairs,
                  int out_dtype, cudaStream_t stream)
{
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = pair_config(attr, P.tiles < pairs ? P.tiles : pairs);
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = px->pdl ? 2 : 1;
    return (int)cudaLaunchKernelEx(&cfg, pick(px->bits, pw->bits, out_dtype), wmap, xmap, P);
}
