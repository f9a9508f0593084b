// Tensor-core inverse path of gbs_dequantize:  xhat = (H^T yhat / sqrt(d'))[0:d],  yhat = q * Delta, one scale per token
// or per group of a power of two coordinates (Section 2.1; inverse by the transpose, Section 2.3).
//
// The rotated row is a U x V matrix of codes Q[u][v] (flat index u V + v; V = 32 for d' <= 4096, 64 up to 8192), and
// H = A (x) H_V with A = H_m (x) H_{2^j}, U <= 128.  A group is at least V wide, so its scale is constant along v:
//
//        xhat = A^T diag(Delta_u) (Q H_V) / sqrt(d').
//
//   * Q H_V in registers, exactly: a code field masked into the low bits of a 16-bit half IS the subnormal half-precision
//     number k * 2^-24, and the sums of V fields stay below 2048 * 2^-24, so the butterflies run in packed half arithmetic
//     (two coordinates per instruction) without a conversion.  Codes are stored as q + 2^(b-1); after H_V the offset sits
//     in coordinate v = 0 alone, where one exact subtraction removes it.
//   * One scale per token: the integers are the fp16 operand as they are, and Delta multiplies once at the end.
//   * Group scales: the operand is Delta_u n, split into two fp16 numbers hi + lo (22 significant bits, relative to the
//     token's largest scale): with s = sh + sl the scale in two halves, hi = rn(n sh), lo = rn(n sl + (n sh - hi)), where
//     n sh - hi is exact in an fma.  A^T then contracts both planes into the same fp32 accumulators.
//   * tcgen05.mma with the plan's fp16 image of A^T, N = 128 columns (128 / V tokens) per tile, accumulators in TMEM; lane
//     u' then holds V consecutive output coordinates of a token: scale, round, 32-byte stores.
// What bounds it: instruction issue of the unpacking (about 290 slots per 32 values with group scales, 230 without)
// against 48 - 100 bytes of HBM traffic per 32 values.  Doing H_V before the contraction in packed halves takes 80
// instructions per 32 values where the fp32 form after the contraction took 124 packed (248 slots).
// 8192 x 3584, 3 bits, groups of 128 -> bf16: 118.5 us on the shared-memory kernel this replaces for group scales, 27 now.
// V = 32 takes four tokens per tile with all sixteen warps on it (two tokens and two groups of warps: 30 us; roles apart, twelve
// warps that unpack and sixteen for the epilogue: 14.2 -> 17.8 us for 4096 rows; sixteen and eight: no change).
// Roles: warp 0 loads the image, warp 1 issues the MMAs, warps 2..17 unpack (ahead) and run the epilogue; warp (q, t) owns
// TMEM lane quadrant q and token t; with V = 64 two groups of eight warps take alternate tiles.  Every wait is bounded.
#include <math.h>
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_tc_common.cuh"
#include "gbs_tc_inv.cuh"

namespace {

constexpr int UMAX = 128;
constexpr int STAGE_COLS = 128;                   // MMA N: 128 / V tokens of V columns
constexpr int ACCS = 4;                           // TMEM accumulators of 128 columns
constexpr int TMEM_COLS = ACCS * STAGE_COLS;
constexpr int A_BYTES = UMAX * UMAX * 2;
constexpr int PLANE_BYTES = UMAX * STAGE_COLS * 2;      // one operand plane of a tile at U = 128
constexpr int EPI_WARPS = 16;
constexpr int THREADS = 32 * (2 + EPI_WARPS);

// V = 32: all sixteen warps work on every tile.  V = 64: a thread owns 64 codes, so eight warps fill a tile and two groups
// take alternate tiles; a stage must belong to one group, or a group would wait on barrier phases it took no part in.
template <int V, bool SPLIT> struct Shape {
    static constexpr int GROUPS = V / 32;
    static constexpr int TOK = STAGE_COLS / V;
    static constexpr int WARPS = EPI_WARPS / GROUPS;            // warps per tile
    static constexpr int PLANES = SPLIT ? 2 : 1;
    static constexpr int STAGES = SPLIT ? (V == 32 ? 3 : 2) : 4;
    static constexpr int AHEAD = V == 32 ? 2 : 1;               // tiles (of its group) a warp unpacks ahead
    static constexpr int SMEM = 1024 + A_BYTES + STAGES * PLANES * PLANE_BYTES + 256;
    static_assert(STAGES % GROUPS == 0 && ACCS % GROUPS == 0, "a stage belongs to one group");
};

struct Bars {
    unsigned long long full[4], empty[4], tfull[ACCS], tempty[ACCS];
    unsigned long long abar;
    unsigned tmem_base;
    volatile int abort_flag;
};

struct InvParams {
    long long n_rows;
    int tok;                      // tokens per tile, TOK at most
    int n_tiles;                  // ceil(n_rows / tok)
    int U, Upad, ksteps;
    int d;                        // output width, a multiple of V
    int code_row_bytes;
    int spr;                      // scales per row
    int glog;                     // log2 of the u-rows per group (group scales)
    int wide;                     // output rows start on 32-byte boundaries
    float norm;                   // 1 / sqrt(d')
    const unsigned char* at_img;  // fp16 image of A^T
    const unsigned char* codes;
    const float* scales;
    void* out;
    int* status;
};

// V codes of one row u -> V/2 packed halves h[4 o + i] = (8 o + i, 8 o + 4 + i), times 2^-24 (LIFT: 2^-10), after H_V; offset removed.
template <int BITS, int V, bool LIFT>
__device__ __forceinline__ void unpack_rotate(const unsigned* w, unsigned h[V / 2])
{
    constexpr int NW = V * BITS / 32;
#pragma unroll
    for (int o = 0; o < V / 8; ++o) rotate_octet<BITS, false, NW, LIFT>(w, o, h + 4 * o);
#pragma unroll
    for (int i = 0; i < V / 2; ++i) h[i] = hpair(h[i]);
#pragma unroll
    for (int s = 4; s < V / 2; s <<= 1)
#pragma unroll
        for (int i = 0; i < V / 2; ++i)
            if ((i & s) == 0) {
                const unsigned a = h[i], b = h[i + s];
                h[i] = hadd2(a, b);
                h[i + s] = hsub2(a, b);
            }
    // low half: V 2^(b-1) times 2^-24, a subnormal, or 2^-10
    constexpr unsigned LOG = (V == 32 ? 5 : 6) + BITS - 1;
    h[0] = hsub2(h[0], LIFT ? (LOG + 5) << 10 : 1u << LOG);
}

// ---------------------------------------------------------------------------------------------
// kernel
// ---------------------------------------------------------------------------------------------
template <int BITS, int V, bool SPLIT, typename OutT>
__global__ void __launch_bounds__(THREADS, 1) k_tc_uv_inv(const __grid_constant__ InvParams P)
{
    typedef Shape<V, SPLIT> SH;
    constexpr int TOK = SH::TOK, STAGES = SH::STAGES, GROUPS = SH::GROUPS, AHEAD = SH::AHEAD;
    constexpr int STAGE_BYTES = SH::PLANES * PLANE_BYTES;
    constexpr int NW = V * BITS / 32;                       // packed words of V codes
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* sm_a = base;
    unsigned char* sm_b = base + A_BYTES;
    Bars* S = reinterpret_cast<Bars*>(base + A_BYTES + STAGES * STAGE_BYTES);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const unsigned slab_bytes = (unsigned)(P.Upad * V * 2);       // a token's operand rows: U lines of V halves

    if (threadIdx.x == 0) {
        mbar_init(&S->abar, 1);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S->full[s], SH::WARPS);
            mbar_init(&S->empty[s], 1);
        }
        for (int s = 0; s < ACCS; ++s) {
            mbar_init(&S->tfull[s], 1);
            mbar_init(&S->tempty[s], SH::WARPS);
        }
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_arrive_expect_tx(&S->abar, A_BYTES);
        bulk_load(sm_a, P.at_img, A_BYTES, &S->abar);         // plan-owned, immutable: needs no ordering
    }
    if (warp == 1) tmem_alloc(&S->tmem_base, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // programmatic dependent launch: the codes and scales may still be being written until this returns
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned tmem_base = S->tmem_base;
    const int n_mine = (P.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // tiles of this CTA

    if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        {
            // fp16 operands: the two type fields of instr_desc (bf16) cleared
            constexpr unsigned IDESC = instr_desc(UMAX, STAGE_COLS) & ~((1u << 7) | (1u << 10));
            constexpr unsigned KSTEP = (16 * V * 2) >> 4;          // sixteen u-lines of V halves
            const unsigned long long ad0 = smem_desc(smem_u32(sm_a), 16, 1024, 2);
            const unsigned long long bd0 = smem_desc(smem_u32(sm_b), slab_bytes, 8 * V * 2, V == 32 ? 4 : 2);
            const unsigned ad_lo0 = (unsigned)ad0, ad_hi = (unsigned)(ad0 >> 32);
            const unsigned bd_lo0 = (unsigned)bd0, bd_hi = (unsigned)(bd0 >> 32);
            bool ok = mbar_wait_warp(&S->abort_flag, &S->abar, 0, P.status, 6);
            for (int it = 0; ok && it < n_mine; ++it) {
                const int s = it % STAGES, c = it % ACCS;
                if (!mbar_wait_warp(&S->abort_flag, &S->full[s], (unsigned)(it / STAGES) & 1u, P.status, 2)) break;
                if (!mbar_wait_warp(&S->abort_flag, &S->tempty[c], ((unsigned)(it / ACCS) & 1u) ^ 1u, P.status, 3)) break;
                tc_fence_after();
                // only the address fields (bytes >> 4, low words) of the descriptors change between k-steps
                const unsigned d_tmem = tmem_base + c * STAGE_COLS;
#pragma unroll
                for (int pl = 0; pl < SH::PLANES; ++pl) {
                    unsigned a_lo = ad_lo0, b_lo = bd_lo0 + (unsigned)(s * STAGE_BYTES + pl * PLANE_BYTES) / 16u;
                    if (pl == 0) umma_f16_words<false>(d_tmem, a_lo, ad_hi, b_lo, bd_hi, IDESC);
                    else umma_f16_words<true>(d_tmem, a_lo, ad_hi, b_lo, bd_hi, IDESC);
                    for (int ks = 1; ks < P.ksteps; ++ks) {
                        a_lo += (ks & 3) ? 2u : (unsigned)((UMAX * 128 - 96) >> 4);
                        b_lo += KSTEP;
                        umma_f16_words<true>(d_tmem, a_lo, ad_hi, b_lo, bd_hi, IDESC);
                    }
                }
                umma_commit(&S->empty[s]);
                umma_commit(&S->tfull[c]);
            }
        }
    } else if (warp >= 2) {
        // ------------------------------ unpack + epilogue ------------------------------
        const int grp = (warp - 2) / SH::WARPS;                    // group of warps: tiles grp, grp + GROUPS, ..
        const int t = ((warp - 2) % SH::WARPS) >> 2;               // token slot inside its tiles
        const int q = warp & 3;                                    // TMEM lane quadrant this warp may access
        const int up = q * 32 + lane;                              // row u of the operand it writes; row u' it reads
        const unsigned taddr0 = tmem_base + ((unsigned)(q * 32) << 16) + t * V;
        const unsigned row_addr = smem_u32(sm_b) + (unsigned)t * slab_bytes + (unsigned)up * (V * 2);
        const unsigned swz = V == 32 ? (unsigned)((up >> 1) & 3) : (unsigned)(up & 7);
        const int n_grp = (n_mine - grp + GROUPS - 1) / GROUPS;    // tiles of this group
        const long long row_first = t < P.tok ? ((long long)blockIdx.x + (long long)grp * gridDim.x) * P.tok + t : P.n_rows;
        const long long row_step = (long long)GROUPS * gridDim.x * TOK;            // fewer than TOK to a tile: one tile per block
        const bool live_u = up < P.U;

        // Packed codes and scales of one tile, fetched two tiles ahead of their unpacking (one tile is less than the latency
        // of a DRAM read).  Nothing here looks at a loaded value: that would stall the warp at the fetch.
        struct Fetched {
            unsigned raw[NW];
            float my_scale, all[SPLIT ? 4 : 1];
        } buf[2];
        auto fetch = [&](int n, Fetched& B) {
            const long long row = row_first + (long long)n * row_step;
#pragma unroll
            for (int i = 0; i < NW; ++i) B.raw[i] = 0u;
            B.my_scale = 0.f;
#pragma unroll
            for (int i = 0; i < (SPLIT ? 4 : 1); ++i) B.all[i] = 0.f;
            if (n >= n_grp || row >= P.n_rows) return;
            const float* sp = P.scales + row * P.spr;
            if (SPLIT) {
                if (live_u) B.my_scale = __ldg(sp + (up >> P.glog));
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (lane + 32 * i < P.spr) B.all[i] = __ldg(sp + lane + 32 * i);
            } else {
                B.my_scale = __ldg(sp);
            }
            if (live_u) {
                const unsigned char* src = P.codes + row * P.code_row_bytes + up * (V * BITS / 8);
                if (BITS == 4) {
#pragma unroll
                    for (int i = 0; i < NW / 4; ++i) {
                        const uint4 v = __ldg(reinterpret_cast<const uint4*>(src) + i);
                        B.raw[4 * i] = v.x; B.raw[4 * i + 1] = v.y; B.raw[4 * i + 2] = v.z; B.raw[4 * i + 3] = v.w;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < NW; ++i) B.raw[i] = __ldg(reinterpret_cast<const unsigned*>(src) + i);
                }
            }
        };

        // the fetched codes -> operand planes of the n-th tile of this group; returns the factor of its epilogue in `fac`
        auto unpack_tile = [&](int n, const Fetched& B, float& fac) -> bool {
            const int it = n * GROUPS + grp, s = it % STAGES;
            unsigned h[V / 2];
            unpack_rotate<BITS, V, SPLIT>(B.raw, h);
            unsigned sh2 = 0u, sl2 = 0u;
            if (SPLIT) {
                // scales relative to 2^e, the power of two below the token's largest: s = Delta 2^(14-e) in (0, 2^15)
                const float big = fmaxf(fmaxf(fabsf(B.all[0]), fabsf(B.all[SPLIT ? 1 : 0])),
                                        fmaxf(fabsf(B.all[SPLIT ? 2 : 0]), fabsf(B.all[SPLIT ? 3 : 0])));
                const unsigned E = max(__reduce_max_sync(0xffffffffu, __float_as_uint(big)) >> 23, 15u);
                const float sf = B.my_scale * __uint_as_float((268u - E) << 23);
                const __half sh = __float2half_rn(sf), sl = __float2half_rn(sf - __half2float(sh));
                sh2 = __half_as_ushort(sh) * 0x10001u;
                sl2 = __half_as_ushort(sl) * 0x10001u;
                fac = P.norm * __uint_as_float((E - 4u) << 23);            // 2^(e-14), and 2^10 of the integers' scaling below
            } else {
                fac = B.my_scale * P.norm * 16777216.f;                      // the halves are integers times 2^-24
            }
            // a warp leaves as one
            const bool ok = mbar_wait(&S->abort_flag, &S->empty[s], ((unsigned)(it / STAGES) & 1u) ^ 1u, P.status, 1);
            if (!__all_sync(0xffffffffu, ok)) return false;
            if (up < P.Upad) {
                const unsigned dst = row_addr + (unsigned)(s * STAGE_BYTES);
#pragma unroll
                for (int c = 0; c < V / 8; ++c) {
                    // rows that pad U to a multiple of 16 hold zero codes: A^T has zero columns there, any finite value will do
                    uint4 hi, lo;
                    unsigned* ph = reinterpret_cast<unsigned*>(&hi);
                    unsigned* pl = reinterpret_cast<unsigned*>(&lo);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (SPLIT) {
                            const unsigned n1 = h[4 * c + e];                              // n * 2^-10
                            ph[e] = hmul2(n1, sh2);
                            pl[e] = hfma2(n1, sl2, hfma2(n1, sh2, hneg2(ph[e])));
                        } else {
                            ph[e] = h[4 * c + e];
                        }
                    }
                    st_shared_v4(dst + ((c ^ swz) << 4), hi);
                    if (SPLIT) st_shared_v4(dst + PLANE_BYTES + ((c ^ swz) << 4), lo);
                }
            }
            // make the generic-proxy writes visible to the tensor cores' (async proxy) reads, then signal
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&S->full[s]);
            return true;
        };

        float fac[AHEAD + 1];
        bool alive = true;
        fetch(0, buf[0]);
        fetch(1, buf[1]);
#pragma unroll
        for (int j = 0; j < AHEAD; ++j) {
            if (alive && j < n_grp) alive = unpack_tile(j, buf[j & 1], fac[j]);
            fetch(j + 2, buf[j & 1]);
        }
        long long row = row_first;
        // one tile: unpack the one AHEAD of it from buffer B, then finish it; false = leave
        auto tile = [&](int n, Fetched& B) -> bool {
            if (n + AHEAD < n_grp) {
                if (!unpack_tile(n + AHEAD, B, fac[AHEAD])) return false;
                fetch(n + AHEAD + 2, B);
            }
            const int it = n * GROUPS + grp, c = it % ACCS;
            const bool ok = mbar_wait(&S->abort_flag, &S->tfull[c], (unsigned)(it / ACCS) & 1u, P.status, 4);
            if (!__all_sync(0xffffffffu, ok)) return false;
            const bool store = row < P.n_rows && up * V < P.d;
            OutT* dst = reinterpret_cast<OutT*>(P.out) + row * (long long)P.d + up * V;
            tc_fence_after();
            float lift = 1.f;
            if (!SPLIT && !(fabsf(fac[0]) <= 3.4028234e38f)) {
                // a scale beyond 2^104 sqrt(d') (or not finite): the power of two on its own
                fac[0] = row < P.n_rows ? __ldg(P.scales + row) * P.norm : 0.f;
                lift = 16777216.f;
            }
#pragma unroll
            for (int half = 0; half < V / 32; ++half) {
                unsigned r[32];
                tmem_ld32_issue(taddr0 + c * STAGE_COLS + half * 32, r);
                tmem_ld_wait(r);
                if (half == V / 32 - 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&S->tempty[c]);
                }
                if (store) {
                    // column 8 o + 2 i + b of the accumulator is coordinate 8 o + i + 4 b
                    float f[32];
#pragma unroll
                    for (int o = 0; o < 4; ++o)
#pragma unroll
                        for (int e = 0; e < 8; ++e) f[8 * o + (e >> 1) + 4 * (e & 1)] = __uint_as_float(r[8 * o + e]) * fac[0];
                    if (!SPLIT && lift != 1.f) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) f[i] *= lift;
                    }
                    store_values<32>(dst + half * 32, f, P.wide != 0);
                }
            }
#pragma unroll
            for (int j = 0; j < AHEAD; ++j) fac[j] = fac[j + 1];
            row += row_step;
            return true;
        };
        for (int n = 0; alive && n < n_grp; n += 2) {
            if (!tile(n, buf[AHEAD & 1])) break;
            if (n + 1 < n_grp && !tile(n + 1, buf[(AHEAD + 1) & 1])) break;
        }
    }

    // ---- teardown: every role leaves its loop (normally or after a wait expired), then TMEM is freed
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

template <int V, bool SPLIT>
cudaError_t launch(const gbs_plan* p, InvParams& P, int out_dtype, cudaStream_t stream)
{
    typedef void (*Kernel)(const InvParams);
    static const Kernel table[2][2] = {
        {k_tc_uv_inv<3, V, SPLIT, float>, k_tc_uv_inv<3, V, SPLIT, __nv_bfloat16>},
        {k_tc_uv_inv<4, V, SPLIT, float>, k_tc_uv_inv<4, V, SPLIT, __nv_bfloat16>}};
    typedef Shape<V, SPLIT> SH;
    {
        // opt in to the large dynamic shared memory once per device (not a stream operation)
        static std::mutex mu;
        static bool done[64] = {false};
        std::lock_guard<std::mutex> lock(mu);
        if (!(p->device >= 0 && p->device < 64 && done[p->device])) {
            for (int i = 0; i < 4; ++i) {
                const cudaError_t e = cudaFuncSetAttribute(table[i >> 1][i & 1], cudaFuncAttributeMaxDynamicSharedMemorySize, SH::SMEM);
                if (e != cudaSuccess) return e;
            }
            if (p->device >= 0 && p->device < 64) done[p->device] = true;
        }
    }
    // Few rows: a tile is filled only as far as that takes no block more than one tile.  A block that restores four rows takes longer than
    // four that restore one each (64 x 4096, groups of 128 -> fp32: 5.9 us with four to a tile, 4.1 with one).
    P.tok = (int)((P.n_rows + p->sm_count - 1) / p->sm_count < SH::TOK ? (P.n_rows + p->sm_count - 1) / p->sm_count : SH::TOK);
    P.n_tiles = (int)((P.n_rows + P.tok - 1) / P.tok);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(P.n_tiles < p->sm_count ? P.n_tiles : p->sm_count));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)SH::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p->pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, table[p->bits - 3][out_dtype == GBS_DTYPE_F32 ? 0 : 1], P);
}

}  // namespace

// The in-register factor V of the inverse path for this shape, or 0: the smallest of 32 and 64 that leaves U <= 128, where
// a scale is constant over V coordinates.
int gbs_tc_uvinv_v(const gbs_plan* p)
{
    if (p->asym) return 0;
    for (int V = 32, lv = 5; V <= 64; V *= 2, ++lv) {
        if (p->k < lv || p->d_pad % V != 0) return 0;
        const int U = p->d_pad / V;
        if (U > UMAX) continue;
        if (U < 16 || p->d % V != 0 || (p->group != 0 && p->group < V)) return 0;
        return p->smem_optin >= Shape<32, true>::SMEM ? V : 0;
    }
    return 0;
}

// The calls this path takes: of the plans that got an image of A^T, all but those the shared-memory kernel does faster.  That kernel's time
// goes with the rows, the width and the order m; here a tile of 128 / V tokens takes much the same whatever the width, and a
// quarter of the lanes or less have rows below d' = 2048.  So with m = 1 and group scales (their operand is two planes) widths up to
// 2048 stay there while the rows are few, in rows per SM: 1024 wide: 6 (bf16) and 24 (fp32), 2048 wide: 2 and 5; 512 wide: always.
// (4 bits, groups of 128, shared memory and here: 5000 x 512 -> bf16: 9.1 and 13.5 us; 600 x 1024 -> bf16: 3.9 and 4.4, 1800: 7.3 and
// 7.0; 2400 x 1024 -> fp32: 9.4 and 9.9, 5000: 17.1 and 16.0; 220 x 2048 -> bf16: 3.3 and 3.5, 400: 3.9 and 3.7; 600 x 2048 -> fp32: 5.5
// and 6.0, 900: 7.0 and 6.3.)  One scale per token and m = 1 is faster here at every width: 100 x 512 -> bf16: 3.6 and 2.7.
bool gbs_tc_uvinv_serves(const gbs_plan* p, int64_t n_rows, int out_dtype)
{
    if (p->inv_v == 0 || p->d_aimg_t == nullptr) return false;
    if (p->group == 0 || p->m != 1 || p->d_pad > 2048) return true;
    const bool f32 = out_dtype == GBS_DTYPE_F32;
    const int per_sm = p->d_pad > 1024 ? (f32 ? 5 : 2) : (f32 ? 24 : 6);
    return p->d_pad > 512 && n_rows > (int64_t)per_sm * p->sm_count;
}

int gbs_tc_uvinv_dequantize(const gbs_plan* p, const void* codes, const float* scales, int64_t n_rows, void* out,
                            int out_dtype, cudaStream_t stream)
{
    if (n_rows > (int64_t)0x7fffffff - 4) return (int)cudaErrorInvalidValue;
    const int V = p->inv_v;
    InvParams P;
    memset(&P, 0, sizeof(P));
    P.n_rows = n_rows;
    P.U = p->d_pad / V;
    P.Upad = (P.U + 15) & ~15;
    P.ksteps = P.Upad / 16;
    P.d = p->d;
    P.code_row_bytes = p->d_pad * p->bits / 8;
    P.spr = p->group ? p->d_pad / p->group : 1;
    while (p->group && (V << P.glog) < p->group) ++P.glog;
    P.wide = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
    P.norm = p->norm;
    P.at_img = p->d_aimg_t;
    P.codes = (const unsigned char*)codes;
    P.scales = scales;
    P.out = out;
    P.status = p->d_status;
    const cudaError_t e = V == 32 ? (p->group ? launch<32, true>(p, P, out_dtype, stream) : launch<32, false>(p, P, out_dtype, stream))
                                  : (p->group ? launch<64, true>(p, P, out_dtype, stream) : launch<64, false>(p, P, out_dtype, stream));
    return (int)e;
}
