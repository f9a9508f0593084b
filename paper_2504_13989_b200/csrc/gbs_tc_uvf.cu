// Tensor-core rotate-quantize of fp32 rows: padded width d' = U V, U = m * 2^j <= 128, V = 32 (d' <= 4096) or 64 (<= 8192).
//
// As for bf16 rows (gbs_tc_uv.cu) the rotation is Y = A X H_V with X the U x V matrix of a row and A = H_m (x) H_{2^j}, but the
// operand is fp32.  A 24-bit significand is exactly three bf16 significands: x = hi + mid + lo, each the top half of what is
// left (two masks and two exact subtractions), so A contracts three bf16 planes into the same fp32 accumulators, smallest
// first, and no input bit is lost.
//   * Sixteen warps load a 4 KB piece of a tile each, lanes side by side, one tile ahead; they split it and write the planes in
//     the layout the MMA reads (N-major, 64- or 128-byte swizzle).  Elements beyond d are zeros (Section 4.2).
//   * tcgen05.mma: 3 U / 16 steps per tile of 128 columns (4 tokens at V = 32, 2 at V = 64), two accumulators in TMEM.
//   * TMEM lane u' holds V outputs of a token.  V = 32: one thread owns them, H_32 is five register butterflies.  V = 64: two
//     warps share them, one taking the sums and one the differences of the two halves before the same five butterflies.
//   * Maxima: group = 32 2^g coordinates, or one scale per token.  Across the warps that share it through shared memory and a
//     named barrier (token: 128 or 256 threads; group at V = 64: the pair of warps); then Delta, rounding, clipping, packing
//     (Sections 2.1, 3.1) from registers.
// What bounds it: 2.07 us per tile of 64 KB in a long batch (5 TB/s), of which 1.6 is one warp's chain of split and epilogue (a tile of one
// token takes 1.75), and about 4.4 us of fill in a short one.  3001 x 4096, 4 bits: 43.7 us on the shared-memory kernel, 17.4 now; 7000 x
// 3584, groups of 128: 117.6 -> 28.3; 7000 x 8192, 4 bits: 63.3.  Tried and slower: loads reissued piece by piece inside the split; tiles
// prefetched into L2 further ahead; the prefetches in a warp of their own that waits for the splits (18.2, 31.4 and 73.3 us); eight warps
// that only split beside sixteen of the epilogue (18.5); fewer tokens per tile (17.3 with three).  No change: twelve such warps, with
// registers moved to the epilogue's; A in tensor memory.
// Every wait is bounded; an expired wait records a code in the plan's status word, and a warp whose wait ran out brings a
// pattern no maximum can have to the barrier it shares, so that all who wait there leave with it.
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_tc_common.cuh"

namespace {

constexpr int UMAX = 128;
constexpr int NCOLS = 128;                        // MMA N: 128 / V tokens of V columns
constexpr int STAGES = 2;
constexpr int ACCS = 2;
constexpr int TMEM_COLS = ACCS * NCOLS;
constexpr int A_BYTES = UMAX * UMAX * 2;
constexpr int PLANE_BYTES = UMAX * NCOLS * 2;     // one bf16 plane of a tile at U = 128
constexpr int STAGE_BYTES = 3 * PLANE_BYTES;      // lo, mid, hi
constexpr int EPI_WARPS = 16;
constexpr int THREADS = 32 * (1 + EPI_WARPS);
constexpr unsigned POISON = 0xffffffffu;          // no maximum of absolute values has the sign bit set

struct __align__(1024) Smem {
    unsigned char a[A_BYTES];
    unsigned char b[STAGES][STAGE_BYTES];
    // maxima exchanged between warps, by tile parity: [token][warp of the token], or V = 64 with groups [token and quadrant][half][group]
    union {
        unsigned tok[2][4][8];
        unsigned grp[2][8][2][16];
    } red;
    unsigned long long full[STAGES], empty[STAGES], tfull[ACCS], tempty[ACCS];
    unsigned long long abar;
    unsigned tmem_base;
    volatile int abort_flag;
};

struct UvfParams {
    long long n_rows, stride;
    int n_tiles;                  // ceil(n_rows / tokens per tile)
    int U, Upad, ksteps;
    int d, d_pad;
    int code_row_bytes;
    int spr;                      // scales per row
    int glog;                     // log2 of the u-rows per group (group scales)
    float c_scale, c_half, norm;
    const float* x;
    const unsigned char* a_img;   // bf16 image of A
    unsigned char* codes;
    float* scales;
    float* y_opt;
    int* status;
};

__device__ __forceinline__ void st_shared_v2(unsigned addr, unsigned a, unsigned b)
{
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ unsigned top_halves(unsigned lo, unsigned hi) { return __byte_perm(lo, hi, 0x7632); }
// what is left of x below its top 16 bits (exact)
__device__ __forceinline__ unsigned below(unsigned x)
{
    return __float_as_uint(__uint_as_float(x) - __uint_as_float(x & 0xffff0000u));
}
// The same for any x: infinities leave a finite number instead of inf - inf, so that their sums stay infinite.  (What a finite x
// leaves is below 2^121; the minimum passes over a NaN.)
__device__ __forceinline__ unsigned below_any(unsigned x) { return __float_as_uint(fminf(__uint_as_float(below(x)), 0x1p121f)); }

template <int BITS, int V, bool GROUPED, bool WANT_Y>
__global__ void __launch_bounds__(THREADS, 1) k_tc_uvf(const __grid_constant__ UvfParams P)
{
    constexpr int TOK = NCOLS / V;                         // tokens per tile
    constexpr int HALVES = V / 32;                         // warps that share a token's lane quadrant
    constexpr int TOK_WARPS = 4 * HALVES;                  // warps of a token
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Smem* S = reinterpret_cast<Smem*>(smem_raw);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const unsigned slab_bytes = (unsigned)(P.Upad * V * 2);      // a token's rows in a plane

    if (threadIdx.x == 0) {
        mbar_init(&S->abar, 1);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S->full[s], EPI_WARPS);
            mbar_init(&S->empty[s], 1);
        }
        for (int s = 0; s < ACCS; ++s) {
            mbar_init(&S->tfull[s], 1);
            mbar_init(&S->tempty[s], EPI_WARPS);
        }
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_arrive_expect_tx(&S->abar, A_BYTES);
        bulk_load(S->a, P.a_img, A_BYTES, &S->abar);          // plan-owned, immutable: needs no ordering
        // the first tile's rows on their way to L2 (and no further) while an earlier kernel may still be writing them (3001 x 4096, 4
        // bits: 17.8 -> 17.4 us)
        for (int t = 0; t < TOK; ++t) {
            const long long row = (long long)blockIdx.x * TOK + t;
            if (row < P.n_rows) prefetch_l2(P.x + row * P.stride, P.d * 4);
        }
    }
    if (warp == 0) tmem_alloc(&S->tmem_base, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // programmatic dependent launch: the rows may still be being written until this returns
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned tmem_base = S->tmem_base;
    const int n_mine = (P.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // tiles of this CTA

    if (warp == 0) {
        // ------------------------------ MMA issuer ------------------------------
        {
            constexpr unsigned IDESC = instr_desc(UMAX, NCOLS);
            constexpr unsigned KSTEP = (16 * V * 2) >> 4;          // sixteen u-lines of V bf16
            const unsigned long long ad0 = smem_desc(smem_u32(S->a), 16, 1024, 2);
            const unsigned long long bd0 = smem_desc(smem_u32(S->b[0]), slab_bytes, 8 * V * 2, V == 32 ? 4 : 2);
            const unsigned ad_lo0 = (unsigned)ad0, ad_hi = (unsigned)(ad0 >> 32);
            const unsigned bd_lo0 = (unsigned)bd0, bd_hi = (unsigned)(bd0 >> 32);
            bool ok = mbar_wait_warp(&S->abort_flag, &S->abar, 0, P.status, 6);
            for (int it = 0; ok && it < n_mine; ++it) {
                const int s = it % STAGES, c = it % ACCS;
                if (!mbar_wait_warp(&S->abort_flag, &S->full[s], (unsigned)(it / STAGES) & 1u, P.status, 2)) break;
                if (!mbar_wait_warp(&S->abort_flag, &S->tempty[c], ((unsigned)(it / ACCS) & 1u) ^ 1u, P.status, 3)) break;
                tc_fence_after();
                // only the address fields (bytes >> 4, low words) of the descriptors change between k-steps
                const unsigned d_tmem = tmem_base + c * NCOLS;
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) {
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
    } else {
        // ------------------------------ split + epilogue ------------------------------
        const int q = warp & 3;                                    // TMEM lane quadrant this warp may access
        const int w = (warp - 1) >> 2;
        const int t = w / HALVES, half = w % HALVES;               // token slot of its tiles, half of the V outputs
        const int up = q * 32 + lane;                              // output row u' it reads
        const int wt = q * HALVES + half;                          // its place among the token's warps
        const int out0 = up * V + half * 32;                       // first coordinate this thread owns
        const unsigned taddr0 = tmem_base + ((unsigned)(q * 32) << 16) + t * V;
        const long long row_first = (long long)blockIdx.x * TOK + t;
        const long long row_step = (long long)gridDim.x * TOK;

        // what it loads: elements e0 + 128 j + 4 lane of the token's row, j < 8, and where they go in a plane
        const int e0 = wt * 1024 + lane * 4;
        const int u0 = e0 / V, b0 = (e0 % V) * 2;                  // operand row and byte in it
        const unsigned dst_first = smem_u32(S->b[0]) + (unsigned)t * slab_bytes + (unsigned)(u0 * V * 2) +
                                   ((((unsigned)b0 >> 4) ^ (V == 32 ? (unsigned)((u0 >> 1) & 3) : (unsigned)(u0 & 7))) << 4) + ((unsigned)b0 & 8u);
        // its rows are sixteen or twice sixteen, and so is Upad's granule
        const bool rows0 = wt * (1024 / V) < P.Upad, rows4 = wt * (1024 / V) + 512 / V < P.Upad;
        const bool whole = wt * 1024 + 1024 <= P.d;
        uint4 x[8];
        auto fetch = [&](int n) {
            const long long row = row_first + (long long)n * row_step;
            const bool in = n < n_mine && row < P.n_rows;
            const float* src = P.x + row * P.stride + e0;
            if (in && whole) {
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = __ldg(reinterpret_cast<const uint4*>(src + 128 * j));
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    x[j] = (in && e0 + 128 * j < P.d) ? __ldg(reinterpret_cast<const uint4*>(src + 128 * j)) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        // The registers hold one tile ahead, for part of a tile's time; DRAM wants more in flight.  Paced by the splits, one tile
        // beyond the loads, by a token's first warp (82.8 -> 70.7 us for 7000 x 8192); further ahead queues in front of other
        // blocks' loads.
        const bool prefetches = wt == 0 && lane == 0;
        auto prefetch = [&](int n) {
            const long long row = row_first + (long long)n * row_step;
            if (prefetches && n < n_mine && row < P.n_rows)
                prefetch_l2(P.x + row * P.stride, P.d * 4);
        };
        auto split_tile = [&](int n) -> bool {
            const int s = n % STAGES;
            const bool ok = mbar_wait(&S->abort_flag, &S->empty[s], ((unsigned)(n / STAGES) & 1u) ^ 1u, P.status, 1);
            if (!__all_sync(0xffffffffu, ok)) return false;
            const unsigned dst0 = dst_first + (unsigned)(s * STAGE_BYTES);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const unsigned x0 = x[j].x, x1 = x[j].y, x2 = x[j].z, x3 = x[j].w;
                const unsigned m0 = below_any(x0), m1 = below_any(x1), m2 = below_any(x2), m3 = below_any(x3);
                const unsigned l0 = below(m0), l1 = below(m1), l2 = below(m2), l3 = below(m3);
                // 128 elements on is 256 bytes on, and two (V = 64) or four rows: that much of the swizzle is a constant
                const unsigned dst = (dst0 ^ (32u * (unsigned)(j & (HALVES == 1 ? 1 : 3)))) + 256u * j;
                if (j < 4 ? rows0 : rows4) {
                    st_shared_v2(dst, top_halves(l0, l1), top_halves(l2, l3));
                    st_shared_v2(dst + PLANE_BYTES, top_halves(m0, m1), top_halves(m2, m3));
                    st_shared_v2(dst + 2 * PLANE_BYTES, top_halves(x0, x1), top_halves(x2, x3));
                }
            }
            // make the generic-proxy writes visible to the tensor cores' (async proxy) reads, then signal
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&S->full[s]);
            return true;
        };

        const bool live_u = up < P.U;
        const int gl = 1 << P.glog;                                // lanes per group
        fetch(0);
        bool alive = split_tile(0);
        fetch(1);
        prefetch(2);
        long long row = row_first;
        for (int n = 0; n < n_mine; ++n, row += row_step) {
            if (alive && n + 1 < n_mine) {
                alive = split_tile(n + 1);
                fetch(n + 2);
                prefetch(n + 3);
            }
            const int c = n % ACCS;
            if (alive) alive = __all_sync(0xffffffffu, mbar_wait(&S->abort_flag, &S->tfull[c], (unsigned)(n / ACCS) & 1u, P.status, 4));
            unsigned r[32];
            unsigned mb = POISON;
            if (alive) {
                tc_fence_after();
                if (V == 32) {
                    tmem_ld32_issue(taddr0 + c * NCOLS, r);
                    tmem_ld_wait(r);
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        unsigned hi[16];
                        tmem_ld16_issue(taddr0 + c * NCOLS + 16 * h, r + 16 * h);
                        tmem_ld16_issue(taddr0 + c * NCOLS + 32 + 16 * h, hi);
                        tmem_ld_wait16x2(r + 16 * h, hi);
                        const float sign = half ? -1.f : 1.f;
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            r[16 * h + e] = __float_as_uint(fmaf(__uint_as_float(hi[e]), sign, __uint_as_float(r[16 * h + e])));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->tempty[c]);
                mb = __float_as_uint(fwht32_absmax(r));
            }
            if (GROUPED) {
                // a group is 2^glog adjacent lanes, of both warps at V = 64
                if (alive) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        if (o < gl) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
                }
                if (V == 64) {
                    unsigned (*slot)[16] = S->red.grp[n & 1][q * 2 + t];
                    if ((lane & (gl - 1)) == 0) slot[half][lane >> P.glog] = mb;
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + q * 2 + t) : "memory");
                    const unsigned other = slot[half ^ 1][lane >> P.glog];
                    mb = max(mb, other);
                }
            } else {
                if (alive) mb = __reduce_max_sync(0xffffffffu, mb);
                unsigned* slot = S->red.tok[n & 1][t];
                if (lane == 0) slot[wt] = mb;
                asm volatile("bar.sync %0, %1;" ::"r"(1 + t), "n"(32 * TOK_WARPS) : "memory");
#pragma unroll
                for (int i = 0; i < TOK_WARPS; ++i) mb = max(mb, slot[i]);
            }
            if (__any_sync(0xffffffffu, mb == POISON)) break;
            const float M = __uint_as_float(mb);
            const float a1 = M > 0.f ? P.c_half / M : 0.f;
            unsigned out[BITS];
            quantize_pack32<BITS>(r, a1, out);
            if (live_u && row < P.n_rows) {
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
    }

    // ---- teardown: every role leaves its loop (normally or after a wait expired), then TMEM is freed
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

typedef void (*UvfKernel)(const UvfParams);
template <int V>
UvfKernel kernel_of(int bits, bool grouped, bool want_y)
{
    static const UvfKernel table[2][2][2] = {
        {{k_tc_uvf<3, V, false, false>, k_tc_uvf<3, V, false, true>}, {k_tc_uvf<3, V, true, false>, k_tc_uvf<3, V, true, true>}},
        {{k_tc_uvf<4, V, false, false>, k_tc_uvf<4, V, false, true>}, {k_tc_uvf<4, V, true, false>, k_tc_uvf<4, V, true, true>}}};
    return table[bits - 3][grouped ? 1 : 0][want_y ? 1 : 0];
}

}  // namespace

// The in-register factor V of the fp32 path for this plan, or 0.  It uses the plan's bf16 image of A = H_m (x) H_{2^j}: the UV
// family's (V = 32) or the wide family's where that has U = d' / 64 (V = 64, groups of at least two lanes).
int gbs_tc_uvf_v(const gbs_plan* p)
{
    if (p->asym || p->smem_optin < (int)sizeof(Smem)) return 0;
    if (p->variant == GBS_VARIANT_TC_UV) return 32;
    if ((p->variant == GBS_VARIANT_TC_UVM || p->variant == GBS_VARIANT_TC_UVR) && p->uvm_glog == 1 &&
        (p->group == 0 || (p->group >= 128 && p->group <= 2048)))
        return 64;
    return 0;
}

// The calls it takes: all of those plans' but the ones that the shared-memory kernel does faster.  That kernel's time goes with the rows,
// the width and the order m; here a tile of 128 / V tokens takes much the same whatever the width.  So with m = 1 a width of 512 stays
// there, 1024 up to 28 rows per SM (64 with group scales), 2048 up to one and a half.  (4 bits, shared memory and here: 5000 x 512:
// 10.9 and 16.7 us; 1200 x 1024: 6.6 and 7.3, 5000: 19.8 and 19.1, with groups of 128: 20.3 and 21.0; 150 x 2048: 3.8 and 4.0, 300:
// 4.5 and 4.2; 16 x 4096: 4.9 and 4.6.)
bool gbs_tc_uvf_serves(const gbs_plan* p, int64_t n_rows)
{
    if (gbs_tc_uvf_v(p) == 0) return false;
    if (p->m != 1 || p->d_pad > 2048) return true;
    if (p->d_pad > 1024) return 2 * n_rows > 3 * (int64_t)p->sm_count;
    return p->d_pad > 512 && n_rows > (p->group ? 64 : 28) * (int64_t)p->sm_count;
}

int gbs_tc_uvf_rotate_quantize(const gbs_plan* p, const void* x, int64_t n_rows, int64_t stride, void* codes, float* scales,
                               float* y_opt, cudaStream_t stream)
{
    if (n_rows > (int64_t)0x7fffffff - 4) return (int)cudaErrorInvalidValue;
    const int V = gbs_tc_uvf_v(p), tok = NCOLS / V;
    UvfParams P;
    memset(&P, 0, sizeof(P));
    P.n_rows = n_rows;
    P.stride = stride;
    P.n_tiles = (int)((n_rows + tok - 1) / tok);
    P.U = p->d_pad / V;
    P.Upad = (P.U + 15) & ~15;
    P.ksteps = P.Upad / 16;
    P.d = p->d;
    P.d_pad = p->d_pad;
    P.code_row_bytes = p->d_pad * p->bits / 8;
    P.spr = p->group ? p->d_pad / p->group : 1;
    while (p->group && (V << P.glog) < p->group) ++P.glog;
    P.c_scale = p->c_scale;
    P.c_half = (float)(1.0 / (2.0 * (double)p->alpha));
    P.norm = p->norm;
    P.x = (const float*)x;
    P.a_img = p->d_aimg;
    P.codes = (unsigned char*)codes;
    P.scales = scales;
    P.y_opt = y_opt;
    P.status = p->d_status;
    {
        // opt in to the large dynamic shared memory once per device (not a stream operation)
        static std::mutex mu;
        static bool done[64] = {false};
        std::lock_guard<std::mutex> lock(mu);
        if (!(p->device >= 0 && p->device < 64 && done[p->device])) {
            for (int i = 0; i < 16; ++i) {
                const UvfKernel k = (i & 8) ? kernel_of<64>(3 + (i & 1), (i & 2) != 0, (i & 4) != 0) : kernel_of<32>(3 + (i & 1), (i & 2) != 0, (i & 4) != 0);
                const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
                if (e != cudaSuccess) return (int)e;
            }
            if (p->device >= 0 && p->device < 64) done[p->device] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(P.n_tiles < p->sm_count ? P.n_tiles : p->sm_count));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = sizeof(Smem);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p->pdl ? 1 : 0;
    const UvfKernel k = V == 32 ? kernel_of<32>(p->bits, p->group != 0, y_opt != nullptr) : kernel_of<64>(p->bits, p->group != 0, y_opt != nullptr);
    return (int)cudaLaunchKernelEx(&cfg, k, P);
}
