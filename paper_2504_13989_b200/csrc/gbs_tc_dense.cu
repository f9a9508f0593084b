// Tensor-core family "DENSE": d' = m, the rotation is the full Paley matrix H_m itself (no Sylvester factor).
//
// Section 5.2.2 names the case: a width of 1536 admits no useful power-of-two split, but 1536 + 8 = 1544 = 1543 + 1
// with 1543 a prime = 3 (mod 4), so Algorithm 2 gives a Hadamard matrix of exactly the expanded order.  There is no
// fast transform for it; Y = X_pad H_m^T is a dense contraction with a +-1 matrix, which is what tensor cores are
// for: bf16 x (+-1) products are exact, the accumulation is fp32 in TMEM.
//
//   * H_m never streams.  Away from row 0 and column 0, Algorithm 2's matrix is Toeplitz: H[n][k] = t(k - n).  In the
//     tensor cores' unswizzled operand layout (core matrices of 8 rows x 16 bytes) the core matrix of rows 8 nb.. and
//     columns 8 kb.. then depends on kb - nb alone, so the whole m x m operand is 2 m / 8 core matrices in a row (49 KB at
//     m = 1544 instead of 4.8 MB), and with the output blocks taken in descending order the descriptor's two strides are
//     both +128 bytes.  A CTA's share (31 KB) stays in shared memory; only the rows of X move.
//   * Column 0 of H (constant -1) is repaired by one more MMA per tile with a 16-column operand whose column 0 holds
//     H[n][0] - t(-n).  Row 0 (2 x_0 - sum of all) is an extra 16-row operand, the same for every k-step, contracted by
//     the last CTA of the cluster, which has the fewest coordinates; it sends the value to the first.
//   * One sweep.  A token's m fp32 values do not fit one SM's TMEM, so a CLUSTER of CTAs takes 128 tokens and each CTA up to
//     512 output coordinates: TMEM lane t holds the CTA's coordinates of token t, and the CTAs exchange their maxima of
//     every token through distributed shared memory before quantizing (Sections 2.1, 3.1): one float per token and pair of CTAs, by st.async, so that
//     the receiver's barrier counts the bytes and no fence stands in between (1.7 us with stores and releasing arrivals, 0.45 now).
//     What a CTA's epilogue has waited for is all that is ever written to it, so it leaves without meeting the others again (0.5 - 0.8 us).
//   * Two warps issue the MMAs, each for half of the columns: one's polls and commits are covered by the other's MMAs.
//   * Packed rows are m b / 8 bytes (579 at m = 1544, b = 3: any alignment): the four warps of a lane quadrant pack its 32 tokens' codes into
//     shared memory, and each writes the CTA's piece of eight rows as words, what is left at either end by bytes.
// What bounds it: the tensor pipe, 2 d m flops per token, and what stands around it.  4096 x 1536, b = 4: 176 us with two sweeps
// over streamed chunks of H on 32 SMs; 27.4 us with one sweep over the Toeplitz operand, of which 13.9 were the MMAs (a poll and
// a commit per 64 columns cost 217 of 1050 cycles: hence 128 columns per stage); 21.0 with a piece of its own for every warp and one
// issuing warp; 18.3 now: first stage 1.0, MMAs 11.7 (0.94 per 128 input coordinates; 9.7 in all, 19 000 cycles, by the tensor pipe's counter), maxima and
// exchange 0.8, quantizer 1.2, stores 1.4.  The number of CTAs per cluster is chosen by cost (pick_split): few wide shares when the batch
// fills the chip, more and narrower ones when it does not.  1 row: 13.4 -> 8.8 us (of which 13 CTAs instead of 7: 4), 772: 14.6 -> 10.9.
// Every wait is bounded; an expired wait records a code in the plan's status word.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_tc_common.cuh"

namespace {

constexpr int TM = 128;                 // tokens per tile (MMA M)
constexpr int KC = 128;                 // input coordinates per stage: two boxes of one 128-byte swizzled line of bf16 per token
constexpr int MAX_STAGES = 3;           // two where a large order's table leaves no room for three
constexpr int A_BOX = TM * 64 * 2;      // 16 KB
constexpr int A_STAGE = 2 * A_BOX;
constexpr int EW = 4;                   // epilogue warps per TMEM lane quadrant: each takes a quarter of the coordinates
constexpr int EPI_WARPS = 4 * EW;
constexpr int N_ISSUERS = 2;
constexpr int THREADS = 32 * (3 + EPI_WARPS);    // producer, issuers (warp 1 and the last one), epilogue
constexpr int TMEM_COLS = 512;
constexpr int MAX_CL = 16;              // CTAs per cluster
constexpr int CORE = 128;               // bytes of a core matrix: 8 rows x 8 bf16
constexpr int ROW0_BYTES = 2 * 4 * CORE;   // row 0 as 16-row operands: 2 at column 0, and all -1

struct Ctl {
    float part[2][EW][TM];              // [tile parity][quarter][token]: maxima of the CTA's own quarters
    float tmax[2][MAX_CL][TM];          // [tile parity][CTA][token]: maxima of every CTA's share, written by their threads
    float y0[2][TM];                    // coordinate 0, from the cluster's last CTA
    unsigned long long full[MAX_STAGES], empty[MAX_STAGES], tfull, tempty, tbar, maxbar[2];
    unsigned tmem_base;
    volatile int abort_flag;
};

struct DenseParams {
    long long n_rows;
    int n_tiles;
    int m;                        // d' = order of H_m
    int cl;                       // CTAs per cluster
    int ncb, ncb_last;            // 8-coordinate output blocks per CTA and of the last CTA, multiples of 4
    int kchunks;                  // ceil(d / 128)
    int ksteps_last;              // MMAs (K = 16) of the last chunk
    int nbp;                      // output blocks the Toeplitz and column tables are laid out for
    int code_row_bytes;
    int stages;
    int stage_words;              // words of a token's row in the packing buffer (odd)
    float c_scale, c_half, norm;
    const unsigned short* x;      // the rows (bf16), for what the tensor map does not show
    long long stride;
    int d;
    const unsigned char* toep;    // core matrices J = kb - nb + nbp - 1
    const unsigned char* row0;    // ROW0_BYTES
    const unsigned char* col0;    // core matrix pairs (column repair, zeros) of block nbp - 1 - i at i
    unsigned char* codes;
    float* scales;
    float* y_opt;
    int* status;
};

// n k-steps of one stage: 32 bytes of the 128-byte line each, four to a box; the operand moves on by `step`
__device__ __forceinline__ void steps(unsigned d_tmem, unsigned long long ad, unsigned long long bd, unsigned step, unsigned idesc, int n)
{
    if (n == KC / 16) {
#pragma unroll
        for (int ks = 0; ks < KC / 16; ++ks)
            umma_f16(d_tmem, ad + (unsigned long long)(2 * (ks & 3) + (ks >> 2) * (A_BOX / 16)), bd + (unsigned long long)(step * ks), idesc, 1u);
    } else {
        for (int ks = 0; ks < n; ++ks) {
            umma_f16(d_tmem, ad, bd, idesc, 1u);
            ad += ks == 3 ? (A_BOX - 96) / 16 : 2;
            bd += step;
        }
    }
}

// A float to another CTA's shared memory, whose barrier there counts its bytes: what a waiter of that barrier sees is ordered by the
// transaction alone.  (An arrival with .release.cluster orders all of the writer's accesses, global ones too.)
__device__ __forceinline__ void peer_send(unsigned addr, float v, unsigned bar_addr)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar_addr) : "memory");
}
// L2 prefetch of the box a later tma_load_2d will fetch (see tma_prefetch_3d)
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int c0, int c1)
{
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(map), "r"(c0), "r"(c1) : "memory");
}

// one column of this thread's TMEM lane
__device__ __forceinline__ unsigned tmem_ld1(unsigned taddr)
{
    unsigned v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=r"(v) : "r"(taddr) : "memory");
    return v;
}
// 128 threads meet; whether any of them says so
__device__ __forceinline__ bool meet_any(int barrier, bool p)
{
    unsigned any;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %2, 0;\n\tbar.red.or.pred p, %1, 128, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(any) : "r"(barrier), "r"(p ? 1u : 0u) : "memory");
    return any != 0;
}
// 32 accumulator columns of four output blocks (descending) into coordinate order
__device__ __forceinline__ void load_chunk(unsigned taddr, unsigned y[32])
{
    unsigned r[32];
    tmem_ld32_issue(taddr, r);
    tmem_ld_wait(r);
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int e = 0; e < 8; ++e) y[8 * o + e] = r[8 * (3 - o) + e];
}

template <int BITS>
__global__ void __launch_bounds__(THREADS, 1) k_tc_dense_rq(const __grid_constant__ CUtensorMap xmap,
                                                            const __grid_constant__ DenseParams P)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* sm_x = base;
    unsigned char* sm_t = sm_x + P.stages * A_STAGE;
    unsigned char* sm_e = sm_t + (P.kchunks * (KC / 8) + P.ncb) * CORE;
    unsigned char* sm_r = sm_e + P.ncb * 2 * CORE;
    unsigned* sm_pack = reinterpret_cast<unsigned*>(sm_r + ROW0_BYTES);
    Ctl* S = reinterpret_cast<Ctl*>(sm_pack + TM * P.stage_words);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();
    const int cluster = (int)blockIdx.x / P.cl, n_clusters = (int)gridDim.x / P.cl;
    const int nb0 = rank * P.ncb;                                  // first output block of this CTA
    const bool last = rank == P.cl - 1;
    const int ncb = last ? P.ncb_last : P.ncb;                     // its blocks, a multiple of 4
    const int toep_n = P.kchunks * (KC / 8) + ncb;                 // core matrices of its share
    // coordinate 0's sixteen columns: behind the last CTA's blocks, or where two blocks of padding would be (blocks descend, so
    // padding comes first)
    const int skip = last && nb0 + ncb - P.m / 8 >= 2 ? 2 : 0;
    const int col_r = skip ? 0 : 8 * ncb;

    const unsigned max_bytes = (unsigned)((P.cl + (rank == 0 ? 1 : 0)) * TM * 4);       // of a tile: a float per token from every CTA, and coordinate 0

    if (threadIdx.x == 0) {
        for (int s = 0; s < P.stages; ++s) {
            mbar_init(&S->full[s], 1);
            mbar_init(&S->empty[s], N_ISSUERS);
        }
        mbar_init(&S->tfull, N_ISSUERS);
        mbar_init(&S->tempty, EPI_WARPS);
        mbar_init(&S->tbar, 1);
        mbar_init(&S->maxbar[0], 1);
        mbar_init(&S->maxbar[1], 1);
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_arrive_expect_tx(&S->maxbar[0], max_bytes);
        mbar_arrive_expect_tx(&S->maxbar[1], max_bytes);
        // plan-owned, immutable tables: need no ordering
        mbar_arrive_expect_tx(&S->tbar, (unsigned)(toep_n * CORE + ncb * 2 * CORE + ROW0_BYTES));
        const int first = P.nbp - nb0 - ncb;
        bulk_load(sm_t, P.toep + (size_t)first * CORE, (unsigned)(toep_n * CORE), &S->tbar);
        bulk_load(sm_e, P.col0 + (size_t)first * 2 * CORE, (unsigned)(ncb * 2 * CORE), &S->tbar);
        bulk_load(sm_r, P.row0, ROW0_BYTES, &S->tbar);
    }
    if (warp == 1) tmem_alloc(&S->tmem_base, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    cluster_sync();                                                // every CTA's barriers are ready for its peers
    tc_fence_after();
    const unsigned tmem_base = S->tmem_base;
    // the first stage on its way from DRAM to L2; nothing reaches this SM before the wait.  (All of the tile's, shared out among the CTAs: no gain.)
    if (threadIdx.x == 0 && cluster < P.n_tiles) {
        tma_prefetch_2d(&xmap, 0, cluster * TM);
        tma_prefetch_2d(&xmap, 64, cluster * TM);
    }
    // programmatic dependent launch: until this returns an earlier kernel may still be writing x or reading the outputs
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int n_mine = cluster < P.n_tiles ? (P.n_tiles - cluster + n_clusters - 1) / n_clusters : 0;

    if (warp == 0) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) {
            int c = 0, s = 0;                                      // stage uses so far, the stage of the next
            unsigned ph = 0;
            bool ok = true;
            for (int i = 0; ok && i < n_mine; ++i) {
                const int row0 = (cluster + i * n_clusters) * TM;
                for (int kc = 0; kc < P.kchunks; ++kc, ++c) {
                    if (!mbar_wait(&S->abort_flag, &S->empty[s], ph ^ 1, P.status, 1)) { ok = false; break; }
                    mbar_arrive_expect_tx(&S->full[s], A_STAGE);
                    tma_load_2d(sm_x + s * A_STAGE, &xmap, &S->full[s], kc * KC, row0);
                    tma_load_2d(sm_x + s * A_STAGE + A_BOX, &xmap, &S->full[s], kc * KC + 64, row0);
                    if (++s == P.stages) { s = 0; ph ^= 1; }
                }
            }
            if (!ok) drain_copies(S->full, P.stages, c);
        }
    } else if (warp == 1 || warp == 2 + EPI_WARPS) {
        // ------------------------------ MMA issuers ------------------------------
        // Each issues for its own columns, all k-steps of a stage, so that one's polls and commits (about 200 cycles a stage) are covered by the other's
        // MMAs.  Fewer than 208 columns stay with the first: an MMA of less than about 100 columns takes no less time.
        {
            const int issuer = warp == 1 ? 0 : 1;
            const int n_all = ncb - skip, n_first = n_all < 26 ? n_all : (n_all / 2 + 1) / 2 * 2, n = issuer == 0 ? n_first : n_all - n_first;
            const int before = issuer == 0 ? 0 : n_first;                           // blocks
            const bool row0s = last && issuer == 1;                                 // coordinate 0 as well
            const unsigned idesc = instr_desc(TM, 8 * n, false);
            constexpr unsigned IDESC_R = instr_desc(TM, 16, false);
            // unswizzled core matrices: leading offset = next 8 columns, stride offset = next 8 rows of the operand
            const unsigned long long td0 = smem_desc(smem_u32(sm_t) + (skip + before) * CORE, CORE, CORE, 0);
            const unsigned long long ed0 = smem_desc(smem_u32(sm_e) + (skip + before) * 2 * CORE, CORE, 2 * CORE, 0);
            const unsigned long long rd0 = smem_desc(smem_u32(sm_r), CORE, 2 * CORE, 0);
            const unsigned tmem = tmem_base + 8 * (skip + before), tmem_r = tmem_base + col_r;
            bool ok = mbar_wait_warp(&S->abort_flag, &S->tbar, 0, P.status, 6);
            int s = 0;
            unsigned ph = 0;
            for (int i = 0; ok && i < n_mine; ++i) {
                // the accumulators fill the CTA's share of TMEM: the next tile waits for the epilogue
                if (!mbar_wait_warp(&S->abort_flag, &S->tempty, (i & 1) ^ 1, P.status, 3)) break;
                tc_fence_after();
                unsigned long long td = td0;
                for (int kc = 0; kc < P.kchunks; ++kc) {
                    if (!mbar_wait_warp(&S->abort_flag, &S->full[s], ph, P.status, 2)) { ok = false; break; }
                    tc_fence_after();
                    const unsigned long long ad = smem_desc(smem_u32(sm_x + s * A_STAGE), 16, 1024, 2);
                    const int ks_n = (kc == P.kchunks - 1) ? P.ksteps_last : KC / 16;
                    if (kc == 0) {
                        // column 0: H[n][0] - t(-n) against x_0, and coordinate 0: 2 x_0 (the other columns of these are zero)
                        if (n) umma_f16(tmem, ad, ed0, idesc, 0u);
                        if (row0s) umma_f16(tmem_r, ad, rd0, IDESC_R, 0u);
                    }
                    // one operand after the other, each in a loop of its own: a condition between two MMAs doubles their time
                    if (n) steps(tmem, ad, td, 2 * CORE / 16, idesc, ks_n);
                    if (row0s) steps(tmem_r, ad, rd0 + 4 * CORE / 16, 0, IDESC_R, ks_n);
                    td += (unsigned long long)(2 * CORE / 16 * (KC / 16));
                    umma_commit(&S->empty[s]);
                    if (++s == P.stages) { s = 0; ph ^= 1; }
                }
                if (ok) umma_commit(&S->tfull);
            }
        }
    } else {
        // ------------------------------ epilogue: one thread = one token and a quarter of the coordinates -----------
        const int q = warp & 3;                            // TMEM lane quadrant this warp may access
        const int h = (warp - 2) >> 2;                     // which quarter of the CTA's coordinates
        const int tok = q * 32 + lane;
        const int chunks = ncb / 4;                        // of 32 coordinates
        const int ch0 = h * chunks / EW, ch1 = (h + 1) * chunks / EW;
        const unsigned lane_base = tmem_base + ((unsigned)(q * 32) << 16);
        const bool has0 = rank == 0 && ch0 == 0 && ch1 > 0;        // coordinate 0 is among this warp's
        const bool sends0 = last && h == 0;
        unsigned* pack = sm_pack + q * 32 * P.stage_words;          // the quadrant's rows
        for (int i = 0; i < n_mine; ++i) {
            const long long row0 = ((long long)cluster + (long long)i * n_clusters) * TM;
            const long long row = row0 + tok;
            const bool live = row < P.n_rows;
            // a warp whose wait ran out still comes to the quadrant's next barrier, where its four warps leave together
            bool ok = __all_sync(0xffffffffu, mbar_wait(&S->abort_flag, &S->tfull, i & 1, P.status, 4));
            float M = 0.f;
            if (ok) {
                tc_fence_after();
                for (int ch = ch0; ch < ch1; ++ch) {
                    const int n_here = P.m - (nb0 + 4 * ch) * 8;           // live coordinates from here on
                    if (n_here <= 0) break;
                    unsigned y[32];
                    load_chunk(lane_base + (unsigned)(8 * (ncb - 4 - 4 * ch)), y);
                    if (has0 && ch == 0) y[0] = 0u;                        // in the maximum of the CTA that has it
                    if (n_here < 32) {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (e >= n_here) y[e] = 0u;                    // coordinates beyond m
                    }
                    M = fmaxf(M, absmax32(y));
                }
                if (sends0) {
                    const float y0 = __uint_as_float(tmem_ld1(lane_base + col_r));
                    M = fmaxf(M, fabsf(y0));
                    peer_send(peer_addr(smem_u32(&S->y0[i & 1][tok]), 0u), y0, peer_addr(smem_u32(&S->maxbar[i & 1]), 0u));
                }
                S->part[i & 1][h][tok] = M;
            }
            if (meet_any(1 + q, !ok)) break;
            // the token's maximum: the quadrant's four warps have theirs together, and each sends it to a quarter of the CTAs (its own among them)
            M = fmaxf(fmaxf(S->part[i & 1][0][tok], S->part[i & 1][1][tok]), fmaxf(S->part[i & 1][2][tok], S->part[i & 1][3][tok]));
            const unsigned mine = smem_u32(&S->tmax[i & 1][rank][tok]), bar = smem_u32(&S->maxbar[i & 1]);
            for (int r = h; r < P.cl; r += EW) peer_send(peer_addr(mine, (unsigned)r), M, peer_addr(bar, (unsigned)r));
            ok = __all_sync(0xffffffffu, cluster_wait(&S->abort_flag, &S->maxbar[i & 1], (unsigned)(i >> 1) & 1u, P.status, 7));
            if (ok) {
                // the barrier's next tile but one.  (No CTA sends for that one before it has the next tile's maxima of all of this CTA's warps.)
                if (warp == 2 && lane == 0 && i + 2 < n_mine) mbar_arrive_expect_tx(&S->maxbar[i & 1], max_bytes);
                for (int r = 0; r < P.cl; ++r) M = fmaxf(M, S->tmax[i & 1][r][tok]);
                const float a1 = __fdividef(P.c_half, fmaxf(M, 1e-30f));
                for (int ch = ch0; ch < ch1; ++ch) {
                    const int n0 = (nb0 + 4 * ch) * 8, n_here = P.m - n0;
                    if (n_here <= 0) break;
                    unsigned y[32];
                    load_chunk(lane_base + (unsigned)(8 * (ncb - 4 - 4 * ch)), y);
                    if (has0 && ch == 0) y[0] = __float_as_uint(S->y0[i & 1][tok]);
                    unsigned out[BITS];
                    quantize_pack32<BITS>(y, a1, out);
#pragma unroll
                    for (int w = 0; w < BITS; ++w) pack[lane * P.stage_words + ch * BITS + w] = out[w];
                    if (P.y_opt && live) {
                        float* yo = P.y_opt + row * (long long)P.m + n0;
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (e < n_here) yo[e] = __uint_as_float(y[e]) * P.norm;
                    }
                }
                // the accumulators have been read: hand TMEM back to the MMA issuers
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->tempty);
                if (rank == 0 && h == 0 && live) {
                    // An infinity among the sixteen elements that meet column 0's repair is multiplied by its zeros there: every rotated
                    // value is NaN, which a maximum passes over.  Its scale is infinite, as for an infinity anywhere else.
                    if (M == 0.f) {
                        const unsigned short* x = P.x + row * P.stride;
                        for (int j = 0; j < 16 && j < P.d; ++j)
                            if ((__ldg(x + j) & 0x7fffu) == 0x7f80u) M = __uint_as_float(0x7f800000u);
                    }
                    P.scales[row] = P.c_scale * M;
                }
            }
            if (meet_any(1 + q, !ok)) break;
            // the CTA's piece of eight rows of the quadrant's 32, as aligned words; what the rows before and after share a word with, by bytes
            const int n_codes = P.m - nb0 * 8 < ncb * 8 ? P.m - nb0 * 8 : ncb * 8;
            const int nbytes = n_codes * BITS / 8;
            const long long first_row = row0 + q * 32 + h * 8;
            const unsigned* rows = pack + h * 8 * P.stage_words;
            unsigned char* piece = P.codes + first_row * P.code_row_bytes + nb0 * BITS;
            const int n_live = P.n_rows - first_row < 8 ? (int)(P.n_rows - first_row) : 8;
#pragma unroll 4
            for (int e = 0; e < n_live; ++e) {
                unsigned char* dst = piece + e * P.code_row_bytes;
                const int off = BITS == 4 ? 0 : (int)(reinterpret_cast<uintptr_t>(dst) & 3u);      // four-bit rows are words
                for (int j = lane; 4 * j - off + 4 <= nbytes; j += 32) {
                    const unsigned hi = rows[e * P.stage_words + j];
                    const unsigned lo = BITS == 4 || j == 0 ? 0u : rows[e * P.stage_words + j - 1];
                    if (off == 0 || j > 0) *reinterpret_cast<unsigned*>(dst + 4 * j - off) = BITS == 4 ? hi : __funnelshift_l(lo, hi, 8 * off);
                }
            }
            if (BITS != 4 && lane < 2 * n_live) {
                const int e = lane >> 1;
                unsigned char* dst = piece + e * P.code_row_bytes;
                const int lead = (int)(-reinterpret_cast<uintptr_t>(dst) & 3u), tail = (nbytes - lead) & 3;
                const unsigned char* src = reinterpret_cast<const unsigned char*>(rows + e * P.stage_words);
                const int at = lane & 1 ? nbytes - tail : 0, n = lane & 1 ? tail : lead;
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    if (b < n) dst[at + b] = src[at + b];
            }
        }
    }

    // ---- teardown.  Peers write to this CTA's shared memory only what its epilogue has waited for, so it may leave once every role has
    // left its loop; after an expired wait it stays until the cluster's CTAs have come here or ended.
    tc_fence_before();
    __syncthreads();
    __syncwarp();
    if (S->abort_flag) cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

// shared memory of a CTA that takes `ncb` output blocks of a contraction over `kchunks` chunks
int smem_bytes(int ncb, int kchunks, int stages, int* stage_words)
{
    const int w = ncb * 8 * 4 / 32 + 1;                            // a row's four-bit codes; odd: different banks
    if (stage_words) *stage_words = w;
    return 1024 + stages * A_STAGE + (kchunks * (KC / 8) + ncb) * CORE + ncb * 2 * CORE + ROW0_BYTES + TM * w * 4 + (int)sizeof(Ctl);
}

typedef void (*DenseKernel)(const CUtensorMap, const DenseParams);
DenseKernel kernel_of(int bits) { return bits == 3 ? k_tc_dense_rq<3> : k_tc_dense_rq<4>; }

// Clusters of `cl` CTAs that run at once (one CTA per SM; a cluster stays inside a GPC, so this can be less than SMs / cl, and none of
// more than eight CTAs need fit), asked of the device together with the opt-in to the large dynamic shared memory and, beyond eight CTAs, to such
// clusters (not stream operations).  -1: the question failed.
int ask_clusters(void* plan, int bits, int cl)
{
    const gbs_plan* p = static_cast<const gbs_plan*>(plan);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p->sm_count / cl * cl));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)p->smem_optin;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cl;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(kernel_of(bits), cudaFuncAttributeMaxDynamicSharedMemorySize, p->smem_optin) != cudaSuccess ||
        (cl > 8 && cudaFuncSetAttribute(kernel_of(bits), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
        cudaOccupancyMaxActiveClusters(&n, kernel_of(bits), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return n;
}

// The answer for one kernel and cluster size, or -1.  Only answers are kept: a question that failed is asked again by the next call.
int clusters_at_once(int* known, int bits, int cl, gbs_cluster_query query, void* ctx)
{
    int* k = known ? known + (bits - 3) * (MAX_CL + 1) + cl : nullptr;               // clusters + 1
    if (k && *k) return *k - 1;
    const int n = query(ctx, bits, cl);
    if (k && n >= 0) *k = n + 1;
    return n;
}

struct Split {
    int ctas, blocks, at_once;    // CTAs that share a token's coordinates, output blocks of each but the last, clusters at once
};

// How many CTAs share a token's coordinates.  An MMA of N columns takes N / 2 cycles (at least about 52), a stage's poll and commit 180 where
// one warp issues and 40 where two do, a tile's exchange and epilogue a few thousand, and the clusters that fit at once take the tiles in
// waves: the split with the least total is taken.  n_rows = 0 only asks whether a split exists.  1544, in us per launch of a graph of ten (calls one by
// one: 4096 rows 18.3), with 13, 10, 6 and 4 CTAs, 4 bits and, in brackets, 3: 1 row 8.8, 9.4, 12.1, 16.0 (9.0, 9.6, 12.2, 16.3); 772: 10.9, 11.0, 13.5, 17.3 (11.7, 11.9, 14.3,
// 18.4); 1400: 16.7, 12.0, 13.7, 17.3 (17.7, 12.8, 14.4, 18.4), with the nine taken 11.4 (12.3); 2600: 24.3, 19.2, 15.0, 18.3 (25.5, 20.2, 15.6, 19.4);
// 4096: 36.4, 26.7, 24.0, 19.4 (37.9, 28.0, 24.5, 20.5); 5500: 48.3, 34.1, 25.2, 31.7 (50.2, 35.6, 25.8, 32.8); 6854: 56.1, 41.3, 34.1, 32.1 (58.1,
// 43.2, 34.8, 33.2).
Split pick_split(int m, int d, int64_t n_rows, int bits, int smem_optin, int* known, gbs_cluster_query query, void* ctx)
{
    const int nb = m / 8, kchunks = (d + KC - 1) / KC;
    const int64_t n_tiles = (n_rows + TM - 1) / TM;
    double best = 0.0;
    Split split = {0, 0, 0};
    for (int ncb = 4; ncb <= 64; ncb += 4) {
        const int cl = (nb + ncb - 1) / ncb, real = nb - (cl - 1) * ncb, last = (real + 3) / 4 * 4;
        if (cl > MAX_CL || (last - real < 2 && 8 * last + 16 > TMEM_COLS) ||      // sixteen columns for coordinate 0 must fit
            smem_bytes(ncb, kchunks, 2, nullptr) > smem_optin)
            continue;
        const int fit = n_rows ? clusters_at_once(known, bits, cl, query, ctx) : 1;
        if (fit < 1) continue;
        const int64_t waves = (n_tiles + fit - 1) / fit;
        const auto chunk = [](int blocks, double more) {
            return 8.0 * ((blocks < 13 ? 52.0 : blocks * 4.0) + more) + (blocks < 26 ? 180.0 : 40.0);
        };
        double step = chunk(last, 52.0);                                          // the last CTA has coordinate 0's MMA as well
        if (cl > 1 && chunk(ncb, 0.0) > step) step = chunk(ncb, 0.0);
        const double cost = (double)waves * (kchunks * step + 4500.0 + 20.0 * ncb);
        if (split.ctas == 0 || cost < best) { best = cost; split = {cl, ncb, fit}; }
    }
    return split;
}

int padded_blocks(int m) { return m / 8 + 64; }                   // a CTA's share may reach beyond the last block

}  // namespace

// The plans this family serves: d' = m (no Sylvester factor), a large Paley order, one scale per token.
bool gbs_tc_dense_supported(const gbs_plan* p)
{
    if (!(p->k == 0 && p->m >= 128 && p->m % 8 == 0 && p->d % 8 == 0 && p->group == 0 && !p->asym && get_encode() != nullptr)) return false;
    return pick_split(p->m, p->d, 0, p->bits, p->smem_optin, nullptr, nullptr, nullptr).ctas != 0;
}

extern "C" int gbs_dense_rule(int m, int d, int64_t n_rows, int bits, int smem_optin, int* known, gbs_cluster_query query, void* ctx, int* blocks)
{
    const Split s = pick_split(m, d, n_rows, bits, smem_optin, known, query, ctx);
    *blocks = s.blocks;
    return s.ctas;
}

// bf16 image of H_m, row-major (row = output coordinate, column = input coordinate): m * m * 2 bytes (the inverse path's
// operand).
void gbs_tc_dense_image(const int8_t* hm, int m, unsigned short* img)
{
    for (size_t i = 0; i < (size_t)m * m; ++i) img[i] = hm[i] < 0 ? 0xBF80 : 0x3F80;
}

size_t gbs_tc_dense_toeplitz_bytes(int m) { return (size_t)((m + KC - 1) / KC * (KC / 8) + padded_blocks(m)) * CORE; }
size_t gbs_tc_dense_col0_bytes(int m) { return (size_t)padded_blocks(m) * 2 * CORE + ROW0_BYTES; }

// The forward path's tables: the Toeplitz core matrices (J = kb - nb + nbp - 1; row r, column c: t(8 (kb - nb) + c - r)) and
// the repair of column 0 (block nbp - 1 - i at i), with row 0 behind it (core matrices: rows 0 .. 7 of columns 0 .. 7 and 8 .. 15,
// then rows 8 .. 15, zero).  t(k - n) = H[n][k] for n, k >= 1; zero where no such pair exists.
void gbs_tc_dense_tables(const int8_t* hm, int m, unsigned short* toep, unsigned short* col0)
{
    const int nbp = padded_blocks(m);
    const int n_core = (int)(gbs_tc_dense_toeplitz_bytes(m) / CORE);
    auto t = [&](int delta) -> int {
        if (delta >= 0) return delta <= m - 2 ? hm[(size_t)m + 1 + delta] : 0;
        return -delta <= m - 2 ? hm[(size_t)(1 - delta) * m + 1] : 0;
    };
    auto bf = [](int v) -> unsigned short { return v == 0 ? 0 : (unsigned short)((v < 0 ? 0x8000 : 0) | (v == 2 || v == -2 ? 0x4000 : 0x3F80)); };
    for (int J = 0; J < n_core; ++J)
        for (int r = 0; r < 8; ++r)
            for (int c = 0; c < 8; ++c) toep[J * 64 + r * 8 + c] = bf(t(8 * (J - nbp + 1) + c - r));
    memset(col0, 0, gbs_tc_dense_col0_bytes(m));
    for (int i = 0; i < nbp; ++i)
        for (int r = 0; r < 8; ++r) {
            const int n = 8 * (nbp - 1 - i) + r;
            if (n >= 1 && n < m) col0[i * 128 + r * 8] = bf((int)hm[(size_t)n * m] - t(-n));
        }
    unsigned short* row0 = col0 + (size_t)nbp * 128;
    for (int v = 0; v < 2; ++v)
        for (int k = 0; k < 16; ++k) row0[v * 256 + (k >> 3) * 64 + (k & 7)] = bf(v ? -1 : (k == 0 ? 2 : 0));
}

int gbs_tc_dense_rotate_quantize(const gbs_plan* p, const void* x, int64_t n_rows, int64_t stride, void* codes,
                                 float* scales, float* y_opt, cudaStream_t stream)
{
    EncodeTiledFn encode = get_encode();
    if (!encode) return (int)cudaErrorNotSupported;
    if (n_rows > (int64_t)0x7fffffff - TM) return (int)cudaErrorInvalidValue;
    CUtensorMap xmap;
    const cuuint32_t estr[2] = {1, 1};
    const cuuint64_t gdim[2] = {(cuuint64_t)p->d, (cuuint64_t)n_rows};
    const cuuint64_t gstr[1] = {(cuuint64_t)(stride * 2)};
    const cuuint32_t box[2] = {64, TM};
    if (encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(x), gdim, gstr, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return (int)cudaErrorInvalidValue;
    DenseParams P;
    memset(&P, 0, sizeof(P));
    P.n_rows = n_rows;
    P.n_tiles = (int)((n_rows + TM - 1) / TM);
    P.m = p->m;
    P.d = p->d;
    P.x = (const unsigned short*)x;
    P.stride = stride;
    P.kchunks = (p->d + KC - 1) / KC;
    P.ksteps_last = ((p->d - (P.kchunks - 1) * KC) + 15) / 16;
    Split split;
    {
        static std::mutex mu;
        static int known[64][2 * (MAX_CL + 1)];
        std::lock_guard<std::mutex> lock(mu);
        split = pick_split(p->m, p->d, n_rows, p->bits, p->smem_optin, p->device >= 0 && p->device < 64 ? known[p->device] : nullptr, ask_clusters,
                           const_cast<gbs_plan*>(p));
    }
    if (split.ctas == 0) return (int)cudaErrorInvalidConfiguration;
    P.cl = split.ctas;
    P.ncb = split.blocks;
    P.ncb_last = ((p->m / 8 - (P.cl - 1) * P.ncb) + 3) / 4 * 4;
    P.nbp = padded_blocks(p->m);
    P.code_row_bytes = p->m * p->bits / 8;
    P.c_scale = p->c_scale;
    P.c_half = (float)(1.0 / (2.0 * (double)p->alpha));
    P.norm = p->norm;
    P.toep = p->d_dense;
    P.col0 = p->d_dense + gbs_tc_dense_toeplitz_bytes(p->m);
    P.row0 = P.col0 + (size_t)padded_blocks(p->m) * 2 * CORE;
    P.codes = (unsigned char*)codes;
    P.scales = scales;
    P.y_opt = y_opt;
    P.status = p->d_status;
    P.stages = smem_bytes(P.ncb, P.kchunks, MAX_STAGES, nullptr) <= p->smem_optin ? MAX_STAGES : 2;
    const int smem = smem_bytes(P.ncb, P.kchunks, P.stages, &P.stage_words);
    const int clusters = P.n_tiles < split.at_once ? P.n_tiles : split.at_once;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * P.cl));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)P.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p->pdl ? 2 : 1;
    return (int)cudaLaunchKernelEx(&cfg, kernel_of(p->bits), xmap, P);
}
