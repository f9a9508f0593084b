// gbs_clip_error for bf16 rows of the UV family by histogram instead of one pass per candidate.
//
// With t = |y| / M (M = the max|y| of the token or group), candidate k quantizes |y| / M to the level l = number of its thresholds
// (j + 1/2) alpha_k / D, j = 0 .. D-1, that t has reached (Sections 2.1, 3.1: rounding to the nearest level, clipping at D).
// With D' = alpha_k / D the error is  M^2 (t - D' l)^2 = M^2 [t^2 - 2 D' t l + D'^2 l^2],  so all K candidates follow from how
// many values (W0) and which sum of t (W1) lie beyond each of the K D thresholds:
//        sum t l = sum_j W1(beyond threshold j),    sum l^2 = sum_j (2 j + 1) W0(beyond threshold j).
// One histogram over the sorted thresholds replaces 5 K operations per value by about 12 whatever K is.
//   * Front end as in gbs_tc_uv.cu: TMA, A X on tcgen05, H_32 in registers, the maximum over a token's four warps.
//   * t becomes a 22-bit integer in the mantissa of one FMA.  Its high bits index a table of cells; an entry holds the
//     number of thresholds below the cell and the low bits of the one threshold inside it, placed so that adding the
//     value's low bits carries into the bin index when the threshold is reached.  Cells are as wide as they can be without two
//     different thresholds in one (512 of them do for ratios k / 64 and 3 bits), and the room that leaves in the table's 64 KB holds copies
//     of an entry side by side, one per lane at 512 cells: lanes then meet in a bank as rarely as the copies allow (one copy of
//     4096 cells: 3.4 cycles per lookup of a warp).  (Where 4096 cells do not part them the call goes to the per-candidate kernel.
//     Thresholds that are one and the same number, such as 1.5 x 0.5 and 0.5 x 1.5 over D, may come
//     out one unit of t apart when the ratios are rounded to floats; they count as one, the lower.)
//   * Two shared-memory atomics per value (count and t) into COPIES interleaved histograms per token, so that a warp's lanes
//     rarely meet: measured 2 cycles per 32 values with 32 copies and 6 with 8.  Everything is an integer: exact in any order.
//   * One scale per token: after a token its 128 threads add the copies up and weigh them with M^2 in fp64.  Nothing is cleared: the words
//     grow modulo 2^32 and a token's part is the difference from the total before it, which its thread keeps.
//   * One scale per group of 128 coordinates or more: the four rows of A X that make up 128 coordinates go to the same lane of the four
//     quadrants, so a warp's lanes belong to different groups and the copy of a lane IS a group's histogram.  The copies are then weighed one by
//     one with their groups' M^2 and cleared; every warp takes a share of the copies of every bin, so that its weights stay in
//     registers.  (A thread per bin instead reads all 32 weights for each of them and leaves a warp idle: 32 768 x 4096, K = 32: 219 us at 3 bits
//     and 321 at 4, against 196 and 277.)  More than 112 thresholds leave room for the histograms of two tokens, not four: two warps then share a
//     lane, each taking half of H_32's outputs.
//   * The t^2 term is the sum of the same integers' squares, in 64 bits, so the three parts of the error belong to one and the same t and
//     may cancel down to the 16 digits of fp64: a candidate that fits a batch exactly is as accurate as the others, wherever it stands in the list.
//     t's rounding is the only approximation.  The integer is within half a unit (2^-23) of the product, and the multiplier, one float per token or
//     group, within 2^-24 of its own size: together at most 1.5 x 2^-23, so that an error E over n values moves by at most 1.5 x 2^-22 M sqrt(n E) +
//     2.25 n 2^-46 M^2.  The integers' part differs from value to value and grows with the square root of n only; the multiplier's is common to a
//     token or group.  Against 64 bits the sums are closer than the per-candidate kernel's, whose Delta is rounded once for all: groups of 128,
//     4096 rows, K = 32, largest relative error 2e-9 - 5e-8 against 6e-8 - 2e-7 on ordinary rows, up to 4e-7 against 2e-5 where a candidate nearly fits.
//   * A stands in tensor memory, so that an MMA reads one operand from shared memory and the table has the other's room.
// What bounds it: the chain of a token's four warps, with the shared-memory port 56 - 63 % busy (per token about 130 cycles of lookups, 330 of
// atomics, 200 of adding up, 450 with groups, 65 of the MMA's operand) and 54 - 65 % of the issue slots taken.  Neither count and sum in one
// atomic (2^24 + t, taken apart again when added up; two histograms in turn and one barrier per token: 148 us where this takes 135)
// nor barriers that warps arrive at early and wait for late (154) nor fewer instructions per value (no change) make it faster.
// 32 768 x 4096, K = 32, 3 bits: 829 us with five fp32 operations per value and candidate; 171.4 with one copy of the table, histograms
// that were cleared for every token (390 cycles with the adding up) and A in shared memory; 135.2 now.  Groups of 128: 839 -> 196 us at 3
// bits, 839 -> 277 at 4; K = 8: 253 -> 162 and 179.
#include <math.h>
#include <string.h>

#include <mutex>

#include "gbs_internal.h"
#include "gbs_tc_common.cuh"

namespace {

constexpr int V = 32, TOK_MAX = 4, UMAX = 128;    // a tile is 4 tokens, or 2
constexpr int STAGES = 2;                          // accumulators; one set of rows in shared memory: a tile takes far longer than its load
constexpr int STAGE_BYTES_MAX = TOK_MAX * UMAX * V * 2;
constexpr int A_COL0 = STAGES * TOK_MAX * V;       // A in tensor memory: a row per lane, two entries per column
constexpr int EPI_WARPS = 16;                      // 16 / TOK of them to a token
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr int TMEM_COLS = 512;
constexpr int T_BITS = 22;                         // t is an integer of 22 bits
constexpr int TABLE_LOG = 14;                      // words of the table of cells: cells x copies
constexpr int MIN_CELL_BITS = 10, MAX_CELL_BITS = 13;          // bits of t inside a cell: 4096 cells x 4 copies .. 512 x 32
constexpr int HIST_TILE = 14336;                   // words of a tile's counts (and of its sums): tokens x bins x copies
constexpr int HIST_WORDS = 2 * (HIST_TILE + TOK_MAX * 32);     // [token][count, sum][one row nobody reads, bins][copy]
constexpr int MAX_BINS = 448;                      // thresholds: K D at most
constexpr unsigned POISON = 0xffffffffu;

struct __align__(1024) Smem {
    unsigned char b[STAGE_BYTES_MAX];
    unsigned hist[HIST_WORDS];
    unsigned lut[1 << TABLE_LOG];
    unsigned red[TOK_MAX][2][4];                   // maxima, by tile parity: a word per warp
    double square[EPI_WARPS];                      // sums of t^2
    unsigned long long full, empty, tfull[STAGES], tempty[STAGES];
    unsigned tmem_base;
    volatile int abort_flag;
    double2 weight[2][TOK_MAX][16];                // groups: M^2 of every copy, by tile parity
    unsigned lane_red[TOK_MAX][2][256];            // groups: maxima, a word per lane
};

struct ClipParams {
    int n_groups;                 // tiles: ceil(n_rows / TOK)
    int Upad, ksteps;
    int K, levels, n_thr;
    int cell_bits;                // the largest number for which no cell holds two different thresholds
    int glog;                     // groups: log2(lanes per group), a lane of four warps having four rows of A X
    float scale;                  // of t as an integer
    float norm2;                  // 1 / d'
    const unsigned char* a_img;
    double* err_sum;
    int* status;
    float alpha[GBS_MAX_CANDIDATES];
    unsigned thr[MAX_BINS];                       // sorted, different, one per cell at most
    unsigned short idx[GBS_MAX_CANDIDATES][7];    // threshold j of candidate k
};

__device__ __forceinline__ unsigned ld_shared(unsigned a)
{
    unsigned v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));          // the table does not change once it is built
    return v;
}

// an integer as a double, by its place in the mantissa of 2^52
__device__ __forceinline__ double exact(unsigned v) { return __hiloint2double(0x43300000, (int)v) - 4503599627370496.0; }

// Tokens of a tile, copies of a histogram (TOK x COPIES x bins is the same for every instantiation: as many copies as the thresholds leave
// room for), one scale per token or per group
template <int TOK, int COPIES, bool GROUPED>
__global__ void __launch_bounds__(THREADS, 1) k_tc_uv_clip(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ ClipParams P)
{
    constexpr int HALVES = 4 / TOK;                               // warps that share a TMEM lane of a token
    constexpr int NV = V / HALVES;                                // values of a thread
    constexpr int TOKEN_WARPS = 4 * HALVES;
    constexpr int STAGE_COLS = TOK * V;
    constexpr int HIST_ROWS = HIST_TILE / TOK;                    // words of a token's counts (and of its sums)
    constexpr int BINS = HIST_ROWS / COPIES;
    // Adding up: a thread takes all copies of a bin, or, with groups, every warp of a token a share (CHUNKS times four) of the copies
    // of every bin, 32 bins at a time.
    constexpr int CHUNKS = GROUPED ? 8 / TOKEN_WARPS : COPIES / 4;
    constexpr int BIN_LANES = GROUPED ? 32 : 32 * TOKEN_WARPS;
    constexpr int PER = (BINS + BIN_LANES - 1) / BIN_LANES;       // bins of a thread
    constexpr int PARTS = GROUPED ? EPI_WARPS : TOK;               // of a bin's total
    static_assert(TOK == 4 || GROUPED, "two warps share a lane only where groups leave no room for four tokens");
    static_assert(!GROUPED || COPIES == 32, "a copy per lane");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Smem* S = reinterpret_cast<Smem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned stage_bytes = (unsigned)(TOK * P.Upad * V * 2);

    if (threadIdx.x == 0) {
        mbar_init(&S->full, 1);
        mbar_init(&S->empty, 1);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&S->tfull[s], 1);
            mbar_init(&S->tempty[s], EPI_WARPS);
        }
        S->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&S->tmem_base, TMEM_COLS);
    for (int i = threadIdx.x; i < HIST_WORDS / 4; i += THREADS) reinterpret_cast<uint4*>(S->hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < EPI_WARPS) S->square[threadIdx.x] = 0.0;
    unsigned* thr = reinterpret_cast<unsigned*>(S->b);             // the first load comes later
    for (int i = threadIdx.x; i < P.n_thr; i += THREADS) thr[i] = P.thr[i];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = S->tmem_base;
    const int copies_log = P.cell_bits + TABLE_LOG - T_BITS;       // of an entry: 4 .. 32, side by side
    if (threadIdx.x < (1 << (T_BITS - MAX_CELL_BITS))) {
        // cell c: thresholds below it, and where the one inside it lies; a run of cells per thread, found by one binary search
        const int run = 1 << (MAX_CELL_BITS - P.cell_bits), c0 = threadIdx.x * run;
        const unsigned in_cell = 1u << P.cell_bits;
        int lo = 0, hi = P.n_thr;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (thr[mid] < ((unsigned)c0 << P.cell_bits)) lo = mid + 1; else hi = mid;
        }
        for (int c = c0; c < c0 + run; ++c) {
            unsigned e = (unsigned)lo << P.cell_bits;
            const unsigned next = lo < P.n_thr ? thr[lo] : 0xffffffffu;
            if ((next >> P.cell_bits) == (unsigned)c) { e += in_cell - (next & (in_cell - 1u)); ++lo; }
            uint4* entry = reinterpret_cast<uint4*>(S->lut + (c << copies_log));
            const int quads = 1 << (copies_log - 2);
            for (int j = 0; j < quads; ++j) entry[(j + lane) & (quads - 1)] = make_uint4(e, e, e, e);   // lanes side by side: different banks
        }
    }
    if (warp >= 2 && warp < 6) {
        // A (plan-owned, immutable: needs no ordering) from its image, two blocks of 64 columns, 128-byte swizzled rows, to tensor memory
        // groups: four neighbouring rows go to the same lane of the four quadrants, so that a warp's lanes belong to 32 different groups
        const int r = GROUPED ? 4 * lane + (warp & 3) : (warp & 3) * 32 + lane;
        const unsigned at = tmem_base + ((unsigned)((warp & 3) * 32) << 16) + A_COL0;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            uint4 w[4];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                w[c] = __ldg(reinterpret_cast<const uint4*>(P.a_img + (h >> 1) * (UMAX * 128) + r * 128 + (((4 * (h & 1) + c) ^ (r & 7)) << 4)));
            tmem_st16(at + h * 16, w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int n_mine = (P.n_groups - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

    double w0[PER], w1[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) w0[i] = w1[i] = 0.0;
    if (warp == 0) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the thresholds were read from where the rows go
            int it = 0;
            for (int g = blockIdx.x; g < P.n_groups; g += gridDim.x, ++it) {
                if (!mbar_wait(&S->abort_flag, &S->empty, (it & 1) ^ 1, P.status, 1)) break;
                mbar_arrive_expect_tx(&S->full, stage_bytes);
                tma_load_3d(S->b, &tmap, &S->full, 0, 0, g * TOK);
            }
            if (S->abort_flag) drain_copies(&S->full, 1, it);
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        {
            constexpr unsigned IDESC = instr_desc(UMAX, STAGE_COLS);
            const unsigned long long bd0 = smem_desc(smem_u32(S->b), (unsigned)(P.Upad * V * 2), 512, 4);
            for (int it = 0; it < n_mine; ++it) {
                const int s = it % STAGES;
                if (!mbar_wait_warp(&S->abort_flag, &S->full, it & 1, P.status, 2)) break;
                if (!mbar_wait_warp(&S->abort_flag, &S->tempty[s], ((it / STAGES) & 1) ^ 1, P.status, 3)) break;
                tc_fence_after();
                // a k-step: eight columns of A's lanes, 1024 bytes of the rows
                const unsigned d_tmem = tmem_base + s * STAGE_COLS;
                for (int ks = 0; ks < P.ksteps; ++ks)
                    umma_f16_ts(d_tmem, tmem_base + A_COL0 + ks * 8, bd0 + (unsigned long long)(ks * (1024 >> 4)), IDESC, ks != 0 ? 1u : 0u);
                umma_commit(&S->empty);
                umma_commit(&S->tfull[s]);
            }
        }
    } else {
        // ------------------------------ histogram ------------------------------
        const int w = warp - 2, t = GROUPED ? w / TOKEN_WARPS : w >> 2, half = (w >> 2) % HALVES, q = warp & 3;
        const int wt = half * 4 + q;                              // of the token's warps
        const int bin0 = GROUPED ? lane : q * 32 + lane;
        const int chunk0 = GROUPED ? lane + wt * CHUNKS : lane;   // eight lanes side by side: different banks
        const unsigned taddr0 = tmem_base + ((unsigned)(q * 32) << 16) + t * V;
        unsigned* hist = S->hist + t * 2 * (HIST_ROWS + 32) + 32;            // behind a row for values below every threshold
        constexpr unsigned BIN_STEP = COPIES * 4;
        constexpr int SUM_OFF = (HIST_ROWS + 32) * 4;
        // bin b (b thresholds reached) is row b - 1: bin 0 lands in the row before the first, which costs less than a predicate
        // (a predicated reduction becomes a branch: 264 us instead of 250)
        const unsigned hb = smem_u32(hist) + (unsigned)(lane % COPIES) * 4u - BIN_STEP;
        const unsigned lut = smem_u32(S->lut) + ((unsigned)(lane & ((1 << copies_log) - 1)) << 2);
        const unsigned cell_mask = (4u << TABLE_LOG) - (4u << copies_log);        // a cell's first byte in the table
        const unsigned low_mask = (1u << P.cell_bits) - 1u;
        const int cell_bits = P.cell_bits;
        // one scale per token: the histograms only ever grow, modulo 2^32, and a token's own counts and sums are what a bin has gained
        // since the token before
        unsigned was0[PER], was[PER][4];
#pragma unroll
        for (int i = 0; i < PER; ++i) was0[i] = was[i][0] = was[i][1] = was[i][2] = was[i][3] = 0u;
        constexpr float MAGIC = 8388608.f;
        constexpr unsigned E = 0x4B000000u;                       // its bit pattern
        double square = 0.0;
        float poison = 0.f;                                       // NaN once a value was not finite
        // What the token of tile `it` left in this thread's bins.  Groups: every copy is another one's; weighed one by one, and cleared.  (The two
        // forms share no code here: written as one they cost tokens 0.8 % and, inlined like the other, groups 1.5 %.)
        auto add_up_groups = [&](int it) {
            double2 weight[CHUNKS][2];
#pragma unroll
            for (int j = 0; j < CHUNKS; ++j) {
                const int jj = (chunk0 + j) % (COPIES / 4);
                weight[j][0] = S->weight[it & 1][t][2 * jj];
                weight[j][1] = S->weight[it & 1][t][2 * jj + 1];
            }
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const int bin = bin0 + BIN_LANES * i;
                if (bin < P.n_thr) {
                    uint4* row = reinterpret_cast<uint4*>(hist + bin * COPIES);
                    uint4* row1 = reinterpret_cast<uint4*>(hist + SUM_OFF / 4 + bin * COPIES);
#pragma unroll
                    for (int j = 0; j < CHUNKS; ++j) {
                        const int jj = (chunk0 + j) % (COPIES / 4);
                        const uint4 x = row[jj], z = row1[jj];
                        row[jj] = row1[jj] = make_uint4(0u, 0u, 0u, 0u);
                        w0[i] = fma(weight[j][0].x, exact(x.x), w0[i]); w1[i] = fma(weight[j][0].x, exact(z.x), w1[i]);
                        w0[i] = fma(weight[j][0].y, exact(x.y), w0[i]); w1[i] = fma(weight[j][0].y, exact(z.y), w1[i]);
                        w0[i] = fma(weight[j][1].x, exact(x.z), w0[i]); w1[i] = fma(weight[j][1].x, exact(z.z), w1[i]);
                        w0[i] = fma(weight[j][1].y, exact(x.w), w0[i]); w1[i] = fma(weight[j][1].y, exact(z.w), w1[i]);
                    }
                }
            }
        };

        for (int it = 0; it < n_mine; ++it) {
            const int s = it % STAGES;
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&S->abort_flag, &S->tfull[s], (it / STAGES) & 1, P.status, 4, false));
            unsigned r[V];
            unsigned mb = POISON;
            if (ok) {
                tc_fence_after();
                tmem_ld32_issue(taddr0 + s * STAGE_COLS, r);
                tmem_ld_wait(r);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S->tempty[s]);
                if constexpr (GROUPED) mb = __float_as_uint(HALVES == 1 ? fwht32_absmax(r) : fwht32_half_absmax(r, half ? -1.f : 1.f));
                else mb = __reduce_max_sync(0xffffffffu, __float_as_uint(fwht32_absmax(r)));
            }
            unsigned* slot = GROUPED ? S->lane_red[t][it & 1] : S->red[t][it & 1];
            if (GROUPED) slot[wt * 32 + lane] = mb;
            else if (lane == 0) slot[q] = mb;
            // The barrier also keeps this token's atomics behind the adding up of the token before.
            asm volatile("bar.sync %0, %1;" ::"r"(1 + t), "n"(32 * TOKEN_WARPS) : "memory");
            if (GROUPED) {
#pragma unroll
                for (int i = 0; i < TOKEN_WARPS; ++i) mb = max(mb, slot[i * 32 + lane]);
            } else {
                mb = max(max(slot[0], slot[1]), max(slot[2], slot[3]));
            }
            if (mb == POISON) break;                               // in every lane
            if (GROUPED)
                for (int o = (1 << P.glog) >> 1; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
            const float M = __uint_as_float(mb);
            if (GROUPED && wt == 0) reinterpret_cast<double*>(S->weight[it & 1][t])[lane] = (double)M * (double)M;
            float lift = 1.f;                                      // scale / M must not overflow
            if (M < 0x1p-96f) {
                lift = 0x1p64f;
#pragma unroll
                for (int i = 0; i < NV; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * lift);
            }
            const float sc = M > 0.f ? P.scale / (M * lift) : 0.f;
            // every value is a signed sum of all that came out of TMEM: the first shows whether one was not finite
            poison = fmaf(__uint_as_float(r[0]), 0.f, poison);
            unsigned long long sq = 0ull;                          // squares below 2^44
            // eight values at a time: their lookups are in flight together
#pragma unroll
            for (int i0 = 0; i0 < NV; i0 += 8) {
                unsigned b[8], e[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    b[i] = __float_as_uint(fmaf(fabsf(__uint_as_float(r[i0 + i])), sc, MAGIC));
                    e[i] = ld_shared(lut + ((b[i] >> (T_BITS - TABLE_LOG - 2)) & cell_mask));
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    b[i] -= E;
                    sq += (unsigned long long)b[i] * b[i];
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const unsigned bin = (e[i] + (b[i] & low_mask)) >> cell_bits;
                    const unsigned at = hb + bin * BIN_STEP;
                    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(at) : "memory");
                    asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(at), "r"(b[i]), "n"(SUM_OFF) : "memory");
                }
            }
            asm volatile("bar.sync %0, %1;" ::"r"(1 + t), "n"(32 * TOKEN_WARPS) : "memory");
            const double m2 = (double)M * (double)M;
            square += m2 * (double)sq;
            if constexpr (GROUPED) {
                add_up_groups(it);
            } else {
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    const int bin = bin0 + BIN_LANES * i;
                    if (bin < P.n_thr) {
                        const uint4* row = reinterpret_cast<const uint4*>(hist + bin * COPIES);
                        const uint4* row1 = reinterpret_cast<const uint4*>(hist + SUM_OFF / 4 + bin * COPIES);
                        unsigned c = 0u;
                        uint4 m = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                        for (int j = 0; j < CHUNKS; ++j) {
                            const int jj = (chunk0 + j) % (COPIES / 4);
                            const uint4 x = row[jj], z = row1[jj];
                            c += (x.x + x.y) + (x.z + x.w);
                            m.x += z.x; m.y += z.y; m.z += z.z; m.w += z.w;
                        }
                        // a component gains at most 1024 values below 2^22: less than 2^32
                        const unsigned long long sum = ((unsigned long long)(m.x - was[i][0]) + (m.y - was[i][1])) +
                                                       ((unsigned long long)(m.z - was[i][2]) + (m.w - was[i][3]));
                        w0[i] += m2 * (double)(c - was0[i]);
                        w1[i] += m2 * (double)sum;
                        was0[i] = c;
                        was[i][0] = m.x; was[i][1] = m.y; was[i][2] = m.z; was[i][3] = m.w;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) square += __shfl_xor_sync(0xffffffffu, square, o);
        if (__any_sync(0xffffffffu, poison != 0.f)) square = __longlong_as_double(0x7ff8000000000000ll);
        if (lane == 0) S->square[w] = square;
    }

    // ---- the block's totals: [bin] over the parts, then from the last threshold down
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
    double* tot = reinterpret_cast<double*>(S->hist);              // [part][2][BINS]
    if (warp >= 2) {
        const int part = GROUPED ? warp - 2 : (warp - 2) / TOKEN_WARPS;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int bin = (GROUPED ? lane : (warp & 3) * 32 + lane) + BIN_LANES * i;
            if (bin < P.n_thr) {
                tot[(part * 2) * BINS + bin] = w0[i];
                tot[(part * 2 + 1) * BINS + bin] = w1[i];
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * P.n_thr; i += THREADS) {
        double* d = tot + (i < P.n_thr ? i : BINS + i - P.n_thr);
        if constexpr (GROUPED) {
            double sum = d[0];
            for (int part = 1; part < PARTS; ++part) sum += d[part * 2 * BINS];
            d[0] = sum;
        } else {
            d[0] = (d[0] + d[2 * BINS]) + (d[4 * BINS] + d[6 * BINS]);
        }
    }
    __syncthreads();
    double* suf = tot + PARTS * 2 * BINS;                          // [2][BINS]: sum over bins b, b + 1, ..
    if (warp < 2) {
        // warp 0 the counts, warp 1 the sums: a contiguous piece per lane, pieces joined from the right
        const int per = (P.n_thr + 31) / 32, b0 = lane * per;
        double s = 0.0;
        for (int b = b0; b < b0 + per && b < P.n_thr; ++b)
            s += tot[warp * BINS + b];
        double after = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double v = __shfl_down_sync(0xffffffffu, after, o);
            if (lane + o < 32) after += v;
        }
        after -= s;                                                // the pieces to the right of this one
        for (int b = (b0 + per < P.n_thr ? b0 + per : P.n_thr) - 1; b >= b0; --b) {
            after += tot[warp * BINS + b];
            suf[warp * BINS + b] = after;
        }
    }
    __syncthreads();
    if (threadIdx.x < P.K) {
        const int k = threadIdx.x;
        const double d = (double)P.alpha[k] / (double)P.levels, scale = (double)P.scale;
        double t2 = 0.0, l1 = 0.0, l2 = 0.0;
        for (int i = 0; i < EPI_WARPS; ++i) t2 += S->square[i];
        for (int j = 0; j < P.levels; ++j) {
            const int b = P.idx[k][j];
            l2 += (double)(2 * j + 1) * suf[b];
            l1 += suf[BINS + b];
        }
        const double err = (t2 / scale - 2.0 * d * l1) / scale + d * d * l2;
        atomicAdd(&P.err_sum[k], (err < 0.0 ? 0.0 : err) * (double)P.norm2);       // what fp64 leaves of an exact fit; NaN stays
    }
}

typedef void (*ClipKernel)(const CUtensorMap, const ClipParams);

}  // namespace

// Scores K clip ratios, or returns GBS_UVCLIP_NOT_SERVED where this path does not apply (groups of 32 or 64, per-row sums, thresholds
// too close to one another, more than 224 of them with groups): the caller then takes the per-candidate kernel.  So it does where that is the faster one, with candidates for
// one of its passes (eight) and few tiles per block, where building the table is what counts.  One scale per token: up to one (64 x 4096, K = 8:
// 6.8 us there, 7.0 here at 3 bits, 7.4 at 4; 600 rows, 4 bits: 11.2 and 10.1).  Groups: up to three (700 rows: 16.5 and 16.7 at 3 bits,
// 18.5 at 4; 2000: 24.9 and 22.8, 24.7).  More candidates take two passes or more there: groups, 1 row, K = 9: 10.2 and 7.2 us at 3 bits, 7.8 at 4, K = 16:
// 10.2 and 7.8, 8.7; 591 rows, K = 16: 12.1 and 10.8, 11.9.
int gbs_tc_uv_clip_histogram(const gbs_plan* p, const void* x, int64_t n_rows, int64_t stride, const float* alphas, int K,
                             double* err_sum, cudaStream_t stream)
{
    EncodeTiledFn encode = get_encode();
    const bool grouped = p->group != 0;
    if (K <= 8 && n_rows <= (int64_t)TOK_MAX * p->sm_count * (grouped ? 3 : 1)) return GBS_UVCLIP_NOT_SERVED;
    if ((grouped && p->group < 4 * V) || !encode || p->smem_optin < (int)sizeof(Smem) || n_rows > (int64_t)0x7fffffff - TOK_MAX)
        return GBS_UVCLIP_NOT_SERVED;
    ClipParams P;
    memset(&P, 0, sizeof(P));
    const int D = p->levels;
    // t = 1 must stay below 2^22 after rounding
    P.scale = 4194304.f - 8.f;
    // the widest cells that no two different thresholds share
    constexpr int CELLS = 1 << (T_BITS - MIN_CELL_BITS);
    constexpr unsigned SAME = 1;                   // alpha rounds to 2^-25, an eighth of a unit; ceil makes one of it
    unsigned T[GBS_MAX_CANDIDATES * 7];
    for (int k = 0; k < K; ++k)
        for (int j = 0; j < D; ++j) {
            const double t = ceil((j + 0.5) / D * (double)alphas[k] * (double)P.scale);
            if (!(t < (double)(1 << T_BITS))) return GBS_UVCLIP_NOT_SERVED;
            T[k * D + j] = (unsigned)t;
        }
    unsigned long long used[CELLS / 64];
    unsigned at[CELLS], last[CELLS];               // the lowest and the highest threshold of a cell
    unsigned short rank[CELLS];
    bool apart = false;
    for (P.cell_bits = MAX_CELL_BITS; P.cell_bits >= MIN_CELL_BITS; --P.cell_bits) {
        memset(used, 0, sizeof(used));
        apart = true;
        for (int i = 0; apart && i < K * D; ++i) {
            const unsigned c = T[i] >> P.cell_bits;
            const bool seen = used[c >> 6] >> (c & 63) & 1;
            at[c] = seen && at[c] < T[i] ? at[c] : T[i];
            last[c] = seen && last[c] > T[i] ? last[c] : T[i];
            apart = last[c] - at[c] <= SAME;
            used[c >> 6] |= 1ull << (c & 63);
        }
        if (apart) break;
    }
    if (!apart) return GBS_UVCLIP_NOT_SERVED;
    for (int w = 0; w < CELLS / 64; ++w)
        for (unsigned long long m = used[w]; m; m &= m - 1) {
            const int c = w * 64 + __builtin_ctzll(m);
            rank[c] = (unsigned short)P.n_thr;
            P.thr[P.n_thr++] = at[c];
        }
    for (int k = 0; k < K; ++k) {
        P.alpha[k] = alphas[k];
        for (int j = 0; j < D; ++j) P.idx[k][j] = rank[T[k * D + j] >> P.cell_bits];
    }
    struct Form {
        ClipKernel kernel;
        int tok, bins;
    };
    static const Form forms[5] = {{k_tc_uv_clip<4, 32, false>, 4, 112}, {k_tc_uv_clip<4, 16, false>, 4, 224}, {k_tc_uv_clip<4, 8, false>, 4, 448},
                                  {k_tc_uv_clip<4, 32, true>, 4, 112}, {k_tc_uv_clip<2, 32, true>, 2, 224}};
    const Form* form = forms + (grouped ? 3 : 0);
    while (form < forms + (grouped ? 5 : 3) && P.n_thr > form->bins) ++form;
    if (form == forms + 5) return GBS_UVCLIP_NOT_SERVED;           // groups: a copy per lane leaves room for 224 thresholds
    CUtensorMap tmap;
    const int U = p->d_pad / V;
    P.Upad = (U + 15) & ~15;
    const cuuint64_t gdim[3] = {(cuuint64_t)V, (cuuint64_t)(p->d / V), (cuuint64_t)n_rows};
    const cuuint64_t gstr[2] = {(cuuint64_t)(V * 2), (cuuint64_t)(stride * 2)};
    const cuuint32_t box[3] = {V, (cuuint32_t)P.Upad, (cuuint32_t)form->tok}, estr[3] = {1, 1, 1};
    if (encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return (int)cudaErrorInvalidValue;
    P.n_groups = (int)((n_rows + form->tok - 1) / form->tok);
    for (int g = p->group / (4 * V); g > 1; g >>= 1) ++P.glog;
    P.ksteps = P.Upad / 16;
    P.K = K;
    P.levels = D;
    P.norm2 = (float)(1.0 / (double)p->d_pad);
    P.a_img = p->d_aimg;
    P.err_sum = err_sum;
    P.status = p->d_status;
    {
        // opt in to the large dynamic shared memory once per device (not a stream operation)
        static std::mutex mu;
        static bool done[64] = {false};
        std::lock_guard<std::mutex> lock(mu);
        if (!(p->device >= 0 && p->device < 64 && done[p->device])) {
            for (const Form& f : forms) {
                const cudaError_t e = cudaFuncSetAttribute(f.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
                if (e != cudaSuccess) return (int)e;
            }
            if (p->device >= 0 && p->device < 64) done[p->device] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(P.n_groups < p->sm_count ? P.n_groups : p->sm_count));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = sizeof(Smem);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p->pdl ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, form->kernel, tmap, P);
}
