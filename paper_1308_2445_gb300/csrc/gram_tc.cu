// Gram products of step 8 on the tensor cores, by exact digit slices, with the accuracy of the double-float
// form checked entry by entry (mixed form: H_R = Z^T ZH, S_R = Z^T ZS, entries a <= b).
//
// The splitting idea is that of Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", Numer. Algorithms 59, 2012), in the
// fixed point of one chunk of rows:
//  - row i of Z is scaled by 2^-r_i and row i of ZH, ZS by 2^r_i, r_i the exponent of the row's largest
//    |Z| entry (the rows of an enriched basis span tens of decades, inversely in Z and in ZH, ZS);
//  - column a of the scaled Z is rounded to a 62-bit integer against its largest entry of the chunk, and
//    cut into 8 balanced base-256 digits d_s in [-128, 127] (the leading one in [-64, 64]), each exact in
//    FP16: slice s holds the digits d_s.  ZH and ZS likewise.
//  - digit products of equal weight 2^(-8 L), L = s + t <= 7, are summed by tcgen05.mma into one FP32
//    accumulator per level; over 256 rows the sums of levels 0-4 stay within 2^24, so they are exact, and
//    the rounding of levels 5-7 is far below the last bit kept.  Levels above 7 are dropped.
//  - every 256 rows the levels are added in 72-bit integers (unit 2^-45 of the leading digit product: 64 bits
//    and a byte of fraction), which hold the whole chunk (at most 8192 rows) without overflow.
// With P the product of the two columns' leading powers of two in the chunk and R its rows, the rounded operands and the
// dropped levels leave about sqrt(R) 2^-60 P, and the rounding of levels 6 and 7 at most 2^-56 P per 256 rows.  That is
// within the double-float form's rounding, 2^-48 sum|z||h|, wherever
//     sum|z||h| >= sqrt(R) 2^-11 P
// (random and same-signed columns on that line, emulated: at most 2^-47.8).  It takes the errors of different rows as
// independent.  Columns that repeat the same digits row after row beside maxima in other rows add them up one way: up to
// 2^-41 of sum|z||h| on the line at R = 8192, 2^-44 at R = 256; constant columns without such maxima lie far above it.
// Search blocks meet the line with bits to spare although a few rows dominate their columns (16^3 case: at
// least 2^-3.8 max|z| max|h|).  The kernel checks it for every entry: it first sums |z||h| (FP16, one MMA
// per step) over one row in 16, the one with the largest scaled ZH entry of its group, a lower bound
// within one or two bits on such blocks.  Entries that fail (none to some dozens of a million on the 32^3
// case) are put on a list and computed in FP64 by k_gram_tc_fixup; a unit (tile and chunk) with more than
// TG_UNIT_FIX of them, or with a non-finite input, is computed there in double-float (gram_df64_tile).
//
// Digit slices are laid out so that one MMA covers several levels: the B slices t = 0, 1, ... of the
// tile's 32 + 32 columns are adjacent along N and level L's accumulator begins at TMEM column 64 L, so
// A_s times the window B_0..B_(7-s) accumulates levels s..7 in MMAs of N up to 256 (measured 1176 clocks
// for the 36 digit products of 16 rows, of which 1152 are the tensor core's minimum; one MMA per product
// would take at least 50 clocks each).
//
// Bound: the integer pipe of the slicers (about 30 integer instructions per value and tile it meets; the
// tensor core waits for them).  n = 334,272, q = 538: 10.0 ms against 40.5 ms for the FP32 pipes;
// n = 47,620, q = 149: 0.28 against 0.64 ms.  Error against 64 bits on such blocks 3e-16 to 8e-16 (q = 538: 2.3e-15),
// float pairs 2e-15.
#include <algorithm>
#include <mutex>
#include <string>

#include "common.h"
#include "df64.h"
#include "gram_tile.h"
#include "slices.h"
#include "tc.h"

namespace hbsd {
namespace {

using df::Seg2d;
using namespace slices;

constexpr int TG_M = 128;                       // columns a of a tile (M of every MMA)
constexpr int TG_B = 32;                        // columns b of a tile, once of ZH and once of ZS
constexpr int TG_BLK = 256;                     // rows per flush of the accumulators
constexpr int TG_STEPS = FLUSH_STEPS;           // MMA steps per flush
constexpr int TG_MAX_BLKS = 32;                 // flushes per chunk: 8192 rows keep the sums below 2^62
constexpr int TG_NS = 3;                        // stage buffers
constexpr int TG_STAGE = DIG * (A_SLICE + B_SLICE);
constexpr int TG_ACC = 2 * TG_B * TG_M;         // sums per unit, 64 bits and a byte of fraction each
constexpr int TG_ATHREADS = 256;                // warps 0-7: slices of Z, flush
constexpr int TG_SLICERS = TG_ATHREADS + 128;   // warps 8-11: slices of ZH and ZS
constexpr int TG_THREADS = TG_SLICERS + 32;     // warp 12: MMA issue
constexpr size_t TG_SMEM = (size_t)TG_NS * TG_STAGE + (size_t)TG_ACC * 9 + 1024;
constexpr int TG_UNIT_FIX = 256;                // failing entries of a unit that are computed one by one
constexpr int TG_EXP_ROWS = 32;                 // rows per CTA of the exponent pass

// a failing entry on the list: its unit (any int), matrix (0: ZH, 1: ZS), columns b and a of the tile
__host__ __device__ constexpr long long tg_entry(int unit, int m, int cb, int ca) {
    return ((long long)unit << 13) | (m << 12) | (cb << 7) | ca;
}
__host__ __device__ constexpr int tg_entry_unit(long long e) { return (int)(e >> 13); }
static_assert(tg_entry_unit(tg_entry(0x7FFFFFFF, 1, TG_B - 1, TG_M - 1)) == 0x7FFFFFFF && tg_entry(1 << 18, 0, 0, 0) > 0,
              "an entry holds every unit");

// rexp[i] = exponent field of max_a |Z(i, a)|; cexp[chunk][0][c] = max over the chunk's rows of the
// exponent field of Z(i, c) minus rexp[i]; cexp[chunk][1..2][c] the same of ZH, ZS plus rexp[i] (memset
// below every real value before); sel[g] = the row of group g (16 rows) with the largest scaled ZH entry, by
// exponent.  One pass over the three blocks; a CTA's second read of its Z rows comes from L1.  32 rows
// per CTA and 16 loads in flight per thread: bound by the latency of the loads (n = 47,620, q = 149:
// 50 us; with 64 rows and 8 loads 78 us).
__global__ void __launch_bounds__(256) k_gram_tc_exps(Seg2d Z, Seg2d ZH, Seg2d ZS, int q, int64_t n, int64_t chunk_rows,
                                                      int* __restrict__ rexp, int* __restrict__ cexp, int* __restrict__ sel) {
    __shared__ int sr[TG_EXP_ROWS], skey[TG_EXP_ROWS / 16];
    const int64_t i0 = (int64_t)blockIdx.x * TG_EXP_ROWS;
    const int rows = (int)min((int64_t)TG_EXP_ROWS, n - i0);
    if (threadIdx.x < TG_EXP_ROWS) sr[threadIdx.x] = 0;
    if (threadIdx.x < TG_EXP_ROWS / 16) skey[threadIdx.x] = 0;
    __syncthreads();
    for (int c = threadIdx.x; c < ((q + 31) & ~31); c += 256) {   // whole warps
        int64_t ld;
        const double* p = Z.column(min(c, q - 1), ld);
        p += i0 * ld;
        for (int r0 = 0; r0 < rows; r0 += 16) {
            int e[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) e[r] = r0 + r < rows ? exp_field(p[(r0 + r) * ld]) : 0;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int m = __reduce_max_sync(0xffffffffu, e[r]);
                if ((threadIdx.x & 31) == r && m > 0) atomicMax(&sr[r0 + r], m);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < rows) rexp[i0 + threadIdx.x] = sr[threadIdx.x];
    int* ce = cexp + (i0 / chunk_rows) * 3 * q;
    for (int t = threadIdx.x; t < ((3 * q + 31) & ~31); t += 256) {
        const int m = min(t, 3 * q - 1) / q, c = min(t, 3 * q - 1) - m * q;
        int64_t ld;
        const double* p = m == 0 ? Z.column(c, ld) : (m == 1 ? ZH.column(c, ld) : ZS.column(c, ld));
        p += i0 * ld;
        int e = (int)0x80808080;
        for (int r0 = 0; r0 < rows; r0 += 16) {
            int x[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) x[r] = r0 + r < rows ? exp_field(p[(r0 + r) * ld]) : 0;
            int key = 0;
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int re = sr[(r0 + r) & (TG_EXP_ROWS - 1)];
                const int v = x[r] == 2047 ? BAD_EXP : (m == 0 ? x[r] - re : x[r] + re);
                if (x[r] != 0) {
                    e = max(e, v);
                    if (m == 1) key = max(key, ((x[r] + re) << 4) | (15 - r));   // the first of equal rows
                }
            }
            key = __reduce_max_sync(0xffffffffu, key);
            if ((threadIdx.x & 31) == 0 && key > 0) atomicMax(&skey[r0 / 16], key);
        }
        if (t < 3 * q && e > __ldcg(ce + t)) atomicMax(ce + t, e);   // the value only grows: most CTAs need no atomic
    }
    __syncthreads();
    if (threadIdx.x < TG_EXP_ROWS / 16 && threadIdx.x * 16 < rows)
        sel[i0 / 16 + threadIdx.x] = (int)(threadIdx.x * 16) + 15 - (skey[threadIdx.x] & 15);   // relative to i0
}

// tile pair p -> (ta, tb): a-tile ta (128 columns) with the b-tiles tb >= 4 ta of nb, ta-major
__device__ __forceinline__ void tg_pair(int p, int nb, int& ta, int& tb) {
    ta = 0;
    while (p >= nb - 4 * ta) {
        p -= nb - 4 * ta;
        ++ta;
    }
    tb = 4 * ta + p;
}

// One unit: 128 columns a x 32 columns b of both products over one chunk of rows, in phases: phase 0 sums
// the guard (one step of 16 selected rows per 256-row block), phase p the block p - 1 (16 steps).  Warps 0-11 cut the
// operands into slices (one thread: 8 rows of one column per step), warp 12 issues the MMAs, warps 0-7
// read the accumulators after each phase.  Three stages: full[s] completes when the slicers have filled
// stage s, empty[s] when the MMAs that read it are done, phasedone when a phase's MMAs are done, accfree
// when its accumulators have been read.  The reading of a phase waits until the slicers are two steps into
// the next one, so that the MMAs find filled stages afterwards.  list[0] counts the units left to k_gram_tc_fixup
// (a wait that gives up leaves its unit there too; units from list[2] on) and list[1] the single entries, in ents.
__global__ void __launch_bounds__(TG_THREADS, 1) k_gram_tc(Seg2d Z, Seg2d ZH, Seg2d ZS, int q, int64_t n,
                                                           int64_t chunk_rows, int nb, const int* __restrict__ rexp,
                                                           const int* __restrict__ cexp, const int* __restrict__ sel,
                                                           double* __restrict__ part, long long* __restrict__ ents,
                                                           int* __restrict__ list) {
    extern __shared__ __align__(1024) uint8_t tg_smem[];
    __shared__ __align__(8) uint64_t full[TG_NS], empty[TG_NS], phasedone, accfree, drain;
    __shared__ uint32_t tslot;
    __shared__ int s_flag, s_cnt, s_base, s_ent[TG_UNIT_FIX];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int ta, tb;
    tg_pair(blockIdx.x, nb, ta, tb);
    const int a0 = ta * TG_M, b0 = tb * TG_B;
    const int64_t r0 = (int64_t)blockIdx.y * chunk_rows, r1 = min(n, r0 + chunk_rows);
    const int steps = (int)((r1 - r0 + 15) / 16), nblk = (steps + TG_STEPS - 1) / TG_STEPS;
    const int total = nblk + steps;
    const int unit = (int)(blockIdx.y * gridDim.x + blockIdx.x);
    const int* ce = cexp + (int64_t)blockIdx.y * 3 * q;
    uint8_t* base = tg_smem + ((1024 - (tc::smem_u32(tg_smem) & 1023)) & 1023);
    long long* sacc = reinterpret_cast<long long*>(base + TG_NS * TG_STAGE);   // [64 columns b][128 columns a]
    uint32_t* slow = reinterpret_cast<uint32_t*>(sacc + TG_ACC);               // [16][128]: fractions, four columns b in a word
    if (tid == 0) {
        for (int i = 0; i < TG_NS; ++i) {
            tc::mbar_init(&full[i], TG_SLICERS / 32);
            tc::mbar_init(&empty[i], 1);
        }
        tc::mbar_init(&phasedone, 1);
        tc::mbar_init(&accfree, TG_ATHREADS / 32);
        tc::mbar_init(&drain, 1);
        s_flag = 0;
        s_cnt = 0;
    }
    // this thread's column: warps 0-7 column a (tid & 127) of Z, warps 8-11 column b of ZH or ZS
    const bool isa = warp < TG_ATHREADS / 32;
    const int bt = tid - TG_ATHREADS, bm = (bt >> 5) & 1;
    const int col = isa ? a0 + (tid & 127) : b0 + (bt & 31);
    const int half = isa ? tid >> 7 : (bt >> 6) & 1;
    const bool live = tid < TG_SLICERS && col < q;
    const int cmax = live ? ce[(isa ? 0 : (1 + bm) * q) + col] : 0;
    __syncthreads();
    if (live && cmax == BAD_EXP) s_flag = 1;
    if (warp == 0) tc::tmem_alloc(&tslot, 512);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = tslot;

    if (s_flag != 0) {
        // non-finite input: the whole unit goes to the fallback
    } else if (warp == TG_SLICERS / 32) {   // ---- MMA issuer
        if (lane == 0) {
            bool ok = true;
            int st = 0, t = 0;
            uint32_t ph = 0;
            for (int p = 0; ok && p <= nblk; ++p) {
                const int end = p == 0 ? nblk : min(total, nblk + p * TG_STEPS);
                // the accumulators of the phase before have been read
                if (p > 0) ok = tc::mbar_wait(&accfree, (uint32_t)((p - 1) & 1), WAIT_NS);
                for (const int first = t; ok && t < end; ++t) {
                    ok = tc::mbar_wait(&full[st], ph, WAIT_NS);
                    if (!ok) break;
                    tc::fence_after_sync();
                    const uint64_t a = tc::smem_desc(tc::smem_u32(base + st * TG_STAGE), 128, 256);
                    const uint64_t b = a + (uint64_t)((DIG * A_SLICE) >> 4);
                    if (p == 0) {
                        if (t == first) mma<0>(tbase, a, b, tc::idesc_f16_f32(TG_M, 2 * TG_B));
                        else mma<1>(tbase, a, b, tc::idesc_f16_f32(TG_M, 2 * TG_B));
                    } else {
                        if (t == first) mma_window<0, 0>(tbase, a, b);
                        else mma_window<0, 1>(tbase, a, b);
                        mma_window<1, 1>(tbase, a, b);
                        mma_window<2, 1>(tbase, a, b);
                        mma_window<3, 1>(tbase, a, b);
                        mma_window<4, 1>(tbase, a, b);
                        mma_window<5, 1>(tbase, a, b);
                        mma_window<6, 1>(tbase, a, b);
                        mma_window<7, 1>(tbase, a, b);
                    }
                    tc::mma_commit(&empty[st]);
                    if (++st == TG_NS) { st = 0; ph ^= 1u; }
                }
                if (ok) tc::mma_commit(&phasedone);
            }
            if (!ok) s_flag = 1;
            tc::mma_drain(&drain, WAIT_NS);
        }
    } else {   // ---- slicers, and (warps 0-7) the reading of the accumulators
        // a thread without a column reads column 0 of its block, with an exponent that shifts it to zero
        int64_t ld;
        const int pc = live ? col : 0;
        const double* p = isa ? Z.column(pc, ld) : (bm ? ZS.column(pc, ld) : ZH.column(pc, ld));
        const int ebase = live ? cmax : 1 << 20;
        const int row_in = isa ? tid & 127 : (bt & 31) + TG_B * bm;   // M or N index in the tile
        const uint32_t soff = (uint32_t)((isa ? 0 : DIG * A_SLICE) + half * 128 + (row_in >> 3) * 256 + (row_in & 7) * 16);
        const int stride = isa ? A_SLICE : B_SLICE;
        const int frow = (warp & 3) * 32 + lane, fm = (warp >> 2) & 1;   // column a, matrix of the reading
        const uint32_t taddr = tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(fm * TG_B);
        long long* facc = sacc + fm * TG_B * TG_M + frow;
        uint32_t* flow = slow + fm * (TG_B / 4) * TG_M + frow;
        if (isa)
#pragma unroll 4
            for (int c = 0; c < TG_B; ++c) {
                facc[c * TG_M] = 0;
                if (c < TG_B / 4) flow[c * TG_M] = 0;
            }
        auto read_phase = [&](int ph) {
            tc::warp_wait(&phasedone, (uint32_t)(ph & 1), WAIT_NS, &s_flag);
            __syncwarp();
            tc::fence_after_sync();
            if (ph == 0) {
                // the guard sums against the chunk's rows (see the head of the file); a column without
                // entries is exact
                const float need = sqrtf((float)(r1 - r0)) * 0x1p-11f;   // in units of the columns' leading powers of two
                const int a = a0 + frow;
                const bool az = a < q && ce[a] >= -4096;
#pragma unroll 1
                for (int c0 = 0; c0 < TG_B; c0 += 8) {
                    uint32_t v[8];
                    tmem_ld8(taddr + (uint32_t)c0, v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const int b = b0 + c0 + c;
                        if (az && b < q && a <= b && ce[(1 + fm) * q + b] >= -4096 && !(__uint_as_float(v[c]) >= need)) {
                            const int k = atomicAdd(&s_cnt, 1);
                            if (k < TG_UNIT_FIX) s_ent[k] = (fm << 12) | ((c0 + c) << 7) | frow;
                        }
                    }
                }
            } else {
#pragma unroll 1
                for (int c0 = 0; c0 < TG_B; c0 += 8) {
                    uint32_t v[8][8];
#pragma unroll
                    for (int l = 0; l < 8; ++l) tmem_ld8(taddr + (uint32_t)(2 * TG_B * l + c0), v[l]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                    for (int c = 0; c < 8; c += 4) {
                        uint32_t w = flow[(c0 + c) / 4 * TG_M];
#pragma unroll
                        for (int d = 0; d < 4; ++d) {
                            const uint32_t l[8] = {v[0][c + d], v[1][c + d], v[2][c + d], v[3][c + d],
                                                   v[4][c + d], v[5][c + d], v[6][c + d], v[7][c + d]};
                            facc[(c0 + c + d) * TG_M] += fold_levels(l, w, d);
                        }
                        flow[(c0 + c) / 4 * TG_M] = w;
                    }
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&accfree);
        };
        // the values and row exponents of the next two steps are on their way while one is sliced
        double x[2][8];
        int4 e[2][2];
        auto fetch = [&](int t, double (&xs)[8], int4 (&es)[2]) {
            if (t >= total) return;
            if (t < nblk) {   // the selected rows of block t
                const int64_t b = r0 + (int64_t)t * TG_BLK;
                int ee[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int64_t g = b + (half * 8 + c) * 16;
                    const int64_t i = g < r1 ? (g & ~(int64_t)(TG_EXP_ROWS - 1)) + sel[g / 16] : r1;
                    xs[c] = i < r1 ? p[i * ld] : 0.0;
                    ee[c] = i < r1 ? rexp[i] : 0;
                }
                es[0] = make_int4(ee[0], ee[1], ee[2], ee[3]);
                es[1] = make_int4(ee[4], ee[5], ee[6], ee[7]);
                return;
            }
            const int64_t i = r0 + (int64_t)(t - nblk) * 16 + half * 8;   // rexp is padded to whole blocks
            es[0] = __ldg(reinterpret_cast<const int4*>(rexp + i));
            es[1] = __ldg(reinterpret_cast<const int4*>(rexp + i + 4));
            const double* pi = p + i * ld;
            if (i + 8 <= r1) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    xs[c] = __ldg(pi);
                    pi += ld;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) xs[c] = i + c < r1 ? p[(i + c) * ld] : 0.0;
            }
        };
        fetch(0, x[0], e[0]);
        fetch(1, x[1], e[1]);
        int st = 0, done = 0, ended = 0, since = 0, next_end = nblk;
        uint32_t ph = 1;
        auto step = [&](int t, double (&xs)[8], int4 (&es)[2]) {
            const int sg = isa ? 1 : -1;
            const int off[8] = {ebase + sg * es[0].x, ebase + sg * es[0].y, ebase + sg * es[0].z, ebase + sg * es[0].w,
                                ebase + sg * es[1].x, ebase + sg * es[1].y, ebase + sg * es[1].z, ebase + sg * es[1].w};
            // the first pass over the stages finds them empty (parity 1 of a fresh barrier is complete)
            tc::warp_wait(&empty[st], ph, WAIT_NS, &s_flag);
            if (t < nblk) slice8_guard(xs, off, base + st * TG_STAGE + soff);
            else slice8(xs, off, base + st * TG_STAGE + soff, stride);
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[st]);   // one arrival per warp
            fetch(t + 2, xs, es);
            if (++st == TG_NS) { st = 0; ph ^= 1u; }
            if (isa) {
                ++since;
                if (done < ended && since >= 2) read_phase(done++);
                if (t + 1 == next_end) {   // a phase's last step
                    ++ended;
                    since = 0;
                    next_end = min(total, next_end + TG_STEPS);
                }
            }
        };
        for (int t = 0; t < total; t += 2) {
            step(t, x[0], e[0]);
            if (t + 1 < total) step(t + 1, x[1], e[1]);
        }
        if (isa)
            while (done < ended) read_phase(done++);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
    const int nfix = s_cnt;
    if (s_flag || nfix > TG_UNIT_FIX) {
        if (tid == 0) list[2 + atomicAdd(list, 1)] = unit;
        return;
    }
    if (nfix > 0) {
        if (tid == 0) s_base = atomicAdd(list + 1, nfix);
        __syncthreads();
        for (int t = tid; t < nfix; t += TG_THREADS)
            ents[s_base + t] = tg_entry(unit, s_ent[t] >> 12, (s_ent[t] >> 7) & (TG_B - 1), s_ent[t] & (TG_M - 1));
    }
    double* out = part + (int64_t)unit * TG_ACC;
    for (int t = tid; t < TG_ACC; t += TG_THREADS) {
        const int a = a0 + (t & (TG_M - 1)), c = t / TG_M, b = b0 + (c & (TG_B - 1));
        if (a < q && b < q) out[t] = scaled_sum(sacc[t], slow[c / 4 * TG_M + (t & (TG_M - 1))], c & 3, ce[a] + ce[(1 + c / TG_B) * q + b] - 2056 - FRAC);
    }
}

// The listed units in double-float, four 32 x 32 tiles each, and the listed entries in FP64, one CTA each
__global__ void __launch_bounds__(GTHREADS, GCTAS) k_gram_tc_fixup(Seg2d Z, Seg2d ZH, Seg2d ZS, int q, int64_t n,
                                                                   int64_t chunk_rows, int nb, int npair, df::f32x2 nz,
                                                                   double* __restrict__ part, const long long* __restrict__ ents,
                                                                   const int* __restrict__ list) {
    __shared__ GramTile sm;
    const int cnt = list[0], nent = list[1];
    for (int w = blockIdx.x; w < 4 * cnt; w += gridDim.x) {
        const int unit = list[2 + (w >> 2)], sub = w & 3;
        const int chunk = unit / npair;
        int ta, tb;
        tg_pair(unit - chunk * npair, nb, ta, tb);
        const int a0 = ta * TG_M + sub * GW, b0 = tb * TG_B;
        if (a0 >= q || a0 > b0) continue;   // tiles above the diagonal only (b0 is a multiple of 32)
        const int64_t r0 = (int64_t)chunk * chunk_rows;
        double* out = part + (int64_t)unit * TG_ACC;
        gram_df64_tile(sm, Z, ZH, ZS, q, a0, b0, GW / 4, false, r0, min(n, r0 + chunk_rows), nz,
                       [&](int m, int a, int b, double v) { out[(m * TG_B + b - b0) * TG_M + (a - ta * TG_M)] = v; });
        __syncthreads();
    }
    double* red = &sm.acc[0][0];
    for (int w = blockIdx.x; w < nent; w += gridDim.x) {
        const long long ent = ents[w];
        const int unit = tg_entry_unit(ent), code = (int)ent, m = (code >> 12) & 1;
        const int chunk = unit / npair;
        int ta, tb;
        tg_pair(unit - chunk * npair, nb, ta, tb);
        const int cb = (code >> 7) & 31, ca = code & 127;
        int64_t lz, lx;
        const double* z = Z.column(ta * TG_M + ca, lz);
        const double* x = m ? ZS.column(tb * TG_B + cb, lx) : ZH.column(tb * TG_B + cb, lx);
        const int64_t r0 = (int64_t)chunk * chunk_rows, r1 = min(n, r0 + chunk_rows);
        double acc = 0.0;
        for (int64_t i = r0 + threadIdx.x; i < r1; i += GTHREADS) acc = fma(z[i * lz], x[i * lx], acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) part[(int64_t)unit * TG_ACC + (m * TG_B + cb) * TG_M + ca] = (red[0] + red[1]) + (red[2] + red[3]);
        __syncthreads();
    }
}

// Sum of the chunks in order; the entry (a, b), a <= b, is used for (b, a) too.
__global__ void __launch_bounds__(256) k_gram_tc_final(const double* __restrict__ part, int nchunks, int npair, int nb, int q,
                                                       double* __restrict__ HR, double* __restrict__ SR) {
    __shared__ double rh[8][33], rs[8][33];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t idx = (int64_t)blockIdx.x * 32 + lane;
    const int b = (int)(idx / q), a = (int)(idx - (int64_t)b * q);   // lanes over the contiguous index a
    const bool on = b < q && a <= b;
    double h = 0.0, s = 0.0;
    if (on) {
        const int ta = a / TG_M, tb = b / TG_B;
        const int pair = ta * nb - 2 * ta * (ta - 1) + tb - 4 * ta;
        const int64_t o = (int64_t)(b - tb * TG_B) * TG_M + (a - ta * TG_M);
        for (int c = g; c < nchunks; c += 8) {
            const double* p = part + ((int64_t)c * npair + pair) * TG_ACC + o;
            h += p[0];
            s += p[TG_B * TG_M];
        }
    }
    rh[g][lane] = h;
    rs[g][lane] = s;
    __syncthreads();
    if (g == 0 && on) {
        double H = 0.0, S = 0.0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            H += rh[t][lane];
            S += rs[t][lane];
        }
        HR[(int64_t)a * q + b] = H;
        SR[(int64_t)a * q + b] = S;
        HR[(int64_t)b * q + a] = H;
        SR[(int64_t)b * q + a] = S;
    }
}

}  // namespace

// tile pairs, and chunks of whole 256-row blocks: the height that ends the last wave of units soonest
struct TgPlan {
    int nb, npair, nch;
    int64_t chunk_rows, units, rpad;
    size_t ints, doubles;   // of the workspace
};
static TgPlan tg_plan(int64_t n, int q) {
    TgPlan g;
    g.nb = ceil_div(q, TG_B);
    g.npair = 0;
    for (int ta = 0; ta * TG_M < q; ++ta) g.npair += g.nb - 4 * ta;
    const int nblk = ceil_div(n, TG_BLK);
    int bpc = 1;
    double best = 1e300;
    for (int k = 1; k <= std::min(nblk, TG_MAX_BLKS); ++k) {
        const double cost = (double)ceil_div((int64_t)g.npair * ceil_div(nblk, k), 152) * (k + 0.4);
        if (cost < best) {
            best = cost;
            bpc = k;
        }
    }
    g.chunk_rows = (int64_t)bpc * TG_BLK;
    g.nch = ceil_div(n, g.chunk_rows);
    g.units = (int64_t)g.nch * g.npair;
    g.rpad = round_up(n, TG_BLK);
    // workspace: sums | listed entries | row exponents | column exponents | guard rows | listed units
    g.ints = (size_t)g.rpad + (size_t)g.nch * 3 * q + (size_t)g.rpad / 16 + 2 + (size_t)g.units;
    g.doubles = (size_t)g.units * (TG_ACC + TG_UNIT_FIX) + g.ints / 2 + 64;
    return g;
}
size_t gram_tc_doubles(int64_t n, int q) { return tg_plan(n, q).doubles; }

int gram2_tc(Session* s, const double* Z0, int64_t ld0, int q0, const double* Z1, int64_t ld1, int q1, const double* H0,
             int64_t ldh0, const double* H1, int64_t ldh1, const double* S0, int64_t lds0, const double* S1, int64_t lds1,
             int64_t n, double* HR, double* SR, cudaStream_t st) {
    const int q = q0 + q1;
    const TgPlan g = tg_plan(n, q);
    const int nb = g.nb, npair = g.npair, nch = g.nch;
    const int64_t chunk_rows = g.chunk_rows, units = g.units, rpad = g.rpad;
    HBSD_TRY(s->df_ws.alloc(g.doubles));
    double* part = s->df_ws.p;
    long long* ents = reinterpret_cast<long long*>(part + units * TG_ACC);
    int* rexp = reinterpret_cast<int*>(ents + units * TG_UNIT_FIX);   // 16-byte aligned: both strides are even
    int* cexp = rexp + rpad;
    int* sel = cexp + (size_t)nch * 3 * q;
    int* list = sel + rpad / 16;
    HBSD_CUDA(cudaMemsetAsync(cexp, 0x80, (size_t)nch * 3 * q * sizeof(int), st));
    HBSD_CUDA(cudaMemsetAsync(list, 0, 2 * sizeof(int), st));
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        attr = cudaFuncSetAttribute(k_gram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TG_SMEM);
    });
    HBSD_CUDA(attr);
    Seg2d Z{Z0, ld0, q0, Z1, ld1}, ZH{H0, ldh0, q0, H1, ldh1}, ZS{S0, lds0, q0, S1, lds1};
    k_gram_tc_exps<<<ceil_div(n, TG_EXP_ROWS), 256, 0, st>>>(Z, ZH, ZS, q, n, chunk_rows, rexp, cexp, sel);
    HBSD_LAUNCHED(s);
    k_gram_tc<<<dim3(npair, nch), TG_THREADS, TG_SMEM, st>>>(Z, ZH, ZS, q, n, chunk_rows, nb, rexp, cexp, sel, part, ents,
                                                              list);
    HBSD_LAUNCHED(s);
    k_gram_tc_fixup<<<152 * GCTAS, GTHREADS, 0, st>>>(Z, ZH, ZS, q, n, chunk_rows, nb, npair, df::NEG_ZERO2, part, ents,
                                                      list);
    HBSD_LAUNCHED(s);
    k_gram_tc_final<<<ceil_div((int64_t)q * q, 32), 256, 0, st>>>(part, nch, npair, nb, q, HR, SR);
    HBSD_LAUNCHED(s);
    return 0;
}

}  // namespace hbsd
