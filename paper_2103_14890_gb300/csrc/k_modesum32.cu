// k_modesum32.cu -- register-blocked FP32 mode sum of eq. CF1 (Sec. 3.3) for
// 2-D velocity grids (N <= 64; N <= 48 in FP64) and 3-D grids with N <= 16.
//
// Work reduction (exact algebra, no approximation):
//   * Q is real, so only k_1 >= 0 is computed (Q-hat_{-k} = conj(Q-hat_k)).
//   * The product f-hat_l f-hat_m is symmetric in (l, m): pairs with l_1 < m_1
//     are summed once with the weight beta-hat(l,m) + beta-hat(m,l); pairs with
//     l_1 = m_1 keep beta-hat(l,m).  So for outputs with first index k_1 only
//     l_1 in [k_1 - h, floor(k_1/2)] is visited and m_1 = k_1 - l_1 >= 0 always
//     lies in the stored half spectrum; f-hat_l with l_1 < 0 is conj(f-hat_{-l}).
//   * A "row" is the line of modes along the last axis with all other indices
//     fixed: (k_1) in 2-D, (k_1, k_2) in 3-D.  Each task's weight stream names
//     the pairs of rows (row of l, row of m) it visits, so the kernel body is
//     the same in both dimensions.
//
// Layout and blocking:
//   * one CTA = one tile of C cells (C = 32, or 16 or 8 for grids whose spectrum
//     does not fit 32 cells in shared memory); the tile's half spectrum
//     (complex FP32, [mode][cell]) sits in shared memory with lane % C = cell,
//     so every weight load is uniform over the lanes that share it and every
//     Fourier load is a conflict-free row of C cells.
//   * a task = (k_1, block of RT consecutive k_2).  With C = 32 a thread owns
//     all RT = R outputs of its cell; with C = 16 the two half-warps split the
//     block, each thread owning R = RT/2 of them.  Walking l_2 upwards slides
//     the window of f-hat_m values (m_2 = k_2 - l_2) down by one, so each step
//     loads one new f-hat_m, one f-hat_l and R weights for 6 R FP32 operations.
//   * each task's weights form a contiguous stream of row pairs, each a
//     16-byte header (which rows of l and m) followed by [l (padded to a
//     multiple of RT)][r]; one row pair is staged into a per-warp
//     shared-memory double buffer with cp.async while the previous one is used.
//   * the rows of the spectrum are stored back to back, with kPad zero columns
//     before the first and after the last row only.  A column index that falls
//     outside [-h, h] therefore reads a neighbouring row's (finite) value or a
//     zero, and always meets a zero weight: the weight stream is zero wherever
//     l_2, m_2 or k_2 leaves K_h.  The host checks that every column touched
//     stays within kPad of [-h, h].
//   * accumulation: plain FP32 along an l_1 row (<= 48 terms), then a TwoSum
//     fold of the row sum into a (hi, lo) pair per output every 4 rows.
//   * several kernel variants (R, warps, C) are compiled; the fastest one for a
//     grid is chosen once by timing (autotune below).
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>
#include <vector>

#include "bz_device.cuh"
#include "bz_internal.h"

namespace bz {

namespace {

// Kernel variants: outputs per thread R along k_2, warps per CTA, cells per
// CTA, cells per thread (pack: 1, or 2 for the packed two-cell kernel, whose
// lanes hold cells c and c + 16 of a 32-cell tile in FP32x2 register pairs),
// wdup: each weight stored twice (w, w) as an FP32x2 operand, pq: the FP32x2
// form with one cell per lane (modesum_pq_kernel), orient: 2 when the two
// halves of a warp (of each of its row groups) hold the same cells and run
// each task plain and mirrored (paired orientations), rows: row pairs of a
// task that a warp sums at a time, one per group of lanes.  Variant ids
// reported by bz_modes_info are index + 1.
struct Variant {
    int R, warps, cells, pack, wdup, pq, orient, rows;
};
constexpr int kNumVariants = kModesumVariants;   // FP32 variants (timed by the autotuner)
// entries 0..9: the FP32 variants; entries 10..12: layouts of the FP64 and FP32X2
// forms (16 bytes per spectrum value): 8-cell tiles, 4-cell tiles for 16^3, and
// two outputs per thread for grids of fewer than 8 points; entry 13: the paired
// 16-cell FP32 variants with two outputs per thread, for small launches
constexpr int kSmallVariant = kNumVariants + 3;
constexpr Variant kVariants[kNumVariants + 4] = {
    {8, 16, 32, 1, 0, 0, 1, 1}, {4, 32, 32, 1, 0, 0, 1, 1}, {4, 16, 16, 1, 0, 0, 1, 1}, {8, 12, 8, 1, 0, 1, 2, 2},
    {4, 16, 32, 2, 1, 0, 1, 1}, {8, 12, 32, 1, 0, 1, 1, 1}, {8, 16, 32, 1, 0, 1, 1, 1}, {8, 16, 16, 1, 0, 1, 2, 1},
    {8, 8, 16, 1, 0, 1, 2, 1},  {8, 4, 16, 1, 0, 1, 2, 1},  {4, 8, 8, 1, 0, 1, 2, 2},   {4, 8, 4, 1, 0, 1, 2, 4},
    {2, 8, 8, 1, 0, 1, 2, 2},   {2, 16, 16, 1, 0, 1, 2, 1}};

// lane groups splitting a task's outputs, and outputs per task (RT)
constexpr int variant_groups(int v) {
    return 32 / kVariants[v].cells * kVariants[v].pack / kVariants[v].orient / kVariants[v].rows;
}
constexpr int variant_rt(int v) { return kVariants[v].R * variant_groups(v); }
// Whether an FP32 variant's tables compute k_2 < 0 on the reflected spectrum
// (every output block of k_2 >= 0 fits within the row: R T <= h + 1); all
// variants that do sum each output in one order, as do all that do not.
constexpr bool variant_reflects(int v, int h) { return kVariants[v].pack == 1 && variant_rt(v) <= h + 1; }
constexpr int kTaskInts = 12;   // ints per task record

constexpr int kPad = 8;         // zero guard columns before the first and after the last row
constexpr int kRowHeadBytes = 16;   // row-pair header in front of each weight row

struct TaskRec {
    int orow, k20, nrows, l2lo, nblk, woff, rfirst;   // rfirst: first r (of RT) this task stores
    int rowf, flags, crow, pad2, pad3;                // rowf: elements per row pair (header + weights);
                                                      // flags: kTask*; crow: row of the conjugate outputs
};

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int NPENDING> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NPENDING) : "memory");
}

// Knuth's TwoSum: s + e == a + b exactly.
template <typename T> __device__ __forceinline__ void two_sum(T a, T b, T &s, T &e) {
    s = a + b;
    T bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Stage `nbytes` bytes (multiple of 16) of a weight row into shared memory.
__device__ __forceinline__ void stage_row(void *dst, const void *src, int nbytes, int lane) {
    char *d = static_cast<char *>(dst);
    const char *g = static_cast<const char *>(src);
    for (int i = lane * 16; i < nbytes; i += 512) cp_async16(d + i, g + i);
    cp_async_commit();
}

// R consecutive weights (16-byte aligned) into registers.
__device__ __forceinline__ void load_w4(float *wv, const float *p) {
    const float4 w4 = *reinterpret_cast<const float4 *>(p);
    wv[0] = w4.x;
    wv[1] = w4.y;
    wv[2] = w4.z;
    wv[3] = w4.w;
}
// One block of RR l_2 steps.  The window of f-hat_m values lives in a 2RR-slot
// register array used under two alternating namings (PH = 0, 1): logical slot
// j is physical slot (j + PH RR) mod 2RR, so moving the window by RR between
// blocks costs no register moves; logical slot j of a block holds the column
// mp + j CS, and output r at step s reads logical slot r - s + RR - 1.
// f-hat_l is read at lp, lp + D, lp + 2 D, ... with D = DIR CS: for DIR = -1
// (l_1 < 0) the row is that of -l_1 read backwards and f-hat_l = conj of the
// value read, which only flips the signs of two FMA operands.  DIR = 0 takes
// the direction at run time (D = dcs, sgn = +/-1 multiplies the value's
// imaginary part): the products are those of DIR = +1 on the conjugated value,
// which are exactly those of DIR = -1 on the value read (negation is exact), so
// the results equal the specialised bodies' bit for bit with half the code.
// The weights of step s are wb[s * WS + r].
//
// RAMP: the first block of a task whose steps start one before the lowest l_2
// of its first output (l2lo = k2_0 - h - 1, outputs k2_0 + r >= 0): pair
// (s, r) lies in K_h exactly when s > r, so only those pairs are evaluated
// (the others have zero weights and would add exact zeros), and the window
// slots it needs are only the RR - 1 it loads itself.
template <typename T, int RR, int CS, int WS, int PH, int DIR, bool RAMP>
__device__ __forceinline__ void block_body(typename C2<T>::type (&win)[2 * RR],
                                           const typename C2<T>::type *__restrict__ mp,
                                           const typename C2<T>::type *__restrict__ lp, int dcs, T sgn,
                                           const T *__restrict__ wb, typename C2<T>::type (&acc)[RR]) {
    using V2 = typename C2<T>::type;
#pragma unroll
    for (int j = 0; j < (RAMP ? RR - 1 : RR); ++j) win[(j + PH * RR) & (2 * RR - 1)] = mp[j * CS];
#pragma unroll
    for (int s = RAMP ? 1 : 0; s < RR; ++s) {
        V2 fl = (DIR == 0) ? lp[s * dcs] : lp[s * DIR * CS];
        if (DIR == 0) fl.y *= sgn;
        T wv[RR];
#pragma unroll
        for (int q = 0; q < RR; q += 4)
            if (!RAMP || q < s) load_w4(wv + q, wb + s * WS + q);
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            if (RAMP && r >= s) continue;
            const V2 b = win[(r - s + RR - 1 + PH * RR) & (2 * RR - 1)];
            const T tx = wv[r] * fl.x, ty = wv[r] * fl.y;       // weight * value read
            if (DIR >= 0) {                                     // acc += w f-hat_l b
                acc[r].x = fma(tx, b.x, acc[r].x);
                acc[r].x = fma(-ty, b.y, acc[r].x);
                acc[r].y = fma(tx, b.y, acc[r].y);
                acc[r].y = fma(ty, b.x, acc[r].y);
            } else {                                            // acc += w conj(value) b
                acc[r].x = fma(tx, b.x, acc[r].x);
                acc[r].x = fma(ty, b.y, acc[r].x);
                acc[r].y = fma(tx, b.y, acc[r].y);
                acc[r].y = fma(-ty, b.x, acc[r].y);
            }
        }
    }
}

// One row pair of a task for this thread's RR outputs:
// acc[r] += sum_l2 w(l2, r) f-hat_l(l2) f-hat_m(k2_0 + r - l2) over nblk
// blocks of RR steps from l2lo.  rowl / rowm point at column 0 of the rows of
// l (or -l) and m (this thread's cell); wrow at this thread's first weight of
// the row.  The blocks run as pairs (PH 0, PH 1) and a last PH 0; with ramp
// (RAMPS only) the first block is the ramp body.
template <typename T, int RR, int CS, int WS, int DIR, bool RAMPS>
__device__ __forceinline__ void row_pass(const typename C2<T>::type *__restrict__ rowl,
                                         const typename C2<T>::type *__restrict__ rowm, const T *__restrict__ wrow,
                                         int nblk, int l2lo, int mbase0, int dir, bool ramp,
                                         typename C2<T>::type (&acc)[RR]) {
    using V2 = typename C2<T>::type;
    V2 win[2 * RR];
    const int dcs = (DIR == 0 ? dir : DIR) * CS;
    const T sgn = (T)dir;
    const V2 *mp = rowm + mbase0 * CS;
    const V2 *lp = rowl + l2lo * dcs;
    int blk = 0;
    bool ramped = false;
    if constexpr (RAMPS) {
        if (ramp) {
            // the ramp block under the PH 1 naming leaves the window exactly
            // as the preload below does for a first block under PH 0
            block_body<T, RR, CS, WS, 1, DIR, true>(win, mp, lp, dcs, sgn, wrow, acc);
            mp -= RR * CS;
            lp += RR * dcs;
            blk = 1;
            ramped = true;
        }
    }
    if (!ramped) {
#pragma unroll
        for (int j = RR; j < 2 * RR - 1; ++j) win[j] = mp[j * CS];
    }
    for (; blk + 1 < nblk; blk += 2) {
        block_body<T, RR, CS, WS, 0, DIR, false>(win, mp, lp, dcs, sgn, wrow + blk * RR * WS, acc);
        block_body<T, RR, CS, WS, 1, DIR, false>(win, mp - RR * CS, lp + RR * dcs, dcs, sgn,
                                                 wrow + (blk + 1) * RR * WS, acc);
        mp -= 2 * RR * CS;
        lp += 2 * RR * dcs;
    }
    if (blk < nblk) block_body<T, RR, CS, WS, 0, DIR, false>(win, mp, lp, dcs, sgn, wrow + blk * RR * WS, acc);
}

// Copy this CTA's cells of the tile's half spectrum into shared memory
// ([kPad + nhalf + kPad][CELLS], zero guards), or with every row's columns
// reversed (rev: mode (row, c) <- (row, -c), the spectrum of f reflected in
// the last velocity axis).  AFTER: in a kernel launched after the one that wrote
// it programmatically.
template <typename V2, int CELLS, bool AFTER = false>
__device__ __forceinline__ void stage_spectrum(uint4 *smem16, const V2 *fhat, int64_t tile, int sub, int nhalf,
                                               int M, bool rev) {
    constexpr int VEC = 16 / (int)sizeof(V2);                    // cells per 16-byte vector
    constexpr int Q4 = CELLS / VEC, ROW = 32 / VEC;              // vectors per mode: this CTA, whole tile
    const uint4 *src = reinterpret_cast<const uint4 *>(fhat + tile * (int64_t)nhalf * 32) + sub * Q4;
    const int body = nhalf * Q4, guard = kPad * Q4;
    for (int i = threadIdx.x; i < body + 2 * guard; i += blockDim.x) {
        const int b = i - guard;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (b >= 0 && b < body) {
            int mode = b / Q4;
            if (rev) {
                const int row = mode / M;
                mode = row * M + (M - 1) - (mode - row * M);
            }
            const uint4 *x = src + mode * ROW + (b % Q4);
            if constexpr (AFTER) v = __ldcg(x);
            else v = *x;
        }
        smem16[i] = v;
    }
}

// Task flags (TaskRec.flags)
constexpr int kTaskRamp = 1;     // first block is the ramp (l2lo = k2_0 - h - 1)
constexpr int kTaskRefl = 2;     // reflected block: on the reflected spectrum (restaged, or read mirrored); output k_2 at column -k_2
constexpr int kTaskConj = 4;     // k_1 = 0 row: also stores conj(Q-hat) at (row crow, column -k_2), k_2 > 0

// The task table: 2 W + 1 offsets (W = warps x split), then the records.
// Warp w's phase-0 tasks are [off[w], off[w + 1]) and its phase-1 tasks
// [off[W + w], off[W + w + 1]); phase 1 (tasks flagged kTaskRefl) runs after
// the CTA has restaged its spectrum reversed.  Tables without reflected
// tasks have an empty phase 1.
template <typename T, int RR, int WARPS, int CELLS, bool RTDIR = false>
__global__ void __launch_bounds__(WARPS * 32, 1) modesum32_kernel(const Mode32Group gd) {
    using V2 = typename C2<T>::type;
    constexpr int G = 32 / CELLS;     // lane groups splitting a task's outputs
    constexpr int RT = RR * G;        // outputs per task
    constexpr int HEAD = kRowHeadBytes / (int)sizeof(T);
    constexpr bool RAMPS = (G == 1);  // ramped tasks need every lane on the same outputs
    extern __shared__ __align__(16) uint4 smem16[];
    // this CTA's instance and tile (instances are ordered longest-first)
    int it = 0;
    while (it + 1 < gd.nitems && (int64_t)blockIdx.x >= gd.tile_start[it + 1]) ++it;
    const Mode32Item &ip = gd.item[it];
    const V2 *__restrict__ fhat = static_cast<const V2 *>(ip.fhat);
    V2 *__restrict__ Qhat = static_cast<V2 *>(ip.Qhat);
    const T *__restrict__ W = static_cast<const T *>(ip.W);
    const int *__restrict__ tasks = ip.tasks;
    const int h = ip.h, M = ip.M, nhalf = ip.nhalf, wrow_max = ip.wrow_max;
    const int64_t n = ip.n;
    // a tile may be split over ip.split CTAs, each taking one part of the
    // task table (the last partial wave of a launch)
    const int64_t cta0 = (int64_t)blockIdx.x - gd.tile_start[it];
    const int part = (int)(cta0 % ip.split);
    const int64_t cta = cta0 / ip.split;
    const int64_t tile = cta / G;                                    // 32-cell tile of the scratch layout
    const int sub = (int)(cta % G);                                  // which CELLS-cell part of it
    V2 *Fs = reinterpret_cast<V2 *>(smem16);                         // [kPad + nhalf + kPad][CELLS]
    T *wsm = reinterpret_cast<T *>(Fs + (size_t)(nhalf + 2 * kPad) * CELLS);   // [warps][2][wrow_max]
    stage_spectrum<V2, CELLS>(smem16, fhat, tile, sub, nhalf, M, false);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cell = lane % CELLS, grp = lane / CELLS;
    T *wbuf0 = wsm + (size_t)warp * 2 * wrow_max;
    T *wbuf1 = wbuf0 + wrow_max;
    const int NW = WARPS * ip.split;                                 // task lists of the table
    int t = tasks[part * WARPS + warp], tend = tasks[part * WARPS + warp + 1];
    bool phase1 = false;
    const TaskRec *trec = reinterpret_cast<const TaskRec *>(tasks + 2 * NW + 1);
    const V2 *F0 = Fs + (size_t)(kPad + h) * CELLS + cell;          // (row 0, column 0) of this cell
    const bool valid = tile * 32 + sub * CELLS + cell < n;          // this lane's cell exists
    V2 *const qt = Qhat + tile * (int64_t)nhalf * 32 + sub * CELLS + cell;   // its (row 0, column -h)

    for (;;) {
        if (t >= tend) {
            // phase 1 (the same for the whole CTA: one table) after a restage;
            // the item's fields are read again from the parameters here rather
            // than kept in registers through the task loop
            if (phase1) break;
            const Mode32Item &iq = gd.item[it];
            const int *tq = iq.tasks;
            const int nw = WARPS * iq.split;
            if (tq[2 * nw] == tq[nw]) break;
            __syncthreads();                                         // every warp is done with the spectrum
            const int64_t c1 = (int64_t)blockIdx.x - gd.tile_start[it];
            const int64_t ct = c1 / iq.split;
            stage_spectrum<V2, CELLS>(smem16, static_cast<const V2 *>(iq.fhat), ct / G, (int)(ct % G), iq.nhalf,
                                      iq.M, true);
            __syncthreads();
            const int w1 = (int)(c1 % iq.split) * WARPS + (int)(threadIdx.x >> 5);
            t = tq[nw + w1];
            tend = tq[nw + w1 + 1];
            phase1 = true;
            continue;
        }
        const TaskRec tk = trec[t++];
        const int rowf = tk.rowf;                         // elements per row pair
        const bool ramp = RAMPS && (tk.flags & kTaskRamp) != 0;
        const T *wsrc = W + tk.woff;
        V2 hi[RR], lo[RR], acc[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r) hi[r] = lo[r] = acc[r] = cmk<V2>(0, 0);
        const int k20 = tk.k20 + grp * RR;                // this thread's first output column
        const int mbase0 = k20 - tk.l2lo - (RR - 1);
        stage_row(wbuf0, wsrc, rowf * (int)sizeof(T), lane);
        for (int i = 0; i < tk.nrows; ++i) {
            const T *wcur = (i & 1) ? wbuf1 : wbuf0;
            if (i + 1 < tk.nrows) {
                stage_row((i & 1) ? wbuf0 : wbuf1, wsrc + (size_t)(i + 1) * rowf, rowf * (int)sizeof(T), lane);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncwarp();
            // row header: element offsets of the rows of l and m, and the
            // direction of l (-1: f-hat_l = conj(f-hat_{-l}), row of -l read backwards)
            const int4 hd = *reinterpret_cast<const int4 *>(wcur);
            const int dir = hd.z > 0 ? 1 : -1;
            if constexpr (RTDIR)
                row_pass<T, RR, CELLS, RT, 0, RAMPS>(F0 + hd.x, F0 + hd.y, wcur + HEAD + grp * RR, tk.nblk * G,
                                                     tk.l2lo, mbase0, dir, ramp, acc);
            else if (dir > 0)
                row_pass<T, RR, CELLS, RT, 1, RAMPS>(F0 + hd.x, F0 + hd.y, wcur + HEAD + grp * RR, tk.nblk * G,
                                                     tk.l2lo, mbase0, dir, ramp, acc);
            else
                row_pass<T, RR, CELLS, RT, -1, RAMPS>(F0 + hd.x, F0 + hd.y, wcur + HEAD + grp * RR, tk.nblk * G,
                                                      tk.l2lo, mbase0, dir, ramp, acc);
            __syncwarp();
            // fold the row sums (<= 4 rows) into (hi, lo)
            if ((i & 3) == 3 || i + 1 == tk.nrows) {
#pragma unroll
                for (int r = 0; r < RR; ++r) {
                    T s, e;
                    two_sum(hi[r].x, acc[r].x, s, e);
                    hi[r].x = s;
                    lo[r].x += e;
                    two_sum(hi[r].y, acc[r].y, s, e);
                    hi[r].y = s;
                    lo[r].y += e;
                    acc[r] = cmk<V2>(0, 0);
                }
            }
        }
        if (valid) {
            // the record's output fields are read again here (volatile: not
            // kept in registers through the row loop)
            const volatile TaskRec *tv = trec + (t - 1);
            const int orow = tv->orow, rfirst = tv->rfirst, flags = tv->flags, crow = tv->crow;
            const int k2o = tv->k20 + grp * RR;
            V2 *out = qt + (int64_t)orow * M * 32;
            const bool refl = (flags & kTaskRefl) != 0, cj = (flags & kTaskConj) != 0;
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                const int k2 = k2o + r;
                if (grp * RR + r >= rfirst && k2 <= h) {
                    const V2 q = cmk<V2>(hi[r].x + lo[r].x, hi[r].y + lo[r].y);
                    out[(refl ? h - k2 : k2 + h) * 32] = q;
                    if (cj && k2 > 0) qt[((int64_t)crow * M + h - k2) * 32] = cmk<V2>(q.x, -q.y);
                }
            }
        }
    }
}

// ---- packed two-cell form ------------------------------------------------------
// The same sums with two cells per thread: lane p of a lane group holds cells
// p and p + 16 of the 32-cell tile, every spectrum entry in shared memory is
// one float4 (re_p, re_{p+16}, im_p, im_{p+16}), and every product and
// accumulation is one FP32x2 instruction (__fmul2_rn / __ffma2_rn: two
// independent IEEE FP32 operations, the same results as two scalar ones).
// Each weight is stored twice, (w, w), so it is an FP32x2 operand as loaded.
// Every lane performs exactly the operations of the scalar kernels, in the
// same order (tx = w a_re, ty = w a_im, re += tx b_re then += (-ty) b_im, im
// += tx b_im then += ty b_re, with the signs of a conjugated f-hat_l for
// l_1 < 0), so its results equal theirs bit for bit and the variants can
// share one batch (whole waves on one, the last wave on another).  The two
// lane groups of a warp split a task's 2 R outputs as in the 16-cell variant.
struct P2Acc {
    float2 re, im;
};

template <int RR, int PH, int DIR>
__device__ __forceinline__ void block_pass_p2(float4 (&win)[2 * RR], const float4 *__restrict__ mp,
                                              const float4 *__restrict__ lp, const float *__restrict__ wb,
                                              P2Acc (&acc)[RR]) {
    constexpr int CS = 16, RT = 2 * RR;
#pragma unroll
    for (int j = 0; j < RR; ++j) win[(j + PH * RR) & (2 * RR - 1)] = mp[j * CS];
#pragma unroll
    for (int s = 0; s < RR; ++s) {
        const float4 av = lp[s * DIR * CS];
        const float2 ar = make_float2(av.x, av.y);
        const float2 ai = make_float2(av.z, av.w), an = make_float2(-av.z, -av.w);
        float2 w2[RR];
#pragma unroll
        for (int q = 0; q < RR; q += 2) {
            const float4 w4 = *reinterpret_cast<const float4 *>(wb + s * 2 * RT + 2 * q);
            w2[q] = make_float2(w4.x, w4.y);
            w2[q + 1] = make_float2(w4.z, w4.w);
        }
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            const float4 bv = win[(r - s + RR - 1 + PH * RR) & (2 * RR - 1)];
            const float2 br = make_float2(bv.x, bv.y), bi = make_float2(bv.z, bv.w);
            const float2 tx = __fmul2_rn(w2[r], ar);
            const float2 ty = __fmul2_rn(w2[r], ai), tn = __fmul2_rn(w2[r], an);   // w a_im, -(w a_im)
            acc[r].re = __ffma2_rn(tx, br, acc[r].re);
            acc[r].re = __ffma2_rn(DIR > 0 ? tn : ty, bi, acc[r].re);
            acc[r].im = __ffma2_rn(tx, bi, acc[r].im);
            acc[r].im = __ffma2_rn(DIR > 0 ? ty : tn, br, acc[r].im);
        }
    }
}

template <int RR, int DIR>
__device__ __forceinline__ void row_pass_p2(const float4 *__restrict__ rowl, const float4 *__restrict__ rowm,
                                            const float *__restrict__ wrow, int nblk, int l2lo, int mbase0,
                                            P2Acc (&acc)[RR]) {
    constexpr int CS = 16, RT = 2 * RR;
    float4 win[2 * RR];
    const float4 *mp = rowm + mbase0 * CS;
    const float4 *lp = rowl + DIR * l2lo * CS;
#pragma unroll
    for (int j = RR; j < 2 * RR - 1; ++j) win[j] = mp[j * CS];
    int blk = 0;
    for (; blk + 1 < nblk; blk += 2) {
        block_pass_p2<RR, 0, DIR>(win, mp, lp, wrow + blk * RR * 2 * RT, acc);
        block_pass_p2<RR, 1, DIR>(win, mp - RR * CS, lp + RR * DIR * CS, wrow + (blk + 1) * RR * 2 * RT, acc);
        mp -= 2 * RR * CS;
        lp += 2 * RR * DIR * CS;
    }
    if (blk < nblk) block_pass_p2<RR, 0, DIR>(win, mp, lp, wrow + blk * RR * 2 * RT, acc);
}

// TwoSum on both lanes of an FP32x2 pair (each lane exact as the scalar form).
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
    s = __fadd2_rn(a, b);
    const float2 bb = __fadd2_rn(s, make_float2(-a.x, -a.y));
    const float2 t = __fadd2_rn(s, make_float2(-bb.x, -bb.y));
    e = __fadd2_rn(__fadd2_rn(a, make_float2(-t.x, -t.y)), __fadd2_rn(b, make_float2(-bb.x, -bb.y)));
}

template <int RR, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) modesum_p2_kernel(const Mode32Group gd) {
    constexpr int G = 2, CS = 16;
    constexpr int HEADF = kRowHeadBytes / (int)sizeof(float);
    extern __shared__ __align__(16) uint4 smem16[];
    int it = 0;
    while (it + 1 < gd.nitems && (int64_t)blockIdx.x >= gd.tile_start[it + 1]) ++it;
    const Mode32Item &ip = gd.item[it];
    const float2 *__restrict__ fhat = static_cast<const float2 *>(ip.fhat);
    float2 *__restrict__ Qhat = static_cast<float2 *>(ip.Qhat);
    const float *__restrict__ W = static_cast<const float *>(ip.W);
    const int *__restrict__ tasks = ip.tasks;
    const int h = ip.h, M = ip.M, nhalf = ip.nhalf, wrow_max = ip.wrow_max;
    const int64_t n = ip.n;
    const int64_t cta0 = (int64_t)blockIdx.x - gd.tile_start[it];
    const int part = (int)(cta0 % ip.split);
    const int64_t tile = cta0 / ip.split;
    float4 *Fs = reinterpret_cast<float4 *>(smem16);                        // [kPad + nhalf + kPad][16]
    float *wsm = reinterpret_cast<float *>(Fs + (size_t)(nhalf + 2 * kPad) * CS);   // [warps][2][wrow_max]
    {
        // the tile's half spectrum as cell pairs (c, c + 16); zero guard rows
        const float2 *src = fhat + tile * (int64_t)nhalf * 32;
        const int rows = nhalf + 2 * kPad;
        for (int i = threadIdx.x; i < rows * CS; i += blockDim.x) {
            const int row = i / CS - kPad, pr = i % CS;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row >= 0 && row < nhalf) {
                const float2 x = src[(int64_t)row * 32 + pr], y = src[(int64_t)row * 32 + pr + 16];
                v = make_float4(x.x, y.x, x.y, y.y);
            }
            Fs[i] = v;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int pr = lane % CS, grp = lane / CS;
    float *wbuf0 = wsm + (size_t)warp * 2 * wrow_max;
    float *wbuf1 = wbuf0 + wrow_max;
    const int vw = part * WARPS + warp;
    const int tbeg = tasks[vw], tend = tasks[vw + 1];
    const TaskRec *trec = reinterpret_cast<const TaskRec *>(tasks + 2 * WARPS * ip.split + 1);
    const float4 *F0 = Fs + (size_t)(kPad + h) * CS + pr;

    for (int t = tbeg; t < tend; ++t) {
        const TaskRec tk = trec[t];
        const int rowf = tk.rowf;
        const float *wsrc = W + tk.woff;
        float2 hre[RR], lre[RR], him[RR], lim[RR];
        P2Acc acc[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            hre[r] = lre[r] = him[r] = lim[r] = make_float2(0.f, 0.f);
            acc[r].re = acc[r].im = make_float2(0.f, 0.f);
        }
        const int k20 = tk.k20 + grp * RR;
        const int mbase0 = k20 - tk.l2lo - (RR - 1);
        stage_row(wbuf0, wsrc, rowf * (int)sizeof(float), lane);
        for (int i = 0; i < tk.nrows; ++i) {
            const float *wcur = (i & 1) ? wbuf1 : wbuf0;
            if (i + 1 < tk.nrows) {
                stage_row((i & 1) ? wbuf0 : wbuf1, wsrc + (size_t)(i + 1) * rowf, rowf * (int)sizeof(float), lane);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncwarp();
            const int4 hd = *reinterpret_cast<const int4 *>(wcur);
            if (hd.z > 0)
                row_pass_p2<RR, 1>(F0 + hd.x, F0 + hd.y, wcur + HEADF + 2 * grp * RR, tk.nblk * G, tk.l2lo, mbase0,
                                   acc);
            else
                row_pass_p2<RR, -1>(F0 + hd.x, F0 + hd.y, wcur + HEADF + 2 * grp * RR, tk.nblk * G, tk.l2lo, mbase0,
                                    acc);
            __syncwarp();
            if ((i & 3) == 3 || i + 1 == tk.nrows) {
#pragma unroll
                for (int r = 0; r < RR; ++r) {
                    float2 sm, e;
                    two_sum2(hre[r], acc[r].re, sm, e);
                    hre[r] = sm;
                    lre[r] = __fadd2_rn(lre[r], e);
                    two_sum2(him[r], acc[r].im, sm, e);
                    him[r] = sm;
                    lim[r] = __fadd2_rn(lim[r], e);
                    acc[r].re = acc[r].im = make_float2(0.f, 0.f);
                }
            }
        }
        const int64_t c0 = tile * 32 + pr, c1 = c0 + 16;
        float2 *out = Qhat + tile * (int64_t)nhalf * 32 + (int64_t)tk.orow * M * 32 + pr;
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            const int k2 = k20 + r;
            if (grp * RR + r >= tk.rfirst && k2 <= h) {
                const float2 re = __fadd2_rn(hre[r], lre[r]), im = __fadd2_rn(him[r], lim[r]);
                if (c0 < n) out[(k2 + h) * 32] = make_float2(re.x, im.x);
                if (c1 < n) out[(k2 + h) * 32 + 16] = make_float2(re.y, im.y);
            }
        }
    }
}

// ---- FP32x2 form with one cell per lane ----------------------------------------
// The sums of modesum32_kernel (tiles of 32 cells, one cell per lane, RR
// outputs per thread, reflected and ramped task tables) with the complex
// product w f-hat_l b (b = f-hat_m from the window) split as
//   U = w b                 (one FP32x2 multiply: (w b_x, w b_y)),
//   P += U f_x, Q += U f_y  (two FP32x2 FMAs; f = f-hat_l, f_y negated for a
//                            conjugated value),
// so that Re = P_x - Q_y and Im = P_y + Q_x.  Three FP32x2 instructions per
// pair in place of six scalar ones, the same six FP32 operations: the kernel
// is bounded by the FMA pipe rather than by instruction issue.  The weights
// are read as in the scalar kernels (16 bytes = four outputs' weights; a
// broadcast 16-byte shared-memory load takes two wavefronts, so a stream of
// (w, w) pairs would make shared memory the bound).  P and Q are folded into the (hi, lo) pair of each output every
// four rows as (P_x - Q_y, P_y + Q_x); the sums differ in rounding from the
// scalar kernels', so the last partial wave of a batch stays on this kernel.
template <int RR, int WS, int PH, bool RAMP, int DIR>
__device__ __forceinline__ void block_pq(float2 (&win)[2 * RR], const float2 *__restrict__ mp, int mcs,
                                         const float2 *__restrict__ lp, int dcs,
                                         const float *__restrict__ wb, float2 (&P)[RR], float2 (&Q)[RR]) {
#pragma unroll
    for (int j = 0; j < (RAMP ? RR - 1 : RR); ++j) win[(j + PH * RR) & (2 * RR - 1)] = mp[j * mcs];
#pragma unroll
    for (int s = RAMP ? 1 : 0; s < RR; ++s) {
        const float2 fl = lp[s * dcs];
        const float fy = DIR > 0 ? fl.y : -fl.y;       // f-hat_l conjugated for DIR < 0
        const float2 fxx = make_float2(fl.x, fl.x), fyy = make_float2(fy, fy);
        // all products U first, then the P and then the Q updates: no FMA
        // waits on the multiply issued just before it
        float wv[RR];
        if constexpr (RR == 2) {
            const float2 w2 = *reinterpret_cast<const float2 *>(wb + s * WS);
            wv[0] = w2.x;
            wv[1] = w2.y;
        } else {
#pragma unroll
            for (int q = 0; q < RR; q += 4)
                if (!RAMP || q < s) load_w4(wv + q, wb + s * WS + q);   // outputs q .. q + 3 before the ramp
        }
        float2 u[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r)
            if (!RAMP || r < s) u[r] = __fmul2_rn(make_float2(wv[r], wv[r]), win[(r - s + RR - 1 + PH * RR) & (2 * RR - 1)]);
#pragma unroll
        for (int r = 0; r < RR; ++r)
            if (!RAMP || r < s) P[r] = __ffma2_rn(u[r], fxx, P[r]);
#pragma unroll
        for (int r = 0; r < RR; ++r)
            if (!RAMP || r < s) Q[r] = __ffma2_rn(u[r], fyy, Q[r]);
    }
}

// One row pair (as row_pass): the ramp block under the PH 1 naming, or the
// preload, then pairs of blocks (PH 0, PH 1) and a last PH 0.  mirror: the
// task of a reflected output block, read from the unreflected spectrum: every
// column index is negated, so f-hat_l and the window run the other way.
template <int RR, int WS, int CS, int DIR>
__device__ __forceinline__ void row_pass_pq(const float2 *__restrict__ rowl, const float2 *__restrict__ rowm,
                                            const float *__restrict__ wrow, int nblk, int l2lo, int mbase0,
                                            bool ramp, bool mirror, float2 (&P)[RR], float2 (&Q)[RR]) {
    float2 win[2 * RR];
    const int dcs = (mirror ? -DIR : DIR) * CS;          // between consecutive l_2
    const int mcs = mirror ? -CS : CS;                   // between consecutive window columns
    const float2 *mp = rowm + mbase0 * mcs;
    const float2 *lp = rowl + l2lo * dcs;
    int blk = 0;
    if (ramp) {
        block_pq<RR, WS, 1, true, DIR>(win, mp, mcs, lp, dcs, wrow, P, Q);
        mp -= RR * mcs;
        lp += RR * dcs;
        blk = 1;
    } else {
#pragma unroll
        for (int j = RR; j < 2 * RR - 1; ++j) win[j] = mp[j * mcs];
    }
    for (; blk + 1 < nblk; blk += 2) {
        block_pq<RR, WS, 0, false, DIR>(win, mp, mcs, lp, dcs, wrow + blk * RR * WS, P, Q);
        block_pq<RR, WS, 1, false, DIR>(win, mp - RR * mcs, mcs, lp + RR * dcs, dcs, wrow + (blk + 1) * RR * WS, P,
                                        Q);
        mp -= 2 * RR * mcs;
        lp += 2 * RR * dcs;
    }
    if (blk < nblk) block_pq<RR, WS, 0, false, DIR>(win, mp, mcs, lp, dcs, wrow + blk * RR * WS, P, Q);
}

// CELLS = 32: one cell per lane; reflected blocks are separate tasks (read
// mirrored).  CELLS = 16 (paired orientations, for grids whose 32-cell
// spectrum does not fit shared memory): lanes c and c + 16 hold cell c, the
// upper half running every task mirrored, i.e. the task's reflected twin with
// the same weights and control flow, so all lanes take the same outputs and
// the ramp applies; the table holds no reflected tasks and k_2 = 0 is the
// lower half's.  CELLS = 8 (grids whose 16-cell spectrum does not fit: 64^2,
// 16^3): the two halves of a warp each do the same for 8 cells, one on the
// even and one on the odd of a task's row pairs (ROWS = 2; the table lists
// them in couples of one read direction), and their sums are added at the end
// of the task.  Consecutive rows lie an odd number of modes apart, so the four
// 64-byte groups of a load fall two and two into the halves of the banks.
template <int RR, int WARPS, int CELLS>
__global__ void __launch_bounds__(WARPS * 32, RR == 2 ? 2 : WARPS <= 4 ? 3 : WARPS <= 8 ? 2 : 1) modesum_pq_kernel(const Mode32Group gd) {
    constexpr bool PAIRED = (CELLS <= 16);
    constexpr int ROWS = PAIRED ? 16 / CELLS : 1;   // row pairs at a time
    constexpr int G = 32 / CELLS;                // CTAs per 32-cell tile
    constexpr int WS = RR;                       // floats per l_2 step
    constexpr int HEAD = kRowHeadBytes / (int)sizeof(float);
    extern __shared__ __align__(16) uint4 smem16[];
    int it = 0;
    while (it + 1 < gd.nitems && (int64_t)blockIdx.x >= gd.tile_start[it + 1]) ++it;
    const Mode32Item &ip = gd.item[it];
    const float2 *fhat = static_cast<const float2 *>(ip.fhat);
    float2 *__restrict__ Qhat = static_cast<float2 *>(ip.Qhat);
    const float *__restrict__ W = static_cast<const float *>(ip.W);
    const int *__restrict__ tasks = ip.tasks;
    const int h = ip.h, M = ip.M, nhalf = ip.nhalf, wrow_max = ip.wrow_max;
    const int64_t cta0 = (int64_t)blockIdx.x - gd.tile_start[it];
    const int part = (int)(cta0 % ip.split);
    const int64_t cta = cta0 / ip.split;
    const int64_t tile = cta / G;
    const int sub = (int)(cta % G);
    float2 *Fs = reinterpret_cast<float2 *>(smem16);                 // [kPad + nhalf + kPad][CELLS]
    float *wsm = reinterpret_cast<float *>(Fs + (size_t)(nhalf + 2 * kPad) * CELLS);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cell = lane % CELLS;
    const bool upper = PAIRED && (lane / CELLS) % 2 == 1;            // runs every task mirrored
    const int rgrp = ROWS > 1 ? lane / (2 * CELLS) : 0;              // its row pair of each couple
    float *wbuf0 = wsm + (size_t)warp * 2 * ROWS * wrow_max;
    float *wbuf1 = wbuf0 + ROWS * wrow_max;
    const int NW = WARPS * ip.split;                 // one phase: every task reads this spectrum
    int t = tasks[part * WARPS + warp], tend = tasks[part * WARPS + warp + 1];
    const TaskRec *trec = reinterpret_cast<const TaskRec *>(tasks + 2 * NW + 1);
    bool staged = false;
    if constexpr (RR == 2) {
        // small launches: the first task's first weights travel while the
        // kernel before this one ends and the spectrum is staged
        griddep_launch();
        staged = t < tend;
        if (staged) stage_row(wbuf0, W + trec[t].woff, ROWS * trec[t].rowf * (int)sizeof(float), lane);
        griddep_wait();
    }
    stage_spectrum<float2, CELLS, RR == 2>(smem16, fhat, tile, sub, nhalf, M, false);
    __syncthreads();
    const float2 *F0 = Fs + (size_t)(kPad + h) * CELLS + cell;
    const bool valid = tile * 32 + sub * CELLS + cell < ip.n;
    float2 *const qt = Qhat + tile * (int64_t)nhalf * 32 + sub * CELLS + cell;

    for (; t < tend;) {
        const TaskRec tk = trec[t++];
        const int rowf = tk.rowf;
        const bool ramp = (tk.flags & kTaskRamp) != 0, mirror = ((tk.flags & kTaskRefl) != 0) != upper;
        const float *wsrc = W + tk.woff;
        float2 hi[RR], lo[RR], P[RR], Q[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r) hi[r] = lo[r] = P[r] = Q[r] = make_float2(0.f, 0.f);
        const int mbase0 = tk.k20 - tk.l2lo - (RR - 1);
        const int nrows = tk.nrows / ROWS, rowb = ROWS * rowf * (int)sizeof(float);
        if (!staged) stage_row(wbuf0, wsrc, rowb, lane);
        staged = false;
        for (int i = 0; i < nrows; ++i) {
            const float *wcur = ((i & 1) ? wbuf1 : wbuf0) + rgrp * rowf;
            if (i + 1 < nrows) {
                stage_row((i & 1) ? wbuf0 : wbuf1, wsrc + (size_t)(i + 1) * (ROWS * rowf), rowb, lane);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncwarp();
            const int4 hd = *reinterpret_cast<const int4 *>(wcur);
            if (hd.z > 0)
                row_pass_pq<RR, WS, CELLS, 1>(F0 + hd.x, F0 + hd.y, wcur + HEAD, tk.nblk, tk.l2lo, mbase0, ramp,
                                              mirror, P, Q);
            else
                row_pass_pq<RR, WS, CELLS, -1>(F0 + hd.x, F0 + hd.y, wcur + HEAD, tk.nblk, tk.l2lo, mbase0, ramp,
                                               mirror, P, Q);
            __syncwarp();
            if ((i & 3) == 3 || i + 1 == nrows) {
#pragma unroll
                for (int r = 0; r < RR; ++r) {
                    // (re, im) TwoSum as FP32x2 operations: the scalar ones, pairwise
                    const float2 a = make_float2(P[r].x - Q[r].y, P[r].y + Q[r].x);
                    float2 sm, e;
                    two_sum2(hi[r], a, sm, e);
                    hi[r] = sm;
                    lo[r] = __fadd2_rn(lo[r], e);
                    P[r] = Q[r] = make_float2(0.f, 0.f);
                }
            }
        }
        if constexpr (ROWS > 1) {
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                const float2 h2 = make_float2(__shfl_xor_sync(0xffffffffu, hi[r].x, 16),
                                              __shfl_xor_sync(0xffffffffu, hi[r].y, 16));
                const float2 l2 = make_float2(__shfl_xor_sync(0xffffffffu, lo[r].x, 16),
                                              __shfl_xor_sync(0xffffffffu, lo[r].y, 16));
                float2 sm, e;
                two_sum2(hi[r], h2, sm, e);
                hi[r] = sm;
                lo[r] = __fadd2_rn(__fadd2_rn(lo[r], l2), e);
            }
        }
        if (valid && rgrp == 0) {
            const volatile TaskRec *tv = trec + (t - 1);
            const int orow = tv->orow, rfirst = tv->rfirst, flags = tv->flags, crow = tv->crow, k20 = tv->k20;
            float2 *out = qt + (int64_t)orow * M * 32;
            const bool refl = ((flags & kTaskRefl) != 0) != upper, cj = (flags & kTaskConj) != 0;
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                const int k2 = k20 + r;
                if (r >= rfirst && k2 <= h && !(upper && k2 == 0)) {
                    const float2 q = make_float2(hi[r].x + lo[r].x, hi[r].y + lo[r].y);
                    out[(refl ? h - k2 : k2 + h) * 32] = q;
                    if (cj && k2 > 0) qt[((int64_t)crow * M + h - k2) * 32] = make_float2(q.x, -q.y);
                }
            }
        }
    }
}

// ---- FP64 and FP32X2 forms -----------------------------------------------------
// Both run the paired orientations of modesum_pq_kernel on tiles of CELLS = 8 or
// 4 cells: a warp holds ROWS = 16 / CELLS groups of lanes, each group its
// CELLS cells plain and mirrored on its own row pair of the task.  Their blocks
// of RR <= 4 outputs divide the half row of 16, 32 and 48 points, so the ramped
// tables leave no padding (the earlier tables for blocks of 8 over the whole
// row summed 1.24 pairs per useful one at 32^2, these 1.04), and two CTAs share
// an SM at 32^2, so that the end of one tile overlaps the other.  4099 cells of
// 32^2 in FP64: 8.76 -> 7.25 ms.
//
// One block of RR l_2 steps and one row pair, as block_pq and row_pass_pq; Term
// supplies the value type (what a spectrum entry is) and the product sums.
template <typename Term, int RR, int PH, bool RAMP>
__device__ __forceinline__ void block_pair(typename Term::Val (&win)[2 * RR], const typename Term::Src mp, int mcs,
                                           const typename Term::Src lp, int dcs, int dir,
                                           const typename Term::W *__restrict__ wb, typename Term::Acc (&acc)[RR]) {
#pragma unroll
    for (int j = 0; j < (RAMP ? RR - 1 : RR); ++j) win[(j + PH * RR) & (2 * RR - 1)] = Term::load(mp, j * mcs);
#pragma unroll
    for (int s = RAMP ? 1 : 0; s < RR; ++s) {
        const typename Term::Val fl = Term::conj(Term::load(lp, s * dcs), dir);
        typename Term::Wt wv[RR];
        Term::template weights<RR>(wv, wb + s * RR * Term::kWPer);
#pragma unroll
        for (int r = 0; r < RR; ++r)
            if (!RAMP || r < s) Term::add(acc[r], wv[r], fl, win[(r - s + RR - 1 + PH * RR) & (2 * RR - 1)]);
    }
}

template <typename Term, int RR, int CS>
__device__ __forceinline__ void row_pass_pair(typename Term::Src rowl, typename Term::Src rowm,
                                              const typename Term::W *__restrict__ wrow, int nblk, int l2lo, int mbase0,
                                              int dir, bool ramp, bool mirror, typename Term::Acc (&acc)[RR]) {
    typename Term::Val win[2 * RR];
    constexpr int WB = RR * RR * Term::kWPer;            // weights of a block
    const int dcs = (mirror ? -dir : dir) * CS;          // between consecutive l_2
    const int mcs = mirror ? -CS : CS;                   // between consecutive window columns
    typename Term::Src mp = Term::at(rowm, mbase0 * mcs), lp = Term::at(rowl, l2lo * dcs);
    int blk = 0;
    if (ramp) {
        block_pair<Term, RR, 1, true>(win, mp, mcs, lp, dcs, dir, wrow, acc);
        mp = Term::at(mp, -RR * mcs);
        lp = Term::at(lp, RR * dcs);
        blk = 1;
    } else {
#pragma unroll
        for (int j = RR; j < 2 * RR - 1; ++j) win[j] = Term::load(mp, j * mcs);
    }
    for (; blk + 1 < nblk; blk += 2) {
        block_pair<Term, RR, 0, false>(win, mp, mcs, lp, dcs, dir, wrow + blk * WB, acc);
        block_pair<Term, RR, 1, false>(win, Term::at(mp, -RR * mcs), mcs, Term::at(lp, RR * dcs), dcs, dir,
                                       wrow + (blk + 1) * WB, acc);
        mp = Term::at(mp, -2 * RR * mcs);
        lp = Term::at(lp, 2 * RR * dcs);
    }
    if (blk < nblk) block_pair<Term, RR, 0, false>(win, mp, mcs, lp, dcs, dir, wrow + blk * WB, acc);
}

// FP64: six operations of the FP64 pipe per pair, which bounds the kernel.
struct Term64 {
    using Val = double2;
    using Src = const double2 *;
    using W = double;
    using Wt = double;
    using Acc = double2;
    static constexpr int kWPer = 1;
    static __device__ __forceinline__ Src at(Src p, int off) { return p + off; }
    static __device__ __forceinline__ Val load(Src p, int off) { return p[off]; }
    static __device__ __forceinline__ Val conj(Val v, int dir) {
        return make_double2(v.x, dir > 0 ? v.y : -v.y);
    }
    template <int RR> static __device__ __forceinline__ void weights(Wt (&w)[RR], const W *__restrict__ p) {
#pragma unroll
        for (int q = 0; q < RR; q += 2) {
            const double2 x = *reinterpret_cast<const double2 *>(p + q);
            w[q] = x.x;
            w[q + 1] = x.y;
        }
    }
    static __device__ __forceinline__ void add(Acc &a, Wt w, const Val &f, const Val &b) {
        const double tx = w * f.x, ty = w * f.y;
        a.x = fma(tx, b.x, a.x);
        a.x = fma(-ty, b.y, a.x);
        a.y = fma(tx, b.y, a.y);
        a.y = fma(ty, b.x, a.y);
    }
};

// FP32X2: double-float arithmetic on the FP32 pipe.  Every value is an
// unevaluated sum hi + lo of two FP32 numbers (|lo| <= u |hi|).  For each term
// w f-hat_l f-hat_m of eq. CF1 the product X = w f-hat_l is formed exactly in
// its high part (TwoProd: fma(a, b, -fl(a b)) is the exact rounding error of
// a b) with the low parts of w and f-hat_l added to its error; each of the four
// real products X b of the complex product is split exactly the same way, its
// high part enters the running sum with its exact error, and every error and
// the cross terms with the low part of b accumulate in a second FP32 sum.  This
// is the compensated dot product ("Dot2") of Ogita, Rump and Oishi (2005),
// accurate as if computed in twice the working precision; the real and
// imaginary parts are the two lanes, and the _rn intrinsics pin the operations.
// The FMA pipe bounds the kernel (70 % busy): 28 FP32x2 operations per pair.
// 4096 cells of 32^2: 1.53 -> 1.22 ms by the tables and the split of the last tiles.
// Not kept: Dekker's three-operation sums on operands ordered by selects (22
// operations, the same numbers) moved the bound to the ALU pipe, 1.55 ms; a
// running sum biased so that it always exceeds the product needs 16 operations
// and took 0.94 ms, but its errors are relative to the bias, 100 times those of
// Dot2 on cells near equilibrium.
struct X2Val {
    float2 h, l;
};
struct X2Src {
    const float2 *p;
    int LO;                                  // from a value's high part to its low part
};
struct X2Wt {
    float h, l;
};
struct X2Acc {
    float2 s, c;
};
struct TermX2 {
    using Val = X2Val;
    using Src = X2Src;
    using W = float;
    using Wt = X2Wt;
    using Acc = X2Acc;
    static constexpr int kWPer = 2;          // a step's high parts, then its low parts
    static __device__ __forceinline__ Src at(Src s, int off) { return Src{s.p + off, s.LO}; }
    static __device__ __forceinline__ Val load(Src s, int off) { return Val{s.p[off], s.p[off + s.LO]}; }
    static __device__ __forceinline__ Val conj(Val v, int dir) {
        if (dir < 0) {
            v.h.y = -v.h.y;
            v.l.y = -v.l.y;
        }
        return v;
    }
    template <int RR> static __device__ __forceinline__ void weights(Wt (&w)[RR], const W *__restrict__ p) {
        if constexpr (RR == 4) {
            const float4 h = *reinterpret_cast<const float4 *>(p), l = *reinterpret_cast<const float4 *>(p + 4);
            w[0] = Wt{h.x, l.x};
            w[1] = Wt{h.y, l.y};
            w[2] = Wt{h.z, l.z};
            w[3] = Wt{h.w, l.w};
        } else {
            static_assert(RR == 2, "2 or 4 outputs per thread");
            const float4 q = *reinterpret_cast<const float4 *>(p);
            w[0] = Wt{q.x, q.z};
            w[1] = Wt{q.y, q.w};
        }
    }
    static __device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
    static __device__ __forceinline__ void add(Acc &a, const Wt &w, const Val &f, const Val &b) {
        const float2 W2 = make_float2(w.h, w.h);
        const float2 X = __fmul2_rn(W2, f.h);
        float2 E = __ffma2_rn(W2, f.h, neg(X));
        E = __ffma2_rn(make_float2(w.l, w.l), f.h, E);
        E = __ffma2_rn(W2, f.l, E);
        // X b = X_x (b_x, b_y) + (-X_y, X_y) (b_y, b_x)
        const float2 bs = make_float2(b.h.y, b.h.x), ls = make_float2(b.l.y, b.l.x);
        const float2 XX = make_float2(X.x, X.x), YN = make_float2(-X.y, X.y);
        const float2 P = __fmul2_rn(XX, b.h);
        float2 d;
        sum_exact(a.s, P, d);
        float2 c = __fadd2_rn(__ffma2_rn(XX, b.h, neg(P)), d);
        const float2 Q = __fmul2_rn(YN, bs);
        sum_exact(a.s, Q, d);
        c = __fadd2_rn(c, __fadd2_rn(__ffma2_rn(YN, bs, neg(Q)), d));
        c = __fadd2_rn(a.c, c);
        c = __ffma2_rn(make_float2(E.x, E.x), b.h, c);
        c = __ffma2_rn(make_float2(-E.y, E.y), bs, c);
        c = __ffma2_rn(XX, b.l, c);
        a.c = __ffma2_rn(YN, ls, c);
    }
    // s <- fl(s + p), d the exact error (TwoSum)
    static __device__ __forceinline__ void sum_exact(float2 &s, float2 p, float2 &d) {
        float2 sm;
        two_sum2(s, p, sm, d);
        s = sm;
    }
};

// The task loop of both forms.  FP64: sums along a row pair fold into (hi, lo)
// by TwoSum every four.  FP32X2: the FP64 spectrum is split into FP32 high and
// low parts as it is staged; its output is rounded to FP32.  A tile may be
// shared by `split` CTAs.
template <bool X2, int RR, int WARPS, int CELLS>
__global__ void __launch_bounds__(WARPS * 32, CELLS == 8 ? 2 : 1) modesum_pair_kernel(const Mode32Group gd) {
    constexpr int G = 32 / CELLS;                // CTAs per 32-cell tile
    constexpr int ROWS = 16 / CELLS;             // row pairs at a time
    constexpr int SLOT = X2 ? 2 : 1;             // floats or doubles per 8-byte slot of the weight stream
    using W = typename std::conditional<X2, float, double>::type;
    using OutV = typename std::conditional<X2, float2, double2>::type;
    extern __shared__ __align__(16) uint4 smem16[];
    int it = 0;
    while (it + 1 < gd.nitems && (int64_t)blockIdx.x >= gd.tile_start[it + 1]) ++it;
    const Mode32Item &ip = gd.item[it];
    const double2 *__restrict__ fhat = static_cast<const double2 *>(ip.fhat);
    const W *__restrict__ Wst = static_cast<const W *>(ip.W);
    const int *__restrict__ tasks = ip.tasks;
    const int h = ip.h, M = ip.M, nhalf = ip.nhalf, wrow_max = ip.wrow_max;
    const int64_t cta0 = (int64_t)blockIdx.x - gd.tile_start[it];
    const int part = (int)(cta0 % ip.split);
    const int64_t cta = cta0 / ip.split;
    const int64_t tile = cta / G;
    const int sub = (int)(cta % G);
    const int rows = nhalf + 2 * kPad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cell = lane % CELLS;
    double2 *Fs = reinterpret_cast<double2 *>(smem16);               // [rows][CELLS]; X2: float2 high, then low parts
    float2 *Fh = reinterpret_cast<float2 *>(smem16);
    W *wsm = reinterpret_cast<W *>(Fs + (size_t)rows * CELLS);       // [warps][2][ROWS wrow_max slots]
    if constexpr (X2) {
        const double2 *src = fhat + tile * (int64_t)nhalf * 32 + sub * CELLS;
        float2 *Fl = Fh + (size_t)rows * CELLS;
        for (int i = threadIdx.x; i < rows * CELLS; i += WARPS * 32) {
            const int row = i / CELLS - kPad, c = i % CELLS;
            float2 hv = make_float2(0.f, 0.f), lv = make_float2(0.f, 0.f);
            if (row >= 0 && row < nhalf) {
                const double2 x = src[(int64_t)row * 32 + c];
                hv.x = __double2float_rn(x.x);
                hv.y = __double2float_rn(x.y);
                lv.x = __double2float_rn(x.x - (double)hv.x);
                lv.y = __double2float_rn(x.y - (double)hv.y);
            }
            Fh[i] = hv;
            Fl[i] = lv;
        }
        __syncthreads();
    } else {
        stage_spectrum<double2, CELLS>(smem16, fhat, tile, sub, nhalf, M, false);
        __syncthreads();
    }
    const bool upper = (lane / CELLS) % 2 == 1;                      // runs every task mirrored
    const int rgrp = lane / (2 * CELLS);                             // its row pair of each ROWS
    W *wbuf0 = wsm + (size_t)warp * 2 * ROWS * wrow_max * SLOT;
    W *wbuf1 = wbuf0 + (size_t)ROWS * wrow_max * SLOT;
    const int NW = WARPS * ip.split;
    int t = tasks[part * WARPS + warp];
    const int tend = tasks[part * WARPS + warp + 1];
    const TaskRec *trec = reinterpret_cast<const TaskRec *>(tasks + 2 * NW + 1);
    const size_t f0 = (size_t)(kPad + h) * CELLS + cell;
    const bool valid = tile * 32 + sub * CELLS + cell < ip.n && rgrp == 0;
    OutV *const qt = static_cast<OutV *>(ip.Qhat) + tile * (int64_t)nhalf * 32 + sub * CELLS + cell;

    for (; t < tend;) {
        const TaskRec tk = trec[t++];
        const int rowb = ROWS * tk.rowf * 8;                         // bytes staged per step
        const bool ramp = (tk.flags & kTaskRamp) != 0;
        const W *wsrc = Wst + (size_t)tk.woff * SLOT;
        const int mbase0 = tk.k20 - tk.l2lo - (RR - 1);
        const int nrows = tk.nrows / ROWS;
        typename std::conditional<X2, X2Acc, double2>::type acc[RR];
        OutV hi[RR], lo[RR];
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            hi[r] = lo[r] = cmk<OutV>(0, 0);
            if constexpr (X2) acc[r] = X2Acc{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            else acc[r] = make_double2(0.0, 0.0);
        }
        stage_row(wbuf0, wsrc, rowb, lane);
        for (int i = 0; i < nrows; ++i) {
            const W *wcur = ((i & 1) ? wbuf1 : wbuf0) + (size_t)rgrp * tk.rowf * SLOT;
            if (i + 1 < nrows) {
                stage_row((i & 1) ? wbuf0 : wbuf1, wsrc + (size_t)(i + 1) * ROWS * tk.rowf * SLOT, rowb, lane);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncwarp();
            const int4 hd = *reinterpret_cast<const int4 *>(wcur);
            constexpr int HEAD = kRowHeadBytes / (int)sizeof(W);
            if constexpr (X2) {
                row_pass_pair<TermX2, RR, CELLS>(X2Src{Fh + f0 + hd.x, rows * CELLS}, X2Src{Fh + f0 + hd.y, rows * CELLS},
                                                 wcur + HEAD, tk.nblk, tk.l2lo, mbase0, hd.z, ramp, upper, acc);
            } else {
                row_pass_pair<Term64, RR, CELLS>(Fs + f0 + hd.x, Fs + f0 + hd.y, wcur + HEAD, tk.nblk, tk.l2lo, mbase0,
                                                 hd.z, ramp, upper, acc);
                if ((i & 3) == 3 || i + 1 == nrows) {
#pragma unroll
                    for (int r = 0; r < RR; ++r) {
                        double sm, e;
                        two_sum(hi[r].x, acc[r].x, sm, e);
                        hi[r].x = sm;
                        lo[r].x += e;
                        two_sum(hi[r].y, acc[r].y, sm, e);
                        hi[r].y = sm;
                        lo[r].y += e;
                        acc[r] = make_double2(0.0, 0.0);
                    }
                }
            }
            __syncwarp();
        }
        // the row groups' sums
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            if constexpr (X2) hi[r] = acc[r].s, lo[r] = acc[r].c;
#pragma unroll
            for (int o = 2 * CELLS; o < 32; o <<= 1) {
                OutV h2, l2;
                h2.x = __shfl_xor_sync(0xffffffffu, hi[r].x, o);
                h2.y = __shfl_xor_sync(0xffffffffu, hi[r].y, o);
                l2.x = __shfl_xor_sync(0xffffffffu, lo[r].x, o);
                l2.y = __shfl_xor_sync(0xffffffffu, lo[r].y, o);
                decltype(h2.x) sm, e;
                two_sum(hi[r].x, h2.x, sm, e);
                hi[r].x = sm;
                lo[r].x = (lo[r].x + l2.x) + e;
                two_sum(hi[r].y, h2.y, sm, e);
                hi[r].y = sm;
                lo[r].y = (lo[r].y + l2.y) + e;
            }
        }
        if (valid) {
            OutV *out = qt + (int64_t)tk.orow * M * 32;
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                const int k2 = tk.k20 + r;
                if (k2 <= h && !(upper && k2 == 0))
                    out[(upper ? h - k2 : k2 + h) * 32] = cmk<OutV>(hi[r].x + lo[r].x, hi[r].y + lo[r].y);
            }
        }
    }
}

// Moves a task of the most loaded warp to another, or swaps it for a shorter
// one, while that lowers the larger of the two loads, the best such step first.
static void even_out(const std::vector<double> &cost, std::vector<int> *per, std::vector<double> &load) {
    const int nw = (int)load.size();
    for (int step = 0; step < 256; ++step) {
        const int a = (int)(std::max_element(load.begin(), load.end()) - load.begin());
        double best = load[a] * (1.0 - 1e-9);
        int bb = -1, bx = -1, by = -1;
        for (int b = 0; b < nw; ++b)
            for (int x = 0; b != a && x < (int)per[a].size(); ++x)
                for (int y = -1; y < (int)per[b].size(); ++y) {
                    const double d = cost[per[a][x]] - (y >= 0 ? cost[per[b][y]] : 0.0);
                    const double m = std::max(load[a] - d, load[b] + d);
                    if (m < best) best = m, bb = b, bx = x, by = y;
                }
        if (bb < 0) break;
        const int i = per[a][bx];
        const double d = cost[i] - (by >= 0 ? cost[per[bb][by]] : 0.0);
        if (by >= 0) {
            std::swap(per[a][bx], per[bb][by]);
        } else {
            per[a].erase(per[a].begin() + bx);
            per[bb].push_back(i);
        }
        load[a] -= d;
        load[bb] += d;
    }
    for (int w = 0; w < nw; ++w)
        std::stable_sort(per[w].begin(), per[w].end(), [&](int x, int y) { return cost[x] > cost[y]; });
}

template <typename T> size_t smem_bytes(const GridView &g, int wrow_max, int v) {
    return 2 * sizeof(T) * (size_t)(g.nhalf + 2 * kPad) * kVariants[v].cells +
           sizeof(T) * (size_t)kVariants[v].warps * 2 * kVariants[v].rows * wrow_max;
}

}  // namespace

// Host part: weight streams and the task table, built once per modes handle.
double beta_host(const bz_modes *m, const int *l, const int *mm);

// Weight stream (with row-pair headers) and task table of one variant, with
// weights of type T; false if the grid is not covered by this variant (another
// variant or the generic kernel serves it).  With T = double and outX2 set, a
// second stream of the same byte layout for the FP32X2 form: the RT doubles of
// each l_2 step become RT FP32 high parts followed by RT FP32 low parts
// (hi = fl32(w), lo = fl32(w - hi)), headers copied as they are.
template <typename T>
static bool build_variant(bz_modes *m, int v, int &rc, void **outW, TaskTables *outT, int *outRowmax,
                          float **outX2 = nullptr) {
    constexpr int HEAD = kRowHeadBytes / (int)sizeof(T);
    const int R = variant_rt(v);                                // outputs per task (RT)
    const int kWarps = kVariants[v].warps;
    const int pack = kVariants[v].pack;                         // cells per lane
    rc = BZ_OK;
    const GridView &gv = m->g->v;
    const int d = gv.dim, h = gv.h, M = gv.M;
    const int rows = kVariants[v].rows;                         // row pairs at a time
    if (!((d == 2 && gv.N <= (rows > 1 && sizeof(T) == 4 ? 64 : 48)) || (d == 3 && gv.N <= 16))) return false;
    // shared memory of the spectrum alone must leave room for the weight buffers
    if (2 * sizeof(T) * (size_t)(gv.nhalf + 2 * kPad) * kVariants[v].cells > 200 * 1024) return false;
    const int nb = (M + R - 1) / R;
    const int lo_col = -h - kPad, hi_col = h + kPad;         // addressable columns
    std::vector<TaskRec> tasks;
    std::vector<T> W;
    std::vector<float> X2;                                  // FP32X2 stream (T = double only)
    const bool want_x2 = outX2 != nullptr && sizeof(T) == 8;
    std::vector<double> stepw(R);
    std::vector<double> cost;
    std::vector<int> phase;                                 // 1: runs on the reflected spectrum
    // reflect: the FP32 variants with one cell per lane whose output blocks
    // fit the row compute k_2 < 0 as k_2 > 0 of the spectrum reflected in the
    // last axis (beta-hat is invariant under that reflection); ramped: with
    // one lane group and R dividing h + 1, every task starts with the ramp
    // block and no step is padding
    const int G = variant_groups(v);
    const bool reflect = (sizeof(T) == 4 || kVariants[v].orient == 2) && variant_reflects(v, h);
    const bool ramped = reflect && G == 1 && (h + 1) % R == 0;
    const bool twins = reflect && kVariants[v].orient == 1;   // paired orientations need no reflected tasks
    // paired orientations compute k_2 < 0 in the mirrored half of every task:
    // only with blocks of k_2 >= 0 (else both halves would write one output)
    if (kVariants[v].orient == 2 && !reflect) return false;
    const int nmid = (d == 3) ? M : 1;                      // values of the middle index (3-D)
    struct Pair { int l[2], m[2]; };                         // leading indices of l and m
    for (int k1 = 0; k1 <= h; ++k1) {
        for (int i2 = 0; i2 < nmid; ++i2) {
            const int k2 = (d == 3) ? i2 - h : 0;
            const int orow = (d == 3) ? k1 * M + i2 : k1;
            std::vector<Pair> pairs;                         // row pairs visited for this output row
            for (int l1 = k1 - h; l1 <= k1 / 2; ++l1) {
                const int m1 = k1 - l1;
                if (d == 2) {
                    pairs.push_back({{l1, 0}, {m1, 0}});
                } else {
                    for (int l2 = std::max(-h, k2 - h); l2 <= std::min(h, k2 + h); ++l2)
                        pairs.push_back({{l1, l2}, {m1, k2 - l2}});
                }
            }
            // groups of `rows` row pairs, the last one filled with copies whose
            // weights are zero; FP32: of one read direction, which its kernel
            // branches on (the FP64 and FP32X2 forms take it lane by lane: 14^2 in
            // FP64 on 9000 cells 1.50 -> 1.43 ms a call)
            std::vector<char> dummy(pairs.size(), 0);
            if (rows > 1) {
                std::vector<Pair> in = pairs;
                pairs.clear();
                dummy.clear();
                for (int neg = 1; neg >= 0; --neg) {
                    for (const Pair &p : in)
                        if ((p.l[0] < 0) == (neg == 1)) pairs.push_back(p), dummy.push_back(0);
                    while ((sizeof(T) == 4 || neg == 0) && pairs.size() % rows)
                        pairs.push_back(pairs.back()), dummy.push_back(1);
                }
            }
            // blocks of R consecutive last-axis outputs.  reflect: the blocks
            // start at 0, R, 2R, ... and cover k_2 >= 0; each is run a second
            // time on the reflected spectrum for k_2 <= 0 (same weights), except
            // in the k_1 = 0 row, whose k_2 < 0 outputs are the conjugates of its
            // k_2 > 0 ones.  Otherwise they tile [-h, h], the last one ending at
            // h (it may overlap the previous block, whose outputs it then does
            // not store) and a block wider than the row starting at -h.
            std::vector<int> starts;
            if (reflect) {
                for (int k = 0; k <= h; k += R) starts.push_back(k);
            } else {
                for (int b = 0; b < nb; ++b) starts.push_back(std::max(-h, std::min(-h + R * b, h - R + 1)));
            }
            int prev_end = -h - 1;
            for (const int k20 : starts) {
                const int k2last = k20 + R - 1;
                int l2lo = 0, nblk = 0, npad = 0;
                if (ramped) {
                    // one step before the lowest l_2 of output k20, through h:
                    // 2h + 2 - k20 steps, a multiple of R when R divides h + 1
                    l2lo = k20 - h - 1;
                    npad = 2 * h + 2 - k20;
                    nblk = npad / R;
                } else {
                    const int lo = std::max(-h, k20 - h), hi = std::min(h, k2last + h);
                    const int len = hi - lo + 1;
                    nblk = (len + R - 1) / R;
                    npad = nblk * R;
                    // place the padded range [l2lo, l2lo + npad - 1] so that every
                    // f-hat_l column and every window column k - l lies within kPad
                    // of [-h, h]
                    bool placed = false;
                    for (int cand = lo - (npad - len); cand <= lo && !placed; ++cand) {
                        const int last = cand + npad - 1;
                        if (cand < lo_col || last > hi_col) continue;
                        if (k20 - last < lo_col || k2last - cand > hi_col) continue;
                        l2lo = cand;
                        placed = true;
                    }
                    if (!placed) return false;
                }
                TaskRec t;
                t.orow = orow;
                t.k20 = k20;
                t.nrows = (int)pairs.size();
                t.l2lo = l2lo;
                t.nblk = nblk;
                t.woff = (int)W.size();
                t.rfirst = reflect ? 0 : std::max(0, prev_end + 1 - k20);
                t.rowf = HEAD + npad * R * (kVariants[v].wdup ? 2 : 1);
                t.flags = (ramped ? kTaskRamp : 0) | (twins && k1 == 0 ? kTaskConj : 0);
                t.crow = (d == 3) ? (M - 1 - i2) : 0;        // k_1 = 0: row of -k (middle index -k_2)
                t.pad2 = t.pad3 = 0;
                prev_end = k2last;
                for (size_t ip = 0; ip < pairs.size(); ++ip) {
                    const Pair &p = pairs[ip];
                    // row of l (that of -l read backwards when l_1 < 0) and row of m
                    const bool neg = p.l[0] < 0;
                    const int a1 = neg ? -p.l[0] : p.l[0], a2 = neg ? -p.l[1] : p.l[1];
                    const int lrow = (d == 3) ? a1 * M + (a2 + h) : a1;
                    const int mrow = (d == 3) ? p.m[0] * M + (p.m[1] + h) : p.m[0];
                    const int cs = kVariants[v].cells / pack;   // shared-memory entries per mode
                    const int head[4] = {lrow * M * cs, mrow * M * cs, neg ? -1 : 1, 0};
                    static_assert(sizeof head == kRowHeadBytes, "16-byte row header");
                    T hw[HEAD];
                    std::memcpy(hw, head, sizeof head);
                    for (int q = 0; q < HEAD; ++q) W.push_back(hw[q]);
                    if (want_x2) {
                        float hf[4];
                        std::memcpy(hf, head, sizeof head);
                        for (int q = 0; q < 4; ++q) X2.push_back(hf[q]);
                    }
                    for (int j = 0; j < npad; ++j) {
                        const int lz = l2lo + j;
                        for (int r = 0; r < R; ++r) {
                            const int kz = k20 + r, mz = kz - lz;
                            double w = 0.0;
                            if (!dummy[ip] && kz <= h && lz >= -h && lz <= h && mz >= -h && mz <= h) {
                                int l[3], mm[3];
                                l[0] = p.l[0];
                                mm[0] = p.m[0];
                                if (d == 3) {
                                    l[1] = p.l[1];
                                    mm[1] = p.m[1];
                                }
                                l[d - 1] = lz;
                                mm[d - 1] = mz;
                                w = beta_host(m, l, mm);
                                if (p.l[0] < p.m[0]) w += beta_host(m, mm, l);
                            }
                            W.push_back((T)w);
                            if (kVariants[v].wdup) W.push_back((T)w);
                            stepw[r] = w;
                        }
                        if (want_x2) {
                            for (int r = 0; r < R; ++r) X2.push_back((float)stepw[r]);
                            for (int r = 0; r < R; ++r) X2.push_back((float)(stepw[r] - (double)(float)stepw[r]));
                        }
                    }
                }
                // evaluated pairs (a ramp skips R (R + 1) / 2 of each row pair's)
                const double c = (double)t.nrows * ((double)npad * R - (ramped ? R * (R + 1) / 2 : 0) + 2.0 * npad);
                tasks.push_back(t);
                cost.push_back(c);
                phase.push_back(0);
                if (twins && k1 > 0) {
                    TaskRec tr = t;                      // the same weights on the reflected spectrum
                    tr.flags = (t.flags & kTaskRamp) | kTaskRefl;
                    tr.rfirst = (k20 == 0) ? 1 : 0;      // k_2 = 0 is the unreflected task's
                    tasks.push_back(tr);
                    cost.push_back(c);
                    phase.push_back(kVariants[v].pq ? 0 : 1);   // the FP32x2 kernel reads it mirrored
                }
            }
        }
    }
    // assignment of tasks to nw warps: longest first to the least loaded, then
    // even_out; the offsets of each warp's list, then the task records
    auto make_table = [&](int nw, float &worst) {
        double longest = 0.0;                               // sum over the phases of the most loaded warp
        std::vector<std::vector<int>> per(2 * nw);
        for (int ph = 0; ph < 2; ++ph) {
            std::vector<int> order;
            for (size_t i = 0; i < tasks.size(); ++i)
                if (phase[i] == ph) order.push_back((int)i);
            std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
            std::vector<double> load(nw, 0.0);
            for (int i : order) {
                int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
                load[w] += cost[i];
                per[ph * nw + w].push_back(i);
            }
            even_out(cost, &per[ph * nw], load);
            longest += *std::max_element(load.begin(), load.end());
        }
        worst = (float)longest;
        std::vector<int> t(2 * nw + 1 + tasks.size() * kTaskInts);
        int pos = 0;
        for (int q = 0; q < 2 * nw; ++q) {
            t[q] = pos;
            for (int i : per[q]) {
                std::memcpy(&t[2 * nw + 1 + (size_t)pos * kTaskInts], &tasks[i], sizeof(TaskRec));
                ++pos;
            }
        }
        t[2 * nw] = pos;
        return t;
    };
    int wrow_max = 0;
    for (auto &t : tasks) wrow_max = std::max(wrow_max, t.rowf);   // staging buffer: one row pair
    if (smem_bytes<T>(gv, wrow_max, v) > 227 * 1024) return false;   // does not fit
    TaskTables tt;
    std::vector<int> tab;
    for (int S = 1; S <= kMaxSplit; ++S) {
        const std::vector<int> t = make_table(kWarps * S, tt.bal[S - 1]);
        tt.off[S - 1] = (int)tab.size();
        tab.insert(tab.end(), t.begin(), t.end());
    }
    double work = 0.0;
    for (double c : cost) work += c;
    tt.work = (float)work;
    T *dW = nullptr;
    int *dT = nullptr;
    float *dX = nullptr;
    cudaError_t e = dev_malloc(&dW, sizeof(T) * W.size());
    if (e == cudaSuccess) e = dev_malloc(&dT, sizeof(int) * tab.size());
    if (e == cudaSuccess) e = cudaMemcpy(dW, W.data(), sizeof(T) * W.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dT, tab.data(), sizeof(int) * tab.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && want_x2) {
        e = dev_malloc(&dX, sizeof(float) * X2.size());
        if (e == cudaSuccess) e = cudaMemcpy(dX, X2.data(), sizeof(float) * X2.size(), cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        dev_free(dW);
        dev_free(dT);
        dev_free(dX);
        rc = cuda_fail(e, "build_kernel_modes: weight stream");
        return false;
    }
    tt.block = dT;
    *outW = dW;
    *outT = tt;
    *outRowmax = wrow_max;
    if (want_x2) *outX2 = dX;
    return true;
}

bool modesum32_available(const bz_modes *m) { return m->d_W32 != nullptr; }

template <typename T, int RR, int WARPS, int CELLS, bool RTDIR = false>
static cudaError_t launch_instance(const Mode32Group &gd, size_t sm, cudaStream_t st) {
    cudaError_t e = allow_dynamic_smem((const void *)modesum32_kernel<T, RR, WARPS, CELLS, RTDIR>, sm);
    if (e != cudaSuccess) return e;
    modesum32_kernel<T, RR, WARPS, CELLS, RTDIR><<<(unsigned)gd.tile_start[gd.nitems], WARPS * 32, sm, st>>>(gd);
    return cudaGetLastError();
}

template <int RR, int WARPS, int CELLS>
static cudaError_t launch_pq(const Mode32Group &gd, size_t sm, cudaStream_t st, bool pdl = false) {
    cudaError_t e = allow_dynamic_smem((const void *)modesum_pq_kernel<RR, WARPS, CELLS>, sm);
    if (e != cudaSuccess) return e;
    if constexpr (RR == 2)
        return launch_after(modesum_pq_kernel<RR, WARPS, CELLS>, (unsigned)gd.tile_start[gd.nitems], WARPS * 32, sm, st,
                            pdl, gd);
    modesum_pq_kernel<RR, WARPS, CELLS><<<(unsigned)gd.tile_start[gd.nitems], WARPS * 32, sm, st>>>(gd);
    return cudaGetLastError();
}

static cudaError_t launch_group(const Mode32Group &gd, int v, size_t sm, cudaStream_t st, bool pdl = false) {
    switch (v) {
        case 0: return launch_instance<float, 8, 16, 32, true>(gd, sm, st);
        case 1: return launch_instance<float, 4, 32, 32>(gd, sm, st);
        case 2: return launch_instance<float, 4, 16, 16>(gd, sm, st);
        case 3: return launch_pq<8, 12, 8>(gd, sm, st);
        case 4: {
            cudaError_t e = allow_dynamic_smem((const void *)modesum_p2_kernel<4, 16>, sm);
            if (e != cudaSuccess) return e;
            modesum_p2_kernel<4, 16><<<(unsigned)gd.tile_start[gd.nitems], 16 * 32, sm, st>>>(gd);
            return cudaGetLastError();
        }
        case 5: return launch_pq<8, 12, 32>(gd, sm, st);
        case 6: return launch_pq<8, 16, 32>(gd, sm, st);
        case 7: return launch_pq<8, 16, 16>(gd, sm, st);
        case 8: return launch_pq<8, 8, 16>(gd, sm, st);
        case 9: return launch_pq<8, 4, 16>(gd, sm, st);
        case kSmallVariant: return launch_pq<2, 16, 16>(gd, sm, st, pdl);
        default: return cudaErrorInvalidValue;
    }
}

static void fill_item(Mode32Item &it, const bz_modes *m, const void *W, const TaskTables &tasks, int rowmax,
                      const void *fhat, void *Qhat, int64_t n, int split = 1) {
    it.split = split;
    const GridView &gv = m->g->v;
    it.fhat = fhat;
    it.Qhat = Qhat;
    it.W = W;
    it.tasks = tasks.block + tasks.off[split - 1];
    it.h = gv.h;
    it.M = gv.M;
    it.nhalf = (int)gv.nhalf;
    it.wrow_max = rowmax;
    it.n = n;
}

// CTAs of an instance of n cells: one per CELLS cells of each 32-cell tile.
static int64_t ctas_for(int v, int64_t n) {
    const int G = 32 / kVariants[v].cells;      // CTAs per 32-cell tile
    return ((n + 31) / 32) * G;
}

// CTAs per SM of a variant's kernel (its launch bounds: the FP32x2 kernels
// with 8 or 4 warps are built for 2 or 3 resident CTAs, the 8-cell FP64 and
// FP32X2 kernels for 2).
static int variant_ctas_per_sm(int v) {
    if (!kVariants[v].pq || (v >= kNumVariants && kVariants[v].cells == 4)) return 1;
    return kVariants[v].warps <= 4 ? 3 : kVariants[v].warps <= 8 ? 2 : 1;
}

// How a launch ends: its first `full` CTAs take a tile each, the tiles after
// them are shared by S CTAs.
struct Tail {
    int64_t full;
    int S;
};

static int sm_count();

// The whole waves of a launch run one CTA per tile; the T CTAs left over would
// keep a part of the SMs busy for as long as a whole wave, so S CTAs share each
// of their tiles.  Every output is computed by one task with the same
// arithmetic, so the results do not depend on S.  S has the least estimated
// time, in units of a CTA's time on a full SM: an SM gets q of the T S CTAs,
// each taking the mean of its share of the work (what counts where other CTAs
// fill its gaps) and of its most loaded warp's part (where they do not), and o
// for its start, chiefly the staged spectrum: `stage` loads per mode.  With several CTAs per SM the last ones end
// apart, by `ragged` times a CTA's length on the mean.  Measured, S = 1 and the
// S taken here: 32^2 in FP32 on 5000, 9000, 19802, 32768 cells 246, 322, 687,
// 1054 us and 185, 290, 632, 1014 (S = 4); 48^2 on 3000, 6000, 13632 cells 735,
// 1110, 2233 us and 497 (4), 938 (2), 2154 (3); 64^2 on 500 and 1500 cells 577,
// 1153 us and 297 (2), 736 (4); 16^3 on 700 and 1400 cells 446, 871 us and
// 295 (5), 528 (6); 32^2 in FP64 on 4099 cells 8.60 ms and 7.54 (2).
static Tail tail_split(const bz_modes *m, int v, const TaskTables &t, int64_t ctas, size_t sm, double stage,
                       double ragged) {
    const int64_t fit = std::max<int64_t>(1, 228 * 1024 / (int64_t)(sm + 1024));
    const int64_t per_sm = std::min<int64_t>(variant_ctas_per_sm(v), fit), sms = sm_count(), wave = sms * per_sm;
    if (per_sm == 1) ragged = 0.0;
    const int G = 32 / kVariants[v].cells;
    int64_t full = ctas / wave * wave;
    full -= full % G;
    const int64_t T = ctas - full;
    if (T == 0) return {ctas, 1};
    const double o = stage * (double)m->g->v.nhalf / t.work;
    auto estimate = [&](int S) {
        const double q = (double)((T * S + sms - 1) / sms);
        return q * (0.5 * (1.0 / S + t.bal[S - 1] / t.bal[0]) + o) + ragged / S;
    };
    Tail r{full, 1};
    double best = estimate(1);
    for (int S = 2; S <= kMaxSplit; ++S)
        if (estimate(S) < (r.S == 1 ? 0.97 : 0.99) * best) {
            best = estimate(S);
            r.S = S;
        }
    return r;
}
// `stage` and `ragged` of the FP32 forms, fitted to the times above; FP64 and
// FP32X2 tasks take 30 and 5 times as long for the same staged bytes, and the
// FP64 pipe is full to the end
constexpr double kStage32 = 4.3, kRagged32 = 0.45, kStage64 = 0.15, kStageX2 = 0.8;

// Appends an instance of n cells to a launch (gd.nitems counts its items): the
// cells of its first `full` CTAs, then those whose tiles S CTAs share.  fsize,
// qsize: bytes per value.  An error, and nothing written, past kMaxGroup items.
static cudaError_t add_items(Mode32Group &gd, const bz_modes *m, int v, const void *W, const TaskTables &t, int rowmax,
                      const void *fhat, size_t fsize, void *Qhat, size_t qsize, int64_t n, Tail tail) {
    const int64_t nm = std::min(n, tail.full * kVariants[v].cells);
    for (int p = 0; p < 2; ++p) {
        const int64_t first = p ? nm : 0, cnt = p ? n - nm : nm, off = first / 32 * m->g->v.nhalf * 32;
        if (cnt <= 0) continue;
        if (gd.nitems >= kMaxGroup) return cudaErrorInvalidValue;
        const int S = p ? tail.S : 1, k = gd.nitems++;
        fill_item(gd.item[k], m, W, t, rowmax, static_cast<const char *>(fhat) + off * fsize,
                  static_cast<char *>(Qhat) + off * qsize, cnt, S);
        gd.tile_start[k + 1] = gd.tile_start[k] + ctas_for(v, cnt) * S;
    }
    return cudaSuccess;
}

static cudaError_t launch_variant(const bz_modes *m, int v, const float2 *fhat, float2 *Qhat, int64_t n,
                                  cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    Mode32Group gd;
    memset(&gd, 0, sizeof gd);
    const cudaError_t e = add_items(gd, m, v, m->var_W[v], m->var_task[v], m->var_rowmax[v], fhat, sizeof(float2), Qhat,
                                    sizeof(float2), n, {ctas_for(v, n), 1});
    if (e != cudaSuccess) return e;
    return launch_group(gd, v, smem_bytes<float>(m->g->v, m->var_rowmax[v], v), st);
}

// FP64 form: paired orientations on 8-cell tiles (variant entry 10), on 4-cell
// tiles where the double spectrum of 8 cells does not fit shared memory (16^3),
// and with two outputs per thread where four overhang the half row (N < 8).
// The FP32X2 form runs on the same layout.
constexpr int kFp64Variants[3] = {10, 11, 12};

bool modesum64_available(const bz_modes *m) { return m->w64 != nullptr; }

template <bool X2, int RR, int WARPS, int CELLS>
static cudaError_t launch_pair(const Mode32Group &gd, size_t sm, cudaStream_t st) {
    cudaError_t e = allow_dynamic_smem((const void *)modesum_pair_kernel<X2, RR, WARPS, CELLS>, sm);
    if (e != cudaSuccess) return e;
    modesum_pair_kernel<X2, RR, WARPS, CELLS><<<(unsigned)gd.tile_start[gd.nitems], WARPS * 32, sm, st>>>(gd);
    return cudaGetLastError();
}

// Spectra of 16 bytes per value (one double, or FP32 high and low parts) and
// weight rows of 8-byte slots in both forms.
template <bool X2>
static cudaError_t launch_pairs(const bz_modes *m, const double2 *fhat, void *Qhat, int64_t n, cudaStream_t st) {
    Mode32Group gd;
    memset(&gd, 0, sizeof gd);
    const int v = m->variant64;
    const size_t sm = smem_bytes<double>(m->g->v, m->rowmax64, v);
    const cudaError_t e = add_items(gd, m, v, X2 ? static_cast<const void *>(m->wx2) : m->w64, m->task64, m->rowmax64, fhat,
                                    sizeof(double2), Qhat, X2 ? sizeof(float2) : sizeof(double2), n,
                                    tail_split(m, v, m->task64, ctas_for(v, n), sm, X2 ? kStageX2 : kStage64, 0.0));
    if (e != cudaSuccess) return e;
    if (m->variant64 == kFp64Variants[0]) return launch_pair<X2, 4, 8, 8>(gd, sm, st);
    if (m->variant64 == kFp64Variants[1]) return launch_pair<X2, 4, 8, 4>(gd, sm, st);
    if (m->variant64 == kFp64Variants[2]) return launch_pair<X2, 2, 8, 8>(gd, sm, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_modesum64(const bz_modes *m, const double2 *fhat, double2 *Qhat, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (!m->w64) return cudaErrorInvalidValue;
    return launch_pairs<false>(m, fhat, Qhat, n, st);
}

bool modesum_x2_available(const bz_modes *m) { return m->wx2 != nullptr && m->variant64 >= 0; }

cudaError_t launch_modesum_x2(const bz_modes *m, const double2 *fhat, float2 *Qhat, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (!modesum_x2_available(m)) return cudaErrorInvalidValue;
    return launch_pairs<true>(m, fhat, Qhat, n, st);
}

bool modesum32_tail_splits(const bz_modes *m) {
    return m->method == 0 && modesum32_available(m) && !m->variant_fixed && kVariants[m->variant].cells == 32;
}

// A variant that holds several CTAs per SM fills only part of each SM in a
// launch of less than half a wave (and a lone wave loses about a sixth: all
// CTAs stage their spectra at once and the SMs empty unevenly).  Its sibling
// with one 16-warp CTA per SM runs the same tasks in the same order
// (bit-identical results), so launches of at most half a wave take it.
static int small_batch_variant(const bz_modes *m, int64_t n) {
    const int v = m->variant;
    if (m->variant_fixed || variant_ctas_per_sm(v) == 1) return v;
    if (n > (int64_t)sm_count() * variant_ctas_per_sm(v) * kVariants[v].cells / 2) return v;
    for (int s = 0; s < kNumVariants; ++s) {
        const Variant &a = kVariants[s], &b = kVariants[v];
        if (s != v && m->var_W[s] && variant_ctas_per_sm(s) == 1 && a.R == b.R && a.cells == b.cells &&
            a.pack == b.pack && a.wdup == b.wdup && a.pq == b.pq && a.orient == b.orient)
            return s;
    }
    return v;
}

// A launch that would give less than one CTA to every SM is bound by the chain
// of one warp's tasks.  The small variant runs the paired 16-cell variants' sums
// (the same terms in the same order, bit-identical results) with two outputs
// per thread: four times the tasks, a third of the chain each, spread over up
// to eight CTAs per tile.  Its steps do fewer FMAs per load, so it is taken where
// the loads of the most loaded warps say that it is faster by a tenth.  64 cells
// of 16^2: 14.6 -> 12.5 us, of 32^2: 82 -> 31 us, of 48^2: 375 -> 93 us.  Returns the CTAs per
// tile, 0 where the other variants are better.
static int small_split(const bz_modes *m, int v, int64_t n) {
    const Variant &k = kVariants[v];
    if (m->variant_fixed || !m->small_W || !k.pq || k.cells != 16 || k.R != 8) return 0;
    const int64_t ctas = ctas_for(kSmallVariant, n), sms = sm_count();
    if (ctas > sms) return 0;
    const float *bal = m->small_task.bal;
    int best = 0;
    double t = 0.9 * m->var_task[v].bal[0];
    for (int S = 1; S <= kMaxSplit; ++S) {
        const double ts = std::max((double)((ctas * S + sms - 1) / sms) * bal[0] / S, (double)bal[S - 1]);
        if (ts < (best ? 0.97 : 1.0) * t) {
            t = ts;
            best = S;
        }
    }
    return best;
}

bool modesum32_small_batches_fast(const bz_modes *m) {
    return m->method == 0 && modesum32_available(m) && small_batch_variant(m, 1) != m->variant;
}

int modesum32_wave_cells_per_sm(const bz_modes *m) {
    if (m->method != 0 || !modesum32_available(m)) return 32;
    return variant_ctas_per_sm(m->variant) * kVariants[m->variant].cells;
}

// One launch for the whole batch: the main part (one tile per CTA) and the
// last partial wave (split tiles, or the 16-cell variant) as two items.
cudaError_t launch_modesum32(const bz_modes *m, const float2 *fhat, float2 *Qhat, int64_t n, cudaStream_t st,
                             bool pdl) {
    if (n <= 0) return cudaSuccess;
    const int sv = small_batch_variant(m, n);
    Mode32Group gd;
    memset(&gd, 0, sizeof gd);
    cudaError_t e;
    if (const int S = small_split(m, sv, n)) {
        e = add_items(gd, m, kSmallVariant, m->small_W, m->small_task, m->small_rowmax, fhat, sizeof(float2), Qhat,
                      sizeof(float2), n, {0, S});
        if (e != cudaSuccess) return e;
        return launch_group(gd, kSmallVariant, smem_bytes<float>(m->g->v, m->small_rowmax, kSmallVariant), st, pdl);
    }
    const Variant &k = kVariants[sv];
    const int64_t ctas = ctas_for(sv, n);
    const size_t sm = smem_bytes<float>(m->g->v, m->var_rowmax[sv], sv);
    const Tail tail = m->variant_fixed && k.rows == 1 ? Tail{ctas, 1}
                                                      : tail_split(m, sv, m->var_task[sv], ctas, sm, kStage32, kRagged32);
    // scalar 32-cell variants: the tiles left over run on the 16-cell variant
    // (twice the CTAs, bit-identical where it sums in the same order), itself with
    // its last ones split: 24^2 on 1949, 7000, 40000 cells 72, 143, 646 us with split
    // 32-cell tiles, 56, 128, 633 so
    if (k.cells == 32 && !m->variant_fixed && tail.full < ctas && !k.pq && k.pack == 1 && m->var_W[2] &&
        variant_reflects(2, m->g->v.h) == variant_reflects(sv, m->g->v.h)) {
        const int64_t nm = tail.full * 32;
        const size_t off = (size_t)nm * m->g->v.nhalf;
        e = launch_variant(m, sv, fhat, Qhat, nm, st);
        if (e != cudaSuccess) return e;
        const size_t s2 = smem_bytes<float>(m->g->v, m->var_rowmax[2], 2);
        e = add_items(gd, m, 2, m->var_W[2], m->var_task[2], m->var_rowmax[2], fhat + off, sizeof(float2), Qhat + off,
                      sizeof(float2), n - nm, tail_split(m, 2, m->var_task[2], ctas_for(2, n - nm), s2, kStage32, kRagged32));
        if (e != cudaSuccess) return e;
        return launch_group(gd, 2, s2, st);
    }
    e = add_items(gd, m, sv, m->var_W[sv], m->var_task[sv], m->var_rowmax[sv], fhat, sizeof(float2), Qhat, sizeof(float2),
                  n, tail);
    if (e != cudaSuccess) return e;
    return launch_group(gd, sv, sm, st);
}

// Heterogeneous instances in one launch; all items must use the same kernel
// variant and be ordered as they should be scheduled (longest first);
// count <= kMaxGroup.
cudaError_t launch_modesum32_group(const bz_modes *const *ms, const float2 *const *fhat, float2 *const *Qhat,
                                   const int64_t *n, int count, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    if (count > kMaxGroup) return cudaErrorInvalidValue;
    const int v = ms[0]->variant;
    Mode32Group gd;
    memset(&gd, 0, sizeof gd);
    size_t sm = 0;
    int64_t whole = 0;
    for (int i = 0; i < count; ++i) {
        if (ms[i]->variant != v) return cudaErrorInvalidValue;
        whole += ctas_for(v, n[i]);
        sm = std::max(sm, smem_bytes<float>(ms[i]->g->v, ms[i]->var_rowmax[v], v));
    }
    for (int i = 0; i < count; ++i) {
        // the launch's last partial wave, as far as it lies in the last instance
        Tail tail{ctas_for(v, n[i]), 1};
        if (i == count - 1 && count < kMaxGroup && (!ms[i]->variant_fixed || kVariants[v].rows > 1)) {
            const Tail all = tail_split(ms[i], v, ms[i]->var_task[v], whole, sm, kStage32, kRagged32);
            if (all.S > 1) tail = {tail.full - std::min(whole - all.full, tail.full), all.S};
        }
        const cudaError_t e = add_items(gd, ms[i], v, ms[i]->var_W[v], ms[i]->var_task[v], ms[i]->var_rowmax[v], fhat[i],
                                        sizeof(float2), Qhat[i], sizeof(float2), n[i], tail);
        if (e != cudaSuccess) return e;
    }
    if (gd.nitems == 0) return cudaSuccess;
    if (sm > 227 * 1024) return cudaErrorInvalidValue;
    return launch_group(gd, v, sm, st);
}

// ---- autotuner ------------------------------------------------------------
// Times every buildable variant once per (dimension, N, SM count) on a
// synthetic batch (zero spectra: the kernel's cost does not depend on the
// values) of twelve 32-cell tiles per SM and keeps the fastest.  Results are
// cached for the process and, when BZ_TUNE_CACHE names a file, in that file as
// lines "dim N sms variant" (variant = index + 1).
static std::mutex g_tune_mu;
static std::map<std::tuple<int, int, int>, int> g_tune;

// SM count of the current device (cached per device; 0 entries are unset).
static int sm_count() {
    static std::atomic<int> cache[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64) {
        const int c = cache[dev].load(std::memory_order_relaxed);
        if (c > 0) return c;
    }
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
    if (dev >= 0 && dev < 64) cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

static void tune_file_load() {
    const char *path = getenv("BZ_TUNE_CACHE");
    if (!path) return;
    FILE *fp = fopen(path, "r");
    if (!fp) return;
    int d, N, sms, id;
    while (fscanf(fp, "%d %d %d %d", &d, &N, &sms, &id) == 4) g_tune[std::make_tuple(d, N, sms)] = id - 1;
    fclose(fp);
}

static void tune_file_store(int d, int N, int sms, int v) {
    const char *path = getenv("BZ_TUNE_CACHE");
    if (!path) return;
    FILE *fp = fopen(path, "a");
    if (!fp) return;
    fprintf(fp, "%d %d %d %d\n", d, N, sms, v + 1);
    fclose(fp);
}

static int autotune(bz_modes *m, int &rc) {
    rc = BZ_OK;
    const GridView &gv = m->g->v;
    int avail[kNumVariants], na = 0;
    for (int v = 0; v < kNumVariants; ++v)
        if (m->var_W[v]) avail[na++] = v;
    if (na == 1) return avail[0];
    const int sms = sm_count();
    const auto key = std::make_tuple(gv.dim, gv.N, sms);
    std::lock_guard<std::mutex> lk(g_tune_mu);
    if (g_tune.empty()) tune_file_load();
    auto it = g_tune.find(key);
    if (it != g_tune.end())
        for (int q = 0; q < na; ++q)
            if (avail[q] == it->second) return avail[q];
    // twelve 32-cell tiles per SM (several waves of every variant, so that
    // neither the tail nor a single wave decides); two rounds over the
    // variants, best of three launches each
    const int64_t n = (int64_t)12 * sms * 32;
    const size_t bytes = 2 * sizeof(float2) * (size_t)((n + 31) / 32) * gv.nhalf * 32;
    void *buf = nullptr;
    cudaError_t e = dev_malloc(&buf, bytes);
    if (e == cudaSuccess) e = cudaMemset(buf, 0, bytes);
    cudaEvent_t a = nullptr, b = nullptr;
    if (e == cudaSuccess) e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    float best[kNumVariants];
    for (int q = 0; q < kNumVariants; ++q) best[q] = 1e30f;
    const float2 *fh = static_cast<const float2 *>(buf);
    float2 *qh = static_cast<float2 *>(buf) + bytes / (2 * sizeof(float2));
    for (int round = 0; round < 2 && e == cudaSuccess; ++round) {
        for (int q = 0; q < na && e == cudaSuccess; ++q) {
            const int v = avail[q];
            e = launch_variant(m, v, fh, qh, n, nullptr);              // warm-up
            for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) {
                e = cudaEventRecord(a, nullptr);
                if (e == cudaSuccess) e = launch_variant(m, v, fh, qh, n, nullptr);
                if (e == cudaSuccess) e = cudaEventRecord(b, nullptr);
                if (e == cudaSuccess) e = cudaEventSynchronize(b);
                float ms = 0.f;
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
                if (e == cudaSuccess) best[v] = std::min(best[v], ms);
            }
        }
    }
    int pick = avail[0];
    for (int q = 1; q < na; ++q)
        if (best[avail[q]] < best[pick]) pick = avail[q];
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    dev_free(buf);
    if (e != cudaSuccess) {
        rc = cuda_fail(e, "build_kernel_modes: autotune");
        return avail[0];
    }
    g_tune[key] = pick;
    tune_file_store(gv.dim, gv.N, sms, pick);
    return pick;
}

int modes_build_fp32_tables(bz_modes *m) {
    m->d_W32 = nullptr;
    m->variant = 0;
    m->variant_fixed = 0;
    m->modesum_variant = 0;
    int rc = BZ_OK;
    bool any = false;
    for (int v = 0; v < kNumVariants; ++v) {
        m->var_W[v] = nullptr;
        m->var_task[v].block = nullptr;
        m->var_rowmax[v] = 0;
        void *w = nullptr;
        if (build_variant<float>(m, v, rc, &w, &m->var_task[v], &m->var_rowmax[v])) {
            m->var_W[v] = static_cast<float *>(w);
            any = true;
        }
        if (rc) return rc;
    }
    // the small variant's tables beside those of the 16-warp paired variant
    m->small_W = nullptr;
    m->small_task.block = nullptr;
    if (m->var_W[7]) {
        void *w = nullptr;
        if (build_variant<float>(m, kSmallVariant, rc, &w, &m->small_task, &m->small_rowmax))
            m->small_W = static_cast<float *>(w);
        if (rc) return rc;
    }
    // FP64 tables where the double spectrum fits shared memory
    m->w64 = nullptr;
    m->task64.block = nullptr;
    m->rowmax64 = 0;
    m->variant64 = -1;
    m->wx2 = nullptr;
    for (int q = 0; q < 3 && m->variant64 < 0; ++q) {
        if (build_variant<double>(m, kFp64Variants[q], rc, &m->w64, &m->task64, &m->rowmax64, &m->wx2))
            m->variant64 = kFp64Variants[q];
        if (rc) return rc;
    }
    if (!any) return BZ_OK;
    const char *force = getenv("BZ_MODESUM_VARIANT");   // fixed choice (1-based id), no timing
    int v = -1;
    if (force) {
        const int id = atoi(force) - 1;
        if (id >= 0 && id < kNumVariants && m->var_W[id]) v = id;
    }
    m->variant_fixed = v >= 0;      // a fixed variant also serves the last partial wave
    if (v < 0) v = autotune(m, rc);
    if (rc) return rc;
    m->variant = v;
    m->d_W32 = m->var_W[v];
    m->w32_rowmax = m->var_rowmax[v];
    m->modesum_variant = m->g->v.dim == 2 && m->g->v.N > 48 ? 0 : v + 1;   // one form only: no choice to report
    return BZ_OK;
}

}  // namespace bz
