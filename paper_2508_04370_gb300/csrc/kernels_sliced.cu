// FP64-accurate Schur-complement updates of large fronts on the bf16 tensor
// cores (the dgemm updates of Sec. 4.4, with FP64 pivots, regularisation and
// refinement unchanged).
//
// The regularised augmented systems of an IPM grow by about 1/delta when a
// dual row is eliminated with a pivot of size delta (and by more at wide
// Theta spreads), so FP32-accurate updates leave errors that refinement
// cannot remove.  These kernels keep the product accurate to about 2^-54 of
// the largest operand entry of each row, like an FP64 product, by exact
// integer arithmetic on the tensor cores (the splitting idea of Ozaki et
// al.):
//
//  1. slicing, in the panel's triangular solve (k_panel_trsm holds each
//     finished row of L in one warp).  Panels are taken in pairs: after the
//     first panel of a pair only the second panel's 32 columns are updated
//     (one chunk); after the second panel the whole trailing part receives
//     both panels' update at once (two chunks, K = 64), which halves the
//     read-modify-write passes over the trailing part and the epilogue work
//     per panel.  Every trailing row r of the two panel operands
//     a_rq = L(r, q) 2^h_q and b_rq = L(r, q) d_q 2^-h_q over the chunks'
//     columns (h_q = floor(log2 |d_q| / 2): an exact balancing of each
//     column, so that a_rq^2 and b_rq^2 are both within a factor 4 of
//     L(r, q)^2 |d_q|, whatever the spread of the pivots) gets one
//     power-of-two scale 2^E_r with |entries| < 2^E_r and is rounded to the
//     56-bit integers X_rq = rint(a_rq 2^(56 - E_r)), written as eight
//     balanced base-2^7 digits X = sum_t x_t 2^(7 (7 - t)), |x_t| <= 64
//     (|x_0| <= 128), each exactly a bf16.  The digits go to a work space in
//     the 128-byte-swizzled K-major image the tensor cores read, one image
//     set per chunk.
//  2. k_update_sliced: a CTA takes runs of 128 x 32 output tiles, each run in one
//     row block, whose digit images arrive once by bulk copies (TMA), and
//     the column tiles' images through two stages; one thread issues, per
//     slice t of the rows, one tcgen05.mma.kind::f16 (K = 16) against the
//     column slices u = 0 .. 7 - t side by side (N = 32 (8 - t)), which adds the
//     36 digit products with t + u <= 7 to eight TMEM accumulators S_d,
//     d = t + u, kept across the chunks.  For a
//     given d at most two products involve x_0 or y_0 (up to 128 x 64) and
//     the others are at most 64 x 64, so |S_d| <= 40960 K <= 2^21.4 for
//     K <= 64 and FP32 accumulation is exact.  The epilogue forms
//     T = sum_d S_d 2^(7 (7 - d)) in 64-bit integers without its low 8 bits
//     (digit_sum.h), the product
//     sum_q a_iq b_jq ~= 2^(E_i + E_j - 63) T
//     as a double built from the integer's bits (one rounding), and
//     subtracts it from the FP64 entry: one FP64 instruction per entry.
// Error per entry: operand rounding 2^-57 and the dropped digit products
// (t + u >= 8) below 2^-55, relative to 2^(E_i + E_j) per column of the
// chunks, and the low bits of T, below 2^-55 once: about
// 2^-52 sqrt(max_q L_iq^2 |d_q| max_q L_jq^2 |d_q|) together;
// FP64 GEMM's is 2^-53 of each |L_iq d_q L_jq|, summed.  Without the
// balancing a panel mixing pivots of size delta and of size 1/delta pairs
// the largest a of one column with the largest b of another, and the
// factorisation of a matrix with that much growth diverges.
#include <cuda_runtime.h>

#include <cstdint>

#include "digit_sum.h"
#include "ipm_dev.h"
#include "tc_common.cuh"
#include "sliced_common.cuh"

namespace ipm {

using namespace sliced;

namespace {


// t 2^e as a double (round half up to 53 bits), built with integer
// operations and without a branch; 0 for t = 0.  far: the result leaves the
// normal range (the caller takes ldexp).
__device__ __forceinline__ double int_scaled(long long t, int e, bool &far) {
    const unsigned long long a = t < 0 ? (unsigned long long)(-t) : (unsigned long long)t;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << (lz & 63);                     // bit 63 set
    const unsigned long long mant = (n >> 11) + ((n >> 10) & 1ull);  // bit 52 set: added to the exponent field below it,
    const int field = 63 - lz + e + 1023;                            // a carry raises the exponent
    far = t != 0 && (unsigned)(field - 1) >= 2045u;
    const unsigned hi = (unsigned)(mant >> 32) + ((unsigned)(field - 1) << 20);
    const double x = __hiloint2double((int)(hi | ((unsigned)(t >> 32) & 0x80000000u)), (int)(unsigned)mant);
    return t != 0 ? x : 0.0;
}

// 128 a + b for accumulators a, b: FP32 integers below 2^22.
__device__ __forceinline__ int32_t acc_pair(uint32_t a, uint32_t b) {
    return sliced::digit_pair(__float_as_uint(__uint_as_float(a) + 12582912.0f),
                              __float_as_uint(__uint_as_float(b) + 12582912.0f));
}

// C(i, j) -= sum_q L(i, q) d_q L(j, q), i >= j, for runs of 128 x 32 tiles.
//
// What bounds a tile (K = 64): the tensor pipe 2,304 cycles (36 products of
// 128 x 32 x 64), the FP64 pipe 2,048 (one subtraction per entry at two per
// clock), the recombination about 2,200 issue slots per SM sub-partition, so
// the three run beside each other: warp 8 copies and issues the MMAs of tile
// n + 1 while four warps recombine tile n from its half of TMEM and the other
// four tile n - 1, eight columns at a time and without branches (with a branch
// per entry the columns' chains of integer instructions did not overlap: 4.1 us
// a tile, now 3.1; 16 warps take 2.9 but leave the next panel's kernels no
// registers on the SM).  One MMA per row slice with N up to 256 reads the row slice
// from shared memory once (544 cycles of shared-memory reads per K = 16; 36 MMAs
// with N = 32 read it 36 times, 1,440).  A CTA keeps going over several row
// blocks: the start of a CTA (TMEM, 160 KB of copies, the first round trips)
// costs as much as four tiles, and the next row block's images arrive while
// the last tiles are recombined.  Registers are held to 112 so that a
// diagonal block or triangular solve of the next panel (256 threads) runs on
// the SM beside it.
// 50-period staircase, per factorisation: the updates take 45 ms of stream time
// beside the panels instead of 69, the factorisation 59.5 ms instead of 73.
constexpr int kSlicedThreads = 288;
constexpr int kChunkA = (int)kSliceOperandBytes;  // digit images of 128 rows, 32 columns of the panel
constexpr int kChunkB = kGroupBytes;              // and of 32 rows (the tile's columns)
constexpr int kSlicedSmem = kSliceChunks * (kChunkA + 2 * kChunkB);

// The tiles of a segment in order.
struct TileCursor {
    const SlicedRun *runs;
    int run, last, t;
    SlicedRun R;
    __device__ __forceinline__ TileCursor(const SlicedRun *r, SlicedSeg g) : runs(r), run(g.first), last(g.last), t(0) {
        R = runs[run];
    }
    __device__ __forceinline__ bool end() const { return run >= last; }
    __device__ __forceinline__ void next() {
        if (++t < R.nt) return;
        t = 0;
        if (++run < last) R = runs[run];
    }
    __device__ __forceinline__ int col() const { return R.j0 + kSliceCols * t; }
    // slice block and row inside it of the tile's columns (as rows of operand B)
    __device__ __forceinline__ int blk_b() const { return R.base + (col() - R.p1) / kSliceRows; }
    __device__ __forceinline__ int row_b() const { return (col() - R.p1) % kSliceRows; }
    __device__ __forceinline__ int blk_a() const { return R.base + (R.i0 - R.p1) / kSliceRows; }
};

__global__ void __maxnreg__(112)
    k_update_sliced(DevPlan P, double *__restrict__ fronts, const SlicedRun *__restrict__ runs,
                    const SlicedSeg *__restrict__ segs, const uint8_t *__restrict__ ws,
                    const int32_t *__restrict__ ws_exp, DevCtl *ctl) {
    extern __shared__ __align__(1024) uint8_t A[];  // [chunk]
    uint8_t *B = A + kSliceChunks * kChunkA;  // [stage][chunk]
    // copies landed (rows per chunk; columns per stage), MMAs of an accumulator
    // done, accumulator read, everything issued done
    __shared__ uint64_t bar_a[kSliceChunks], bar_b[2], bar_full[2], bar_empty[2], bar_end;
    __shared__ uint32_t tbase;
    const SlicedSeg seg = segs[blockIdx.x];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto copy_a = [&](const TileCursor &c) {
        for (int ch = 0; ch < c.R.kc; ch++) {
            tc::mbar_expect_tx(&bar_a[ch], kChunkA);
            tc::bulk_g2s(A + ch * kChunkA, ws + (int64_t)c.blk_a() * kSliceBlockBytes + ch * kSliceChunkBytes, kChunkA,
                         &bar_a[ch]);
        }
    };
    auto copy_b = [&](const TileCursor &c, int st) {
        const uint8_t *src = ws + (int64_t)c.blk_b() * kSliceBlockBytes + kSliceOperandBytes + c.row_b() / 32 * kChunkB;
        tc::mbar_expect_tx(&bar_b[st], (uint32_t)(c.R.kc * kChunkB));
        for (int ch = 0; ch < c.R.kc; ch++)
            tc::bulk_g2s(B + (st * kSliceChunks + ch) * kChunkB, src + ch * kSliceChunkBytes, kChunkB, &bar_b[st]);
    };
    if (tid == 256) {
        for (int q = 0; q < 2; q++) {
            tc::mbar_init(&bar_a[q], 1);
            tc::mbar_init(&bar_b[q], 1);
            tc::mbar_init(&bar_full[q], 1);
            tc::mbar_init(&bar_empty[q], 4);
        }
        tc::mbar_init(&bar_end, 1);
        tc::fence_mbar_init();
    }
    if (warp == 0) tc::tmem_alloc(&tbase, 512);  // two sets of 8 accumulators x 32 columns
    if (tid == 256) {
        // the first tile's images are on their way before the CTA meets
        TileCursor c(runs, seg);
        copy_a(c);
        copy_b(c, 0);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tbase;
    if (warp == 8) {
        if (lane == 0) {
            TileCursor c(runs, seg), cc(runs, seg);  // the tile to multiply, the tile to copy
            int copied = 1;                          // column tiles whose copy was issued
            cc.next();
            if (!cc.end()) {
                copy_b(cc, 1);
                copied = 2;
                cc.next();
            }
            int pa[kSliceChunks] = {0, 0};       // parity of the next copy of each row chunk
            bool wait_a[kSliceChunks] = {false, false};
            for (int ch = 0; ch < c.R.kc; ch++) wait_a[ch] = true;
            bool ok = true;
            auto need = [&](uint64_t *bar, int parity, int why) {
                if (ok && !tc::mbar_wait(bar, parity)) {
                    atomicOr(&ctl->status, kStatTimeout | why);
                    ok = false;
                }
                return ok;
            };
            for (int n = 0; !c.end() && ok; n++, c.next()) {
                const int st = n & 1, use = n >> 1, kc = c.R.kc;
                const uint32_t acc = tmem + 256u * st;
                if (n > 0 && c.t == 0) {
                    // a new row block, once the last one's MMAs are done
                    if (!need(&bar_full[st ^ 1], ((n - 1) >> 1) & 1, kStatWaitMma)) break;
                    copy_a(c);
                    for (int ch = 0; ch < kc; ch++) wait_a[ch] = true;
                }
                if (n >= 2) need(&bar_empty[st], (use - 1) & 1, kStatWaitMma);
                need(&bar_b[st], use & 1, kStatWaitCopy);
#pragma unroll
                for (int ch = 0; ch < kSliceChunks; ch++) {
                    if (ch >= kc) continue;
                    if (wait_a[ch] && need(&bar_a[ch], pa[ch], kStatWaitCopy)) {
                        pa[ch] ^= 1;
                        wait_a[ch] = false;
                    }
                    if (!ok) continue;
                    tc::fence_after_sync();
                    const uint32_t a0 = tc::smem_u32(A + ch * kChunkA);
                    const uint32_t b0 = tc::smem_u32(B + (st * kSliceChunks + ch) * kChunkB);
#pragma unroll
                    for (int kk = 0; kk < 2; kk++)
#pragma unroll
                        for (int t = 0; t < kSlices; t++)
                            tc::mma_bf16(acc + (uint32_t)(t * kSliceCols),
                                         tc::smem_desc(a0 + (t >> 1) * (uint32_t)kSlicePairBytes + (t & 1) * 64 + kk * 32),
                                         tc::smem_desc64(b0 + kk * 32), tc::idesc_bf16(kSliceRows, kSliceCols * (kSlices - t)),
                                         (ch > 0 || t > 0 || kk > 0) ? 1u : 0u);
                }
                if (!ok) break;
                tc::commit_to(&bar_full[st]);
                // the stage of tile n - 1 is free once its MMAs are done
                if (n >= 1 && !cc.end() && need(&bar_full[st ^ 1], ((n - 1) >> 1) & 1, kStatWaitMma)) {
                    copy_b(cc, st ^ 1);
                    copied++;
                    cc.next();
                }
            }
            // every copy landed and every MMA done before the CTA gives up its
            // shared memory and TMEM (a wait that failed is waited for once more)
            if (!ok) {
                for (int ch = 0; ch < kSliceChunks; ch++)
                    if (wait_a[ch]) tc::mbar_wait(&bar_a[ch], pa[ch]);
                for (int n = copied > 2 ? copied - 2 : 0; n < copied; n++) tc::mbar_wait(&bar_b[n & 1], (n >> 1) & 1);
            }
            tc::commit_to(&bar_end);
            if (!tc::mbar_wait(&bar_end, 0)) {
                atomicOr(&ctl->status, kStatTimeout | kStatWaitMma);
                tc::mbar_wait(&bar_end, 0);
            }
        }
    } else {
        // warps 0-3 recombine the even tiles, 4-7 the odd ones (a segment of one
        // tile: 16 columns each); a warp reads the 32 TMEM lanes (rows) of its quarter
        const int quarter = warp & 3, group = warp >> 2, r = quarter * 32 + lane;
        // a tile as this thread sees it: its row's entries, the row's scale and
        // (lane c) the scale of column c; the row's columns end at cmax
        struct Tile {
            double *row;
            int j0, cmax, Ea, eb;
        };
        auto load = [&](const TileCursor &c) {
            Tile t;
            const int row = c.R.i0 + r, f = P.sn_f[c.R.s], ld = P.sn_ld[c.R.s];
            t.j0 = c.col();
            t.row = fronts + P.sn_off[c.R.s] + row + (int64_t)t.j0 * ld;
            t.cmax = row < f ? min(f, row + 1) : 0;
            t.Ea = ws_exp[((int64_t)c.blk_a() * kSliceRows + r) * 2];
            t.eb = ws_exp[((int64_t)c.blk_b() * kSliceRows + c.row_b() + lane) * 2 + 1];
            return t;
        };
        auto fetch = [&](const Tile &t, int ld, int c0, double (&v)[8]) {
#pragma unroll
            for (int c = 0; c < 8; c++) v[c] = t.j0 + c0 + c < t.cmax ? t.row[(int64_t)(c0 + c) * ld] : 0.0;
        };
        TileCursor c(runs, seg);
        const bool alone = c.R.nt == 1 && seg.last - seg.first == 1;
        const int c_first = alone ? 16 * group : 0, c_last = alone ? c_first + 16 : kSliceCols;
        if (!alone && group == 1) c.next();
        Tile cur{}, nxt{};
        int ldc = 0, ldn = 0;
        double ev[8], en[8];
        if (!c.end()) {
            cur = load(c);
            ldc = P.sn_ld[c.R.s];
            fetch(cur, ldc, c_first, ev);
        }
        for (int n = alone ? 0 : group; !c.end(); n += 2) {
            const int st = n & 1;
            c.next();
            if (!alone && !c.end()) c.next();
            const bool more = !c.end();
            if (more) {
                nxt = load(c);
                ldn = P.sn_ld[c.R.s];
            }
            bool ok = tc::mbar_wait(&bar_full[st], (n >> 1) & 1);
            if (!ok) atomicOr(&ctl->status, kStatTimeout | kStatWaitMma);
            ok = __all_sync(0xffffffffu, ok);  // warp-uniform: the TMEM loads below are warp-collective
            if (!ok) break;
            tc::fence_after_sync();
            const uint32_t lane_base = tmem + 256u * st + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
            for (int c0 = c_first; c0 < c_last; c0 += 8) {
                // the next eight entries are on their way while these are formed
                if (c0 + 8 < c_last) fetch(cur, ldc, c0 + 8, en);
                else if (more) fetch(nxt, ldn, c_first, en);
                // T = sum_d S_d 2^(7 (7 - d)), kept as T 2^-8 (|.| < 2^62): the bits
                // dropped are far below the truncation of the digit products with
                // t + u >= 8.  S_4..S_7 first, to keep the registers low.
                uint32_t v[4][8];
                int64_t t[8];
#pragma unroll
                for (int d = 0; d < 4; d++) tc::tmem_ld8(lane_base + (uint32_t)((d + 4) * kSliceCols + c0), v[d]);
                tc::tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 8; c++)
                    t[c] = sliced::digit_low(acc_pair(v[0][c], v[1][c]), acc_pair(v[2][c], v[3][c]));
#pragma unroll
                for (int d = 0; d < 4; d++) tc::tmem_ld8(lane_base + (uint32_t)(d * kSliceCols + c0), v[d]);
                tc::tmem_wait_ld();
                if (c0 + 8 == c_last && more) {
                    // this warp's part of the accumulator is read
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&bar_empty[st]);
                }
#pragma unroll
                for (int c = 0; c < 8; c++)
                    t[c] = sliced::digit_sum(t[c], acc_pair(v[0][c], v[1][c]), acc_pair(v[2][c], v[3][c]));
                double x[8];
                unsigned far = 0;
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    bool out;
                    x[c] = int_scaled(t[c], cur.Ea + __shfl_sync(0xffffffffu, cur.eb, c0 + c) - 55, out);
                    far |= (unsigned)out << c;
                }
                if (__any_sync(0xffffffffu, far)) {  // (also lanes beyond the front: harmless)
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        const int e = cur.Ea + __shfl_sync(0xffffffffu, cur.eb, c0 + c) - 55;
                        if ((far >> c) & 1u) x[c] = ldexp((double)t[c], e);
                    }
                }
#pragma unroll
                for (int c = 0; c < 8; c++) ev[c] -= x[c];
#pragma unroll
                for (int c = 0; c < 8; c++)
                    if (cur.j0 + c0 + c < cur.cmax) cur.row[(int64_t)(c0 + c) * ldc] = ev[c];
#pragma unroll
                for (int c = 0; c < 8; c++) ev[c] = en[c];
            }
            cur = nxt;
            ldc = ldn;
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

void launch_update_sliced(const DevPlan &P, double *fronts, const SlicedRun *runs, const SlicedSeg *segs,
                          int32_t count, const uint8_t *ws, const int32_t *ws_exp, DevCtl *ctl, cudaStream_t st) {
    if (count <= 0) return;
    static uint64_t attr = 0;
    if (first_on_device(attr))
        cudaFuncSetAttribute(k_update_sliced, cudaFuncAttributeMaxDynamicSharedMemorySize, kSlicedSmem);
    k_update_sliced<<<count, kSlicedThreads, kSlicedSmem, st>>>(P, fronts, runs, segs, ws, ws_exp, ctl);
}


}  // namespace ipm
